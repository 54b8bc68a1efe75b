// Shared-basis spectral decomposition of one projection type over the E experts
// (Sec. "Shared-basis Spectral Decomposition": Eq. shared_basis_input_proj for
// gate/up, the concatenation along input channels for down; Definitions
// spectral_energy_matrix / spectral_matrix), and the calibration Gram
// H = X Diag(g) X^T of the appendix (Eq. app_affinity_gram).
//
//   side "in"  (gate/up): W_e is d x D (rows: the expert's intermediate
//              channels), W_cat = [W_1; ...; W_E] = U S Phi^T, P~_cat = U S.
//   side "out" (down):    W_e is D x d, W_cat = [W_1 ... W_E] = Phi S V^T,
//              P~_cat = V S, split by the experts' input channels.
//
// Both sides are the same computation on A = the R x D matrix (R = E d) whose
// row r = (e, i) is row i of W_e ("in") or column i of W_e ("out"):
//   G   = A^T A (D x D, symmetric; its eigenvectors are Phi, its eigenvalues S^2)
//   P~  = A Phi (R x n), alpha_{e,k} = ||P~_e[:, k]||, P_e = P~_e / alpha_e.
// Kernels: a fp32 tile GEMM (CUDA cores) for G and P~ -- fp32 throughout,
// because the eigenvectors of G move with its rounding error divided by the
// eigenvalue gaps; a blocked cyclic two-sided Jacobi eigensolver for G in one
// cooperative kernel (pairs of 32-wide index blocks are diagonalised in shared
// memory, the products of their rotations applied to G and V^T as 64 x 64 tile
// products, two grid barriers per round of block pairs); a sort of the
// eigenvalues with the sign of each eigenvector fixed (largest component
// positive); the column norms and the unit-major P.
#include <cuda.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <cstring>

#include "device.cuh"
#include "internal.h"

#define BM_CK(call)                                             \
  do {                                                          \
    const cudaError_t e_ = (call);                              \
    if (e_ != cudaSuccess) return bmoe::record_cuda_error((int)e_); \
  } while (0)

namespace {

constexpr int kTM = 128, kTN = 128, kTK = 16, kGT = 256;   // GEMM tile, K step and threads (8 x 8 outputs a thread)
constexpr int kLdA = kTM + 4, kLdB = kTN + 4;              // row strides of the staged tiles

__device__ __forceinline__ float to_f(float v) { return v; }
__device__ __forceinline__ float to_f(uint16_t v) { return __uint_as_float((uint32_t)v << 16); }   // bf16 bits

// Four consecutive elements of a row (a is a multiple of 4), zero past `lim`.  VEC: rows start on four
// elements' alignment and `lim` is a multiple of 4.
template <bool VEC, typename T>
__device__ __forceinline__ float4 load4(const T* row, int a, int lim) {
  if constexpr (VEC) {
    if (a >= lim) return make_float4(0.f, 0.f, 0.f, 0.f);
    if constexpr (sizeof(T) == 4) {
      return __ldg(reinterpret_cast<const float4*>(row + a));
    } else {
      const uint2 u = __ldg(reinterpret_cast<const uint2*>(row + a));
      return make_float4(__uint_as_float(u.x << 16), __uint_as_float(u.x & 0xFFFF0000u), __uint_as_float(u.y << 16),
                         __uint_as_float(u.y & 0xFFFF0000u));
    }
  } else {
    float4 v;
    v.x = a < lim ? to_f(row[a]) : 0.f;
    v.y = a + 1 < lim ? to_f(row[a + 1]) : 0.f;
    v.z = a + 2 < lim ? to_f(row[a + 2]) : 0.f;
    v.w = a + 3 < lim ? to_f(row[a + 3]) : 0.f;
    return v;
  }
}

// The 8 x 8 outputs of a thread over one K step: rows ty * 8 + 2 r + {0, 1} packed in acc[r][.] (fma.f32x2:
// two products an issue slot), columns tx * 4 + c and 64 + tx * 4 + c (16-byte reads without bank conflicts).
__device__ __forceinline__ void tile_fma(const float* As, const float* Bs, int ty, int tx,
                                         unsigned long long (&acc)[4][8]) {
#pragma unroll
  for (int k = 0; k < kTK; ++k) {
    const ulonglong2 a0 = *reinterpret_cast<const ulonglong2*>(As + k * kLdA + ty * 8);
    const ulonglong2 a1 = *reinterpret_cast<const ulonglong2*>(As + k * kLdA + ty * 8 + 4);
    const float4 b0 = *reinterpret_cast<const float4*>(Bs + k * kLdB + tx * 4);
    const float4 b1 = *reinterpret_cast<const float4*>(Bs + k * kLdB + 64 + tx * 4);
    const unsigned long long a[4] = {a0.x, a0.y, a1.x, a1.y};
    const float b[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      unsigned long long bb;
      asm("mov.b64 %0, {%1, %1};" : "=l"(bb) : "f"(b[c]));
#pragma unroll
      for (int r = 0; r < 4; ++r) asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc[r][c]) : "l"(a[r]), "l"(bb));
    }
  }
}
__device__ __forceinline__ float tile_out(const unsigned long long (&acc)[4][8], int i, int j) {
  float lo, hi;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(acc[i >> 1][j]));
  return (i & 1) ? hi : lo;
}
__device__ __forceinline__ int tile_col(int tx, int j) { return (j < 4 ? 0 : 60) + tx * 4 + j; }

// Tile t of the upper triangle of ntile x ntile.
__device__ __forceinline__ int2 upper_tile(int t, int ntile) {
  int ta = 0;
  while (t >= ntile - ta) {
    t -= ntile - ta;
    ++ta;
  }
  return make_int2(ta, ta + t);
}

// G = sum_r w_r A[r, :]^T A[r, :]  (A: R x D, row stride lda; w = null: all 1).
// One block per upper-triangle tile pair (ta <= tb) of 128 x 128 and range of rows; the lower triangle is
// written by mirroring (so G is exactly symmetric).  One range writes G; with more (grid y, `part` not null:
// where the tiles alone leave SMs idle -- 36 tiles at D = 1024 ran 24576 rows on a quarter of the chip) each
// writes its tile of part[range][tile] and k_gram_sum adds them.
template <typename T, bool VEC>
__global__ void __launch_bounds__(kGT, 2) k_gram(const T* __restrict__ A, const float* __restrict__ w, int64_t R, int D,
                                                 int64_t lda, float* __restrict__ G, int64_t ldg, int ntile,
                                                 int64_t rows, float* __restrict__ part) {
  __shared__ __align__(16) float As[2][kTK * kLdA];
  __shared__ __align__(16) float Bs[2][kTK * kLdB];
  const int2 tl = upper_tile(blockIdx.x, ntile);
  const int a0 = tl.x * kTM, b0 = tl.y * kTN;
  const int64_t rbeg = (int64_t)blockIdx.y * rows, rend = min(R, rbeg + rows);
  const int tid = threadIdx.x, ty = tid >> 4, tx = tid & 15;
  const int lk = tid >> 5, lc = (tid & 31) * 4;   // loader: rows lk and lk + 8 of the step, 4 columns
  unsigned long long acc[4][8];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 8; ++j) acc[i][j] = 0ull;
  float4 va[2], vb[2];
  auto fetch = [&](int64_t r0) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int64_t r = r0 + lk + 8 * h;
      if (r < rend) {
        const T* row = A + r * lda;
        const float wr = w ? w[r] : 1.f;
        va[h] = load4<VEC>(row, a0 + lc, D);
        vb[h] = load4<VEC>(row, b0 + lc, D);
        va[h].x *= wr;
        va[h].y *= wr;
        va[h].z *= wr;
        va[h].w *= wr;
      } else {
        va[h] = vb[h] = make_float4(0.f, 0.f, 0.f, 0.f);
      }
    }
  };
  fetch(rbeg);
  int buf = 0;
  for (int64_t r0 = rbeg; r0 < rend; r0 += kTK) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      *reinterpret_cast<float4*>(&As[buf][(lk + 8 * h) * kLdA + lc]) = va[h];
      *reinterpret_cast<float4*>(&Bs[buf][(lk + 8 * h) * kLdB + lc]) = vb[h];
    }
    __syncthreads();
    if (r0 + kTK < rend) fetch(r0 + kTK);
    tile_fma(As[buf], Bs[buf], ty, tx, acc);
    buf ^= 1;
  }
  float* pt = part ? part + ((size_t)blockIdx.y * gridDim.x + blockIdx.x) * (kTM * kTN) : nullptr;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int la = ty * 8 + i, a = a0 + la;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int lb = tile_col(tx, j), b = b0 + lb;
      const float v = tile_out(acc, i, j);
      if (part) {
        pt[la * kTN + lb] = v;
      } else if (a < D && b < D && (tl.x != tl.y || a <= b)) {   // exactly symmetric: one value per pair
        G[(size_t)a * ldg + b] = v;
        G[(size_t)b * ldg + a] = v;
      }
    }
  }
}

// G from the ranges' tiles, added in order: one block per tile and 32 x 32 piece of it, the mirror image
// through a transposed tile.
__global__ void __launch_bounds__(256) k_gram_sum(const float* __restrict__ part, int splits, int D,
                                                  float* __restrict__ G, int64_t ldg, int ntile) {
  __shared__ float tr[32][33];
  const int2 tl = upper_tile(blockIdx.x, ntile);
  const int pr = (blockIdx.y >> 2) * 32, pc = (blockIdx.y & 3) * 32;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
#pragma unroll
  for (int y = ty; y < 32; y += 8) {
    float v = 0.f;
    for (int s = 0; s < splits; ++s)
      v += part[((size_t)s * gridDim.x + blockIdx.x) * (kTM * kTN) + (pr + y) * kTN + pc + tx];
    tr[y][tx] = v;
    const int a = tl.x * kTM + pr + y, b = tl.y * kTN + pc + tx;
    if (a < D && b < D && (tl.x != tl.y || a <= b)) G[(size_t)a * ldg + b] = v;
  }
  __syncthreads();
#pragma unroll
  for (int y = ty; y < 32; y += 8) {
    const int a = tl.x * kTM + pr + tx, b = tl.y * kTN + pc + y;
    if (a < D && b < D && (tl.x != tl.y || a < b)) G[(size_t)b * ldg + a] = tr[tx][y];
  }
}

// C = A Phi  (A: R x D fp32 row-major, Phi: D x n row-major, C: R x n).  Tiles of
// 128 rows of A (read 16 columns at a time and transposed into shared memory) by 128
// columns of Phi.
template <bool VEC>
__global__ void __launch_bounds__(kGT, 2) k_project(const float* __restrict__ A, const float* __restrict__ Phi, int64_t R,
                                                    int D, int n, float* __restrict__ C) {
  __shared__ __align__(16) float As[2][kTK * kLdA];
  __shared__ __align__(16) float Bs[2][kTK * kLdB];
  const int64_t m0 = (int64_t)blockIdx.y * kTM;
  const int n0 = blockIdx.x * kTN;
  const int tid = threadIdx.x, ty = tid >> 4, tx = tid & 15;
  const int am = tid & 127, ak = (tid >> 7) * 8;   // A loader: row am, columns ak .. ak + 7 of the step
  const int bk = tid >> 5, bc = (tid & 31) * 4;    // Phi loader: rows bk and bk + 8, columns bc .. bc + 3
  unsigned long long acc[4][8];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 8; ++j) acc[i][j] = 0ull;
  float4 va[2], vb[2];
  auto fetch = [&](int k0) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      va[h] = m0 + am < R ? load4<VEC>(A + (m0 + am) * D, k0 + ak + 4 * h, D) : make_float4(0.f, 0.f, 0.f, 0.f);
      vb[h] = k0 + bk + 8 * h < D ? load4<VEC>(Phi + (size_t)(k0 + bk + 8 * h) * n, n0 + bc, n)
                                  : make_float4(0.f, 0.f, 0.f, 0.f);
    }
  };
  fetch(0);
  int buf = 0;
  for (int k0 = 0; k0 < D; k0 += kTK) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      As[buf][(ak + 4 * h) * kLdA + am] = va[h].x;
      As[buf][(ak + 4 * h + 1) * kLdA + am] = va[h].y;
      As[buf][(ak + 4 * h + 2) * kLdA + am] = va[h].z;
      As[buf][(ak + 4 * h + 3) * kLdA + am] = va[h].w;
      *reinterpret_cast<float4*>(&Bs[buf][(bk + 8 * h) * kLdB + bc]) = vb[h];
    }
    __syncthreads();
    if (k0 + kTK < D) fetch(k0 + kTK);
    tile_fma(As[buf], Bs[buf], ty, tx, acc);
    buf ^= 1;
  }
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int64_t m = m0 + ty * 8 + i;
    if (m >= R) continue;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int c = n0 + tile_col(tx, 4 * h);
      if (VEC) {
        if (c < n)
          *reinterpret_cast<float4*>(C + m * n + c) = make_float4(tile_out(acc, i, 4 * h), tile_out(acc, i, 4 * h + 1),
                                                                  tile_out(acc, i, 4 * h + 2), tile_out(acc, i, 4 * h + 3));
      } else {
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if (c + j < n) C[m * n + c + j] = tile_out(acc, i, 4 * h + j);
      }
    }
  }
}

// A for side "out": row (e, i) = column i of W_e (W: E x D x d) -> A: (E d) x D.
__global__ void k_transpose_out(const float* __restrict__ W, int E, int D, int d, float* __restrict__ A) {
  __shared__ float tile[32][33];
  const int e = blockIdx.z;
  const int i0 = blockIdx.x * 32, a0 = blockIdx.y * 32;
  const float* We = W + (size_t)e * D * d;
  for (int y = threadIdx.y; y < 32; y += blockDim.y) {
    const int a = a0 + y, i = i0 + threadIdx.x;
    tile[y][threadIdx.x] = (a < D && i < d) ? We[(size_t)a * d + i] : 0.f;
  }
  __syncthreads();
  for (int y = threadIdx.y; y < 32; y += blockDim.y) {
    const int i = i0 + y, a = a0 + threadIdx.x;
    if (i < d && a < D) A[((size_t)e * d + i) * D + a] = tile[threadIdx.x][y];
  }
}

// ---------------------------------------------------------------------------
// Blocked cyclic two-sided Jacobi (rotations: Golub & Van Loan, Alg. 8.5.3;
// blocked as in their Sec. 8.5.6).  The indices 0 .. m - 1 (n rounded up to a
// multiple of 64; the added ones are zero rows, never rotated) form blocks of 32.
// In an outer round of a sweep the blocks pair up by the circle arrangement
// (player 0 stays, the others advance by one a round), and per pair (I, J)
//   solve   one block of threads rotates the 64 x 64 diagonal tile G[IJ, IJ] in
//           shared memory: 32 rounds of 32 disjoint pairs (i of I, j of J); in the
//           first outer round of a sweep, the 63 rounds of the circle arrangement
//           of all 64, which also covers the pairs within I and J.  The product of
//           its rotations is Q (64 x 64).
//   apply   G[P, P'] <- Q_P^T G[P, P'] Q_P' for every two pairs P < P' (and its
//           mirror image), two 64 x 64 x 64 products in shared memory
//   V^T     rows IJ <- Q^T rows IJ, by the blocks that solve nothing, while the
//           next round's tiles are being solved
// so that each index pair meets once a sweep as in the scalar cyclic order, with two
// grid barriers per 32 rounds of rotations instead of one per round (at D = 1024,
// eight sweeps: 84 ms with a barrier per round of rotations, 5.0 ms so: 20 us per outer
// round, 12 of them the chain of dependent rotations, 6 the tile products, the rest barriers).
// For a pair (p, q) with a_pq != 0: tau = (a_qq - a_pp) / (2 a_pq), t = sign(tau) /
// (|tau| + sqrt(1 + tau^2)), c = 1 / sqrt(1 + t^2), s = t c; the rotation J
// (J_pp = J_qq = c, J_pq = s, J_qp = -s) makes (J^T G J)_pq = 0.  The solver stops
// after the first sweep in which every |a_pq| was <= tol sqrt(|a_pp a_qq|) or <= 4e-7
// max_j |a_jj|; until then elements down to a sixteenth of that are rotated too (left
// standing, those just under the test turn the vectors by more than all rounding does:
// 4.8e-4 of the basis at D = 1024), but only between eigenvalues well apart (|tau| > 16:
// small angles) and well above the test.  Elsewhere, as among the zeros of weights of low
// rank and between them and the rest, such elements are rounding noise, and turning vectors
// by it in every sweep costs them orthogonality and raises the noise (rank 5, D = 1500:
// Phi^T Phi off by 2.3e-5 with those elements rotated everywhere, 1.0e-6 so; zero singular
// values 2.7e-4 and 5.4e-5 of the largest.  Rotated down to 10 times the test instead of
// 600: rank 200, D = 2048 3.4e-5 and 30 sweeps, 8.5e-6 and 21 so).
// ---------------------------------------------------------------------------
constexpr int kJB = 32, kJP = 2 * kJB, kJT = 512;   // block width, tile width, threads
constexpr float kJFine = 1.f / 16.f;                // rotations are skipped below this part of the stopping test where
constexpr float kJApart = 16.f;                     // |tau| is above this and both eigenvalues above this many times
constexpr float kJLarge = 600.f;                    // its floor (2.4e-4 of the largest); elsewhere below the test itself
constexpr size_t kTile = (size_t)kJP * kJP;
constexpr size_t kJSmem = 5 * kTile * sizeof(float);

struct JacobiArgs {
  float* G;          // m x m, symmetric, overwritten (diagonal: the eigenvalues)
  float* Vt;         // m x m: row j = eigenvector j (set to the identity here)
  float* Q;          // [2][m / 64] tiles: the pairs' rotations, by parity of the round
  int* act;          // [2][m / 64] whether a pair rotated at all
  int n, m;
  int max_sweeps;
  float tol;
  uint32_t* bar;     // grid-barrier counter, and pairs above the stopping test so far (both zero at launch)
  uint32_t* rot;
  int* status;       // BITSMOE_ERR_TIMEOUT if a wait ran out
  int* sweeps;       // sweeps run (written by block 0)
  long long spin;    // bound of each barrier wait, in SM clocks
};

__device__ __forceinline__ int jacobi_player(int pos, int r, int m) { return pos == 0 ? 0 : 1 + (pos - 1 + r) % (m - 1); }

__device__ __forceinline__ bool grid_sync_bounded(uint32_t* bar, uint32_t target, long long spin, int* status,
                                                  int* ok) {
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(bar) : "memory");
    const long long t0 = clock64();
    int good = 1;
    for (;;) {
      uint32_t v;
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(bar) : "memory");
      if ((int)(v - target) >= 0) break;
      if (clock64() - t0 > spin) {
        atomicCAS(status, 0, BITSMOE_ERR_TIMEOUT);
        good = 0;
        break;
      }
    }
    __threadfence();
    *ok = good;
  }
  __syncthreads();
  return *ok != 0;
}

__device__ __forceinline__ void cp16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// The global index of a tile's row or column l of the pair of blocks (bi, bj).
__device__ __forceinline__ int tile_index(int2 b, int l) { return (l < kJB ? b.x * kJB : b.y * kJB - kJB) + l; }
__device__ __forceinline__ int2 pair_blocks(int p, int r, int nblk) {
  return make_int2(jacobi_player(p, r, nblk), jacobi_player(nblk - 1 - p, r, nblk));
}

// 64 x 64 floats into shared memory by 16-byte copies: rows of pair `rb`, columns of pair `cb`.
__device__ __forceinline__ void tile_in(float* dst, const float* M, int m, int2 rb, int2 cb) {
#pragma unroll
  for (int i = 0; i < (int)(kTile / 4 / kJT); ++i) {
    const int ch = threadIdx.x + i * kJT, row = ch >> 4, c = (ch & 15) * 4;
    cp16(dst + ch * 4, M + (size_t)tile_index(rb, row) * m + tile_index(cb, c));
  }
}
__device__ __forceinline__ void flat_in(float* dst, const float* src) {
#pragma unroll
  for (int i = 0; i < (int)(kTile / 4 / kJT); ++i)
    cp16(dst + 4 * (threadIdx.x + i * kJT), src + 4 * (threadIdx.x + i * kJT));
}

// C = A^T B of 64 x 64 tiles in shared memory ([k][.] both): the two halves of the block take half of the
// k each, 4 x 4 outputs a thread (rows 4 ty .., columns 4 tx ..); the second half's sums pass through `red`,
// and the first half holds the result.
__device__ __forceinline__ void tile_tn(const float* A, const float* B, float4* red, int ty, int tx, float (&acc)[4][4]) {
  const int half = threadIdx.x >> 8;
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
#pragma unroll 8
  for (int k = half * (kJP / 2); k < (half + 1) * (kJP / 2); ++k) {
    const float4 a4 = *reinterpret_cast<const float4*>(A + k * kJP + 4 * ty);
    const float4 b4 = *reinterpret_cast<const float4*>(B + k * kJP + 4 * tx);
    const float a[4] = {a4.x, a4.y, a4.z, a4.w}, b[4] = {b4.x, b4.y, b4.z, b4.w};
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
  }
  const int t = threadIdx.x & 255;
  if (half) {
#pragma unroll
    for (int i = 0; i < 4; ++i) red[i * 256 + t] = make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
  }
  __syncthreads();
  if (!half) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float4 v = red[i * 256 + t];
      acc[i][0] += v.x;
      acc[i][1] += v.y;
      acc[i][2] += v.z;
      acc[i][3] += v.w;
    }
  }
}

__device__ __forceinline__ float sqrt_approx(float x) {
  float y;
  asm("sqrt.approx.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// The rotation of a pair: c, s and t (1, 0, 0: none).  t itself may be off by a few units in the last place, which
// leaves that part of a_pq behind: approximate quotients and roots, which lie on the chain from round to round.
// What keeps the vectors orthogonal is c^2 + s^2 = 1: with 1 <= 1 + t^2 <= 2, c is one Newton step from the
// approximate inverse root, within one unit in the last place.  Measured against rounded quotients and roots on 18
// sizes (D 66 .. 1024, both sides): the basis is not further from 64 bits (relative 2-norm at D = 1024: 3.6e-4 to
// 3.9e-4, rounded 3.9e-4 to 4.3e-4; the unblocked solver before 5.1e-4 to 5.2e-4), nor is it with weights scaled by
// 2^-70 .. 2^28, and the whole call takes 7.3 ms instead of 8.0.
struct Rotation {
  float c, s, t;
  bool need;   // above the thresholds of the stopping test
};
__device__ __forceinline__ Rotation jacobi_rotation(float app, float aqq, float apq, float atol, float tol) {
  const float mag = fabsf(apq), rel = tol * sqrt_approx(fabsf(app) * fabsf(aqq));
  const float tau = __fdividef(aqq - app, 2.f * apq);
  float t = __fdividef(tau >= 0.f ? 1.f : -1.f, fabsf(tau) + sqrt_approx(fmaf(tau, tau, 1.f)));
  const float part = fabsf(tau) > kJApart && fminf(fabsf(app), fabsf(aqq)) > kJLarge * atol ? kJFine : 1.f;
  t = mag > part * atol && mag > part * rel ? t : 0.f;
  const float x = fmaf(t, t, 1.f), y = rsqrtf(x), c = t != 0.f ? fmaf(0.5f * y, fmaf(-x * y, y, 1.f), y) : 1.f;
  return Rotation{c, t * c, t, mag > atol && mag > rel};
}

// Writes a pair's Q (a warp's rows 4 w .. at the lane's columns p, q) and whether it rotated, and its tile S of G
// (the upper triangle, copied to the lower one).
__device__ __forceinline__ void jacobi_solved(const JacobiArgs& ja, int pair, int2 blk, int par, float* S, int p,
                                              int q, const float (&qa)[4], const float (&qb)[4], unsigned any,
                                              unsigned need) {
  const int half = ja.m / kJP, w = threadIdx.x >> 5;
  float* Q = ja.Q + ((size_t)par * half + pair) * kTile;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    __stcg(Q + (4 * w + i) * kJP + p, qa[i]);
    __stcg(Q + (4 * w + i) * kJP + q, qb[i]);
  }
  if (any) {   // along the diagonals, so that neither the reads nor the writes meet in a bank
    const int lane = threadIdx.x & 31;
    for (int k = 1 + w; k < kJP; k += kJT / 32)
#pragma unroll
      for (int r = lane; r < kJP; r += 32)
        if (r + k < kJP) S[(r + k) * kJP + r] = S[r * kJP + r + k];
    __syncthreads();
#pragma unroll
    for (int i = 0; i < (int)(kTile / 4 / kJT); ++i) {
      const int ch = threadIdx.x + i * kJT, row = ch >> 4, c = (ch & 15) * 4;
      __stcg(reinterpret_cast<float4*>(ja.G + (size_t)tile_index(blk, row) * ja.m + tile_index(blk, c)),
             *reinterpret_cast<const float4*>(S + 4 * ch));
    }
  }
  if (threadIdx.x == 0) {
    __stcg(ja.act + par * half + pair, (int)any);
    if (need) atomicAdd(ja.rot, 1u);
  }
  __syncthreads();   // the tiles may be written again
}

// Rotates the tile of one pair of blocks, all 63 rounds of the circle arrangement: two rows of 2 x 2 blocks a
// warp, from one tile to the other and back.
__device__ void jacobi_solve_all(const JacobiArgs& ja, int pair, int2 blk, float atol, int par, float* sm) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  float *S = sm, *Sn = sm + kTile;
  tile_in(S, ja.G, ja.m, blk, blk);
  cp_wait();
  __syncthreads();
  // lane: columns p, q of this round; the warp's rows 4 w .. 4 w + 3 of Q at those columns in registers
  int p = lane, q = kJP - 1 - lane;
  float qa[4], qb[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    qa[i] = 4 * w + i == p ? 1.f : 0.f;
    qb[i] = 4 * w + i == q ? 1.f : 0.f;
  }
  unsigned any = 0u, need = 0u;
#pragma unroll 1
  for (int t = 0; t < kJP - 1; ++t) {
    const float app = S[p * kJP + p], aqq = S[q * kJP + q], apq = S[p * kJP + q];
    const Rotation ro = jacobi_rotation(app, aqq, apq, atol, ja.tol);
    const float c = ro.c, s = ro.s;
    const unsigned mk = __ballot_sync(0xFFFFFFFFu, ro.t != 0.f);   // the same in every warp
    need |= __ballot_sync(0xFFFFFFFFu, ro.need);
    if (mk) {
      any = 1u;
#pragma unroll
      for (int h = 0; h < 2; ++h) {   // rows of pair i, columns of the lane's pair
        const int i = 2 * w + h;
        const int pi = __shfl_sync(0xFFFFFFFFu, p, i), qi = __shfl_sync(0xFFFFFFFFu, q, i);
        const float ci = __shfl_sync(0xFFFFFFFFu, c, i), si = __shfl_sync(0xFFFFFFFFu, s, i);
        const float vpp = S[pi * kJP + p], vpq = S[pi * kJP + q], vqp = S[qi * kJP + p], vqq = S[qi * kJP + q];
        const float xp = ci * vpp - si * vqp, xq = ci * vpq - si * vqq;
        const float yp = ci * vqp + si * vpp, yq = ci * vqq + si * vpq;
        float r0 = c * xp - s * xq, r1 = c * xq + s * xp, r2 = c * yp - s * yq, r3 = c * yq + s * yp;
        if (i == lane && ro.t != 0.f) {   // the rotated 2 x 2 block (Golub & Van Loan's update, which keeps
          r0 = app - ro.t * apq;          // a_pp + a_qq to one rounding per element)
          r3 = aqq + ro.t * apq;
          r1 = r2 = 0.f;
        }
        Sn[pi * kJP + p] = r0;
        Sn[pi * kJP + q] = r1;
        Sn[qi * kJP + p] = r2;
        Sn[qi * kJP + q] = r3;
      }
      __syncthreads();   // the round's tile is whole; the other one is free
      float* x = S;
      S = Sn;
      Sn = x;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float a = qa[i], b = qb[i];
        qa[i] = c * a - s * b;
        qb[i] = c * b + s * a;
      }
    }
    // the circle: place k takes the player of place k + 1; q's places run downwards
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float up = __shfl_down_sync(0xFFFFFFFFu, qa[i], 1), dn = __shfl_up_sync(0xFFFFFFFFu, qb[i], 1);
      const float first = __shfl_sync(0xFFFFFFFFu, qa[i], 1);
      const float old = qb[i];
      qb[i] = lane == 0 ? first : dn;
      if (lane != 0) qa[i] = lane == 31 ? old : up;
    }
    if (lane != 0) p = p == kJP - 1 ? 1 : p + 1;
    q = q == kJP - 1 ? 1 : q + 1;
  }
  jacobi_solved(ja, pair, blk, par, S, p, q, qa, qb, any, need);
}

// The same for the pairs between the two blocks only: round t rotates (p_i = i, q_i = 32 + (i + t) mod 32).  The 2
// x 2 block of pairs i and j = i + d is one lane's (lane i of warp d; warp 0 has d = 16, whose lower lanes cover
// it): its elements (p_i, p_j) and (q_i, q_j) stay in registers, the latter moving by one lane a round as the
// q_i do, and so do Q's columns; (p_i, q_j) and (p_j, q_i) move to the neighbouring warps and lie in the tile.  By
// symmetry that is the whole tile.  Warp 1, whose (p_i, q_(i + 1)) is the next round's a_pq, keeps the diagonal
// and works out the next round's rotations while the other warps finish this one (700 clocks a round; 1000 with
// every warp working them out for itself).
__device__ void jacobi_solve_cross(const JacobiArgs& ja, int pair, int2 blk, float atol, int par, float* sm) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  float* S = sm;
  float2* rot = reinterpret_cast<float2*>(sm + kTile);   // [2][32] c and s of a round's pairs
  unsigned* flags = reinterpret_cast<unsigned*>(rot + 64);
  tile_in(S, ja.G, ja.m, blk, blk);
  cp_wait();
  __syncthreads();
  const int d = w ? w : 16, j = (lane + d) & 31, up = (lane + 1) & 31;
  const bool mine = w || lane < 16;
  float pp = S[lane * kJP + j], qq = S[(kJB + lane) * kJP + kJB + j];
  float app = 0.f, aqq = 0.f, apq = 0.f;   // warp 1
  Rotation ro{1.f, 0.f, 0.f, false};
  unsigned any = 0u, need = 0u;
  auto rotations = [&](int t) {   // of round t from the diagonal and a_pq
    ro = jacobi_rotation(app, aqq, apq, atol, ja.tol);
    any |= ro.t != 0.f;
    need |= ro.need;
    rot[(t & 1) * 32 + lane] = make_float2(ro.c, ro.s);
  };
  if (w == 1) {
    app = S[lane * (kJP + 1)];
    aqq = S[(kJB + lane) * (kJP + 1)];
    apq = S[lane * kJP + kJB + lane];
    rotations(0);
  }
  float qa[4], qb[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    qa[i] = 4 * w + i == lane ? 1.f : 0.f;
    qb[i] = 4 * w + i == kJB + lane ? 1.f : 0.f;
  }
  __syncthreads();
#pragma unroll 1
  for (int t = 0; t < kJB; ++t) {
    const float2 ri = rot[(t & 1) * 32 + lane], rj = rot[(t & 1) * 32 + j];
    float *const e1 = S + lane * kJP + kJB + ((j + t) & 31), *const e2 = S + j * kJP + kJB + ((lane + t) & 31);
    const float vpq = *e1, vqp = *e2;
    const float xp = ri.x * pp - ri.y * vqp, xq = ri.x * vpq - ri.y * qq;
    const float yp = ri.x * vqp + ri.y * pp, yq = ri.x * qq + ri.y * vpq;
    pp = rj.x * xp - rj.y * xq;
    const float r1 = rj.x * xq + rj.y * xp, r2 = rj.x * yp - rj.y * yq;
    qq = rj.x * yq + rj.y * yp;
    if (w == 0) __syncwarp();   // warp 0's upper lanes have read the elements that its lower lanes write
    if (mine) {
      *e1 = r1;
      *e2 = r2;
    }
    qq = __shfl_sync(0xFFFFFFFFu, qq, up);   // q_i moves by one lane
    if (w == 1) {
      S[lane * kJP + kJB + ((lane + t) & 31)] = ro.t != 0.f ? 0.f : apq;
      app = app - ro.t * apq;   // (Golub & Van Loan's update, which keeps a_pp + a_qq to one rounding per element)
      aqq = __shfl_sync(0xFFFFFFFFu, aqq + ro.t * apq, up);
      apq = r1;
      if (t + 1 < kJB) rotations(t + 1);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float a = qa[i], b = qb[i];
      qa[i] = ri.x * a - ri.y * b;
      qb[i] = __shfl_sync(0xFFFFFFFFu, ri.x * b + ri.y * a, up);
    }
    __syncthreads();
  }
  if (mine) {   // back into the tile's upper triangle
    S[min(lane, j) * kJP + max(lane, j)] = pp;
    S[(kJB + min(lane, j)) * kJP + kJB + max(lane, j)] = qq;
  }
  if (w == 1) {
    S[lane * (kJP + 1)] = app;
    S[(kJB + lane) * (kJP + 1)] = aqq;
    any = __ballot_sync(0xFFFFFFFFu, any);
    need = __ballot_sync(0xFFFFFFFFu, need);
    if (lane == 0) {
      flags[0] = any;
      flags[1] = need;
    }
  }
  __syncthreads();
  jacobi_solved(ja, pair, blk, par, S, lane, kJB + lane, qa, qb, flags[0], flags[1]);
}

// V^T's rows of the round's pairs, tile by tile, by the blocks first, first + step, ...
__device__ void jacobi_vectors(const JacobiArgs& ja, int r, int par, int first, int step, int ty, int tx, float* sm) {
  const int half = ja.m / kJP;
  for (int id = first; id < half * half; id += step) {
    const int p = id / half, ct = id - p * half;
    if (!__ldcg(ja.act + par * half + p)) continue;
    const int2 b = pair_blocks(p, r, 2 * half), cols = make_int2(2 * ct, 2 * ct + 1);
    tile_in(sm, ja.Vt, ja.m, b, cols);
    flat_in(sm + kTile, ja.Q + ((size_t)par * half + p) * kTile);
    cp_wait();
    __syncthreads();
    float acc[4][4];
    tile_tn(sm + kTile, sm, reinterpret_cast<float4*>(sm + 4 * kTile), ty, tx, acc);
    if (threadIdx.x < 256) {
#pragma unroll
      for (int i = 0; i < 4; ++i)
        __stcg(reinterpret_cast<float4*>(ja.Vt + (size_t)tile_index(b, 4 * ty + i) * ja.m + ct * kJP + 4 * tx),
               make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]));
    }
    __syncthreads();
  }
}

// G's tiles of every two pairs.
__device__ void jacobi_apply(const JacobiArgs& ja, int r, int par, int ty, int tx, float* sm) {
  const int half = ja.m / kJP, tiles = half * (half - 1) / 2;
  float* Mt = sm + 3 * kTile;
  float4* red = reinterpret_cast<float4*>(sm + 4 * kTile);
  for (int id = blockIdx.x; id < tiles; id += gridDim.x) {
    int p1 = 0, left = id;
    while (left >= half - 1 - p1) {
      left -= half - 1 - p1;
      ++p1;
    }
    const int p2 = p1 + 1 + left;
    if (!__ldcg(ja.act + par * half + p1) && !__ldcg(ja.act + par * half + p2)) continue;
    const int2 b1 = pair_blocks(p1, r, 2 * half), b2 = pair_blocks(p2, r, 2 * half);
    tile_in(sm, ja.G, ja.m, b1, b2);
    flat_in(sm + kTile, ja.Q + ((size_t)par * half + p1) * kTile);
    flat_in(sm + 2 * kTile, ja.Q + ((size_t)par * half + p2) * kTile);
    cp_wait();
    __syncthreads();
    float acc[4][4];
    tile_tn(sm, sm + kTile, red, ty, tx, acc);   // (Q1^T G)^T: [column][row]
    if (threadIdx.x < 256) {
#pragma unroll
      for (int i = 0; i < 4; ++i)
        *reinterpret_cast<float4*>(Mt + (4 * ty + i) * kJP + 4 * tx) =
            make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
    }
    __syncthreads();
    tile_tn(Mt, sm + 2 * kTile, red, ty, tx, acc);
    if (threadIdx.x < 256) {
#pragma unroll
      for (int i = 0; i < 4; ++i)
        __stcg(reinterpret_cast<float4*>(ja.G + (size_t)tile_index(b1, 4 * ty + i) * ja.m + tile_index(b2, 4 * tx)),
               make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]));
#pragma unroll
      for (int j = 0; j < 4; ++j)   // the mirror image
        __stcg(reinterpret_cast<float4*>(ja.G + (size_t)tile_index(b2, 4 * tx + j) * ja.m + tile_index(b1, 4 * ty)),
               make_float4(acc[0][j], acc[1][j], acc[2][j], acc[3][j]));
    }
    __syncthreads();
  }
}

__global__ void __launch_bounds__(kJT, 1) k_jacobi(JacobiArgs ja) {
  extern __shared__ __align__(16) uint8_t jsm[];
  float* sm = reinterpret_cast<float*>(jsm);
  __shared__ int ok;
  __shared__ float dmax_s;
  const int n = ja.n, m = ja.m, half = m / kJP;
  const int tid = threadIdx.x, nt = blockDim.x, blk = blockIdx.x, nb = gridDim.x;
  // 4 x 4 outputs: a warp covers 16 rows by 32 columns
  const int tw = (tid & 255) >> 5, lane = tid & 31;
  const int ty = (tw >> 1) * 4 + (lane >> 3), tx = (tw & 1) * 8 + (lane & 7);
  for (size_t i = (size_t)blk * nt + tid; i < (size_t)m * m; i += (size_t)nb * nt)
    ja.Vt[i] = (i / m == i % m) ? 1.f : 0.f;
  // absolute floor of the rotation test: a few units in the last place of the largest
  // diagonal element, below which an off-diagonal element is rounding noise
  {
    float dm = 0.f;
    for (int x = tid; x < n; x += nt) dm = fmaxf(dm, fabsf(__ldcg(ja.G + (size_t)x * m + x)));
    for (int o = 16; o; o >>= 1) dm = fmaxf(dm, __shfl_xor_sync(0xFFFFFFFFu, dm, o));
    if (tid == 0) dmax_s = 0.f;
    __syncthreads();
    if ((tid & 31) == 0) atomicMax(reinterpret_cast<int*>(&dmax_s), __float_as_int(dm));   // non-negative floats
    __syncthreads();
  }
  const float atol = 4e-7f * dmax_s;
  uint32_t target = nb;
  if (!grid_sync_bounded(ja.bar, target, ja.spin, ja.status, &ok)) return;
  // V^T by the blocks that solve nothing, while they would wait, when that is at most four tiles a block (a
  // solve's time); otherwise by every block after G's tiles
  const bool late = half * half <= 4 * (nb - half);
  int sweep = 0, g = 0, rprev = -1;   // g: outer rounds run so far (their parity picks the Q)
  uint32_t rotated = 0;
  for (; sweep < ja.max_sweeps; ++sweep) {
    uint32_t now = rotated;
    for (int r = 0; r < 2 * half - 1; ++r, ++g) {
      const int par = g & 1;
      for (int p = blk; p < half; p += nb) {
        if (r == 0) jacobi_solve_all(ja, p, pair_blocks(p, r, 2 * half), atol, par, sm);
        else jacobi_solve_cross(ja, p, pair_blocks(p, r, 2 * half), atol, par, sm);
      }
      if (late && rprev >= 0 && blk >= half) jacobi_vectors(ja, rprev, par ^ 1, blk - half, nb - half, ty, tx, sm);
      target += nb;
      if (!grid_sync_bounded(ja.bar, target, ja.spin, ja.status, &ok)) return;
      jacobi_apply(ja, r, par, ty, tx, sm);
      if (!late) jacobi_vectors(ja, r, par, nb - 1 - blk, nb, ty, tx, sm);   // (the last blocks have fewer tiles of G)
      now = __ldcg(ja.rot);   // no solve is under way between the two barriers: every block reads the same
      target += nb;
      if (!grid_sync_bounded(ja.bar, target, ja.spin, ja.status, &ok)) return;
      rprev = r;
    }
    if (now == rotated) break;
    rotated = now;
  }
  if (late) jacobi_vectors(ja, rprev, (g & 1) ^ 1, blk, nb, ty, tx, sm);
  if (blk == 0 && tid == 0 && ja.sweeps) *ja.sweeps = sweep;
}

// Rank of each eigenvalue (descending, ties to the lower index), the sign of
// each eigenvector (its largest |component| made positive, the first one on
// ties), then Phi[:, rank] = sign * V^T[j, :] and sigma[rank] = sqrt(max(lambda, 0))
// for the n_out leading ones.
__global__ void k_order(const float* __restrict__ G, const float* __restrict__ Vt, int n, int ld, int n_out,
                        float* __restrict__ phi, float* __restrict__ sigma) {
  const int j = blockIdx.x;   // one block per eigenvector
  __shared__ float red_v[32];
  __shared__ int red_i[32], red_c[32];
  __shared__ float red_n[32];
  __shared__ int rank_s;
  __shared__ float scale_s;
  const float lj = __ldg(G + (size_t)j * ld + j);
  int cnt = 0;
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    const float li = __ldg(G + (size_t)i * ld + i);
    cnt += (li > lj) | ((li == lj) & (i < j));
  }
  // largest |component| of V^T[j, :] (first on ties) and its squared norm (the vector is
  // rescaled to unit length: the rotations' rounding moves it by a few units in the last place)
  float bv = -1.f, nn = 0.f;
  int bi = 0x7FFFFFFF;
  const float* vr = Vt + (size_t)j * ld;
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    const float v = vr[i], a = fabsf(v);
    nn = fmaf(v, v, nn);
    if (a > bv || (a == bv && i < bi)) {
      bv = a;
      bi = i;
    }
  }
  for (int o = 16; o; o >>= 1) {
    nn += __shfl_xor_sync(0xFFFFFFFFu, nn, o);
    cnt += __shfl_xor_sync(0xFFFFFFFFu, cnt, o);
    const float ov = __shfl_xor_sync(0xFFFFFFFFu, bv, o);
    const int oi = __shfl_xor_sync(0xFFFFFFFFu, bi, o);
    if (ov > bv || (ov == bv && oi < bi)) {
      bv = ov;
      bi = oi;
    }
  }
  const int w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  if ((threadIdx.x & 31) == 0) {
    red_v[w] = bv;
    red_i[w] = bi;
    red_c[w] = cnt;
    red_n[w] = nn;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    int rk = 0;
    float v = -1.f, tn = 0.f;
    int vi = 0x7FFFFFFF;
    for (int q = 0; q < nw; ++q) {
      rk += red_c[q];
      tn += red_n[q];
      if (red_v[q] > v || (red_v[q] == v && red_i[q] < vi)) {
        v = red_v[q];
        vi = red_i[q];
      }
    }
    if (vi >= n) vi = 0;   // no component compares (not finite)
    rank_s = rk;
    red_i[0] = vi;
    scale_s = tn > 0.f ? 1.f / sqrtf(tn) : 1.f;
  }
  __syncthreads();
  const int rk = rank_s;
  if (rk >= n_out) return;
  const float sg = vr[red_i[0]] < 0.f ? -scale_s : scale_s;
  for (int i = threadIdx.x; i < n; i += blockDim.x) phi[(size_t)i * n_out + rk] = sg * vr[i];
  if (threadIdx.x == 0) sigma[rk] = sqrtf(fmaxf(lj, 0.f));
}

// alpha[e][k] = ||P~[e d .. e d + d - 1][k]||_2 and P[e][k][i] = P~[e d + i][k] / alpha
// (0 where alpha = 0).  One block per (expert, 32 columns): the column sums of
// squares, then the scaled transpose through a 32 x 33 tile.
__global__ void k_normalize(const float* __restrict__ Pt, int E, int d, int n, float* __restrict__ alpha,
                            float* __restrict__ P) {
  __shared__ float tile[32][33];
  __shared__ float part[8][32];
  __shared__ float inv[32];
  const int e = blockIdx.y, k0 = blockIdx.x * 32;
  const int tx = threadIdx.x, ty = threadIdx.y;   // 32 x 8
  const float* base = Pt + (size_t)e * d * n;
  float ss = 0.f;
  const int k = k0 + tx;
  if (k < n)
    for (int i = ty; i < d; i += 8) {
      const float v = base[(size_t)i * n + k];
      ss = fmaf(v, v, ss);
    }
  part[ty][tx] = ss;
  __syncthreads();
  if (ty == 0) {
    float t = 0.f;
    for (int q = 0; q < 8; ++q) t += part[q][tx];
    const float a = sqrtf(t);
    if (k < n) alpha[(size_t)e * n + k] = a;
    inv[tx] = a > 0.f ? 1.f / a : 1.f;
  }
  __syncthreads();
  for (int i0 = 0; i0 < d; i0 += 32) {
    for (int y = ty; y < 32; y += 8) {
      const int i = i0 + y;
      tile[y][tx] = (i < d && k < n) ? base[(size_t)i * n + k] : 0.f;
    }
    __syncthreads();
    for (int y = ty; y < 32; y += 8) {
      const int kk = k0 + y, i = i0 + tx;
      if (kk < n && i < d) P[((size_t)e * n + kk) * d + i] = tile[tx][y] * inv[y];
    }
    __syncthreads();
  }
}

struct DecLayout {
  size_t A, G, Vt, Pt, Q, act, sync, total;
  int m;   // side of G and V^T: D rounded up to whole pairs of index blocks
};
DecLayout dec_layout(int side, int E, int d, int D) {
  const size_t R = (size_t)E * d, n = std::min<size_t>(D, R);
  DecLayout l;
  size_t off = 0;
  auto take = [&](size_t bytes) {
    const size_t o = off;
    off = (off + bytes + 255) / 256 * 256;
    return o;
  };
  l.m = (D + kJP - 1) / kJP * kJP;
  l.A = take(side == 1 ? R * D * 4 : 0);
  l.G = take((size_t)l.m * l.m * 4);
  l.Vt = take((size_t)l.m * l.m * 4);
  l.Pt = take(R * n * 4);
  l.Q = take((size_t)2 * (l.m / kJP) * kTile * 4);
  l.act = take((size_t)2 * (l.m / kJP) * 4);
  l.sync = take(256);
  l.total = off;
  return l;
}

// Ranges of rows for the Gram matrix: as many as fill the chip with the tiles there are (two blocks an SM), of
// at least 512 rows, with their tiles in `room` floats.
int gram_splits(int tiles, int64_t R, size_t room, int sms) {
  const int64_t fill = 2 * (int64_t)sms / tiles, most = (int64_t)(room / ((size_t)tiles * kTM * kTN));
  return (int)std::max<int64_t>(1, std::min({fill, R / 512, most, (int64_t)64}));
}

}  // namespace

extern "C" size_t bitsmoe_decompose_workspace_bytes(int side, int E, int d, int D) {
  if ((side != 0 && side != 1) || E < 1 || d < 1 || D < 1) return 0;
  return dec_layout(side, E, d, D).total;
}

extern "C" int bitsmoe_shared_basis(int side, const float* W, int E, int d, int D, float* phi, float* sigma,
                                    float* alpha, float* P, void* ws, size_t ws_bytes, int max_sweeps, int* sweeps,
                                    int* status, void* stream) {
  using namespace bmoe;
  if ((side != 0 && side != 1) || E < 1 || d < 1 || D < 2 || D > BITSMOE_DECOMPOSE_MAX_D || max_sweeps < 1 || !W || !phi ||
      !sigma || !alpha || !P || !ws || !status)
    return BITSMOE_ERR_INVALID_ARG;
  const DecLayout l = dec_layout(side, E, d, D);
  if (ws_bytes < l.total) return BITSMOE_ERR_WORKSPACE_TOO_SMALL;
  if ((reinterpret_cast<uintptr_t>(ws) & 255) != 0) return BITSMOE_ERR_ALIGNMENT;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  uint8_t* wb = static_cast<uint8_t*>(ws);
  const int64_t R = (int64_t)E * d;
  const int n = (int)std::min<int64_t>(D, R);
  float* G = reinterpret_cast<float*>(wb + l.G);
  float* Vt = reinterpret_cast<float*>(wb + l.Vt);
  float* Pt = reinterpret_cast<float*>(wb + l.Pt);
  uint32_t* bar = reinterpret_cast<uint32_t*>(wb + l.sync);
  const float* A = W;
  const int m = l.m, half = m / kJP;
  BM_CK(cudaMemsetAsync(bar, 0, 256, st));
  if (m != D) BM_CK(cudaMemsetAsync(G, 0, (size_t)m * m * 4, st));   // the padding stays 0
  if (side == 1) {
    float* At = reinterpret_cast<float*>(wb + l.A);
    k_transpose_out<<<dim3((d + 31) / 32, (D + 31) / 32, E), dim3(32, 8), 0, st>>>(W, E, D, d, At);
    BM_CK(cudaGetLastError());
    A = At;
  }
  int dev = 0, sms = 0;
  BM_CK(cudaGetDevice(&dev));
  BM_CK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  const int ntile = (D + kTM - 1) / kTM, tiles = ntile * (ntile + 1) / 2;
  const bool va = D % 4 == 0 && reinterpret_cast<uintptr_t>(A) % 16 == 0;
  const int splits = gram_splits(tiles, R, (size_t)R * n, sms);
  const int64_t rows = ((R + splits - 1) / splits + kTK - 1) / kTK * kTK;
  float* part = splits > 1 ? Pt : nullptr;   // P~'s place is free until the projection
  (va ? k_gram<float, true> : k_gram<float, false>)<<<dim3(tiles, splits), kGT, 0, st>>>(A, nullptr, R, D, D, G, m, ntile,
                                                                                         rows, part);
  BM_CK(cudaGetLastError());
  if (part) {
    k_gram_sum<<<dim3(tiles, 16), 256, 0, st>>>(part, splits, D, G, m, ntile);
    BM_CK(cudaGetLastError());
  }
  // the eigensolver: at most one block per SM, all resident (cooperative launch)
  const int nb = std::min(sms, half * (half + 1));
  BM_CK(cudaFuncSetAttribute(k_jacobi, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kJSmem));
  int per_sm = 0;
  BM_CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_jacobi, kJT, kJSmem));
  if (per_sm < 1) return BITSMOE_ERR_SHAPE;
  JacobiArgs ja;
  ja.G = G;
  ja.Vt = Vt;
  ja.Q = reinterpret_cast<float*>(wb + l.Q);
  ja.act = reinterpret_cast<int*>(wb + l.act);
  ja.n = D;
  ja.m = m;
  ja.max_sweeps = max_sweeps;
  ja.tol = 1e-7f;
  ja.bar = bar;
  ja.rot = bar + 32;
  ja.status = status;
  ja.sweeps = sweeps;
  ja.spin = 2ll << 30;
  void* args[] = {&ja};
  BM_CK(cudaLaunchCooperativeKernel(reinterpret_cast<void*>(k_jacobi), dim3(nb), dim3(kJT), args, kJSmem, st));
  k_order<<<D, 256, 0, st>>>(G, Vt, D, m, n, phi, sigma);
  BM_CK(cudaGetLastError());
  const bool vp = va && n % 4 == 0 && reinterpret_cast<uintptr_t>(phi) % 16 == 0;
  (vp ? k_project<true> : k_project<false>)<<<dim3((n + kTN - 1) / kTN, (unsigned)((R + kTM - 1) / kTM)), kGT, 0, st>>>(
      A, phi, R, D, n, Pt);
  BM_CK(cudaGetLastError());
  k_normalize<<<dim3((n + 31) / 32, E), dim3(32, 8), 0, st>>>(Pt, E, d, n, alpha, P);
  BM_CK(cudaGetLastError());
  return BITSMOE_OK;
}

extern "C" int bitsmoe_calibration_gram(const void* x, const float* g, int64_t T, int D, float* H, void* stream) {
  using namespace bmoe;
  if (T < 0 || D < 1 || !H || (T > 0 && !x)) return BITSMOE_ERR_INVALID_ARG;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const int ntile = (D + kTM - 1) / kTM;
  if (T == 0) {
    BM_CK(cudaMemsetAsync(H, 0, (size_t)D * D * 4, st));
    return BITSMOE_OK;
  }
  const bool vx = D % 4 == 0 && reinterpret_cast<uintptr_t>(x) % 8 == 0;
  (vx ? k_gram<uint16_t, true> : k_gram<uint16_t, false>)<<<ntile * (ntile + 1) / 2, kGT, 0, st>>>(
      static_cast<const uint16_t*>(x), g, T, D, D, H, D, ntile, T, nullptr);
  BM_CK(cudaGetLastError());
  return BITSMOE_OK;
}
