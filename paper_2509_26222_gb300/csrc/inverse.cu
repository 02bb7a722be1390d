// Explicit inverse of the float32 Cholesky factor and solves by products.
//
// The refined solves of the mixed-precision update apply the float32 factor
// many times per frame (the weight increment, and the covariance columns of
// the centers that leave the active block).  A blocked substitution is a
// chain of a/64 dependent steps per application.  For active blocks of a few
// thousand centers it is cheaper to form Z = L^{-1} once per factorization,
// in log2(a/64) levels of independent products, and to apply
// H^{-1} ~ Z^T Z as two products that run on every SM at once:
//
//   level b (b = 128, 256, ...): for every diagonal pair of b/2-blocks
//     [L11 0; L21 L22]^{-1} = [Z11 0; -Z22 L21 Z11  Z22]
//   (T = L21 Z11, then Z21 = -Z22 T; Z11, Z22 come from the level below and
//   the 64 x 64 blocks from the factorization itself).
//
// Z has the factor's shape (row-major, leading dimension ldz) with zeros
// above the diagonal; its transpose follows it in the same buffer (rows
// n .. 2n - 1).  The solves are Y = Z F followed by F = Z^T Y.
#include <cuda_runtime.h>

#include "common.cuh"
#include "tc_util.cuh"
#include "tiles.cuh"

namespace rbf {
namespace {

constexpr int TG = 64;       // output tile (rows and columns)
constexpr int TK = 32;       // K chunk staged in shared memory
constexpr int TLD = TG + 4;  // padded row of the staged chunks
constexpr int GEMV_M = 8;    // right-hand sides handled by the matrix-vector kernels

// Element (r, c) of a row-major matrix, or of the transpose of one.
struct Mat {
  const float* p;
  int64_t ld;
  bool t;
};

// acc += A[i0 + 0..63, kb..ke) * B[kb..ke, j0 + 0..63) for rows < M and
// columns < N; 256 threads, each a 4 x 4 block of the tile.  The next chunk
// is fetched into registers while the current one is multiplied.
__device__ __forceinline__ void tile_mma(float (&acc)[4][4], const Mat A, const Mat B, int64_t i0, int64_t j0,
                                         int64_t M, int64_t N, int64_t kb, int64_t ke, float (*As)[TLD],
                                         float (*Bs)[TLD]) {
  const int tid = threadIdx.x, ty = tid >> 4, tx = tid & 15;
  float ra[8], rb[8];
  auto fetch = [&](int64_t k0) {
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      int idx = tid + 256 * e;  // 0 .. 2047
      int r, kk;
      if (A.t) { r = idx & (TG - 1); kk = idx >> 6; }
      else { kk = idx & (TK - 1); r = idx >> 5; }
      int64_t gi = i0 + r, gk = k0 + kk;
      ra[e] = (gi < M && gk < ke) ? (A.t ? A.p[gk * A.ld + gi] : A.p[gi * A.ld + gk]) : 0.f;
      int cc;
      if (B.t) { kk = idx & (TK - 1); cc = idx >> 5; }
      else { cc = idx & (TG - 1); kk = idx >> 6; }
      int64_t gj = j0 + cc;
      gk = k0 + kk;
      rb[e] = (gj < N && gk < ke) ? (B.t ? B.p[gj * B.ld + gk] : B.p[gk * B.ld + gj]) : 0.f;
    }
  };
  auto stash = [&]() {
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      int idx = tid + 256 * e;
      int r, kk;
      if (A.t) { r = idx & (TG - 1); kk = idx >> 6; }
      else { kk = idx & (TK - 1); r = idx >> 5; }
      As[kk][r] = ra[e];
      int cc;
      if (B.t) { kk = idx & (TK - 1); cc = idx >> 5; }
      else { cc = idx & (TG - 1); kk = idx >> 6; }
      Bs[kk][cc] = rb[e];
    }
  };
  if (kb >= ke) return;
  fetch(kb);
  for (int64_t k0 = kb; k0 < ke; k0 += TK) {
    stash();
    __syncthreads();
    if (k0 + TK < ke) fetch(k0 + TK);
#pragma unroll 8
    for (int kk = 0; kk < TK; ++kk) {
      float4 a4 = *reinterpret_cast<const float4*>(&As[kk][ty * 4]);
      float4 b4 = *reinterpret_cast<const float4*>(&Bs[kk][tx * 4]);
      float av[4] = {a4.x, a4.y, a4.z, a4.w};
      float bv[4] = {b4.x, b4.y, b4.z, b4.w};
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < 4; ++v) acc[u][v] = fmaf(av[u], bv[v], acc[u][v]);
    }
    __syncthreads();
  }
}

// C = alpha acc, or C += alpha acc with atomics (the two halves of a K range
// split in two: 0 + a + b equals 0 + b + a exactly, so the result does not
// depend on which half lands first)
__device__ __forceinline__ void tile_store(const float (&acc)[4][4], float alpha, float* C, int64_t ldc, int64_t i0,
                                           int64_t j0, int64_t M, int64_t N, bool add = false) {
  const int tid = threadIdx.x, ty = tid >> 4, tx = tid & 15;
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    int64_t i = i0 + ty * 4 + u;
    if (i >= M) continue;
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      int64_t j = j0 + tx * 4 + v;
      if (j < N) {
        if (add) atomicAdd(C + i * ldc + j, alpha * acc[u][v]);
        else C[i * ldc + j] = alpha * acc[u][v];
      }
    }
  }
}

// Copy the 64 x 64 diagonal inverses into Z (whose other entries are zero).
__global__ void k_inv_diag(const float* __restrict__ Zd, int64_t n, float* __restrict__ Z, int64_t ldz) {
  after_previous();
  int64_t q = blockIdx.x;
  int64_t k = q * 64;
  int kb = (int)((n - k) < 64 ? (n - k) : 64);
  for (int e = threadIdx.x; e < 64 * 64; e += blockDim.x) {
    int i = e >> 6, t = e & 63;
    if (i < kb && t <= i) Z[(k + i) * ldz + k + t] = Zd[q * 64 * 64 + e];
  }
}

// One level of the doubling: pair p covers rows [p b, p b + b); its upper
// half has h1 = b/2 rows, its lower half h2 = min(b/2, n - p b - b/2).
// kind 0: T21 = L21 Z11 (Z11 lower: only k >= j contributes);
// kind 1: Z21 = -Z22 T21 (Z22 lower: only k <= i contributes).
// split = 2: blockIdx.z = 2 p + half, each half of the K range adds its
// partial product into the (zeroed) output.
__global__ void __launch_bounds__(256) k_trtri_level(int kind, int64_t b, int64_t n, const float* __restrict__ W,
                                                     int64_t ldw, float* __restrict__ Z, int64_t ldz,
                                                     float* __restrict__ T, int split) {
  __shared__ __align__(16) float As[TK][TLD];
  __shared__ __align__(16) float Bs[TK][TLD];
  after_previous();
  const int64_t p = split == 2 ? (blockIdx.z >> 1) : blockIdx.z;
  const int half = split == 2 ? (int)(blockIdx.z & 1) : -1;
  const int64_t r1 = p * b, h1 = b / 2, r2 = r1 + h1;
  const int64_t h2 = (n - r2) < h1 ? (n - r2) : h1;
  if (h2 <= 0) return;
  const int64_t i0 = (int64_t)blockIdx.y * TG, j0 = (int64_t)blockIdx.x * TG;
  if (i0 >= h2 || j0 >= h1) return;
  float acc[4][4] = {};
  int64_t kb, ke;
  if (kind == 0) {
    kb = j0;
    ke = h1;
  } else {
    kb = 0;
    ke = (i0 + TG) < h2 ? (i0 + TG) : h2;
  }
  if (half >= 0) {
    int64_t mid = kb + ((ke - kb) / 2 + TK - 1) / TK * TK;
    if (mid > ke) mid = ke;
    if (half == 0) ke = mid;
    else kb = mid;
  }
  if (kind == 0) {
    Mat A{W + r2 * ldw + r1, ldw, false};
    Mat B{Z + r1 * ldz + r1, ldz, false};
    tile_mma(acc, A, B, i0, j0, h2, h1, kb, ke, As, Bs);
    tile_store(acc, 1.f, T + r2 * ldz + r1, ldz, i0, j0, h2, h1, half >= 0);
  } else {
    Mat A{Z + r2 * ldz + r2, ldz, false};
    Mat B{T + r2 * ldz + r1, ldz, false};
    tile_mma(acc, A, B, i0, j0, h2, h1, kb, ke, As, Bs);
    tile_store(acc, -1.f, Z + r2 * ldz + r1, ldz, i0, j0, h2, h1, half >= 0);
  }
}

// The same products for the levels whose half has TT_MIN rows or more, on the
// tensor cores: one 128 x 128 tile of the output per CTA, C = A B with float32
// operands split into three bfloat16 slices (h, m, l) on their way into shared
// memory and their products accumulated in float32 in tensor memory.
//
// The large levels are nearly all of the n^3 / 3 multiply-adds.  On the float32
// pipe 64 x 64 tiles reach 16 to 20 TFLOP/s there, bound by their shared-memory
// loads.  Here a chunk of K = 64 costs a CTA 24 or 32 instructions of
// 128 x 128 x 16 and the split of 2 x 8,192 floats; two CTAs on an SM overlap the
// two.  B comes as rows of K, so a thread splits two neighbouring rows and stores
// pairs, which makes B K-major.  At half-size 512 this kernel takes as long as the
// float32 tiles (48 + 52 us and 41 + 58 for the two products): the line is at 1024.
// Whole inverse, float32 tiles and now: n = 1,810 225 / 164 us, 2,500 517 / 266,
// 3,750 936 / 425, 5,000 1,959 / 899.
//
// No further from 64 bits than float32 multiply-adds (0.77 to 1.00 times, block by
// block), because
//  * the product h h and the small ones have an accumulator each: added to one,
//    every small product was rounded to the sum of the large ones (2.1 to 2.4);
//  * where a level has fewer tiles than two per SM and two CTAs take half of K
//    each, they are a cluster and swap halves of their accumulators, which are
//    added before the one rounding (rounded apart and added in memory: up to 1.03);
//  * the first product, whose errors the second one amplifies, takes all products
//    but l l, the second one h h, h m, m h, h l, l h and m m (these six for both:
//    up to 1.0004).
// (One accumulator, six products and sums in memory: 160, 258, 434 and 950 us.)
constexpr int TT_MIN = 1024;
constexpr int TT_K = 64;
constexpr int TT_SLICE = 128 * TT_K * 2;             // bytes of a 128 x 64 bf16 slice
constexpr uint32_t TT_COLS = 256;
constexpr int TT_ROW = 128 * 4 + 32;                 // bytes of a staged output row (padded over the banks)
constexpr int TT_TURN = 32 * 36 * 4;                 // bytes of a warp's 32 x 32 floats on their way to the peer
constexpr int TT_SMEM = 128 * TT_ROW + 8 * TT_TURN + 1024;  // the operands (6 slices) lie in the same place
static_assert(128 * TT_ROW + 8 * TT_TURN >= 6 * TT_SLICE, "operands");

// x and y as three bfloat16 each (24 bits, every slice rounded to nearest; a NaN
// stays one), slice t of x in the low and of y in the high half of q[t].  (With the
// rounding as an integer addition, inverse of 3,750 rows 474 us; with the
// conversion instruction 443.)
__device__ __forceinline__ void split3(float x, float y, uint32_t (&q)[3]) {
#pragma unroll
  for (int t = 0; t < 3; ++t) {
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(q[t]) : "f"(y), "f"(x));
    x -= __uint_as_float(q[t] << 16);
    y -= __uint_as_float(q[t] & 0xffff0000u);
  }
}

__global__ void __launch_bounds__(256, 2) k_trtri_tc(int kind, int64_t b, int64_t n, const float* __restrict__ W,
                                                     int64_t ldw, float* __restrict__ Z, int64_t ldz,
                                                     float* __restrict__ T, int split, int* __restrict__ status) {
  extern __shared__ uint8_t tt_raw[];
  __shared__ uint64_t mbar;
  __shared__ uint32_t tmem_slot;
  __shared__ int ok_s;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t p = split == 2 ? (blockIdx.z >> 1) : blockIdx.z;
  const int64_t r1 = p * b, h1 = b / 2, r2 = r1 + h1;
  const int64_t h2 = (n - r2) < h1 ? (n - r2) : h1;
  const int64_t i0 = (int64_t)blockIdx.y * 128, j0 = (int64_t)blockIdx.x * 128;
  if (h2 <= 0 || i0 >= h2 || j0 >= h1) return;
  // K range: kind 0 T21 = L21 Z11 (Z11 lower: k >= j0), kind 1 Z21 = -Z22 T21 (Z22 lower: k < i0 + 128)
  int64_t kb = kind == 0 ? j0 : 0;
  const int64_t kn = kind == 0 ? h1 : h2;  // rows of B
  int64_t ke = kind == 0 ? h1 : ((i0 + 128) < h2 ? (i0 + 128) : h2);
  if (split == 2) {
    int64_t mid = kb + ((ke - kb) / 2 + TT_K - 1) / TT_K * TT_K;
    if (mid > ke) mid = ke;
    if (blockIdx.z & 1) kb = mid;
    else ke = mid;
  }
  const bool some = kb < ke;  // (the second half of a short K may be empty)
  const float* A = kind == 0 ? W + r2 * ldw + r1 : Z + r2 * ldz + r2;
  const int64_t lda = kind == 0 ? ldw : ldz;
  const float* B = kind == 0 ? Z + r1 * ldz + r1 : T + r2 * ldz + r1;
  float* C = (kind == 0 ? T : Z) + r2 * ldz + r1;
  uint8_t* sm = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(tt_raw) + 1023) & ~(uintptr_t)1023);
  after_previous();
  if (warp == 0) tc::tmem_alloc(&tmem_slot, TT_COLS);
  if (tid == 0) tc::mbar_init(&mbar, 1);
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  const uint32_t tmem = tmem_slot;
  // A: rows tid / 16 + 16 q, 4 columns from 4 (tid % 16); B: row pairs 4 (warp % 8) + lane / 8, 4 columns from
  // 32 q + 4 (lane % 8): whole 128-byte lines in every load
  const int ar = tid >> 4, ac = (tid & 15) * 4;
  const int kp = 4 * warp + (lane >> 3), jl = lane & 7;
  float4 av[8], b0[4], b1[4];
  auto fetch = [&](int64_t k0) {
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
    const float* pa = A + (i0 + ar) * lda + k0 + ac;
    // (columns past the matrix but inside the padded row hold zeros or are times a zero row of B)
#pragma unroll
    for (int q = 0; q < 8; ++q)
      av[q] = (i0 + ar + 16 * q < h2 && k0 + ac < kn) ? *reinterpret_cast<const float4*>(pa + 16 * q * lda) : zero;
    const int64_t k = k0 + 2 * kp;
    const float* pb = B + k * ldz + j0 + 4 * jl;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      b0[q] = k < kn ? *reinterpret_cast<const float4*>(pb + 32 * q) : zero;
      b1[q] = k + 1 < kn ? *reinterpret_cast<const float4*>(pb + ldz + 32 * q) : zero;
    }
  };
  // component (e + jl / 2) % 4 first: the eight lanes of a row pair then store to
  // rows of eight different swizzle phases, so that a warp's stores meet 32 banks
  auto rotated = [&](const float4& v, float (&x)[4]) {
    const bool r1 = (jl >> 1) & 1, r2 = (jl >> 2) & 1;
    const float t[4] = {r1 ? v.y : v.x, r1 ? v.z : v.y, r1 ? v.w : v.z, r1 ? v.x : v.w};
    x[0] = r2 ? t[2] : t[0];
    x[1] = r2 ? t[3] : t[1];
    x[2] = r2 ? t[0] : t[2];
    x[3] = r2 ? t[1] : t[3];
  };
  uint32_t phase = 0;
  bool ok = true;
  auto wait = [&]() {  // the products of the last chunk
    if (tid == 0) {
      long long it = 0;
      bool got;
      while (!(got = tc::mbar_try_wait(&mbar, phase)) && ++it < tc::WAIT_LIMIT) {
      }
      if (!got) {
        atomicOr(status, DEV_TIMEOUT);
        // one more bounded chance to drain before the operands and TMEM are given back
        for (it = 0; !tc::mbar_try_wait(&mbar, phase) && it < tc::WAIT_LIMIT; ++it) {
        }
      }
      ok_s = got ? 1 : 0;
    }
    __syncthreads();
    tc::fence_after();
    ok = ok_s != 0;
    phase ^= 1;
  };
  if (some) fetch(kb);
  for (int64_t k0 = kb; k0 < ke && ok; k0 += TT_K) {
    if (k0 > kb) wait();
    if (!ok) break;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      uint32_t lo[3], hi[3];
      split3(av[q].x, av[q].y, lo);
      split3(av[q].z, av[q].w, hi);
      const uint32_t off = tc::sw128_offset(ar + 16 * q, ac >> 3) + 2 * (ac & 7);
#pragma unroll
      for (int t = 0; t < 3; ++t)
        *reinterpret_cast<uint2*>(sm + t * TT_SLICE + off) = make_uint2(lo[t], hi[t]);
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      float x[4], y[4];
      rotated(b0[q], x);
      rotated(b1[q], y);
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        uint32_t w[3];
        split3(x[e], y[e], w);
        const int j = 32 * q + 4 * jl + ((e + (jl >> 1)) & 3);
        const uint32_t off = tc::sw128_offset(j, kp >> 2) + 4 * (kp & 3);
#pragma unroll
        for (int t = 0; t < 3; ++t)
          *reinterpret_cast<uint32_t*>(sm + (3 + t) * TT_SLICE + off) = w[t];
      }
    }
    tc::fence_proxy_async();
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    if (tid == 0) {
      const int pa[8] = {0, 0, 1, 0, 1, 2, 1, 2}, pb[8] = {0, 1, 0, 2, 1, 0, 2, 1};
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        if (q >= 6 && kind != 0) break;
        const uint64_t ad = tc::sdesc_sw128(tc::smem_u32(sm + pa[q] * TT_SLICE));
        const uint64_t bd = tc::sdesc_sw128(tc::smem_u32(sm + (3 + pb[q]) * TT_SLICE));
#pragma unroll
        for (int kk = 0; kk < TT_K / 16; ++kk)
          tc::mma_bf16(tmem + (q ? 128u : 0u), ad + (uint64_t)(2 * kk), bd + (uint64_t)(2 * kk),
                       (k0 > kb || q > 1 || kk > 0) ? 1u : 0u);
      }
      tc::mma_commit(&mbar);
    }
    if (k0 + TT_K < ke) fetch(k0 + TT_K);
  }
  if (ok && some) wait();
  // epilogue: warp w reads TMEM lanes 32 (w % 4) .., puts a row a lane where the
  // operands were (they are read), and a thread a row sends it off in one bulk store
  const float alpha = kind == 0 ? 1.f : -1.f;
  const int lr = 32 * (warp & 3) + lane, q = warp >> 2;
  const uint32_t tl = tmem + ((uint32_t)(32 * (warp & 3)) << 16);
  float v[32], v2[32];
  auto load = [&](int col) {
    tc::tmem_ld32(tl + (uint32_t)col, v);
    tc::tmem_ld32(tl + (uint32_t)(128 + col), v2);
#pragma unroll
    for (int e = 0; e < 32; ++e) {
      if (!some) v[e] = v2[e] = 0.f;
    }
  };
  auto send = [&](int col, int bytes) {
    tc::fence_proxy_async();
    __syncthreads();
    if (tid < 128 && i0 + tid < h2)
      asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(C + (i0 + tid) * ldz + j0 + col),
                   "r"(tc::smem_u32(sm + tid * TT_ROW)), "r"(bytes)
                   : "memory");
    asm volatile("cp.async.bulk.commit_group;\n\tcp.async.bulk.wait_group 0;" ::: "memory");
  };
  if (split == 2) {
    // columns 64 rank .. + 63 are this CTA's: the others' two accumulators go to the peer
    const uint32_t rank = blockIdx.z & 1;
    tc::cluster_arrive();
    load(64 * (int)(rank ^ 1) + 32 * q);
    tc::cluster_wait();  // both have read their operands
    // turned in shared memory, so that eight lanes store the 128 bytes of a row (with
    // a row a lane, in pieces of 16 bytes, the inverse of 3,750 rows took 441 us)
    const uint32_t to = tc::cluster_addr(tc::smem_u32(sm), rank ^ 1);
    float* st = reinterpret_cast<float*>(sm + 128 * TT_ROW + warp * TT_TURN);
    auto give = [&](const float (&x)[32], uint32_t off) {
#pragma unroll
      for (int e = 0; e < 32; e += 4)
        *reinterpret_cast<float4*>(st + lane * 36 + e) = make_float4(x[e], x[e + 1], x[e + 2], x[e + 3]);
      __syncwarp();
#pragma unroll
      for (int t = 0; t < 32; t += 4) {
        const int r = t + (lane >> 3);
        const float4 y = *reinterpret_cast<const float4*>(st + r * 36 + 4 * (lane & 7));
        tc::cluster_store4(to + (uint32_t)((32 * (warp & 3) + r) * TT_ROW) + off + 16u * (lane & 7), y.x, y.y, y.z, y.w);
      }
      __syncwarp();
    };
    give(v, 128u * q);
    give(v2, 256u + 128u * q);
    tc::cluster_arrive();
    load(64 * (int)rank + 32 * q);
    tc::cluster_wait();
    float* sr = reinterpret_cast<float*>(sm + lr * TT_ROW) + 32 * q;
#pragma unroll
    for (int e = 0; e < 32; e += 4) {
      const float4 a = *reinterpret_cast<const float4*>(sr + e), c = *reinterpret_cast<const float4*>(sr + 64 + e);
      auto sum = [&](float x, float y, int k) {
        const FF s = ff_two_sum(v[e + k], x);
        return alpha * (s.hi + (s.lo + (v2[e + k] + y)));
      };
      *reinterpret_cast<float4*>(sr + e) = make_float4(sum(a.x, c.x, 0), sum(a.y, c.y, 1), sum(a.z, c.z, 2), sum(a.w, c.w, 3));
    }
    if (ok) send(64 * (int)rank, 256);
  } else if (ok) {
#pragma unroll 1
    for (int cb = 0; cb < 2; ++cb) {
      const int col = 64 * q + 32 * cb;
      load(col);
      float* sr = reinterpret_cast<float*>(sm + lr * TT_ROW) + col;
#pragma unroll
      for (int e = 0; e < 32; e += 4)
        *reinterpret_cast<float4*>(sr + e) = make_float4(alpha * (v[e] + v2[e]), alpha * (v[e + 1] + v2[e + 1]),
                                                         alpha * (v[e + 2] + v2[e + 2]), alpha * (v[e + 3] + v2[e + 3]));
    }
    send(0, 512);
  }
  tc::fence_before();
  __syncthreads();
  if (warp == 0) tc::tmem_dealloc(tmem, TT_COLS);
}

// Y = Z F (forward, Z lower) or Y = Zt F (backward, Zt = Z^T upper) for
// m > GEMV_M right-hand sides; F, Y row-major n x m.  blockIdx.z splits K; partial
// products go to P[z] and are summed by k_sum_partials.
__global__ void __launch_bounds__(256) k_inv_apply(bool backward, int64_t n, int64_t m, const float* __restrict__ Z,
                                                   int64_t ldz, const float* __restrict__ F, float* __restrict__ P,
                                                   int nsplit) {
  __shared__ __align__(16) float As[TK][TLD];
  __shared__ __align__(16) float Bs[TK][TLD];
  const int64_t i0 = (int64_t)blockIdx.y * TG, j0 = (int64_t)blockIdx.x * TG;
  int64_t kb = backward ? i0 : 0;
  int64_t ke = backward ? n : ((i0 + TG) < n ? (i0 + TG) : n);
  int64_t len = ke - kb;
  int64_t chunk = ((len + nsplit - 1) / nsplit + TK - 1) / TK * TK;
  int64_t sb = kb + (int64_t)blockIdx.z * chunk;
  int64_t se = (sb + chunk) < ke ? (sb + chunk) : ke;
  float acc[4][4] = {};
  Mat A{Z, ldz, false};  // Z (forward) or its transpose stored row-major (backward)
  Mat B{F, m, false};
  if (sb < se) tile_mma(acc, A, B, i0, j0, n, m, sb, se, As, Bs);
  tile_store(acc, 1.f, P + (int64_t)blockIdx.z * n * m, m, i0, j0, n, m);
}

__global__ void k_sum_partials(const float* __restrict__ P, int nsplit, int64_t tot, float* __restrict__ Y) {
  int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= tot) return;
  float s = 0.f;
  for (int z = 0; z < nsplit; ++z) s += P[z * tot + e];
  Y[e] = s;
}

// Y = A F for m <= GEMV_M with A = Z (lower: row i over k <= i) or A = Z^T
// stored transposed (upper: row i over k >= i): one warp per row, lanes over
// the row, eight loads of A in flight per lane.  With Xd set, the result is
// added to the float64 Xd instead of stored to Y.
template <bool UPPER>
__global__ void __launch_bounds__(256) k_inv_gemv(int64_t n, int m, const float* __restrict__ A, int64_t lda,
                                                  const float* __restrict__ F, float* __restrict__ Y,
                                                  double* __restrict__ Xd) {
  after_previous();
  const int lane = threadIdx.x & 31;
  const int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (i >= n) return;
  const int64_t lo = UPPER ? i : 0, hi = UPPER ? n : i + 1;
  float acc[GEMV_M];
#pragma unroll
  for (int j = 0; j < GEMV_M; ++j) acc[j] = 0.f;
  const float* ar = A + i * lda;
  for (int64_t k0 = lo + lane; k0 < hi; k0 += 256) {
    float z[8], f[8][GEMV_M];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      int64_t k = k0 + 32 * u;
      bool ok = k < hi;
      z[u] = ok ? ar[k] : 0.f;
#pragma unroll
      for (int j = 0; j < GEMV_M; ++j) f[u][j] = (ok && j < m) ? F[k * m + j] : 0.f;
    }
#pragma unroll
    for (int u = 0; u < 8; ++u)
#pragma unroll
      for (int j = 0; j < GEMV_M; ++j) acc[j] = fmaf(z[u], f[u][j], acc[j]);
  }
#pragma unroll
  for (int j = 0; j < GEMV_M; ++j) {
    if (j >= m) break;
    float v = acc[j];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0) {
      if (Xd) Xd[i * m + j] += (double)v;
      else Y[i * m + j] = v;
    }
  }
}

// Zt = Z^T (n x n, both with leading dimension ld), 32 x 32 tiles
__global__ void k_transpose32(const float* __restrict__ Z, int64_t n, int64_t ld, float* __restrict__ Zt) {
  __shared__ float t[32][33];
  after_previous();
  const int64_t bx = (int64_t)blockIdx.x * 32, by = (int64_t)blockIdx.y * 32;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;  // 32 x 8 threads
  for (int r = ty; r < 32; r += 8) {
    int64_t i = by + r, j = bx + tx;
    t[r][tx] = (i < n && j < n) ? Z[i * ld + j] : 0.f;
  }
  __syncthreads();
  for (int r = ty; r < 32; r += 8) {
    int64_t i = bx + r, j = by + tx;
    if (i < n && j < n) Zt[i * ld + j] = t[tx][r];
  }
}

// Y[i][u] = Z[i][pos[u]]: the product of Z with unit columns
__global__ void k_gather_cols(const float* __restrict__ Z, int64_t n, int64_t ld, const int32_t* __restrict__ pos,
                              int64_t m, float* __restrict__ Y) {
  int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= n * m) return;
  int64_t i = e / m, u = e % m;
  Y[e] = Z[i * ld + pos[u]];
}

unsigned cdiv(int64_t a, int64_t b) { return (unsigned)((a + b - 1) / b); }

}  // namespace

// K slices of the inverse apply: as many as fill the co-resident CTAs of
// the GPU once (the tiles alone leave most SMs idle for a few right-hand
// sides), at least 4 chunks of K each and at most 8.
static int apply_split(Ctx* c, int64_t tiles, int64_t n) {
  static int cap[64] = {0};
  const int dev = c->device & 63;
  if (!cap[dev]) {
    int occ = 0, sms = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_inv_apply, 256, 0) != cudaSuccess || occ < 1) occ = 1;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, c->device) != cudaSuccess || sms < 1) sms = 1;
    cap[dev] = occ * sms;
  }
  int64_t ns = cap[dev] / (tiles > 0 ? tiles : 1);
  const int64_t most = n / (4 * TK);
  if (ns > most) ns = most;
  if (ns > 8) ns = 8;
  return ns < 1 ? 1 : (int)ns;
}

rbf_status trtri_mixed(Ctx* c, const float* W, int64_t ldw, int64_t n, const float* Zd, float* Z, int64_t ldz,
                       cudaStream_t s) {
  if (n <= 0) return RBF_OK;
  Buf& tb = c->scratch(65);
  RBF_TRY(tb.ensure((size_t)n * ldz * sizeof(float)));
  float* T = tb.as<float>();
  StageTimer st(c, RBF_STAGE_INVERSE, s, (double)n * n * n / 3.0);
  RBF_CUDA(cudaMemsetAsync(Z, 0, (size_t)n * ldz * sizeof(float), s));
  RBF_CUDA(cudaMemsetAsync(T, 0, (size_t)n * ldz * sizeof(float), s));  // levels write disjoint blocks
  const bool early = not_capturing(s);
  RBF_CUDA(launch_early(early, k_inv_diag, cdiv(n, 64), 256, 0, s, Zd, n, Z, ldz));
  for (int64_t b = 128; b / 2 < n; b *= 2) {
    int64_t h = b / 2;
    if (h >= TT_MIN) {
      static bool attr[64] = {false};
      if (!attr[c->device & 63]) {
        RBF_CUDA(cudaFuncSetAttribute(k_trtri_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, TT_SMEM));
        attr[c->device & 63] = true;
      }
      // fewer tiles than two per SM: K in two halves, by a pair of CTAs
      const int64_t tt = (int64_t)cdiv(h, 128) * cdiv(h, 128) * cdiv(n, b);
      const int sp = tt < 2 * 152 ? 2 : 1;
      for (int kind = 0; kind < 2; ++kind) {
        RBF_CUDA(launch_early_z(early, (unsigned)sp, k_trtri_tc, dim3(cdiv(h, 128), cdiv(h, 128), (unsigned)(cdiv(n, b) * sp)),
                                256, TT_SMEM, s, kind, b, n, W, ldw, Z, ldz, T, sp, c->dflag.as<int>()));
      }
      continue;
    }
    // levels whose tiles do not fill the GPU twice split K in two halves
    const int64_t tiles = (int64_t)cdiv(h, TG) * cdiv(h, TG) * cdiv(n, b);
    const int split = (tiles < 2 * 152 && h >= 256) ? 2 : 1;
    dim3 grid(cdiv(h, TG), cdiv(h, TG), (unsigned)(cdiv(n, b) * split));
    for (int kind = 0; kind < 2; ++kind) {
      RBF_CUDA(launch_early(early, k_trtri_level, grid, 256, 0, s, kind, b, n, W, ldw, Z, ldz, T, split));
    }
  }
  // Z^T stored row-major, so that products with Z^T read rows too
  RBF_CUDA(launch_early(early, k_transpose32, dim3(cdiv(n, 32), cdiv(n, 32)), 256, 0, s, (const float*)Z, n, ldz, Z + n * ldz));
  return RBF_OK;
}

rbf_status inv_solve(Ctx* c, const float* Z, int64_t ldz, int64_t n, float* F, int64_t m, cudaStream_t s) {
  if (n <= 0 || m <= 0) return RBF_OK;
  Buf& yb = c->scratch(66);
  RBF_TRY(yb.ensure((size_t)n * m * sizeof(float)));
  float* Y = yb.as<float>();
  StageTimer st(c, RBF_STAGE_INVAPPLY, s, 2.0 * (double)n * n * m);
  const float* Zt = Z + n * ldz;
  if (m <= GEMV_M) {
    { k_inv_gemv<false><<<cdiv(n * 32, 256), 256, 0, s>>>(n, (int)m, Z, ldz, F, Y, nullptr); ::rbf::note_launch(); }
    RBF_CUDA(cudaGetLastError());
    { k_inv_gemv<true><<<cdiv(n * 32, 256), 256, 0, s>>>(n, (int)m, Zt, ldz, Y, F, nullptr); ::rbf::note_launch(); }
    RBF_CUDA(cudaGetLastError());
    return RBF_OK;
  }
  int64_t tiles = (int64_t)cdiv(n, TG) * cdiv(m, TG);
  int nsplit = apply_split(c, tiles, n);
  Buf& pb = c->scratch(67);
  RBF_TRY(pb.ensure((size_t)nsplit * n * m * sizeof(float)));
  float* P = pb.as<float>();
  dim3 grid(cdiv(m, TG), cdiv(n, TG), nsplit);
  unsigned nr = cdiv(n * m, 256);
  { k_inv_apply<<<grid, 256, 0, s>>>(false, n, m, Z, ldz, F, P, nsplit); ::rbf::note_launch(); }
  RBF_CUDA(cudaGetLastError());
  { k_sum_partials<<<nr, 256, 0, s>>>(P, nsplit, n * m, Y); ::rbf::note_launch(); }
  RBF_CUDA(cudaGetLastError());
  { k_inv_apply<<<grid, 256, 0, s>>>(true, n, m, Zt, ldz, Y, P, nsplit); ::rbf::note_launch(); }
  RBF_CUDA(cudaGetLastError());
  { k_sum_partials<<<nr, 256, 0, s>>>(P, nsplit, n * m, F); ::rbf::note_launch(); }
  RBF_CUDA(cudaGetLastError());
  return RBF_OK;
}

// X += Z^T (Z R) for m <= GEMV_M right-hand sides, R and X float64: R is
// rounded to float32 once (a float64 operand inside the matrix-vector loop
// would convert it once per row, on GB300's narrow float64 pipe), and the
// float64 accumulation happens in the second matrix-vector launch.
__global__ void k_round_f32(const double* __restrict__ R, int64_t cnt, float* __restrict__ F) {
  after_previous();
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < cnt) F[i] = (float)R[i];
}

rbf_status inv_solve_acc(Ctx* c, const float* Z, int64_t ldz, int64_t n, const double* R, double* X, int64_t m,
                         cudaStream_t s) {
  if (n <= 0 || m <= 0) return RBF_OK;
  if (m > GEMV_M) return fail(RBF_EINVAL, "inv_solve_acc: at most %d right-hand sides", GEMV_M);
  Buf& yb = c->scratch(66);
  RBF_TRY(yb.ensure((size_t)2 * n * m * sizeof(float)));
  float* Y = yb.as<float>();
  float* F = Y + n * m;
  StageTimer st(c, RBF_STAGE_INVAPPLY, s, 2.0 * (double)n * n * m);
  const float* Zt = Z + n * ldz;
  const bool early = not_capturing(s);
  const unsigned g = cdiv(n * 32, 256);
  RBF_CUDA(launch_early(early, k_round_f32, cdiv(n * m, 256), 256, 0, s, R, n * m, F));
  RBF_CUDA(launch_early(early, k_inv_gemv<false>, g, 256, 0, s, n, (int)m, Z, ldz, (const float*)F, Y, (double*)nullptr));
  RBF_CUDA(launch_early(early, k_inv_gemv<true>, g, 256, 0, s, n, (int)m, Zt, ldz, (const float*)Y, (float*)nullptr, X));
  return RBF_OK;
}

// F = Z^T (Z E_P) for unit columns E_P at positions pos (n x m, row-major):
// the first product is a gather of columns of Z.
rbf_status inv_solve_unit(Ctx* c, const float* Z, int64_t ldz, int64_t n, const int32_t* pos, int64_t m, float* F,
                          cudaStream_t s) {
  if (n <= 0 || m <= 0) return RBF_OK;
  Buf& yb = c->scratch(66);
  RBF_TRY(yb.ensure((size_t)n * m * sizeof(float)));
  float* Y = yb.as<float>();
  StageTimer st(c, RBF_STAGE_INVAPPLY, s, (double)n * n * m);
  const float* Zt = Z + n * ldz;
  { k_gather_cols<<<cdiv(n * m, 256), 256, 0, s>>>(Z, n, ldz, pos, m, Y); ::rbf::note_launch(); }
  RBF_CUDA(cudaGetLastError());
  if (m <= GEMV_M) {
    { k_inv_gemv<true><<<cdiv(n * 32, 256), 256, 0, s>>>(n, (int)m, Zt, ldz, Y, F, nullptr); ::rbf::note_launch(); }
    RBF_CUDA(cudaGetLastError());
    return RBF_OK;
  }
  int64_t tiles = (int64_t)cdiv(n, TG) * cdiv(m, TG);
  int nsplit = apply_split(c, tiles, n);
  Buf& pb = c->scratch(67);
  RBF_TRY(pb.ensure((size_t)nsplit * n * m * sizeof(float)));
  float* P = pb.as<float>();
  dim3 grid(cdiv(m, TG), cdiv(n, TG), nsplit);
  { k_inv_apply<<<grid, 256, 0, s>>>(true, n, m, Zt, ldz, Y, P, nsplit); ::rbf::note_launch(); }
  RBF_CUDA(cudaGetLastError());
  { k_sum_partials<<<cdiv(n * m, 256), 256, 0, s>>>(P, nsplit, n * m, F); ::rbf::note_launch(); }
  RBF_CUDA(cudaGetLastError());
  return RBF_OK;
}

}  // namespace rbf
