// Dense FP64 linear algebra for the active-block update (Sec. III-C).
//
// The update needs the Cholesky factor of the information matrix of the
// active rows (the matrix whose inverse Eq. kf_w_update applies), triangular
// solves with it, a partial factorization (Schur complement) to drop centers
// that leave the active block, and a few small products.  All matrices are
// row-major with a leading dimension; only lower triangles are referenced
// where a matrix is symmetric.
//
//  potrf_lower: right-looking blocked Cholesky, block 16, one launch per block
//    column: the panel of this column and the trailing update of the previous
//    one run side by side (k_potrf_step).  Stopping after nfactor columns
//    leaves the Schur complement in the trailing block.
//  trsm_lower: L X = B or L^T X = B for many right-hand sides with one
//    cooperative launch: a CTA owns one block row of a few right-hand sides
//    and waits on a flag per block row and column chunk (bounded spin; a
//    timeout sets a status bit) before consuming a solved block.
#include <math.h>

#include <type_traits>

#include "common.cuh"
#include "recip.cuh"

namespace rbf {

constexpr int NB = 32;   // block of the triangular solves
constexpr int PB = 16;   // block column of the factorization
constexpr int UT = 32;   // tile of the trailing update
constexpr int PT = 256;  // threads of a factorization CTA

// ---------------------------------------------------------------------------
// Step k of the factorization, one CTA per SM.
//
// What bounds it: a float64 warp instruction holds its quarter of the SM for
// 64 cycles whatever its number of active lanes (measured: 65 cycles for one
// warp, dependent or not; 1.68 lanes a cycle for an SM with 8 warps), so the
// factorization is bound by the float64 pipe while the trailing block is large,
// and by the serial chain of the diagonal tile when it is small.  Therefore
//  * block columns of 16: the work every CTA repeats (the diagonal tile) grows
//    with the cube of the block, the number of launches only with its inverse;
//  * look-ahead in one launch: the first CTAs apply panel k - 1 to block column
//    k, factor its diagonal tile (each for itself) and solve their rows, and
//    then join the others, who apply panel k - 1 to the columns behind it in
//    32 x 32 tiles drawn from a counter.  The two parts touch disjoint columns;
//  * the diagonal tile is eliminated as V D^-1 V^T, without a square root in the
//    chain, by one warp: lane (i, h) holds row i and the columns 2c + h; the
//    columns are scaled to L = V D^-1/2 at the end.
// Against three launches per 32-wide panel (a chain with a barrier per operation,
// a copy of the tile, 64 x 64 trailing tiles): three frames of a = 1,810, the
// first banded, 16.7 -> 7.2 ms; a = 256, 630 -> 191 us.  A step without trailing
// work takes 12 us, of which the chain of the diagonal tile is about 5.  The next
// step's blocks are placed while a step runs (launch_early): 14.3 -> 11.7 us from
// step to step, the three frames 11.3 -> 10.3 ms in all.
// ---------------------------------------------------------------------------
struct PotrfStep {
  double* A;
  int64_t lda, k;    // first column of this block column
  int64_t ne, pe;    // row ends (band) of this panel and of the previous one
  int kb, kp;        // widths of this block column (0: none) and of the previous one (0: none)
  int npanel;        // CTAs that share the panel
  int tiles;         // trailing tiles
  double* dt;        // factored diagonal tile of this step (16 x 16), if several CTAs read it
  const double* dtp; // that of the previous step, to be copied into A, or null
  int* next;         // tile counter, 0 before the launch
  int* flag;
};

__global__ void __launch_bounds__(PT) k_potrf_step(PotrfStep P) {
  __shared__ double D[PB][PB + 1];   // diagonal tile, then V
  __shared__ double U[PB][PB + 1];   // V D^-1
  __shared__ double Lk[PB][PB + 1];  // L[k block, k - 1]
  __shared__ double rs[PB];          // D^-1/2
  __shared__ double Pi[2][PB][UT + 1], Pj[2][PB][UT + 1];
  __shared__ int nxt[2], redo;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  after_previous();
  double* __restrict__ A = P.A;
  const int64_t lda = P.lda, k = P.k, k0 = k + P.kb;
  const int kb = P.kb, kp = P.kp;
  if (P.dtp && blockIdx.x == gridDim.x - 1) {
    const int i = tid >> 4, j = tid & 15;
    if (i < kp && j <= i) A[(k - kp + i) * lda + k - kp + j] = P.dtp[tid];
  }
  if ((int)blockIdx.x < P.npanel) {
    const int i = tid >> 4, j = tid & 15;
    double dv = (i < kb && j <= i) ? A[(k + i) * lda + k + j] : (i == j ? 1.0 : 0.0);
    Lk[i][j] = (i < kb && j < kp) ? A[(k + i) * lda + k - kp + j] : 0.0;
    int64_t r = k0 + (int64_t)blockIdx.x * PB + i;
    double x = (r < P.ne && j < kb) ? A[r * lda + k + j] : 0.0;
    double(*Lr)[UT + 1] = Pi[0];  // L[rows, k - 1], transposed
    Lr[j][i] = (r < P.pe && j < kp) ? A[r * lda + k - kp + j] : 0.0;
    __syncthreads();
    if (kp) {
      double acc = 0.0;
#pragma unroll
      for (int t = 0; t < PB; ++t) acc = fma(Lk[i][t], Lk[j][t], acc);
      if (i < kb && j <= i) dv -= acc;
    }
    D[i][j] = dv;
    __syncthreads();
    // in: D; out: D = V, U = V D^-1, rs.  Warp 0; true if a pivot lies outside the
    // range of rcp_pos (nothing of the result is used then, unless ANY).
    auto eliminate = [&](auto any) {
      constexpr bool ANY = decltype(any)::value;
      const int ri = lane & 15, h = lane >> 4;
      double a[PB / 2];
#pragma unroll
      for (int c = 0; c < PB / 2; ++c) a[c] = D[ri][2 * c + h];
      __syncwarp();
      bool bad = false, odd = false;
#pragma unroll
      for (int t = 0; t < PB; ++t) {
        const double v = __shfl_sync(0xffffffffu, a[t >> 1], ri + 16 * (t & 1));  // column t of row ri
        double d = __shfl_sync(0xffffffffu, v, t);
        if (!(d > 0.0)) {
          bad = true;
          d = 1.0;
        }
        odd |= !rcp_pos_range(d);
        const double u = ANY ? v / d : v * rcp_pos(d);
        if (h == 0) {
          D[ri][t] = ri == t ? d : v;
          U[ri][t] = u;
        }
#pragma unroll
        for (int c = t >> 1; c < PB / 2; ++c) {
          const double vk = __shfl_sync(0xffffffffu, v, 2 * c + h);
          if (2 * c + h > t) a[c] = fma(-u, vk, a[c]);
        }
      }
      if (bad && (ANY || !odd) && lane == 0 && blockIdx.x == 0) atomicOr(P.flag, DEV_NOT_SPD);
      __syncwarp();
      if (h == 0) rs[ri] = rsqrt(D[ri][ri]);
      return odd;
    };
    if (warp == 0) {
      const bool odd = eliminate(std::false_type{});
      if (lane == 0) redo = odd ? 1 : 0;
    }
    if (kp) {  // the rows' own update, beside the chain of the diagonal tile
      double acc = 0.0;
#pragma unroll
      for (int t = 0; t < PB; ++t) acc = fma(Lr[t][i], Lk[j][t], acc);
      x -= acc;
    }
    __syncthreads();
    if (redo) {  // a subnormal, huge or infinite pivot: again, with the language's division
      D[i][j] = dv;
      __syncthreads();
      if (warp == 0) eliminate(std::true_type{});
      __syncthreads();
    }
    if (blockIdx.x == 0) {
      double l = j <= i ? D[i][j] * rs[j] : 0.0;  // D rsqrt(D) on the diagonal
      if (i == j && isinf(D[i][i])) l = D[i][i];  // (an infinite ridge: its weight stays zero)
      if (P.npanel > 1) P.dt[tid] = l;
      else if (i < kb && j <= i) A[(k + i) * lda + k + j] = l;  // this CTA alone has read the tile
    }
    double ur[PB - 1];
#pragma unroll
    for (int t = 0; t < PB - 1; ++t) ur[t] = U[j][t];
    const double rj = rs[j];
    for (int64_t g = blockIdx.x;;) {
#pragma unroll
      for (int t = 0; t < PB - 1; ++t) {
        const double xt = __shfl_sync(0xffffffffu, x, (lane & 16) + t);
        if (j > t) x = fma(-xt, ur[t], x);
      }
      if (r < P.ne && j < kb) A[r * lda + k + j] = x * rj;
      g += P.npanel;
      if (k0 + g * PB >= P.ne) break;
      r = k0 + g * PB + i;
      x = (r < P.ne && j < kb) ? A[r * lda + k + j] : 0.0;
      if (kp) {
        __syncthreads();
        Lr[j][i] = (r < P.pe && j < kp) ? A[r * lda + k - kp + j] : 0.0;
        __syncthreads();
        double acc = 0.0;
#pragma unroll
        for (int t = 0; t < PB; ++t) acc = fma(Lr[t][i], Lk[j][t], acc);
        x -= acc;
      }
    }
    __syncthreads();  // Lr is staged over below
  }
  // trailing tiles (ti >= tj) of rows [k0, pe): C -= P P^T with the previous
  // panel P; the next tile's operands are on their way while this one's
  // products run.
  if (P.tiles == 0) return;
  const int tx = tid & 15, ty = tid >> 4;
  double pi[2], pj[2], cv[4];
  int64_t i0 = 0, j0 = 0;
  auto fetch = [&](int b, int64_t& fi, int64_t& fj) {
    int ti = (int)((sqrtf(8.f * (float)b + 1.f) - 1.f) * 0.5f);
    while ((ti + 1) * (ti + 2) / 2 <= b) ++ti;
    while (ti * (ti + 1) / 2 > b) --ti;
    fi = k0 + (int64_t)ti * UT;
    fj = k0 + (int64_t)(b - ti * (ti + 1) / 2) * UT;
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int64_t ra = fi + ty + 16 * u, rb = fj + ty + 16 * u;
      pi[u] = (ra < P.pe && tx < kp) ? A[ra * lda + k - kp + tx] : 0.0;
      pj[u] = (rb < P.pe && tx < kp) ? A[rb * lda + k - kp + tx] : 0.0;
#pragma unroll
      for (int v = 0; v < 2; ++v) {
        const int64_t ri = fi + 2 * ty + u, cj = fj + tx + 16 * v;
        cv[2 * u + v] = (ri < P.pe && cj <= ri) ? A[ri * lda + cj] : 0.0;
      }
    }
  };
  if (tid == 0) nxt[0] = atomicAdd(P.next, 1);
  __syncthreads();
  int b = nxt[0], par = 0;
  if (b >= P.tiles) return;
  fetch(b, i0, j0);
  while (b < P.tiles) {
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      Pi[par][tx][ty + 16 * u] = pi[u];
      Pj[par][tx][ty + 16 * u] = pj[u];
    }
    double c[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) c[q] = cv[q];
    if (tid == 0) nxt[par ^ 1] = atomicAdd(P.next, 1);
    __syncthreads();
    const int bn = nxt[par ^ 1];
    const int64_t ci = i0, cj0 = j0;
    if (bn < P.tiles) fetch(bn, i0, j0);
#pragma unroll
    for (int t = 0; t < PB; ++t) {
      const double a0 = Pi[par][t][2 * ty], a1 = Pi[par][t][2 * ty + 1];
      const double b0 = Pj[par][t][tx], b1 = Pj[par][t][tx + 16];
      c[0] = fma(-a0, b0, c[0]);
      c[1] = fma(-a0, b1, c[1]);
      c[2] = fma(-a1, b0, c[2]);
      c[3] = fma(-a1, b1, c[3]);
    }
#pragma unroll
    for (int u = 0; u < 2; ++u)
#pragma unroll
      for (int v = 0; v < 2; ++v) {
        const int64_t ri = ci + 2 * ty + u, cj = cj0 + tx + 16 * v;
        if (ri < P.pe && cj <= ri) A[ri * lda + cj] = c[2 * u + v];
      }
    b = bn;
    par ^= 1;
  }
}

static int dense_sms(int dev) {
  static int sms[64] = {0};
  int& v = sms[dev & 63];
  if (!v && (cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || v <= 0)) v = 152;
  return v;
}

rbf_status potrf_lower(Ctx* c, double* A, int64_t n, int64_t lda, int64_t nfactor, bool mixed,
                       cudaStream_t s, int64_t bw) {
  (void)mixed;
  if (n <= 0 || nfactor <= 0) return RBF_OK;
  const int64_t steps = (nfactor + PB - 1) / PB;
  const int sms = dense_sms(c->device);
  // two diagonal tiles, then one tile counter per launch
  Buf& dt = c->scratch(30);
  RBF_TRY(dt.ensure(2 * PB * PB * sizeof(double) + (size_t)(steps + 1) * sizeof(int)));
  int* next = reinterpret_cast<int*>(dt.as<double>() + 2 * PB * PB);
  RBF_CUDA(cudaMemsetAsync(next, 0, (size_t)(steps + 1) * sizeof(int), s));
  StageTimer st(c, RBF_STAGE_PANEL, s, potrf_work(n, nfactor, bw));  // panels and trailing updates share the launches
  const bool early = not_capturing(s);
  PotrfStep P;
  P.A = A;
  P.lda = lda;
  P.flag = c->dflag.as<int>();
  P.kp = 0;
  P.pe = 0;
  P.dtp = nullptr;
  for (int64_t q = 0; q <= steps; ++q) {
    P.k = q * PB < nfactor ? q * PB : nfactor;
    P.kb = (int)((nfactor - P.k) < PB ? (nfactor - P.k) : PB);  // 0: the last panel's update only
    const int64_t k0 = P.k + P.kb;
    // rows beyond the band are zero in this panel and untouched by its update
    P.ne = P.kb ? ((k0 + bw) < n ? (k0 + bw) : n) : P.k;
    const int64_t groups = (P.ne - k0 + PB - 1) / PB;
    P.npanel = P.kb ? (int)(groups < 1 ? 1 : (groups < sms ? groups : sms)) : 0;
    const int64_t T = P.pe > k0 ? (P.pe - k0 + UT - 1) / UT : 0;
    P.tiles = P.kp ? (int)(T * (T + 1) / 2) : 0;
    P.dt = dt.as<double>() + (q & 1) * PB * PB;
    P.next = next + q;
    int64_t grid = (int64_t)P.npanel + P.tiles;
    if (grid > sms) grid = sms;
    if (grid < 1) {
      if (!P.dtp) break;
      grid = 1;
    }
    RBF_CUDA(launch_early(early && q > 0, k_potrf_step, dim3((unsigned)grid), dim3(PT), 0, s, P));
    P.dtp = P.npanel > 1 ? P.dt : nullptr;
    P.kp = P.kb;
    P.pe = P.ne;
  }
  return RBF_OK;
}

// ---------------------------------------------------------------------------
// Sync-free blocked triangular solve with many right-hand sides.
// ---------------------------------------------------------------------------
constexpr int TS_THREADS = 256;
constexpr long long TS_SPIN_LIMIT = 1LL << 22;

__device__ __forceinline__ int ld_acquire(const int* p) {
  int v;
  asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_release(int* p, int v) {
  asm volatile("st.release.gpu.global.b32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// Inverses of the 32 x 32 diagonal blocks of L, one CTA each, identity beyond a
// ragged last block: the 16 x 16 halves by substitution (a warp each, lane =
// column), Z21 = -Z22 (L21 Z11) by all threads.  The solves apply them as
// products (10 us a factor).  Formed inside every CTA of every solve, with a
// division per entry, they were most of the 153 us of a solve of 256 unknowns
// (now 22 us).
__global__ void __launch_bounds__(TS_THREADS) k_diag_inv(const double* __restrict__ L, int64_t ldl, int64_t n,
                                                         double* __restrict__ Z) {
  __shared__ double T[NB][NB + 1], Zs[NB][NB + 1], Y[16][17];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t r0 = (int64_t)blockIdx.x * NB;
  for (int e = tid; e < NB * NB; e += TS_THREADS) {
    const int i = e / NB, j = e % NB;
    T[i][j] = (r0 + i < n && j <= i) ? L[(r0 + i) * ldl + r0 + j] : (i == j ? 1.0 : 0.0);
    Zs[i][j] = 0.0;
  }
  __syncthreads();
  if (warp < 2 && lane < 16) {
    const int o = 16 * warp;
    const double rd = 1.0 / T[o + lane][o + lane];
    double z[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      double acc = i == lane ? 1.0 : 0.0;
#pragma unroll
      for (int t = 0; t < i; ++t) acc = fma(-T[o + i][o + t], z[t], acc);
      z[i] = acc * __shfl_sync(0xffffu, rd, i);
      if (i >= lane) Zs[o + i][o + lane] = z[i];
    }
  }
  __syncthreads();
  const int i = tid >> 4, j = tid & 15;
  double acc = 0.0;
#pragma unroll
  for (int t = 0; t < 16; ++t) acc = fma(T[16 + i][t], Zs[t][j], acc);
  Y[i][j] = acc;
  __syncthreads();
  acc = 0.0;
#pragma unroll
  for (int t = 0; t < 16; ++t) acc = fma(-Zs[16 + i][16 + t], Y[t][j], acc);
  Zs[16 + i][j] = acc;
  __syncthreads();
  for (int e = tid; e < NB * NB; e += TS_THREADS) Z[(int64_t)blockIdx.x * NB * NB + e] = Zs[e / NB][e % NB];
}

// Solves op(L) X = B in place: item (lk, ch) is block row lk (in the order of
// the solve) of the TW right-hand sides of chunk ch.  A CTA walks its items in
// ascending order, block rows first, so that every wait is for an earlier item
// of a co-resident CTA.  A thread keeps the partial sum of one row and one
// right-hand side over a share of the columns in a register until the row is
// done; the next block of L is loaded while the current one is used.
// Narrow chunks (4 right-hand sides, 8 above 64) because a step of the chain
// costs 32 x 32 x TW products on one SM's slow float64 pipe.  At a = 1,810 the
// solves of three frames (six with one right-hand side, two with about 50, which
// took two launches of 32) went from 8.9 to 1.5 ms: 0.16 ms each and 0.30 ms each.
template <int TW>
__global__ void __launch_bounds__(TS_THREADS) k_trsm_syncfree(const double* __restrict__ L, int64_t ldl, int64_t n,
                                                              const double* __restrict__ Z, double* B, int64_t ldb,
                                                              int64_t m, int64_t nch, bool transpose, int64_t bwb,
                                                              int* flags, int epoch, int* status,
                                                              long long spin_limit, int wait_xor) {
  constexpr int KS = 8 / TW;  // shares of the columns
  __shared__ double Ls[NB][NB + 1];
  __shared__ double Xs[NB][TW];
  __shared__ int bail;
  const int tid = threadIdx.x, ti = tid >> 3, tg = tid & 7;
  const int ks = tg % KS, j = tg / KS;
  const int64_t nblk = (n + NB - 1) / NB;
  if (tid == 0) bail = 0;
  __syncthreads();
  for (int64_t it = blockIdx.x; it < nblk * nch; it += gridDim.x) {
    const int64_t lk = it / nch, ch = it % nch;
    const int64_t r = transpose ? (nblk - 1 - lk) : lk, r0 = r * NB, c0 = ch * TW;
    const int rb = (int)((n - r0) < NB ? (n - r0) : NB);
    const int mc = (int)((m - c0) < TW ? (m - c0) : TW);
    // op(L)[r, cb]: thread (ti, tg) loads 4 entries, contiguous over tg
    double lv[4];
    auto load_l = [&](int64_t lc) {
      const int64_t cb = transpose ? (nblk - 1 - lc) : lc, cc0 = cb * NB;
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int t = tg + 8 * u;  // forward: L[r0 + ti, cc0 + t]; transposed: L[cc0 + ti, r0 + t]
        if (!transpose) lv[u] = (ti < rb && cc0 + t < n) ? L[(r0 + ti) * ldl + cc0 + t] : 0.0;
        else lv[u] = (cc0 + ti < n && t < rb) ? L[(cc0 + ti) * ldl + r0 + t] : 0.0;
      }
    };
    double acc = 0.0;
    int64_t lc = (lk - bwb) > 0 ? (lk - bwb) : 0;  // blocks outside the band are zero
    if (lc < lk) load_l(lc);
    for (; lc < lk; ++lc) {
      const int64_t cb = transpose ? (nblk - 1 - lc) : lc, cc0 = cb * NB;
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        if (!transpose) Ls[ti][tg + 8 * u] = lv[u];
        else Ls[tg + 8 * u][ti] = lv[u];
      }
      if (lc + 1 < lk) load_l(lc + 1);
      if (tid == 0) {
        long long spins = 0;
        while (ld_acquire(flags + ch * nblk + cb) != (epoch ^ wait_xor)) {
          if (++spins > spin_limit) {
            atomicOr(status, DEV_TIMEOUT);
            bail = 1;
            break;
          }
        }
      }
      __syncthreads();
      if (bail) return;
      if (tid < NB * TW) {
        const int t = tid / TW, q = tid % TW;
        Xs[t][q] = (cc0 + t < n && q < mc) ? __ldcg(B + (cc0 + t) * ldb + c0 + q) : 0.0;
      }
      __syncthreads();
#pragma unroll
      for (int q = 0; q < NB / KS; ++q) acc = fma(Ls[ti][ks + KS * q], Xs[ks + KS * q][j], acc);
      __syncthreads();
    }
    // x = D^{-1} (b - acc)
#pragma unroll
    for (int o = 1; o < KS; o <<= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    const double* Zr = Z + r * NB * NB;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const double z = Zr[ti * NB + tg + 8 * u];
      if (!transpose) Ls[ti][tg + 8 * u] = z;
      else Ls[tg + 8 * u][ti] = z;
    }
    if (ks == 0) Xs[ti][j] = (ti < rb && j < mc) ? __ldcg(B + (r0 + ti) * ldb + c0 + j) - acc : 0.0;
    __syncthreads();
    double x = 0.0;
#pragma unroll
    for (int q = 0; q < NB / KS; ++q) x = fma(Ls[ti][ks + KS * q], Xs[ks + KS * q][j], x);
#pragma unroll
    for (int o = 1; o < KS; o <<= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    if (ks == 0 && ti < rb && j < mc) B[(r0 + ti) * ldb + c0 + j] = x;
    __syncthreads();
    if (tid == 0) {
      __threadfence();  // cumulative: orders the block's stores (seen through the barrier) before the flag
      st_release(flags + ch * nblk + r, epoch);
    }
  }
}

// Inverses of the diagonal blocks of a factor, for the solves that follow.
static rbf_status diag_inverses(Ctx* c, const double* L, int64_t n, int64_t ldl, cudaStream_t s) {
  const int64_t nblk = (n + NB - 1) / NB;
  Buf& zb = c->scratch(99);
  RBF_TRY(zb.ensure((size_t)nblk * NB * NB * sizeof(double)));
  { k_diag_inv<<<(unsigned)nblk, TS_THREADS, 0, s>>>(L, ldl, n, zb.as<double>()); ::rbf::note_launch(); }
  RBF_CUDA(cudaGetLastError());
  return RBF_OK;
}

template <int TW>
static rbf_status trsm_launch(Ctx* c, const double* L, int64_t n, int64_t ldl, double* B, int64_t m, int64_t ldb,
                              bool transpose, cudaStream_t s, int64_t bw) {
  int64_t nblk = (n + NB - 1) / NB, nch = (m + TW - 1) / TW;
  const size_t fbytes = (size_t)(nblk * nch) * sizeof(int);
  if (c->sync_flags.bytes < fbytes) {
    RBF_TRY(c->sync_flags.ensure(fbytes));
    RBF_CUDA(cudaMemsetAsync(c->sync_flags.p, 0, c->sync_flags.bytes, s));
    c->epoch = 0;
  }
  static int max_blocks_dev[64] = {0};
  int& max_blocks = max_blocks_dev[c->device & 63];
  if (!max_blocks) {
    int per_sm = 0;
    RBF_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_trsm_syncfree<TW>, TS_THREADS, 0));
    max_blocks = per_sm * dense_sms(c->device);
  }
  int64_t grid = nblk * nch < max_blocks ? nblk * nch : max_blocks;
  if (grid < 1) return fail(RBF_ECUDA, "trsm: no co-resident blocks");
  const double* Z = c->scratch(99).as<double>();
  int* flags = c->sync_flags.as<int>();
  int* status = c->dflag.as<int>();
  int epoch = (int)(++c->epoch);
  int64_t bwb = bw >= n ? nblk : bw / NB + 2;
  long long lim = c->spin_limit > 0 ? c->spin_limit : TS_SPIN_LIMIT;
  int wx = c->wait_xor;
  void* args[] = {(void*)&L,   (void*)&ldl,       (void*)&n,   (void*)&Z,     (void*)&B,     (void*)&ldb,    (void*)&m,
                  (void*)&nch, (void*)&transpose, (void*)&bwb, (void*)&flags, (void*)&epoch, (void*)&status, (void*)&lim,
                  (void*)&wx};
  RBF_CUDA(cooperative_launch((const void*)k_trsm_syncfree<TW>, dim3((unsigned)grid), dim3(TS_THREADS), args, 0, s));
  return RBF_OK;
}

rbf_status trsm_lower(Ctx* c, const double* L, int64_t n, int64_t ldl, double* B, int64_t m,
                      int64_t ldb, bool transpose, cudaStream_t s, int64_t bw, bool have_inv) {
  if (n <= 0 || m <= 0) return RBF_OK;
  if (!have_inv) RBF_TRY(diag_inverses(c, L, n, ldl, s));
  if (m == 1) return trsm_launch<1>(c, L, n, ldl, B, m, ldb, transpose, s, bw);
  if (m <= 64) return trsm_launch<4>(c, L, n, ldl, B, m, ldb, transpose, s, bw);
  return trsm_launch<8>(c, L, n, ldl, B, m, ldb, transpose, s, bw);
}

// ---------------------------------------------------------------------------
// Inverse of a small SPD matrix (m <= SPD_SMALL_MAX) in one CTA by symmetric
// sweeps without pivoting (the pivots are the diagonals of successive Schur
// complements, positive for an SPD matrix): sweep k takes A_ij - A_ik A_jk / p
// off every entry, A_ik / p in column k and -1 / p at the pivot, and leaves
// -A^{-1} after the last.  Only the lower triangle is kept, rows i and m - 1 - i
// in one pass of m + 1 lanes: the float64 pipe of one SM bounds it (three
// inverses of orders up to 51: 255 -> 175 us).  In place, row-major m x m.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_spd_inverse_small(double* __restrict__ G, int m, int* __restrict__ flag) {
  extern __shared__ double gj[];  // A (m x (m + 1)), then the pivot column and its multiples
  const int ld = m + 1;
  double* A = gj;
  double* c = gj + (int64_t)m * ld;
  double* f = c + m;
  const int tid = threadIdx.x;
  for (int e = tid; e < m * m; e += blockDim.x) A[(e / m) * ld + e % m] = G[e];
  __syncthreads();
  for (int k = 0; k < m; ++k) {
    if (tid < m) {
      double p = A[k * ld + k];
      if (!(p > 0.0)) {
        if (tid == 0) atomicOr(flag, DEV_NOT_SPD);
        p = 1.0;
      }
      const double v = tid >= k ? A[tid * ld + k] : A[k * ld + tid], rp = 1.0 / p;
      c[tid] = v;
      f[tid] = tid == k ? -rp : v * rp;
    }
    __syncthreads();
    for (int r = tid >> 5; 2 * r < m; r += 8) {  // rows r and m - 1 - r
      const int rb = m - 1 - r;
      for (int q = tid & 31; q <= m; q += 32) {
        const int i = q <= r ? r : rb, j = q <= r ? q : q - (r + 1);
        if (q > r && (rb == r || j > rb)) break;  // the middle row of an odd m has no partner
        double v;
        if (i == k) v = f[j];
        else if (j == k) v = f[i];
        else v = fma(-f[i], c[j], A[i * ld + j]);
        A[i * ld + j] = v;
      }
    }
    __syncthreads();
  }
  for (int e = tid; e < m * m; e += blockDim.x) {
    const int i = e / m, j = e % m;
    G[e] = -(i >= j ? A[i * ld + j] : A[j * ld + i]);
  }
}

rbf_status spd_inverse_small(Ctx* c, double* G, int64_t m, cudaStream_t s) {
  if (m <= 0 || m > SPD_SMALL_MAX) return fail(RBF_EINVAL, "spd_inverse_small: m must be in [1, %d]", SPD_SMALL_MAX);
  size_t smem = (size_t)(m * (m + 1) + 2 * m) * sizeof(double);
  static bool attr[64] = {false};
  if (!attr[c->device & 63]) {
    size_t mx = (size_t)(SPD_SMALL_MAX * (SPD_SMALL_MAX + 1) + 2 * SPD_SMALL_MAX) * sizeof(double);
    RBF_CUDA(cudaFuncSetAttribute(k_spd_inverse_small, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)mx));
    attr[c->device & 63] = true;
  }
  { k_spd_inverse_small<<<1, 256, smem, s>>>(G, (int)m, c->dflag.as<int>()); ::rbf::note_launch(); }
  RBF_CUDA(cudaGetLastError());
  return RBF_OK;
}

// ---------------------------------------------------------------------------
// Small FP64 GEMM: C = alpha op(A) op(B) + beta C (row-major).
// ---------------------------------------------------------------------------
constexpr int GT = 32;
__global__ void __launch_bounds__(256) k_gemm_f64(bool ta, bool tb, int64_t m, int64_t n, int64_t k,
                                                  double alpha, const double* __restrict__ A,
                                                  int64_t lda, const double* __restrict__ B,
                                                  int64_t ldb, double beta, double* __restrict__ Cm,
                                                  int64_t ldc) {
  __shared__ double As[GT][GT + 1];
  __shared__ double Bs[GT][GT + 1];
  int64_t i0 = (int64_t)blockIdx.y * GT, j0 = (int64_t)blockIdx.x * GT;
  int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;  // 8 rows of threads, 4 outputs each
  double acc[4] = {0, 0, 0, 0};
  for (int64_t k0 = 0; k0 < k; k0 += GT) {
    for (int e = threadIdx.x; e < GT * GT; e += blockDim.x) {
      int r = e / GT, q = e % GT;
      int64_t ia = i0 + r, ka = k0 + q;
      double va = 0.0;
      if (ia < m && ka < k) va = ta ? A[ka * lda + ia] : A[ia * lda + ka];
      As[r][q] = va;
      int64_t kb = k0 + r, jb = j0 + q;
      double vb = 0.0;
      if (kb < k && jb < n) vb = tb ? B[jb * ldb + kb] : B[kb * ldb + jb];
      Bs[r][q] = vb;
    }
    __syncthreads();
#pragma unroll 8
    for (int t = 0; t < GT; ++t) {
      double b = Bs[t][tx];
#pragma unroll
      for (int u = 0; u < 4; ++u) acc[u] = fma(As[ty * 4 + u][t], b, acc[u]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    int64_t i = i0 + ty * 4 + u, j = j0 + tx;
    if (i < m && j < n) {
      double prev = beta != 0.0 ? Cm[i * ldc + j] : 0.0;
      Cm[i * ldc + j] = alpha * acc[u] + beta * prev;
    }
  }
}

// Partial products over a slice of k (split-K) for small outputs with long k.
__global__ void __launch_bounds__(256) k_gemm_splitk(bool ta, bool tb, int64_t m, int64_t n, int64_t k,
                                                     int64_t kchunk, const double* __restrict__ A,
                                                     int64_t lda, const double* __restrict__ B,
                                                     int64_t ldb, double* __restrict__ part) {
  int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= m * n) return;
  int64_t i = e / n, j = e % n;
  int64_t k0 = (int64_t)blockIdx.y * kchunk, k1 = k0 + kchunk < k ? k0 + kchunk : k;
  double acc = 0.0;
  for (int64_t t = k0; t < k1; ++t) {
    double a = ta ? A[t * lda + i] : A[i * lda + t];
    double b = tb ? B[j * ldb + t] : B[t * ldb + j];
    acc = fma(a, b, acc);
  }
  part[(int64_t)blockIdx.y * m * n + e] = acc;
}

__global__ void k_gemm_reduce(int64_t m, int64_t n, int nsplit, const double* __restrict__ part, double alpha,
                              double beta, double* __restrict__ Cm, int64_t ldc) {
  int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= m * n) return;
  double acc = 0.0;
  for (int q = 0; q < nsplit; ++q) acc += part[(int64_t)q * m * n + e];
  int64_t i = e / n, j = e % n;
  double prev = beta != 0.0 ? Cm[i * ldc + j] : 0.0;
  Cm[i * ldc + j] = alpha * acc + beta * prev;
}

rbf_status gemm_f64(Ctx* c, bool ta, bool tb, int64_t m, int64_t n, int64_t k, double alpha, const double* A,
                    int64_t lda, const double* B, int64_t ldb, double beta, double* Cm, int64_t ldc,
                    cudaStream_t s, int slot) {
  if (m <= 0 || n <= 0) return RBF_OK;
  int64_t tiles = ((m + GT - 1) / GT) * ((n + GT - 1) / GT);
  if (tiles < 64 && k > 512) {
    int64_t kchunk = 64;
    int64_t nsplit = (k + kchunk - 1) / kchunk;
    if (nsplit > 4096) {
      nsplit = 4096;
      kchunk = (k + nsplit - 1) / nsplit;
      nsplit = (k + kchunk - 1) / kchunk;
    }
    Buf& part = c->scratch(slot);
    RBF_TRY(part.ensure((size_t)nsplit * m * n * sizeof(double)));
    dim3 grid((unsigned)((m * n + 255) / 256), (unsigned)nsplit);
    { k_gemm_splitk<<<grid, 256, 0, s>>>(ta, tb, m, n, k, kchunk, A, lda, B, ldb, part.as<double>()); ::rbf::note_launch(); }
    RBF_CUDA(cudaGetLastError());
    { k_gemm_reduce<<<(unsigned)((m * n + 255) / 256), 256, 0, s>>>(m, n, (int)nsplit, part.as<double>(), alpha,
                                                                 beta, Cm, ldc); ::rbf::note_launch(); }
    RBF_CUDA(cudaGetLastError());
    return RBF_OK;
  }
  dim3 grid((unsigned)((n + GT - 1) / GT), (unsigned)((m + GT - 1) / GT));
  { k_gemm_f64<<<grid, 256, 0, s>>>(ta, tb, m, n, k, alpha, A, lda, B, ldb, beta, Cm, ldc); ::rbf::note_launch(); }
  RBF_CUDA(cudaGetLastError());
  return RBF_OK;
}

// r = b - H x for a symmetric H stored in full (one warp per row, its band only).
__global__ void __launch_bounds__(256) k_symv_residual(const double* __restrict__ H, int64_t n, int64_t ld, int64_t bw,
                                                       const double* __restrict__ x,
                                                       const double* __restrict__ b,
                                                       double* __restrict__ r) {
  after_previous();
  int lane = threadIdx.x & 31;
  int64_t row = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (row >= n) return;
  double acc = 0.0;
  const int64_t j1 = row + bw < n ? row + bw + 1 : n;
  for (int64_t j = (row > bw ? row - bw : 0) + lane; j < j1; j += 32) acc = fma(H[row * ld + j], x[j], acc);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
  if (lane == 0) r[row] = b[row] - acc;
}

rbf_status symv_residual(const double* H, int64_t n, int64_t ld, const double* x, const double* b,
                         double* r, cudaStream_t s, int64_t bw) {
  if (n <= 0) return RBF_OK;
  RBF_CUDA(launch_early(not_capturing(s), k_symv_residual, (unsigned)((n * 32 + 255) / 256), 256, 0, s, H, n, ld, bw, x, b, r));
  return RBF_OK;
}

}  // namespace rbf
