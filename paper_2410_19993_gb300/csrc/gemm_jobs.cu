// gemm_jobs.cu -- batched dense kernels of the cyclic-reduction factor and substitution on the
// CUDA cores: job-list GEMMs (FP32 or FP64) and Gauss-Jordan inversion of symmetric M-matrices.
//
// Every level of block cyclic reduction over the columns is a batch of independent dense M x M
// operations on different column blocks: inverses of the blocks it eliminates and products
// that form the couplings and Schur complements of the blocks it keeps.  A launch processes one
// list of such jobs; the host builds the lists once per factorization plan.
#include <math.h>

#include "common.cuh"
#include "kernels.h"

namespace xbar {

// ---------------------------------------------------------------------------------------------
// Job-list GEMM, TS x TS output tiles, 256 threads: thread (ty, tx) computes rows ty + 16 r and columns
// tx + 16 c (r, c < TS / 16); K is staged through shared memory in slabs of 16.
// ---------------------------------------------------------------------------------------------
constexpr int kGK = 16;

template <typename T, int TS>
__global__ void __launch_bounds__(256) gemm_jobs_kernel(const GemmJob<T>* __restrict__ jobs, int m, int n,
                                                        int tiles_n) {
  constexpr int CW = TS / 16;
  __shared__ T As[kGK][TS + 1];
  __shared__ T Bs[kGK][TS + 4];
  const GemmJob<T>& jb = jobs[blockIdx.y];
  const int i0 = (blockIdx.x / tiles_n) * TS, j0 = (blockIdx.x % tiles_n) * TS;
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  T acc[CW][CW];
#pragma unroll
  for (int r = 0; r < CW; ++r)
#pragma unroll
    for (int c = 0; c < CW; ++c) acc[r][c] = (T)0;

  // the K slabs of all segments in order; the next slab's values are loaded into registers while
  // the current one is multiplied
  T ra[CW], rb[CW];
  auto load = [&](int s, int k0) {
    const T* A = jb.A[s];
    const T* B = jb.B[s];
    const int lda = jb.lda[s], ldb = jb.ldb[s], K = jb.k[s], ta = jb.ta[s], tb = jb.tb[s];
#pragma unroll
    for (int u = 0; u < CW; ++u) {  // A slab: rows i0..i0+TS-1, k k0..k0+15
      const int t = tid + 256 * u;
      int i, kk;
      if (ta) { kk = t / TS; i = t % TS; }   // A[kk][i]: consecutive threads along i
      else { i = t >> 4; kk = t & 15; }      // A[i][kk]: consecutive threads along kk
      const int gi = i0 + i, gk = k0 + kk;
      ra[u] = (gi < m && gk < K) ? (ta ? A[(size_t)gk * lda + gi] : A[(size_t)gi * lda + gk]) : (T)0;
    }
#pragma unroll
    for (int u = 0; u < CW; ++u) {  // B slab: k k0..k0+15, columns j0..j0+TS-1
      const int t = tid + 256 * u;
      int j, kk;
      if (tb) { j = t >> 4; kk = t & 15; }       // B[j][kk]
      else { kk = t / TS; j = t % TS; }          // B[kk][j]
      const int gj = j0 + j, gk = k0 + kk;
      rb[u] = (gj < n && gk < K) ? (tb ? B[(size_t)gj * ldb + gk] : B[(size_t)gk * ldb + gj]) : (T)0;
    }
  };
  auto store = [&](int s) {
    const int ta = jb.ta[s], tb = jb.tb[s];
#pragma unroll
    for (int u = 0; u < CW; ++u) {
      const int t = tid + 256 * u;
      if (ta) As[t / TS][t % TS] = ra[u];
      else As[t & 15][t >> 4] = ra[u];
    }
#pragma unroll
    for (int u = 0; u < CW; ++u) {
      const int t = tid + 256 * u;
      if (tb) Bs[t & 15][t >> 4] = rb[u];
      else Bs[t / TS][t % TS] = rb[u];
    }
  };
  const int nseg = jb.nseg;
  int s = 0, k0 = 0;
  if (nseg > 0 && jb.k[0] > 0) load(0, 0);
  while (s < nseg) {
    const int cs = s;
    store(cs);
    __syncthreads();
    k0 += kGK;  // advance to the next slab and prefetch it
    if (k0 >= jb.k[s]) {
      k0 = 0;
      ++s;
    }
    if (s < nseg) load(s, k0);
#pragma unroll
    for (int kk = 0; kk < kGK; ++kk) {
      T a[CW], b[CW];
#pragma unroll
      for (int r = 0; r < CW; ++r) a[r] = As[kk][ty + 16 * r];
#pragma unroll
      for (int c = 0; c < CW; ++c) b[c] = Bs[kk][tx + 16 * c];
#pragma unroll
      for (int r = 0; r < CW; ++r)
#pragma unroll
        for (int c = 0; c < CW; ++c) acc[r][c] = fma(a[r], b[c], acc[r][c]);
    }
    __syncthreads();
  }
  const T alpha = jb.alpha;
#pragma unroll
  for (int r = 0; r < CW; ++r) {
    const int gi = i0 + ty + 16 * r;
    if (gi >= m) continue;
#pragma unroll
    for (int c = 0; c < CW; ++c) {
      const int gj = j0 + tx + 16 * c;
      if (gj >= n) continue;
      T v = alpha * acc[r][c];
      if (jb.Cin) v += jb.Cin[(size_t)gi * jb.ldcin + gj];
      jb.C[(size_t)gi * jb.ldc + gj] = v;
    }
  }
}

// Tile size: the largest of 64, 32 and 16 that neither pads the matrix by more than the next smaller one
// would nor leaves fewer than two blocks per SM.  A block's time is its multiply-adds per thread times
// the K depth (an FP64 multiply-add of the block's eight warps takes 152 cycles), so a level of few small
// jobs wants many blocks: the 32 x 32 FP64 blocks of a 256 x 32 map took 54 us a launch in one 64 x 64
// tile each and take 9 us in 16 x 16 tiles; a level with hundreds of tiles loses nothing.
template <typename T>
cudaError_t launch_gemm_jobs(const GemmJob<T>* jobs_dev, int njobs, int m, int n, int nsm, cudaStream_t st) {
  if (njobs <= 0 || m <= 0 || n <= 0) return cudaSuccess;
  if (njobs > 65535) return cudaErrorInvalidValue;
  auto tiles = [](int x, int ts) { return (x + ts - 1) / ts; };
  int ts = 64;
  while (ts > 16) {
    const int h = ts / 2;
    const bool pads = tiles(m, ts) * ts > tiles(m, h) * h || tiles(n, ts) * ts > tiles(n, h) * h;
    if (!pads && (long long)njobs * tiles(m, ts) * tiles(n, ts) >= 2 * nsm) break;
    ts = h;
  }
  const int tm = tiles(m, ts), tn = tiles(n, ts);
  const dim3 grid(tm * tn, njobs);
  if (ts == 16) gemm_jobs_kernel<T, 16><<<grid, 256, 0, st>>>(jobs_dev, m, n, tn);
  else if (ts == 32) gemm_jobs_kernel<T, 32><<<grid, 256, 0, st>>>(jobs_dev, m, n, tn);
  else gemm_jobs_kernel<T, 64><<<grid, 256, 0, st>>>(jobs_dev, m, n, tn);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------------------------
// Job-list matrix-vector products: NV (1, 2, 4, 8 or 16) columns, tb = 0, ldb = ldc = ldcin = NV.  Bound
// by reading each block of the factor once, so a block of 256 threads takes 16 rows of a product and
// keeps many loads in flight: a warp reads two rows along K (ta = 0; the lanes' partial sums meet at the
// end) or, transposed, two values of K for 16 columns.  The vectors go through shared memory.
// One vector of a 256 x 256 map: 77 us a launch as a product padded to 16 columns in 64-row tiles.
// ---------------------------------------------------------------------------------------------
constexpr int kVR = 16;    // rows of the result per block
constexpr int kVK = 128;   // K values per staged chunk

// sums of NS values over the 32 lanes; afterwards lane l holds, in v[0], the sum of value l / (32 / NS')
// with NS' = NS rounded up to a power of two (NS <= 32)
template <typename T, int NS>
__device__ __forceinline__ void lane_sums(T (&v)[NS], int lane) {
  int n = NS;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    if (n > 1) {
      const bool up = (lane & o) != 0;
#pragma unroll
      for (int k = 0; k < NS / 2; ++k)
        if (k < n / 2) {
          const T send = up ? v[k] : v[k + n / 2], keep = up ? v[k + n / 2] : v[k];
          v[k] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
      n >>= 1;
    } else {
      v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
    }
  }
}

template <typename T, int NV>
__global__ void __launch_bounds__(256) gemv_jobs_kernel(const GemmJob<T>* __restrict__ jobs, int m) {
  __shared__ T bs[kVK][NV];
  __shared__ T red0[kVR][NV];
  __shared__ T red1[8][kVR][NV];
  const GemmJob<T>& jb = jobs[blockIdx.y];
  const int i0 = blockIdx.x * kVR;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int ia = i0 + 2 * warp;                           // ta = 0: this warp's two rows
  const int it = i0 + (lane & 15), kt = 2 * warp + (lane >> 4);  // ta = 1: column, first K value
  T acc0[2 * NV], acc1[NV];
#pragma unroll
  for (int v = 0; v < 2 * NV; ++v) acc0[v] = (T)0;
#pragma unroll
  for (int v = 0; v < NV; ++v) acc1[v] = (T)0;
  const int nseg = jb.nseg;
  for (int s = 0; s < nseg; ++s) {
    const T* A = jb.A[s];
    const T* B = jb.B[s];
    const int lda = jb.lda[s], K = jb.k[s], ta = jb.ta[s];
    for (int k0 = 0; k0 < K; k0 += kVK) {
      const int kc = min(kVK, K - k0);
      __syncthreads();
      for (int t = tid; t < kVK * NV; t += 256)
        (&bs[0][0])[t] = t < kc * NV ? B[(size_t)k0 * NV + t] : (T)0;
      // this chunk's part of A, loaded before the barrier
      T a[8];
      if (!ta) {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int k = lane + 32 * u;
          a[u] = (ia < m && k < kc) ? A[(size_t)ia * lda + k0 + k] : (T)0;
          a[4 + u] = (ia + 1 < m && k < kc) ? A[(size_t)(ia + 1) * lda + k0 + k] : (T)0;
        }
      } else {
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const int k = kt + 16 * u;
          a[u] = (it < m && k < kc) ? A[(size_t)(k0 + k) * lda + it] : (T)0;
        }
      }
      __syncthreads();
      if (!ta) {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          if (32 * u >= kc) break;  // uniform
#pragma unroll
          for (int v = 0; v < NV; ++v) {
            const T b = bs[lane + 32 * u][v];
            acc0[v] = fma(a[u], b, acc0[v]);
            acc0[NV + v] = fma(a[4 + u], b, acc0[NV + v]);
          }
        }
      } else {
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          if (16 * u >= kc) break;  // uniform
#pragma unroll
          for (int v = 0; v < NV; ++v) acc1[v] = fma(a[u], bs[kt + 16 * u][v], acc1[v]);
        }
      }
    }
  }
  lane_sums<T, 2 * NV>(acc0, lane);
  {
    constexpr int rep = 32 / (2 * NV);
    const int k = lane / rep;
    if (lane % rep == 0) red0[2 * warp + k / NV][k % NV] = acc0[0];
  }
#pragma unroll
  for (int v = 0; v < NV; ++v) acc1[v] += __shfl_xor_sync(0xffffffffu, acc1[v], 16);
  if (lane < 16)
#pragma unroll
    for (int v = 0; v < NV; ++v) red1[warp][lane][v] = acc1[v];
  __syncthreads();
  for (int t = tid; t < kVR * NV; t += 256) {
    const int r = t / NV, v = t % NV, i = i0 + r;
    if (i >= m) continue;
    T x = red0[r][v];
#pragma unroll
    for (int w = 0; w < 8; ++w) x += red1[w][r][v];
    x *= jb.alpha;
    if (jb.Cin) x += jb.Cin[(size_t)i * NV + v];
    jb.C[(size_t)i * NV + v] = x;
  }
}

template <typename T>
cudaError_t launch_gemv_jobs(const GemmJob<T>* jobs_dev, int njobs, int m, int nv, cudaStream_t st) {
  if (njobs <= 0 || m <= 0) return cudaSuccess;
  if (njobs > 65535) return cudaErrorInvalidValue;
  const dim3 grid((m + kVR - 1) / kVR, njobs);
  switch (nv) {
    case 1: gemv_jobs_kernel<T, 1><<<grid, 256, 0, st>>>(jobs_dev, m); break;
    case 2: gemv_jobs_kernel<T, 2><<<grid, 256, 0, st>>>(jobs_dev, m); break;
    case 4: gemv_jobs_kernel<T, 4><<<grid, 256, 0, st>>>(jobs_dev, m); break;
    case 8: gemv_jobs_kernel<T, 8><<<grid, 256, 0, st>>>(jobs_dev, m); break;
    case 16: gemv_jobs_kernel<T, 16><<<grid, 256, 0, st>>>(jobs_dev, m); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------------------------
// Gauss-Jordan inversion in registers, eliminating panels of 8 pivots at a time.  The matrix
// (padded with the identity to NT x NT) is held by 32 NT / RPT threads: thread (ty, tx) owns rows
// ty + (NT/RPT) r (r < RPT) and columns tx + 32 c (c < NT/32).  For the panel of pivots P..P+7, with
// D = A[P:P+8, P:P+8], panel rows R = A[P:P+8, :] and panel columns C = A[:, P:P+8]:
//     R' = D^-1 R outside the pivot columns and D^-1 inside them,
//     A[i, :] <- A[i, :] - C[i, :] R' outside the pivot columns and -C[i, :] D^-1 inside them
// for the rows i outside the panel, which is the product of the 8 single-pivot sweep operators;
// after all panels the inverse is in place.  No pivoting: the matrices are symmetric M-matrices
// (positive definite), so every pivot is positive.  The owners publish R and C to shared memory,
// one warp forms R' there (8 dependent sweep steps on 8 rows), and every thread applies the rank-8
// update to its own elements; the shared buffers alternate between panels, so each panel costs
// two block barriers.  All register indices are compile-time constants (the panel loop is unrolled).
// ---------------------------------------------------------------------------------------------
template <typename T, int NT, int RPT>
__global__ void __launch_bounds__(NT / RPT * 32) gj_kernel(const GjJob<T>* __restrict__ jobs, int n) {
  constexpr int RG = NT / RPT;  // row groups = warps
  constexpr int CB = NT / 32;   // columns per lane
  constexpr int PW = 8;        // pivots per panel
  __shared__ __align__(16) T PR[2][PW][NT];   // panel rows, then R'
  __shared__ __align__(16) T PC[2][NT][PW];   // panel columns
  const GjJob<T> jb = jobs[blockIdx.x];
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  T a[RPT][CB];
#pragma unroll
  for (int r = 0; r < RPT; ++r) {
    const int i = ty + RG * r;
#pragma unroll
    for (int c = 0; c < CB; ++c) {
      const int mm = tx + 32 * c;
      a[r][c] = (i < n && mm < n) ? jb.src[(size_t)i * jb.lds + mm] : (i == mm ? (T)1 : (T)0);
    }
  }
  // the panel loop is not unrolled (code size): registers of a runtime row or column index are
  // picked by short compare chains
#pragma unroll 1
  for (int pn = 0; pn < NT / PW; ++pn) {
    const int P0 = pn * PW;
    if (P0 >= n) break;  // uniform: identity padding needs no steps
    const int b = pn & 1;
    // (1) publish the panel rows and columns
#pragma unroll
    for (int k = 0; k < PW; ++k) {
      const int row = P0 + k;
      if (ty == row % RG) {
        const int rk = row / RG;
#pragma unroll
        for (int c = 0; c < CB; ++c) {
          T v = a[0][c];
#pragma unroll
          for (int r = 1; r < RPT; ++r)
            if (r == rk) v = a[r][c];
          PR[b][k][tx + 32 * c] = v;
        }
      }
    }
    {
      const int ck = P0 / 32;  // the 8 panel columns lie in one 32-column block
      const int k = tx - (P0 & 31);
      if (k >= 0 && k < PW) {
#pragma unroll
        for (int r = 0; r < RPT; ++r) {
          T v = a[r][0];
#pragma unroll
          for (int c = 1; c < CB; ++c)
            if (c == ck) v = a[r][c];
          PC[b][ty + RG * r][k] = v;
        }
      }
    }
    __syncthreads();
    // (2) one warp: R' = D^-1 R (8 sweep steps on the panel rows, two at a time, in registers; lane l holds
    // columns l + 32 c of the 8 rows, the pivot column's values come by shuffle from its lane)
    if (ty == 0) {
      T pr[PW][CB];
#pragma unroll
      for (int k = 0; k < PW; ++k)
#pragma unroll
        for (int c = 0; c < CB; ++c) pr[k][c] = PR[b][k][tx + 32 * c];
      const int ck = P0 / 32, src = P0 & 31;
#pragma unroll
      for (int k = 0; k < PW; k += 2) {  // two pivots at a time: one round of shuffles
        T f0[PW], f1[PW];  // columns P0 + k, P0 + k + 1 of the 8 rows (lanes src + k, + 1, slot ck)
#pragma unroll
        for (int l = 0; l < PW; ++l) {
          T v = pr[l][0];
#pragma unroll
          for (int c = 1; c < CB; ++c)
            if (c == ck) v = pr[l][c];
          f0[l] = __shfl_sync(0xffffffffu, v, src + k);
          f1[l] = __shfl_sync(0xffffffffu, v, src + k + 1);
        }
        const T p00 = f0[k], p01 = f1[k], p10 = f0[k + 1], p11 = f1[k + 1];
        // each pivot with its own reciprocal, the second one that of the Schur complement: solving for both rows
        // by the 2 x 2 determinant rounds once more and errs by 3.9e-8 instead of 1.7e-8 (64 rows)
        const T i0 = (T)1 / p00, t = p01 * i0, i1 = (T)1 / fma(-p10, t, p11);
#pragma unroll
        for (int c = 0; c < CB; ++c) {
          const bool in0 = (tx == src + k) && (c == ck), in1 = (tx == src + k + 1) && (c == ck);
          const T r0 = in0 ? (T)1 : in1 ? (T)0 : pr[k][c], r1 = in1 ? (T)1 : in0 ? (T)0 : pr[k + 1][c];
          const T h0 = r0 * i0, g1 = fma(-p10, h0, r1) * i1, g0 = fma(-t, g1, h0);
#pragma unroll
          for (int l = 0; l < PW; ++l) {
            if (l == k || l == k + 1) continue;
            pr[l][c] = fma(-f1[l], g1, fma(-f0[l], g0, in0 || in1 ? (T)0 : pr[l][c]));
          }
          pr[k][c] = g0;
          pr[k + 1][c] = g1;
        }
      }
#pragma unroll
      for (int k = 0; k < PW; ++k)
#pragma unroll
        for (int c = 0; c < CB; ++c) PR[b][k][tx + 32 * c] = pr[k][c];
    }
    __syncthreads();
    // (3) every thread: rank-8 update of its elements; R' of its columns is read once per panel, the
    // panel-column values C[i, :] once per row (a shared-memory broadcast: i is uniform in a warp)
    T rp[PW][CB];
#pragma unroll
    for (int k = 0; k < PW; ++k)
#pragma unroll
      for (int c = 0; c < CB; ++c) rp[k][c] = PR[b][k][tx + 32 * c];
#pragma unroll
    for (int r = 0; r < RPT; ++r) {
      const int i = ty + RG * r;
      if (i >= P0 && i < P0 + PW) {  // panel row: R'
        const int k = i - P0;
#pragma unroll
        for (int c = 0; c < CB; ++c) {
          T v = rp[0][c];
#pragma unroll
          for (int kk = 1; kk < PW; ++kk)
            if (kk == k) v = rp[kk][c];
          a[r][c] = v;
        }
        continue;
      }
      T cr[PW];
#pragma unroll
      for (int k = 0; k < PW; ++k) cr[k] = PC[b][i][k];
#pragma unroll
      for (int c = 0; c < CB; ++c) {
        const int mm = tx + 32 * c;
        T v = (mm >= P0 && mm < P0 + PW) ? (T)0 : a[r][c];
#pragma unroll
        for (int k = 0; k < PW; ++k) v = fma(-cr[k], rp[k][c], v);
        a[r][c] = v;
      }
    }
  }
#pragma unroll
  for (int r = 0; r < RPT; ++r) {
    const int i = ty + RG * r;
    if (i >= n) continue;
#pragma unroll
    for (int c = 0; c < CB; ++c) {
      const int mm = tx + 32 * c;
      if (mm < n) jb.dst[(size_t)i * jb.ldd + mm] = a[r][c];
    }
  }
}

// Single-pivot variant for FP64 (its register budget does not allow the panel form at 128 rows).  Thread
// (ty, tx) owns rows ty + (NT/8) r (r < 8) and columns tx + 32 c (c < NT/32); each step applies one
// sweep operator (a_qq <- 1/a_qq, a_qm <- a_qm/a_qq, a_iq <- -a_iq/a_qq, a_im <- a_im - a_iq a_qm/a_qq) with
// the pivot row and column published through double-buffered shared memory (one barrier per step).
// Bound by FP64 issue (64 cycles an instruction and sub-partition), so a step issues as few as it can:
// the short reciprocal, one product per column (the pivot column takes the reciprocal itself and a
// zero to add to, so that it needs none of its own) and one multiply-add per element.
template <int NT>
__global__ void __launch_bounds__(NT * 4) gj1_kernel(const GjJob<double>* __restrict__ jobs, int n) {
  constexpr int RG = NT / 8;   // row groups = warps
  constexpr int CB = NT / 32;  // columns per lane
  __shared__ double prow[2][NT], pcol[2][NT];
  const GjJob<double> jb = jobs[blockIdx.x];
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  double a[8][CB];
#pragma unroll
  for (int r = 0; r < 8; ++r) {
    const int i = ty + RG * r;
#pragma unroll
    for (int c = 0; c < CB; ++c) {
      const int mm = tx + 32 * c;
      a[r][c] = (i < n && mm < n) ? jb.src[(size_t)i * jb.lds + mm] : (i == mm ? 1.0 : 0.0);
    }
  }
#pragma unroll
  for (int aq = 0; aq < 8; ++aq) {
    for (int rq = 0; rq < RG; ++rq) {
      const int q = rq + RG * aq;
      if (q >= n) break;  // uniform: identity padding needs no steps
      const int buf = q & 1, cq = q & 31, bq = q >> 5;
      if (ty == rq) {
#pragma unroll
        for (int c = 0; c < CB; ++c) prow[buf][tx + 32 * c] = a[aq][c];
      }
      if (tx == cq) {
#pragma unroll
        for (int r = 0; r < 8; ++r) {
          double v = a[r][0];
#pragma unroll
          for (int c = 1; c < CB; ++c)
            if (c == bq) v = a[r][c];
          pcol[buf][ty + RG * r] = v;
        }
      }
      __syncthreads();
      const double inv = pivot_rcp(prow[buf][q]);
      double f[CB], cs[8];
#pragma unroll
      for (int c = 0; c < CB; ++c) f[c] = tx == cq && c == bq ? inv : prow[buf][tx + 32 * c] * inv;
#pragma unroll
      for (int r = 0; r < 8; ++r) cs[r] = pcol[buf][ty + RG * r];
#pragma unroll
      for (int r = 0; r < 8; ++r)
#pragma unroll
        for (int c = 0; c < CB; ++c) a[r][c] = fma(-cs[r], f[c], tx == cq && c == bq ? 0.0 : a[r][c]);
      if (ty == rq) {  // pivot row
#pragma unroll
        for (int c = 0; c < CB; ++c) a[aq][c] = f[c];
      }
    }
  }
#pragma unroll
  for (int r = 0; r < 8; ++r) {
    const int i = ty + RG * r;
    if (i >= n) continue;
#pragma unroll
    for (int c = 0; c < CB; ++c) {
      const int mm = tx + 32 * c;
      if (mm < n) jb.dst[(size_t)i * jb.ldd + mm] = a[r][c];
    }
  }
}

template <typename T>
cudaError_t launch_gj_inverse(const GjJob<T>* jobs_dev, int njobs, int n, unsigned* status, cudaStream_t st) {
  (void)status;
  if (njobs <= 0 || n <= 0) return cudaSuccess;
  if constexpr (sizeof(T) == 8) {  // FP64: single-pivot steps
    if (n <= 32) gj1_kernel<32><<<njobs, 128, 0, st>>>(jobs_dev, n);
    else if (n <= 64) gj1_kernel<64><<<njobs, 256, 0, st>>>(jobs_dev, n);
    else if (n <= 128) gj1_kernel<128><<<njobs, 512, 0, st>>>(jobs_dev, n);
    else return cudaErrorInvalidValue;
  } else {
    if (n <= 32) gj_kernel<T, 32, 8><<<njobs, 128, 0, st>>>(jobs_dev, n);
    else if (n <= 64) gj_kernel<T, 64, 8><<<njobs, 256, 0, st>>>(jobs_dev, n);
    else if (n <= 128) gj_kernel<T, 128, 8><<<njobs, 512, 0, st>>>(jobs_dev, n);
    else return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

template cudaError_t launch_gemm_jobs<float>(const GemmJob<float>*, int, int, int, int, cudaStream_t);
template cudaError_t launch_gemm_jobs<double>(const GemmJob<double>*, int, int, int, int, cudaStream_t);
template cudaError_t launch_gemv_jobs<float>(const GemmJob<float>*, int, int, int, cudaStream_t);
template cudaError_t launch_gemv_jobs<double>(const GemmJob<double>*, int, int, int, cudaStream_t);
template cudaError_t launch_gj_inverse<float>(const GjJob<float>*, int, int, unsigned*, cudaStream_t);
template cudaError_t launch_gj_inverse<double>(const GjJob<double>*, int, int, unsigned*, cudaStream_t);

}  // namespace xbar
