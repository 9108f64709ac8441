// factor64.cu -- FP64 block Thomas factorization of the word-line system, eliminated from both ends
// (Sec. II-C: one decomposition per conductance map).
//
// The word-line system is block tridiagonal over the N columns (assemble.cu: dense M x M blocks C_j,
// couplings -g_w I).  Its elimination runs as two independent chains that meet in column m:
//     left   Z_0 = C_0,          Z_j = C_j - g_w^2 X_{j-1}                 j = 1 .. m-1
//     right  Z_{N-1} = C_{N-1},  Z_j = C_j - g_w^2 X_{j+1}                 j = N-2 .. m+1
//     meet   Z_m = C_m - g_w^2 X_{m-1} - g_w^2 X_{m+1},                     X_j = Z_j^{-1},
// which halves the sequential depth of the one-ended chain for the same work.  Diagonals are formed
// without subtraction from the grounded row sums
//     sigma_j = h_j + [j = 0] g_s + g_w X_prev sigma_prev (+ the same from the right in column m),
//     Z_ii = sigma_i + g_w [a neighbour remains] + sum_{k != i} |Z_ik|
// (the GTH idea for M-matrices; all terms >= 0).
//
// What bounds it.  An FP64 instruction takes 64 cycles of an SM sub-partition whatever the number of
// active lanes, a dependent chain advances one operation per 64 cycles, and a scalar pivot of the
// inversion is such a chain (reciprocal, scale, update: ~450 cycles).  So the M pivots of every
// column are the critical path, and everything else is moved off it:
//   * per chain one block (the pivot block's) does nothing but invert 16 x 16 pivot blocks: from the
//     not yet updated rows of the next panel and the inverse it has just computed it forms the next
//     pivot block itself, so it never waits for a row update (one panel of look-ahead);
//   * the rows are spread over Mp / R worker blocks, R rows each, one thread per column with the R
//     values in registers; a worker applies panel q (row - (row[P] D^-1) R_P) when D_q^-1 arrives and
//     publishes the rows the others need next.  Panel rows go from L2 straight to the registers of
//     the thread that owns the column.
// Exchange is through L2 with monotonic counters (release / acquire at device scope) instead of
// block barriers; every wait is bounded.  Slots alternate with the parity of the column step: a slot
// is rewritten two steps later, when every worker, each of which owns rows of some panel, has
// published rows of the step between and therefore has read it.
//
// Measured against the previous kernel (one chain, a group barrier per panel and every block
// inverting the pivot block): 16 x 16 284 -> 60 us, 64 x 64 3.50 -> 1.14 ms, 256 x 256 61.7 -> 17.0 ms
// (the FP64 work alone is 7.2 ms).  A panel takes 17-18k cycles: 10.5k for the 16 pivots, 3.4-4.2k for the
// next pivot block's two products, the rest waiting for its rows; at 256 rows the workers' update
// (9k) and their waits are as long.
#include <math.h>

#include "common.cuh"
#include "kernels.h"

namespace xbar {

namespace {

constexpr int kPB = 16;  // pivots per panel

// counters in global memory, one 32-byte sector each
constexpr int kFlagStride = 8;
constexpr int kMaxPanels = 64;
constexpr int kFlagAbort = 0, kFlagDone = kFlagStride, kFlagChain = 2 * kFlagStride;
constexpr int kChainFlags = (1 + 2 * kMaxPanels) * kFlagStride;  // D, then R[q], then S[q]
constexpr int kFlagWords = kFlagChain + 2 * kChainFlags;

__device__ __forceinline__ unsigned ld_acquire(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
// release at device scope: the writes of the block's threads before the barrier that precedes the call
// are visible to whoever acquires the new value
__device__ __forceinline__ void add_release(unsigned* p) {
  asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(p) : "memory");
}

// bounded wait until *f >= target (one thread); false when it expires or another block gave up
__device__ __forceinline__ bool wait_count(const unsigned* f, unsigned target, unsigned* flags, unsigned* status,
                                           uint64_t limit) {
  if ((int)(ld_acquire(f) - target) >= 0) return true;
  const uint64_t t0 = globaltimer_ns();
  while ((int)(ld_acquire(f) - target) < 0) {
    if (globaltimer_ns() - t0 > limit) {
      set_status(status, XBAR_DEV_TIMEOUT);
      atomicExch(flags + kFlagAbort, 1u);
      return false;
    }
    if (*reinterpret_cast<volatile unsigned*>(flags + kFlagAbort)) return false;
  }
  return true;
}

// named barriers of the inversion: warps 0 .. 4
template <int ID>
__device__ __forceinline__ void bar5_sync() { asm volatile("bar.sync %0, 160;" ::"n"(ID) : "memory"); }
template <int ID>
__device__ __forceinline__ void bar5_arrive() { asm volatile("bar.arrive %0, 160;" ::"n"(ID) : "memory"); }
constexpr int kBarRow = 1, kBarInv = 3, kBarAll = 5;  // the first two by the parity of the pivot

template <int MP>
struct GjShared {
  double row[2][MP], diag[2], inv[2];
};

// In-place Gauss-Jordan inversion of a symmetric positive definite MP x MP matrix, no pivoting, by five
// warps.  Lanes of warps 0 .. 3 hold column `col` of rows r0 .. r0 + RW - 1 and apply the pivots; warp 4
// computes the reciprocals: the next pivot is  d_{q+1,q+1} - a_{q,q+1}^2 / pv_q,  so it needs pivot
// row q and that diagonal entry only and runs beside the update by pivot q.  Only the pivot row
// is exchanged (shared memory): the swept part of the matrix is antisymmetric to the rest, so
// column q is the pivot row with the sign of the rows already swept turned.  16 x 16: 13.2k cycles
// with every warp forming the reciprocal itself (a barrier, reciprocal and update in turn).
template <int MP, int RW>
__device__ __forceinline__ void gj_invert(double (&d)[RW], int r0, int col, int warp, GjShared<MP>& sh) {
  if (warp == 4) {
    bar5_sync<kBarRow>();
    double inv = pivot_rcp(sh.row[0][0]);
    sh.inv[0] = inv;  // every lane the same value
    bar5_arrive<kBarInv>();
#pragma unroll
    for (int q = 0; q < MP - 1; ++q) {
      const double rc = sh.row[q & 1][q + 1];
      inv = pivot_rcp(fma(-(rc * rc), inv, sh.diag[q & 1]));
      sh.inv[(q + 1) & 1] = inv;
      if (q & 1) {
        bar5_arrive<kBarInv>();
        bar5_sync<kBarRow>();
      } else {
        bar5_arrive<kBarInv + 1>();
        bar5_sync<kBarRow + 1>();
      }
    }
    return;
  }
  if (r0 == 0) sh.row[0][col] = d[0];
#pragma unroll
  for (int r = 0; r < RW; ++r)
    if (r0 + r == 1 && col == 1) sh.diag[0] = d[r];
#pragma unroll
  for (int q = 0; q < MP; ++q) {
    const int b = q & 1;
    if (b) bar5_sync<kBarRow + 1>();
    else bar5_sync<kBarRow>();
    const double rc = sh.row[b][col];
    double cq[RW];
#pragma unroll
    for (int r = 0; r < RW; ++r) cq[r] = sh.row[b][r0 + r];
    if (b) bar5_sync<kBarInv + 1>();
    else bar5_sync<kBarInv>();
    const double inv = sh.inv[b];
    const bool incol = col == q;
    const double f = incol ? inv : rc * inv;  // row q after the sweep
#pragma unroll
    for (int r = 0; r < RW; ++r) {
      const double c = r0 + r < q ? cq[r] : -cq[r];
      const double v = fma(c, f, incol ? 0.0 : d[r]);
      d[r] = r0 + r == q ? f : v;
    }
    if (q + 1 < MP) {
#pragma unroll
      for (int r = 0; r < RW; ++r) {
        if (r0 + r == q + 1) sh.row[b ^ 1][col] = d[r];
        if (r0 + r == q + 2 && col == q + 2) sh.diag[b ^ 1] = d[r];
      }
    }
  }
}

// sums of NV values over the W consecutive lanes of a group (W a power of two >= NV); afterwards a
// lane holds, in v[0], the sum of value  (lane % W) / (W / NV)
template <int NV, int W>
__device__ __forceinline__ void group_sums(double (&v)[NV], int lane) {
  int n = NV;
#pragma unroll
  for (int o = W / 2; o > 0; o >>= 1) {
    if (n > 1) {
      const bool up = (lane & o) != 0;
#pragma unroll
      for (int k = 0; k < NV / 2; ++k)
        if (k < n / 2) {
          const double send = up ? v[k] : v[k + n / 2], keep = up ? v[k + n / 2] : v[k];
          v[k] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
      n >>= 1;
    } else {
      v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
    }
  }
}

// column of step s of a chain
__device__ __forceinline__ int chain_col(int chain, int s, int N) { return chain == 0 ? s : N - 1 - s; }

}  // namespace

// ---- blocks of 16 rows: one block of five warps per chain, the matrix in registers -----------------
__global__ void __launch_bounds__(160) factor64_small_kernel(Factor64Params p) {
  constexpr int MP = kPB, RW = 2;
  const int chain = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int col = lane & 15, r0 = warp * 4 + (lane >> 4) * 2;
  const bool holds = warp < 4;  // warp 4 only computes the pivots' reciprocals
  const int M = p.M, N = p.N, m = p.meet;
  const int nsteps = chain == 0 ? m + 1 : N - 1 - m;
  const bool right = m < N - 1;
  const double gw = p.gw, gw2 = gw * gw;
  const uint64_t limit = wait_limit(p.status);
  __shared__ GjShared<MP> gj;
  __shared__ double sig[2][MP], offs[MP], sgs[MP], diag[MP];
  double* gsig = p.buf;  // sigma of the right chain's last column
  double a[RW], c[RW];
#pragma unroll
  for (int r = 0; r < RW; ++r) a[r] = 0.0;
  double h = 0.0;  // thread i: h of row i
  auto load_c = [&](int s) {
    const int j = chain_col(chain, s, N);
    if (holds) {
      const double* C = p.Coff + ((size_t)j * MP + r0) * MP + col;
#pragma unroll
      for (int r = 0; r < RW; ++r) c[r] = C[r * MP];
    }
    if (tid < M) h = p.h[(size_t)j * MP + tid] + (j == 0 ? p.gsrc : 0.0);
  };
  load_c(0);
  for (int s = 0; s < nsteps; ++s) {
    const int j = chain_col(chain, s, N);
    const bool meet = chain == 0 && s == m;
    if (meet && right) {
      const bool ok = tid != 0 || wait_count(p.flags + kFlagDone, 1u, p.flags, p.status, limit);
      if (!__syncthreads_and(ok)) return;
    }
    if (holds) {
      // Z_j without its diagonal; per row the sums of |Z_ik| and of X_prev sigma_prev
      const double sk = s > 0 ? sig[(s - 1) & 1][col] : 0.0;
      double v[2 * RW];
#pragma unroll
      for (int r = 0; r < RW; ++r) {
        const int i = r0 + r;
        const bool off = i < M && col < M && i != col;
        double z = fma(-gw2, a[r], c[r]), sg = a[r] * sk;
        if (meet && right) {
          const double x = __ldcg(p.X + ((size_t)(m + 1) * MP + i) * MP + col);
          z = fma(-gw2, x, z);
          sg = fma(x, __ldcg(gsig + col), sg);
        }
        a[r] = off ? z : 0.0;
        v[r] = fabs(a[r]);
        v[RW + r] = sg;
      }
      constexpr int rep = MP / (2 * RW);
      group_sums<2 * RW, MP>(v, lane);
      const int k = (lane & (MP - 1)) / rep;
      if ((lane & (rep - 1)) == 0) {
        if (k < RW) offs[r0 + k] = v[0];
        else sgs[r0 + k - RW] = v[0];
      }
    }
    __syncthreads();
    if (tid < MP) {
      const bool real = tid < M;
      const double sg = real ? fma(gw, sgs[tid], h) : 0.0;
      sig[s & 1][tid] = sg;
      diag[tid] = real ? sg + (meet ? 0.0 : gw) + offs[tid] : 1.0;
    }
    __syncthreads();
    if (holds)
#pragma unroll
      for (int r = 0; r < RW; ++r)
        if (r0 + r == col) a[r] = diag[col];
    if (s + 1 < nsteps) load_c(s + 1);  // in flight during the inversion
    gj_invert<MP, RW>(a, r0, col, warp, gj);
    if (holds) {
      double* Xo = p.X + ((size_t)j * MP + r0) * MP + col;
#pragma unroll
      for (int r = 0; r < RW; ++r) Xo[r * MP] = a[r];
    }
  }
  if (chain == 1) {
    if (tid < MP) gsig[tid] = sig[(nsteps - 1) & 1][tid];
    __syncthreads();
    if (tid == 0) add_release(p.flags + kFlagDone);
  }
}

// ---- larger blocks -----------------------------------------------------------------------------------
namespace {

// per-chain scratch in global memory (doubles)
struct ChainBuf {
  double *R, *S, *D, *sig;
};
__host__ __device__ inline size_t chain_doubles(int Mp) {
  return 2 * (size_t)Mp * Mp + 2 * (size_t)Mp * 32 + 2 * (size_t)Mp * kPB + 2 * (size_t)Mp;
}
__device__ __forceinline__ ChainBuf chain_buf(double* base, int chain, int Mp) {
  ChainBuf b;
  b.R = base + chain * chain_doubles(Mp);      // [2][panel][16][Mp] panel rows when the panel starts
  b.S = b.R + 2 * (size_t)Mp * Mp;             // [2][panel][16][32] rows P_q, columns P_{q-1} and P_q, one
                                               // panel earlier: what the next pivot block is formed from
  b.D = b.S + 2 * (size_t)Mp * 32;             // [2][panel][16][16] inverse pivot blocks
  b.sig = b.D + 2 * (size_t)Mp * kPB;          // [2][Mp]
  return b;
}

// the block that inverts the pivot blocks of one chain: warps 0 .. 3 hold the matrix, warp 4 computes
// the reciprocals and publishes, warp 5 fetches the next panel's rows meanwhile
__device__ void pivot_chain(const Factor64Params& p, int chain, int nsteps, int owners, uint64_t limit) {
  constexpr int SP = 33;  // row pitch of the fetched 16 x 32 block
  __shared__ double S[2][kPB * SP];
  __shared__ double Dm[kPB][kPB + 1], W1[kPB][kPB + 1], Bm[kPB][kPB + 1];
  __shared__ GjShared<kPB> gj;
  __shared__ unsigned fail;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int Mp = p.Mp, np = Mp / kPB, total = nsteps * np;
  const ChainBuf cb = chain_buf(p.buf, chain, Mp);
  unsigned* fl = p.flags + kFlagChain + chain * kChainFlags;
  unsigned* fS = fl + (1 + kMaxPanels) * kFlagStride;
  if (tid == 0) fail = 0;
  __syncthreads();
  auto fetch = [&](int c) {  // one warp
    const int s = c / np, q = c - s * np;
    bool ok = true;
    if (lane == 0) ok = wait_count(fS + q * kFlagStride, (unsigned)(s + 1) * owners, p.flags, p.status, limit);
    ok = __shfl_sync(0xffffffffu, ok, 0);
    __syncwarp();  // lane 0's acquire orders the other lanes' reads (a shuffle orders no memory)
    if (!ok) {
      if (lane == 0) fail = 1;
      return;
    }
    const double* src = cb.S + ((size_t)(s & 1) * np + q) * kPB * 32;
    double* dst = S[c & 1];
#pragma unroll
    for (int t = 0; t < kPB; ++t) dst[t * SP + lane] = __ldcg(src + t * 32 + lane);
  };
  if (warp == 5) fetch(0);
  const int col = lane & 15, r0 = (warp & 3) * 4 + (lane >> 4) * 2;
  // the symmetric product: thread t < 128 forms element t of the lower triangle (row by row), warp 4
  // the last eight (row 15, columns 8 .. 15) with four lanes each
  int ti = 0;
  while ((ti + 1) * (ti + 2) / 2 <= tid) ++ti;
  const int tj = tid - ti * (ti + 1) / 2;
  for (int c = 0; c < total; ++c) {
    __syncthreads();
    if (fail) return;
    const int s = c / np, q = c - s * np;
    if (warp <= 4) {
      const double* Sc = S[c & 1];
      double d[2] = {0.0, 0.0};
      if (q == 0) {
        if (warp < 4) {
          d[0] = Sc[r0 * SP + 16 + col];
          d[1] = Sc[(r0 + 1) * SP + 16 + col];
        }
      } else {  // D_q = A_qq - A_qp D_p^-1 A_qp^T, p the panel before
        if (warp < 4) {
          double w0 = 0.0, w1 = 0.0;
#pragma unroll
          for (int k = 0; k < kPB; ++k) {
            const double dk = Dm[k][col];
            w0 = fma(Sc[r0 * SP + k], dk, w0);
            w1 = fma(Sc[(r0 + 1) * SP + k], dk, w1);
          }
          W1[r0][col] = w0;
          W1[r0 + 1][col] = w1;
        }
        bar5_sync<kBarAll>();
        if (warp < 4) {
          double v = Sc[ti * SP + 16 + tj];
#pragma unroll
          for (int k = 0; k < kPB; ++k) v = fma(-W1[ti][k], Sc[tj * SP + k], v);
          Bm[ti][tj] = v;
          Bm[tj][ti] = v;
        } else {
          const int cj = 8 + (lane >> 2), k0 = (lane & 3) * 4;
          double v = 0.0;
#pragma unroll
          for (int k = 0; k < 4; ++k) v = fma(-W1[15][k0 + k], Sc[cj * SP + k0 + k], v);
          v += __shfl_xor_sync(0xffffffffu, v, 1);
          v += __shfl_xor_sync(0xffffffffu, v, 2);
          if ((lane & 3) == 0) {
            v += Sc[15 * SP + 16 + cj];
            Bm[15][cj] = v;
            Bm[cj][15] = v;
          }
        }
        bar5_sync<kBarAll>();
        d[0] = Bm[r0][col];
        d[1] = Bm[r0 + 1][col];
      }
      gj_invert<kPB, 2>(d, r0, col, warp, gj);
      if (warp < 4) {
        double* Dg = cb.D + ((size_t)(s & 1) * np + q) * kPB * kPB;
        Dg[r0 * kPB + col] = d[0];
        Dg[(r0 + 1) * kPB + col] = d[1];
        Dm[r0][col] = d[0];  // the last reads of Dm are two barriers back
        Dm[r0 + 1][col] = d[1];
      }
      bar5_sync<kBarAll>();
      if (tid == 128) add_release(fl);
    } else if (warp == 5 && c + 1 < total) {
      fetch(c + 1);
    }
  }
}

}  // namespace

// R rows per worker block, KC columns per thread.  Grid: chains x (1 + Mp / R) blocks, cooperative.
template <int R, int KC>
__global__ void __launch_bounds__(256, 1) factor64_kernel(Factor64Params p) {
  const int Mp = p.Mp, M = p.M, N = p.N, m = p.meet, np = Mp / kPB;
  const int G = Mp / R;
  const int chain = blockIdx.x / (G + 1), role = blockIdx.x - chain * (G + 1);
  const int nsteps = chain == 0 ? m + 1 : N - 1 - m;
  const bool right = m < N - 1;
  const uint64_t limit = wait_limit(p.status);
  constexpr int owners = kPB / R;  // worker blocks per panel
  if (role == 0) {
    pivot_chain(p, chain, nsteps, owners, limit);
    return;
  }
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nt = blockDim.x, nwarps = nt >> 5;
  const int row0 = (role - 1) * R, qo = row0 / kPB, lr = row0 - qo * kPB;  // own rows, their panel
  const ChainBuf cb = chain_buf(p.buf, chain, Mp);
  unsigned* fD = p.flags + kFlagChain + chain * kChainFlags;
  unsigned* fR = fD + kFlagStride;
  unsigned* fS = fD + (1 + kMaxPanels) * kFlagStride;
  const double gw = p.gw, gw2 = gw * gw;
  __shared__ double pa[R][kPB], pe[R][32];
  __shared__ __align__(16) double W[R][kPB];
  __shared__ double red[8][2 * R], tot[2 * R], diag[R];
  double a[KC][R];
#pragma unroll
  for (int c = 0; c < KC; ++c)
#pragma unroll
    for (int r = 0; r < R; ++r) a[c][r] = 0.0;
  // the next column's inputs, in flight while this column's last panel is applied
  double cpre[R], hpre = 0.0;
  auto prefetch = [&](int s) {
    const int j = chain_col(chain, s, N);
    if (KC == 1 && tid < Mp)
#pragma unroll
      for (int r = 0; r < R; ++r) cpre[r] = p.Coff[((size_t)j * Mp + row0 + r) * Mp + tid];
    if (tid < R && row0 + tid < M) hpre = p.h[(size_t)j * Mp + row0 + tid] + (j == 0 ? p.gsrc : 0.0);
  };
  prefetch(0);

  for (int s = 0; s < nsteps; ++s) {
    const int j = chain_col(chain, s, N), par = s & 1;
    const bool meet = chain == 0 && s == m;
    double* Rb = cb.R + (size_t)par * Mp * Mp;
    double* Sb = cb.S + (size_t)par * Mp * 32;
    const double* Db = cb.D + (size_t)par * Mp * kPB;
    const bool from_right = meet && right;
    if (from_right) {
      const bool ok = tid != 0 || wait_count(p.flags + kFlagDone, (unsigned)G, p.flags, p.status, limit);
      if (!__syncthreads_and(ok)) return;
    }
    // ---- Z_j: off-diagonal, row sums, diagonal -------------------------------------------------
    {
      const double* C = p.Coff + ((size_t)j * Mp + row0) * Mp;
      const double* sp = cb.sig + (size_t)(par ^ 1) * Mp;
      const double* Xr = p.X + ((size_t)(m + 1) * Mp + row0) * Mp;
      const double* sr = chain_buf(p.buf, 1, Mp).sig + (size_t)((N - 2 - m) & 1) * Mp;
      double v[2 * R];
#pragma unroll
      for (int r = 0; r < 2 * R; ++r) v[r] = 0.0;
#pragma unroll
      for (int c = 0; c < KC; ++c) {
        const int k = tid + c * nt;
        if (k < Mp) {
          const double sk = s > 0 ? __ldcg(sp + k) : 0.0;
          const double skr = from_right ? __ldcg(sr + k) : 0.0;
#pragma unroll
          for (int r = 0; r < R; ++r) {
            const int i = row0 + r;
            double z = fma(-gw2, a[c][r], KC == 1 ? cpre[r] : C[(size_t)r * Mp + k]);
            v[R + r] = fma(a[c][r], sk, v[R + r]);
            if (from_right) {
              const double x = __ldcg(Xr + (size_t)r * Mp + k);
              z = fma(-gw2, x, z);
              v[R + r] = fma(x, skr, v[R + r]);
            }
            a[c][r] = (i < M && k < M && k != i) ? z : 0.0;
            v[r] += fabs(a[c][r]);
          }
        }
      }
      group_sums<2 * R, 32>(v, lane);
      constexpr int rep = 32 / (2 * R);
      if ((lane & (rep - 1)) == 0) red[warp][lane / rep] = v[0];
      __syncthreads();
      if (tid < 2 * R) {
        double t = red[0][tid];
        for (int w = 1; w < nwarps; ++w) t += red[w][tid];
        tot[tid] = t;
      }
      __syncthreads();
      if (tid < R) {
        const int i = row0 + tid;
        const bool real = i < M;
        const double sg = real ? fma(gw, tot[R + tid], hpre) : 0.0;
        cb.sig[(size_t)par * Mp + i] = sg;
        diag[tid] = real ? sg + (meet ? 0.0 : gw) + tot[tid] : 1.0;
      }
      __syncthreads();
#pragma unroll
      for (int c = 0; c < KC; ++c) {
        const int k = tid + c * nt;
#pragma unroll
        for (int r = 0; r < R; ++r)
          if (k == row0 + r) a[c][r] = diag[r];
      }
    }
    auto put_rows = [&]() {  // own rows of panel qo, before it is applied
#pragma unroll
      for (int c = 0; c < KC; ++c) {
        const int k = tid + c * nt;
        if (k < Mp)
#pragma unroll
          for (int r = 0; r < R; ++r) Rb[(size_t)(row0 + r) * Mp + k] = a[c][r];
      }
    };
    auto signal = [&](unsigned* f) {  // after a __syncthreads that follows the writes
      if (tid == 0) add_release(f);
    };
    if (qo <= 1) {
      if (qo == 0) put_rows();
      const unsigned cc = (unsigned)(tid - (qo - 1) * kPB);  // columns P_{qo-1}, P_qo (< 32 <= nt)
      if (cc < 32u)
#pragma unroll
        for (int r = 0; r < R; ++r) Sb[((size_t)qo * kPB + lr + r) * 32 + cc] = a[0][r];
      __syncthreads();
      signal(fS + qo * kFlagStride);
      if (qo == 0) signal(fR);
    }
    // ---- panels ------------------------------------------------------------------------------
    for (int q = 0; q < np; ++q) {
      const int P0 = q * kPB;
      const bool rowin = qo == q;
      const bool early = qo == q + 2;  // the pivot block after next is formed from these rows
      if (q == np - 1 && s + 1 < nsteps) prefetch(s + 1);
      {
        const bool ok = tid != 0 || wait_count(fR + q * kFlagStride, (unsigned)(s + 1) * owners, p.flags, p.status, limit);
        if (!__syncthreads_and(ok)) return;
      }
      double x[kPB];  // this thread's column of the panel rows
      auto load_col = [&](int c) {
        const int k = tid + c * nt;
        if (k < Mp)
#pragma unroll
          for (int u = 0; u < kPB; ++u) x[u] = __ldcg(Rb + (size_t)(P0 + u) * Mp + k);
      };
      load_col(0);
#pragma unroll
      for (int c = 0; c < KC; ++c) {
        const unsigned kk = (unsigned)(tid + c * nt - P0);
        if (kk < (unsigned)kPB)
#pragma unroll
          for (int r = 0; r < R; ++r) pa[r][kk] = a[c][r];
        if (early && kk - kPB < 32u)
#pragma unroll
          for (int r = 0; r < R; ++r) pe[r][kk - kPB] = a[c][r];
      }
      // rows of the pivot block after next: their columns of panels q+1 and q+2 are updated first, one
      // element per thread, because the pivot chain waits for them
      double xe[kPB];
      const int er = tid / 32, ec = tid & 31;
      if (early && er < R)
#pragma unroll
        for (int u = 0; u < kPB; ++u) xe[u] = __ldcg(Rb + (size_t)(P0 + u) * Mp + P0 + kPB + ec);
      {
        const bool ok = tid != 0 || wait_count(fD, (unsigned)(s * np + q + 1), p.flags, p.status, limit);
        if (!__syncthreads_and(ok)) return;
      }
      // W = own rows[P] D^-1 (rows of the panel itself: -D^-1, so that one update serves both); KS lanes
      // share an element
      const double* D = Db + (size_t)q * kPB * kPB;
      constexpr int KS = 128 / (R * kPB);
      if (tid < 128) {
        const int o = tid / KS, ks = tid % KS, r = o / kPB, u = o % kPB;
        double w = 0.0;
        if (rowin) {
          w = -__ldcg(D + (lr + r) * kPB + u);
        } else {
          double dk[kPB / KS];
#pragma unroll
          for (int k = 0; k < kPB / KS; ++k) dk[k] = __ldcg(D + (ks * (kPB / KS) + k) * kPB + u);
#pragma unroll
          for (int k = 0; k < kPB / KS; ++k) w = fma(pa[r][ks * (kPB / KS) + k], dk[k], w);
#pragma unroll
          for (int o2 = KS / 2; o2 > 0; o2 >>= 1) w += __shfl_xor_sync(0xffffffffu, w, o2);
        }
        if (ks == 0) W[r][u] = w;
      }
      __syncthreads();
      if (early) {
        if (er < R) {
          double v = pe[er][ec];
#pragma unroll
          for (int u = 0; u < kPB; ++u) v = fma(-W[er][u], xe[u], v);
          Sb[((size_t)qo * kPB + lr + er) * 32 + ec] = v;
        }
        __syncthreads();
        signal(fS + qo * kFlagStride);
      }
      auto update = [&](int c) {
        const unsigned kk = (unsigned)(tid + c * nt - P0);
        const bool cin = kk < (unsigned)kPB;
#pragma unroll
        for (int r = 0; r < R; ++r) {
          double acc = rowin ? 0.0 : a[c][r];
#pragma unroll
          for (int u = 0; u < kPB; u += 2) {
            const double2 w2 = *reinterpret_cast<const double2*>(&W[r][u]);
            acc = fma(-w2.x, x[u], acc);
            acc = fma(-w2.y, x[u + 1], acc);
          }
          a[c][r] = cin ? -W[r][kk] : acc;
        }
      };
#pragma unroll
      for (int c = 0; c < KC; ++c) {
        if (c > 0) load_col(c);
        if (tid + c * nt < Mp) update(c);
      }
      if (qo == q + 1) {
        put_rows();
        __syncthreads();
        signal(fR + qo * kFlagStride);
      }
    }
    double* Xo = p.X + ((size_t)j * Mp + row0) * Mp;
#pragma unroll
    for (int c = 0; c < KC; ++c) {
      const int k = tid + c * nt;
      if (k < Mp)
#pragma unroll
        for (int r = 0; r < R; ++r) Xo[(size_t)r * Mp + k] = a[c][r];
    }
  }
  if (chain == 1) {
    __syncthreads();
    if (tid == 0) add_release(p.flags + kFlagDone);
  }
}

size_t factor64_buf_bytes(int Mp) {
  return (Mp == kPB ? (size_t)Mp : 2 * chain_doubles(Mp)) * sizeof(double);
}
size_t factor64_flag_bytes() { return kFlagWords * sizeof(unsigned); }

cudaError_t launch_factor64(const Factor64Params& p, cudaStream_t st) {
  const int Mp = p.Mp;
  if (Mp < 16 || Mp % kPB || Mp > kMaxPanels * kPB || p.N < 1 || p.meet < 0 || p.meet >= p.N)
    return cudaErrorInvalidValue;
  cudaError_t err = cudaMemsetAsync(p.flags, 0, factor64_flag_bytes(), st);
  if (err != cudaSuccess) return err;
  const int chains = p.meet < p.N - 1 ? 2 : 1;
  cudaLaunchConfig_t cfg = {};
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  if (Mp == kPB) {
    cfg.gridDim = dim3(chains);
    cfg.blockDim = dim3(160);
    cfg.numAttrs = chains > 1 ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, factor64_small_kernel, p);
  }
  const int R = p.rows, KC = Mp <= 256 ? 1 : Mp <= 512 ? 2 : 4;
  if (R != 8 && (Mp > 256 || (R != 4 && (R != 2 || Mp > 128)))) return cudaErrorInvalidValue;
  cfg.gridDim = dim3(chains * (Mp / R + 1));
  const int cols = (Mp + KC - 1) / KC;
  cfg.blockDim = dim3(R == 8 || cols > 192 ? 256 : 192);
  cfg.numAttrs = 1;
  if (R == 2) return cudaLaunchKernelEx(&cfg, factor64_kernel<2, 1>, p);
  if (R == 4) return cudaLaunchKernelEx(&cfg, factor64_kernel<4, 1>, p);
  if (KC == 1) return cudaLaunchKernelEx(&cfg, factor64_kernel<8, 1>, p);
  if (KC == 2) return cudaLaunchKernelEx(&cfg, factor64_kernel<8, 2>, p);
  return cudaLaunchKernelEx(&cfg, factor64_kernel<8, 4>, p);
}

}  // namespace xbar
