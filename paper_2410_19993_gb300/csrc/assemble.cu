// assemble.cu -- nodal-system assembly for the column-block formulation.
//
// The nodal matrix of Sec. II-A (Eqs. 1-7) couples, inside bit line j, the
// bit-line nodes u(:,j) in a tridiagonal chain T_j (segments g_b, the open top
// of Eq. 3, the sense resistor g_o at the bottom) and each u(i,j) to its
// word-line node w(i,j) through G_ij; word-line nodes couple to the next
// column through g_w.  Eliminating u(:,j) inside the column leaves, on the
// word-line nodes of column j, the dense block
//     C_j = diag(dW_j) - diag(G_j) T_j^{-1} diag(G_j)
// and the current of bit line j becomes a linear functional of w(:,j):
//     I_j = g_o u(M,j) = h_j . w_j,   h_j = g_o G_j o (T_j^{-1} e_M).
// Everything about T_j^{-1} is obtained from two subtraction-free pivot
// recurrences (top-down and bottom-up "grounded parts" of the chain), so all
// quantities keep full relative accuracy.
#include <math.h>

#include "common.cuh"
#include "kernels.h"

namespace xbar {

// Gc[j][i] = G[i][j] (row-major M x N input), zero in the padding rows i >= M.  With `status`
// set, every entry is also checked (finite and >= 0) and XBAR_DEV_BADINPUT recorded otherwise.
__global__ void asm_gc_kernel(MapDev m, const double* __restrict__ G, unsigned* status) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int j = blockIdx.y;
  if (i >= m.Mp || j >= m.N) return;
  const double g = i < m.M ? G[(size_t)i * m.N + j] : 0.0;
  if (status && !(g >= 0.0 && g <= 1.79e308)) set_status(status, XBAR_DEV_BADINPUT);
  m.Gc[(size_t)j * m.Mp + i] = g;
}

// The pivot recurrences of T_j are chains of linear-fractional maps, x -> g_b (G + x) / (G + x + g_b)
// (top-down: alpha_i from alpha_{i-1} with G = G_{i-1}; bottom-up: beta_i from beta_{i+1} with
// G = G_{i+1}).  A map is the 2 x 2 matrix [[g_b, g_b G], [1, G + g_b]] acting on (x, 1), and a chain of
// them is the matrix product: all entries are >= 0, so products keep full relative accuracy.  One warp
// takes a direction of a bit line: each lane composes the maps of its segment of rows, a warp scan composes
// the segments, and each lane then walks only its own rows from the value the scan gives at their start.
struct Mob {
  double a, b, c, d;  // x -> (a x + b) / (c x + d)
};
__device__ __forceinline__ Mob mob_id() { return {1.0, 0.0, 0.0, 1.0}; }
__device__ __forceinline__ Mob mob_step(double G, double gb) { return {gb, gb * G, 1.0, G + gb}; }
// x 2^-sh for x >= 0, on the integer pipe (an FP64 instruction costs 64 cycles of issue): exact, zero where
// the result would be below the normal range (2^-1000 of the largest entry)
__device__ __forceinline__ double shift_exp(double x, int sh) {
  const int hi = __double2hiint(x), e = (hi >> 20) - sh;
  return e > 0 && hi >= (1 << 20) ? __hiloint2double(hi - sh * (1 << 20), __double2loint(x)) : 0.0;
}
// X o Y, rescaled by a power of two (exact) so that the largest entry is in [1/2, 1)
__device__ __forceinline__ Mob mob_mul(const Mob& X, const Mob& Y) {
  const Mob r{X.a * Y.a + X.b * Y.c, X.a * Y.b + X.b * Y.d, X.c * Y.a + X.d * Y.c, X.c * Y.b + X.d * Y.d};
  const int sh = (max(max(__double2hiint(r.a), __double2hiint(r.b)), max(__double2hiint(r.c), __double2hiint(r.d))) >> 20) - 1022;
  if (sh > 1024) return r;  // an entry overflowed: infinities and NaN pass on as they are
  return {shift_exp(r.a, sh), shift_exp(r.b, sh), shift_exp(r.c, sh), shift_exp(r.d, sh)};
}
__device__ __forceinline__ double mob_apply(const Mob& X, double x) { return (X.a * x + X.b) / (X.c * x + X.d); }
__device__ __forceinline__ Mob shfl_up_mob(const Mob& X, int k) {
  return {__shfl_up_sync(0xffffffffu, X.a, k), __shfl_up_sync(0xffffffffu, X.b, k),
          __shfl_up_sync(0xffffffffu, X.c, k), __shfl_up_sync(0xffffffffu, X.d, k)};
}
__device__ __forceinline__ Mob shfl_down_mob(const Mob& X, int k) {
  return {__shfl_down_sync(0xffffffffu, X.a, k), __shfl_down_sync(0xffffffffu, X.b, k),
          __shfl_down_sync(0xffffffffu, X.c, k), __shfl_down_sync(0xffffffffu, X.d, k)};
}

// One block of two warps per bit line j: warp 0 top-down, warp 1 bottom-up, side by side; lane L of each owns
// rows [L K, L K + K), K = ceil(M / 32).  Bound by the chain of FP64 operations of a lane, the divisions
// above all (440 cycles each), so a row divides once per direction: the pivot d = G + alpha + g_b (or
// G + beta + g_b) is also the denominator of the next step of the recurrence.  Then all threads form the
// rows' diagonal of T^-1 and h.  256 rows: 55 us with one warp walking both directions and five
// divisions a row, 25 us this way; 16 rows 23 -> 12 us.
constexpr int kColThreads = 64;
constexpr int kColMax = 1024;
__global__ void __launch_bounds__(kColThreads) asm_columns_kernel(MapDev m) {
  __shared__ double alphas[kColMax], betas[kColMax], qs_[kColMax];
  const int lane = threadIdx.x & 31, dir = threadIdx.x >> 5;
  const int j = blockIdx.x;
  const int M = m.M, N = m.N, Mp = m.Mp;
  const double gs = m.gs, gw = m.gw, gb = m.gb, go = m.go;
  const double* Gc = m.Gc + (size_t)j * Mp;
  double* dW = m.dW + (size_t)j * Mp;
  double* tha = m.tha + (size_t)j * Mp;
  double* thc = m.thc + (size_t)j * Mp;
  double* tdiag = m.tdiag + (size_t)j * Mp;
  double* rho = m.rho + (size_t)j * Mp;
  double* h = m.h + (size_t)j * Mp;
  const int K = (M + 31) / 32;
  const int i0 = min(lane * K, M), i1 = min(i0 + K, M);

  if (dir == 0) {
    // top-down: pivots d-_i = G_i + alpha_i + (i < M-1 ? g_b : g_o),
    //           alpha_0 = 0, alpha_i = g_b t / (t + g_b), t = G_{i-1} + alpha_{i-1}
    // this lane's maps produce alpha_i for i0 < i <= i1 (i <= M - 1)
    Mob P = mob_id();
    for (int i = i0 + 1; i <= i1 && i <= M - 1; ++i) P = mob_mul(mob_step(Gc[i - 1], gb), P);
#pragma unroll
    for (int k = 1; k < 32; k <<= 1) {  // inclusive scan: P = S_L o S_{L-1} o ... o S_0
      if (k * K >= M) break;            // uniform: the lanes that far up hold nothing
      const Mob Y = shfl_up_mob(P, k);
      if (lane >= k) P = mob_mul(P, Y);
    }
    Mob E = shfl_up_mob(P, 1);  // the maps before this lane's rows
    if (lane == 0) E = mob_id();
    double alpha = mob_apply(E, 0.0);  // alpha_{i0}
    for (int i = i0; i < i1; ++i) {
      const double g = Gc[i], t = g + alpha;
      const double inv = 1.0 / (t + (i < M - 1 ? gb : go));
      const double c = gb * inv;
      dW[i] = g + (j == 0 ? gs : gw) + (j < N - 1 ? gw : 0.0);
      tha[i] = g * inv;
      thc[i] = c;
      alphas[i] = alpha;
      alpha = t * c;  // alpha_{i+1} (unused after the last row)
    }
  } else {
    // bottom-up: pivots d+_i = G_i + beta_i + (i > 0 ? g_b : 0),
    //            beta_{M-1} = g_o, beta_i = g_b t / (t + g_b), t = G_{i+1} + beta_{i+1}
    // this lane's maps produce beta_i for i0 <= i < i1 (i <= M - 2)
    Mob Q = mob_id();
    for (int i = i0; i < min(i1, M - 1); ++i) Q = mob_mul(Q, mob_step(Gc[i + 1], gb));  // g_i0 o ... o g_top
#pragma unroll
    for (int k = 1; k < 32; k <<= 1) {  // inclusive suffix scan: Q = T_L o T_{L+1} o ... o T_31
      if (k * K >= M) break;
      const Mob Y = shfl_down_mob(Q, k);
      if (lane + k < 32) Q = mob_mul(Q, Y);
    }
    Mob U = shfl_down_mob(Q, 1);  // the maps below this lane's rows
    if (lane == 31) U = mob_id();
    // rho_i = g_b / d+_i;  q_i = prod_{k=i+1}^{M-1} rho_k
    double beta = mob_apply(U, go);  // beta_{i1} (g_o when i1 >= M - 1)
    if (i1 > i0 && i1 - 1 < M - 1) {  // beta_{i1-1}
      const double t = Gc[i1] + beta;
      beta = gb * t / (t + gb);
    } else {
      beta = go;
    }
    double rp = 1.0;  // product of rho over this lane's rows
    for (int i = i1 - 1; i >= i0; --i) {
      const double t = Gc[i] + beta;
      const double r = gb / (t + (i > 0 ? gb : 0.0));
      betas[i] = beta;
      rho[i] = r;
      rp *= r;
      beta = t * r;  // beta_{i-1} (unused before the first row)
    }
    double qs = rp;  // suffix product over lanes L .. 31
#pragma unroll
    for (int k = 1; k < 32; k <<= 1) {
      const double y = __shfl_down_sync(0xffffffffu, qs, k);
      if (lane + k < 32) qs *= y;
    }
    double q = __shfl_down_sync(0xffffffffu, qs, 1);  // rows below this lane's
    if (lane == 31) q = 1.0;
    for (int i = i1 - 1; i >= i0; --i) {
      if (i < i1 - 1) q *= rho[i + 1];
      qs_[i] = q;
    }
  }
  __syncthreads();
  // diag(T^-1)_i = 1 / (G_i + alpha_i + beta_i);  h_i = g_o G_i diag(T^-1)_i q_i
  for (int i = threadIdx.x; i < Mp; i += kColThreads) {
    if (i < M) {
      const double g = Gc[i], t = 1.0 / (g + alphas[i] + betas[i]);
      tdiag[i] = t;
      h[i] = go * g * t * qs_[i];
    } else {
      dW[i] = 1.0;
      tha[i] = 0.0;
      thc[i] = 0.0;
      tdiag[i] = 0.0;
      rho[i] = 0.0;
      h[i] = 0.0;
    }
  }
}

// Equilibration and coupling vectors of one (j, i).
__device__ __forceinline__ void asm_scale(const MapDev& m, int i, int j) {
  const int Mp = m.Mp;
  const size_t o = (size_t)j * Mp + i;
  const bool real = i < m.M;
  const double s = real ? 1.0 / sqrt(m.dW[o]) : 1.0;
  const double snext = (real && j + 1 < m.N) ? 1.0 / sqrt(m.dW[o + Mp]) : 0.0;
  const double e_eq = (real && j + 1 < m.N) ? m.gw * s * snext : 0.0;
  const double e_pl = (real && j + 1 < m.N) ? m.gw : 0.0;
  m.s_eq[o] = s;
  m.e_eq[o] = e_eq;
  m.e_pl[o] = e_pl;
  m.hs_eq[o] = s * m.h[o];
  m.s32[o] = (float)s;
  m.e32[o] = (float)e_eq;
  m.hs32[o] = (float)(s * m.h[o]);
  auto pair = [](double x) {
    const float hi = (float)x;
    return make_float2(hi, (float)(x - (double)hi));
  };
  m.Gc2[o] = pair(m.Gc[o]);
  m.h2[o] = pair(m.h[o]);
  m.tha2[o] = pair(m.tha[o]);
  m.thc2[o] = pair(m.thc[o]);
  if (j == 0) {
    m.src_eq[i] = real ? m.gs * s : 0.0;
    m.src_pl[i] = real ? m.gs : 0.0;
    m.src32[i] = (float)(real ? m.gs * s : 0.0);
  }
}

// Off-diagonal of C_j: Coff_j[i][k] = -G_i G_k T^-1_{ik} (i != k), zero on the diagonal and in padding, in the
// precision T the factor reads (FP32 factors round each entry once either way).  The block is
// symmetric, so only k > i is computed:  T^-1_{ik} = tdiag_i prod_{m=i+1}^{k} rho_m, one running product and one
// scaling per entry (two FP64 operations; the FP64 pipe bounds the kernel).  A warp takes 32 rows, a lane
// per row, and walks k in chunks of 32: entry (k, i) is stored at once (consecutive lanes, consecutive i),
// entry (i, k) through a shared-memory tile.  256 x 256: 162 us with both triangles computed, 55 us this way.
// Blocks past the rows of C form the scales and couplings (asm_scale), in the same launch.
constexpr int kCoffThreads = 128;
template <typename T>
__global__ void __launch_bounds__(kCoffThreads) asm_coff_kernel(MapDev m, int coff_blocks) {
  __shared__ T tiles[kCoffThreads / 32][32][33];
  const int j = blockIdx.y, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int M = m.M, Mp = m.Mp;
  if ((int)blockIdx.x >= coff_blocks) {
    const int i = ((int)blockIdx.x - coff_blocks) * kCoffThreads + (int)threadIdx.x;
    if (i < Mp) asm_scale(m, i, j);
    return;
  }
  const int i0 = (blockIdx.x * (kCoffThreads / 32) + warp) * 32, i = i0 + lane;
  if (i0 >= Mp) return;  // whole warps; no block barrier below
  T(*tile)[33] = tiles[warp];
  T* C = reinterpret_cast<T*>(m.Coff) + (size_t)j * Mp * Mp;
  const double* Gc = m.Gc + (size_t)j * Mp;
  const double* rho = m.rho + (size_t)j * Mp;
  double p = i < M ? -Gc[i] * m.tdiag[(size_t)j * Mp + i] : 0.0;
  for (int k0 = i0; k0 < Mp; k0 += 32) {
    const int kn = min(32, Mp - k0);
#pragma unroll 8
    for (int q = 0; q < kn; ++q) {
      const int k = k0 + q;
      T v = (T)0;
      if (k > i && k < M) {
        p *= rho[k];
        v = (T)(p * Gc[k]);
      }
      if (k > i && i < Mp) C[(size_t)k * Mp + i] = v;
      tile[lane][q] = v;
    }
    __syncwarp();
    const int k = k0 + lane;
    for (int r = 0; r < 32; ++r)
      if (k < Mp && k >= i0 + r) C[(size_t)(i0 + r) * Mp + k] = tile[r][lane];
    __syncwarp();
  }
}

cudaError_t launch_store_g(const MapDev& m, const double* G_dev, unsigned* status, cudaStream_t st) {
  dim3 g((m.Mp + 127) / 128, m.N);
  asm_gc_kernel<<<g, 128, 0, st>>>(m, G_dev, status);
  return cudaGetLastError();
}

cudaError_t launch_assemble(const MapDev& m, bool f32, cudaStream_t st) {
  if (m.Mp > kColMax) return cudaErrorInvalidValue;
  asm_columns_kernel<<<m.N, kColThreads, 0, st>>>(m);
  const int cb = (m.Mp + kCoffThreads - 1) / kCoffThreads;
  const dim3 grid(2 * cb, m.N);
  if (f32) asm_coff_kernel<float><<<grid, kCoffThreads, 0, st>>>(m, cb);
  else asm_coff_kernel<double><<<grid, kCoffThreads, 0, st>>>(m, cb);
  return cudaGetLastError();
}

__global__ void d2f_kernel(const double* a, float* b, size_t n) {
  for (size_t k = blockIdx.x * (size_t)blockDim.x + threadIdx.x; k < n; k += (size_t)gridDim.x * blockDim.x)
    b[k] = (float)a[k];
}

cudaError_t launch_d2f(const double* a, float* b, size_t n, cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  int blocks = (int)((n + 255) / 256);
  if (blocks > 4096) blocks = 4096;
  d2f_kernel<<<blocks, 256, 0, st>>>(a, b, n);
  return cudaGetLastError();
}

}  // namespace xbar
