// sweep_few.cu -- forward and back substitution of a few input vectors (Sec. II-C), a thread-block
// cluster per chain and panel of NV vectors.
//
// Same recurrences and the same two launches as sweep.cu (inward along the two elimination chains, then
// the meeting column and outward).  With a few vectors a step is a matrix-vector product and the
// N dependent steps are a chain of latencies: one block per panel reads all of X_j through one SM
// (28 us a step for a 256 x 256 FP64 block, 39k cycles of which are the SM's FP64 pipe), and a
// 64-vector tensor-core panel takes as long for one vector as for 64 (5.2 us).  Here block g of a
// cluster of C = Mp / RR holds rows [g RR, (g+1) RR) of every X_j: they arrive by bulk copies a few steps
// ahead, two or one rows per warp are multiplied with the whole running vector, and the block's RR new
// elements go to every block of the cluster by asynchronous shared-memory stores that complete on
// the receiver's mbarrier (transaction bytes).  The running vector is double-buffered: a block sends
// element s + 2 only after it has received s + 1 from every block, each of which has then read s.
//
// The currents' dot products are left as one partial sum per block and column in the z scratch, where
// the block's own first row was (its z is consumed; the three columns around the meeting one, whose z
// the other chain's cluster still reads, use rows of the meeting column's slot, which holds no z),
// and a small kernel adds them in order.
//
// Measured: one vector of 256 x 256 in FP64 14.3 -> 0.7 ms a solve (7.1 with one block per chain);
// rule and widths at sweep_few_plan.
#include <math.h>

#include "common.cuh"
#include "kernels.h"

namespace xbar {

namespace {

constexpr int kFewWarps = 8;                         // warps that multiply; one more sums the currents
constexpr int kFewThreads = (kFewWarps + 1) * 32;
constexpr int kFewRing = 4;                          // at most this many X_j slices in flight

__device__ __forceinline__ uint32_t few_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void few_cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t few_peer(uint32_t local, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(local), "r"(rank));
  return r;
}
// asynchronous 16-byte store to a block of the cluster, counted in bytes on that block's mbarrier
__device__ __forceinline__ void st_async16(uint32_t addr, uint4 v, uint32_t bar) {
  asm volatile(
      "st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(addr),
      "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w), "r"(bar)
      : "memory");
}

// bounded wait for phase `parity`, acquire at cluster scope
__device__ __forceinline__ bool few_wait(uint64_t* bar, unsigned parity, unsigned* status, uint64_t limit) {
  auto done = [&]() {
    uint32_t d;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.test_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(d)
        : "r"(smem_addr(bar)), "r"(parity)
        : "memory");
    return d != 0;
  };
  if (done()) return true;
  const uint64_t t0 = globaltimer_ns();
  unsigned k = 0;
  while (!done()) {
    if ((++k & 255u) == 0 && globaltimer_ns() - t0 > limit) {
      set_status(status, XBAR_DEV_TIMEOUT);
      return false;
    }
  }
  return true;
}

// sums of NS values (a power of two <= 32) over the 32 lanes; lane l then holds sum l / (32 / NS) in v[0]
template <typename T, int NS>
__device__ __forceinline__ void warp_sums(T (&v)[NS], int lane) {
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

// where the partial current of block g for column j (panel vector b) waits in z
__host__ __device__ inline size_t few_partial(int j, int m, int g, int RR, int Mp, int Bpad, int b) {
  const int d = j - m;
  const bool near = d >= -1 && d <= 1;
  return ((size_t)(near ? m : j) * Mp + (size_t)g * RR + (near ? d + 1 : 0)) * Bpad + b;
}

__host__ __device__ constexpr int few_depth(int RR, int Mp, int elem) {
  return RR * Mp * elem > 24 * 1024 ? 3 : kFewRing;
}

}  // namespace

// Grid (panels x C, chains), cluster (C, 1, 1).  Chain of a block: blockIdx.y + chain0.  kOut: the meeting
// column and the outward part.
template <typename T, int NV, int RR, bool kOut>
__global__ void __launch_bounds__(kFewThreads) sweep_few_kernel(SweepParams<T> p, int C, int chain0) {
  constexpr int RW = RR / kFewWarps;  // rows per multiplying warp
  constexpr int NE = RR * NV;         // elements of the running vector this block produces
  const int Mp = p.Mp, N = p.N, Bpad = p.Bpad, m = p.meet;
  const int chain = (int)blockIdx.y + chain0;
  const int nsteps = (chain == 0 ? m : N - 1 - m) + (kOut ? 1 : 0);
  const int jdir = (chain == 0) == kOut ? -1 : 1, jstart = kOut ? m : (chain == 0 ? 0 : N - 1);
  auto col_of = [&](int s) { return jstart + jdir * s; };
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int g = (int)few_rank(), row0 = g * RR;
  const int b0 = (int)(blockIdx.x / C) * NV;
  const int depth = few_depth(RR, Mp, sizeof(T));

  extern __shared__ __align__(128) unsigned char smem_raw[];
  T* ring = reinterpret_cast<T*>(smem_raw);           // [depth][RR][Mp]
  T* vin = ring + (size_t)depth * RR * Mp;            // [2][Mp][NV]
  __shared__ __align__(8) uint64_t full[kFewRing], vbar[2];
  __shared__ __align__(16) T vout[NE];
  __shared__ T ybuf[NE], cbuf[2][NE];
  static_assert(NE * sizeof(T) % 16 == 0, "whole 16-byte pieces");
  __shared__ unsigned fail;

  if (p.skip && *p.skip) return;  // the same for every block
  const uint64_t wlim = wait_limit(p.status);
  if (tid == 0) {
    for (int k = 0; k < kFewRing; ++k) mbar_init(&full[k], 1);
    mbar_init(&vbar[0], 1);
    mbar_init(&vbar[1], 1);
    fail = 0;
    fence_mbar_init();
  }
  const unsigned slice = (unsigned)(RR * Mp * sizeof(T));
  auto fetch = [&](int s) {  // one thread
    mbar_arrive_expect_tx(&full[s % depth], slice);
    bulk_g2s(ring + (size_t)(s % depth) * RR * Mp, p.X + ((size_t)col_of(s) * Mp + row0) * Mp, slice, &full[s % depth]);
  };
  few_cluster_sync();  // every block's mbarriers exist before a peer's stores arrive on them
  if (tid == 0)
    for (int s = 0; s < depth && s < nsteps; ++s) fetch(s);

  // the whole input of step 0: the right-hand side of its column and, in the meeting column, both chains' z
  const bool from_left = kOut && m > 0, from_right = kOut && !p.V && m + 1 < N;
  for (int t = tid; t < Mp * NV; t += kFewThreads) {
    const int i = t / NV, b = b0 + t % NV;
    T v;
    if (p.V) v = (jstart == 0 && i < p.M && b < p.B) ? p.src[i] * (T)p.V[(size_t)b * p.M + i] : (T)0;
    else v = p.rhs[((size_t)jstart * Mp + i) * Bpad + b];
    if (from_left) v = fma(p.e[(size_t)(m - 1) * Mp + i], p.z[((size_t)(m - 1) * Mp + i) * Bpad + b], v);
    if (from_right) v = fma(p.e[(size_t)m * Mp + i], p.z[((size_t)(m + 1) * Mp + i) * Bpad + b], v);
    vin[t] = v;
  }
  // element threads (tid < NE): row i, vector b; operands of the next step's epilogue, one step ahead
  const int ei = row0 + tid / NV, eb = b0 + tid % NV;
  const bool elem = tid < NE;
  const bool zout = kOut && (chain == 0 || !p.V);
  T ecpl = (T)0, zin = (T)0, rin = (T)0, hs = (T)0;
  auto load_operands = [&](int s) {
    if (!elem) return;
    const int j = col_of(s);
    const bool more = s + 1 < nsteps;
    if (more) ecpl = p.e[(size_t)min(j, col_of(s + 1)) * Mp + ei];
    if (zout && s > 0) zin = p.z[((size_t)j * Mp + ei) * Bpad + eb];
    if (!kOut && more && p.rhs) rin = p.rhs[((size_t)col_of(s + 1) * Mp + ei) * Bpad + eb];
    if (kOut) hs = p.hs[(size_t)j * Mp + ei];
  };
  load_operands(0);
  __syncthreads();

  int s_end = nsteps;
  for (int s = 0; s < nsteps; ++s) {
    const int j = col_of(s);
    const bool more = s + 1 < nsteps;
    const bool have_w = kOut && (s > 0 || chain == 0);  // w_m is reported by the left cluster
    if (warp < kFewWarps) {
      bool ok = true;
      if (s > 0) {
        if (tid == 0) mbar_arrive_expect_tx(&vbar[s & 1], (unsigned)(Mp * NV * sizeof(T)));
        ok = few_wait(&vbar[s & 1], (unsigned)(((s - 1) >> 1) & 1), p.status, wlim);
      }
      ok = ok && mbar_spin_bounded(&full[s % depth], (unsigned)((s / depth) & 1), p.status, wlim, 0);
      if (!ok) fail = 1;
      const T* x = ring + (size_t)(s % depth) * RR * Mp + (size_t)warp * RW * Mp;
      const T* v = vin + (size_t)(s & 1) * Mp * NV;
      T acc[RW * NV];
#pragma unroll
      for (int k = 0; k < RW * NV; ++k) acc[k] = (T)0;
#pragma unroll 4
      for (int k = lane; k < Mp; k += 32) {
        T xv[RW];
#pragma unroll
        for (int r = 0; r < RW; ++r) xv[r] = x[r * Mp + k];
#pragma unroll
        for (int q = 0; q < NV; ++q) {
          const T vv = v[k * NV + q];
#pragma unroll
          for (int r = 0; r < RW; ++r) acc[r * NV + q] = fma(xv[r], vv, acc[r * NV + q]);
        }
      }
      warp_sums<T, RW * NV>(acc, lane);
      constexpr int rep = 32 / (RW * NV);
      if (lane % rep == 0) ybuf[warp * RW * NV + lane / rep] = acc[0];
    }
    __syncthreads();
    if (fail) {
      s_end = s;  // slices s .. s + depth - 1 have been asked for
      break;
    }
    if (elem) {
      T y = ybuf[tid];
      if (!kOut) {
        p.z[((size_t)j * Mp + ei) * Bpad + eb] = y;
      } else if (zout && s > 0) {
        y += zin;
      }
      if (more) vout[tid] = !kOut && p.rhs ? fma(ecpl, y, rin) : ecpl * y;
      if (have_w) {
        const size_t o = ((size_t)j * Mp + ei) * Bpad + eb;
        if (p.w) p.w[o] = y;
        if constexpr (sizeof(T) == 4) {
          if (p.w1out) p.w1out[o] = p.s32[(size_t)j * Mp + ei] * y;
        }
        cbuf[s & 1][tid] = hs * y;
      }
    }
    __syncthreads();
    if (tid == 0 && s + depth < nsteps) {
      fence_proxy_async_smem();
      fetch(s + depth);
    }
    if (more) {
      const uint32_t dst = smem_addr(vin + ((size_t)((s + 1) & 1) * Mp + row0) * NV), bar = smem_addr(&vbar[(s + 1) & 1]);
      constexpr int NP = NE * (int)sizeof(T) / 16;  // 16-byte pieces of the block's elements
      for (int t = tid; t < NP * C; t += kFewThreads) {
        const int peer = t / NP, k = t - peer * NP;
        st_async16(few_peer(dst + 16u * k, (uint32_t)peer), reinterpret_cast<const uint4*>(vout)[k],
                   few_peer(bar, (uint32_t)peer));
      }
      load_operands(s + 1);
    }
    if (kOut && warp == kFewWarps && have_w) {  // this block's part of the currents of column j
      constexpr int parts = 32 / NV < RR ? 32 / NV : RR;
      const int q = lane % NV, part = lane / NV;
      T c = (T)0;
      if (part < parts)
#pragma unroll
        for (int r = 0; r < RR / parts; ++r) c += cbuf[s & 1][(part * (RR / parts) + r) * NV + q];
#pragma unroll
      for (int o = NV; o < parts * NV; o <<= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
      if (lane < NV) p.z[few_partial(j, m, g, RR, Mp, Bpad, b0 + lane)] = c;
    }
  }
  // No block leaves while a copy or a peer's store may still arrive in its shared memory.  A run that
  // completes has received everything sent to it.  After a wait that ran out, the slices in flight are
  // waited for (bounded), and a pause on either side of the barrier lets the stores land that nothing
  // waits for: this block's in its peers, then its peers' here.
  auto pause = [&]() {
    if (!fail) return;
    const uint64_t t0 = globaltimer_ns();
    while (globaltimer_ns() - t0 < 200000) __nanosleep(1000);
  };
  if (fail && tid == 0)
    for (int f = s_end; f < s_end + depth && f < nsteps; ++f)
      mbar_wait_bounded(&full[f % depth], (unsigned)((f / depth) & 1), p.status, 2000000000ull);
  pause();
  few_cluster_sync();
  pause();
}

// I_j(b) = sum of the C partial sums, in order (I = dI, or I += dI with the maximum relative change)
template <typename T>
__global__ void few_currents_kernel(SweepParams<T> p, int C, int RR) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (p.skip && *p.skip) return;
  float rel = 0.0f;
  if (t < p.B * p.N) {
    const int b = t % p.B, j = t / p.B;
    T c = (T)0;
    for (int g = 0; g < C; ++g) c += p.z[few_partial(j, p.meet, g, RR, p.Mp, p.Bpad, b)];
    const double dI = (double)c;
    if (!isfinite(dI)) set_status(p.status, XBAR_DEV_NONFINITE);
    double* Ip = p.I + (size_t)b * p.N + j;
    if (p.accumulate) {
      const double In = *Ip + dI;
      *Ip = In;
      rel = (float)(fabs(dI) / fmax(fabs(In), 1e-300));
    } else {
      *Ip = dI;
    }
  }
  if (p.max_rel) {
    for (int o = 16; o > 0; o >>= 1) rel = fmaxf(rel, __shfl_xor_sync(0xffffffffu, rel, o));
    if ((threadIdx.x & 31) == 0 && rel > 0.0f) atomic_max_nonneg(p.max_rel, rel);
  }
}

// Widths.  Both chains' clusters of every panel run at once (2 panels C <= SMs), with as few vectors a
// panel as that allows: a step's products take NV Mp RR / 1.7 cycles in FP64 (16 rows of 256: 2.4k a
// vector) beside about 1.2k of exchange.  Eight rows a block up to 128 rows, where the cluster still
// fits, else sixteen.  Wider batches go to the panels of sweep.cu / sweep_tc.cu.  At the border, a solve with eight
// vectors a panel against one on panels: 256 rows, 32 vectors: FP64 4.10 ms (33 vectors on panels 7.10), mixed
// 2.05 (3.88); 128 rows, 72 vectors: FP64 1.15 (1.80), mixed 0.84 (0.98); 64 rows, 152 vectors: 0.41 (0.50) and
// 0.44 (0.53); 16 rows, 608 vectors: mixed 0.27 (0.32).
FewPlan sweep_few_plan(int Mp, int B, int nsm) {
  FewPlan f;
  if (Mp > 256 || B < 1) return f;
  for (int nv = 1; nv <= 8; nv *= 2)
    for (int rr = (Mp >= 32 && Mp <= 128) ? 8 : 16; rr <= 16; rr *= 2) {
      const long long panels = (B + nv - 1) / nv;
      if (2 * panels * (Mp / rr) <= nsm) {
        f.nv = nv;
        f.rr = rr;
        return f;
      }
    }
  return f;
}

template <typename T, int NV, int RR, bool kOut>
static cudaError_t launch_part(const SweepParams<T>& p, int chains, int chain0, cudaStream_t st) {
  const int C = p.Mp / RR, panels = p.Bpad / NV;
  const size_t smem = ((size_t)few_depth(RR, p.Mp, sizeof(T)) * RR + 2 * NV) * p.Mp * sizeof(T);
  auto kern = sweep_few_kernel<T, NV, RR, kOut>;
  cudaError_t err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (err == cudaSuccess && C > 8) err = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (err != cudaSuccess) return err;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(panels * C, chains);
  cfg.blockDim = dim3(kFewThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = C;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, p, C, chain0);
}

template <typename T, int NV, int RR>
static cudaError_t launch_few(const SweepParams<T>& p, cudaStream_t st) {
  const bool left = p.meet > 0, right = p.meet < p.N - 1;
  const bool right_in = right && p.rhs;  // an input vector enters at column 0 only
  if (left || right_in) {
    const cudaError_t err = launch_part<T, NV, RR, false>(p, left && right_in ? 2 : 1, left ? 0 : 1, st);
    if (err != cudaSuccess) return err;
  }
  const bool first = p.rhs && p.first_only;
  const cudaError_t err = launch_part<T, NV, RR, true>(p, right && !first ? 2 : 1, 0, st);
  if (err != cudaSuccess || first) return err;
  few_currents_kernel<T><<<(p.B * p.N + 127) / 128, 128, 0, st>>>(p, p.Mp / RR, RR);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_sweep_few(const SweepParams<T>& p, FewPlan f, cudaStream_t st) {
  if (f.nv < 1 || p.Mp > 256 || p.Mp % f.rr || p.Bp != f.nv || p.Bpad % f.nv || p.B > p.Bpad || p.B < 1 || p.meet < 0 ||
      p.meet >= p.N || (!p.V && !p.rhs) || (long long)p.B * p.N > 0x7fffff00ll)
    return cudaErrorInvalidValue;
  switch (f.nv * 100 + f.rr) {
    case 108: return launch_few<T, 1, 8>(p, st);
    case 116: return launch_few<T, 1, 16>(p, st);
    case 208: return launch_few<T, 2, 8>(p, st);
    case 216: return launch_few<T, 2, 16>(p, st);
    case 408: return launch_few<T, 4, 8>(p, st);
    case 416: return launch_few<T, 4, 16>(p, st);
    case 808: return launch_few<T, 8, 8>(p, st);
    case 816: return launch_few<T, 8, 16>(p, st);
    default: return cudaErrorInvalidValue;
  }
}

template cudaError_t launch_sweep_few<float>(const SweepParams<float>&, FewPlan, cudaStream_t);
template cudaError_t launch_sweep_few<double>(const SweepParams<double>&, FewPlan, cudaStream_t);

}  // namespace xbar
