// factor_cluster.cu -- the block Thomas factorization of factor.cu on a thread-block cluster.
//
// Same mathematics as factor.cu (Z_j = C_j - g_w^2 X_prev, X_j = Z_j^{-1}, diagonals from the grounded row
// sums sigma_j), for FP32 factors with 32 <= Mp <= 256, eliminated from both ends: columns 0 .. m-1 and N-1 ..
// m+1 are two independent chains, one cluster each, and a second launch inverts the meeting column
//     Z_m = C_m - g_w^2 X_{m-1} - g_w^2 X_{m+1}.
// The factor is bound by the latency of its chain (16 dependent panels a column on 16 SMs), so half the
// chain is half the time: 12.25 -> 6.2 ms at 256 x 256, 2.85 -> 1.45 ms at 128 x 128, on twice the SMs
// (4.87 and 1.31 ms with the early hand-over and the shared coefficient broadcasts below).  Few columns, and
// the tiles of a crowded batch, are eliminated from one end (one_chain in api.cu).
// In a cluster of C blocks block g holds rows [g R, (g+1) R) of the current matrix in registers, one
// thread per column (R = 16, C = Mp / R).
// The in-place blocked Gauss-Jordan inversion uses panels of R rows, so panel p is exactly block p's
// rows.  With R_p the owner's rows when panel p starts and D_p^-1 the inverse of their pivot block,
// Gauss-Jordan replaces the owner's rows by D_p^-1 R_p (D_p^-1 in the pivot columns) and every other
// block's rows by  row - W' R_p  (-W' in the pivot columns), W' = row[P] D_p^-1.  So the other blocks
// need only R_p and D_p^-1, not the owner's formed rows.  What they need travels in three parts, each as
// early as it exists, because every hand-over costs more than the arithmetic it feeds:
//   * the owner's rows go to its slot of a global (L2-resident) buffer already before panel p-1 is applied
//     to them; each peer's mbarrier is signalled (arrive with release at cluster scope) and its threads
//     load their own column straight into registers.  (Pulling panels from the owner's shared memory
//     instead makes all peers drain one SM's port at once and is several times slower.)
//   * the owner's W' for panel p-1 (1 KB) follows when D_{p-1}^-1 is known, by asynchronous stores to every
//     peer's shared memory that complete on the peer's mbarrier (transaction bytes); with it each thread
//     applies panel p-1, whose column it still holds, to its column of the owner's rows: R_p.  That doubles
//     the multiply-adds and takes the rows' update, store, signal and load (5k cycles together) off
//     the chain;
//   * D_p^-1 (1 KB) goes from the inverting warp the same way, to the next owner first.
// The next owner forms W' and its updated pivot block first and one warp inverts it while the others
// apply the panel (look-ahead).  The chain from panel to panel is then  D^-1 arrives, W', pivot block,
// inversion.  Updates run one thread per column on pairs of rows (packed FP32 multiply-adds, coefficients
// broadcast from shared memory).  Every wait is bounded; a block whose wait expires records
// XBAR_DEV_TIMEOUT and stops waiting but keeps the cluster barrier sequence (one per column step).
#include <math.h>

#include "common.cuh"
#include "kernels.h"

namespace xbar {

namespace {

constexpr int kWork = 128;             // threads of the row work: two columns and two pivot-block elements each
constexpr int kInvWarp = kWork / 32;   // one more warp inverts pivot blocks meanwhile
constexpr int kThreads = kWork + 32;
constexpr int kRows = 16;
static_assert(kThreads == 160, "named barriers");
static_assert(2 * kWork == kRows * kRows, "two elements of a pivot block per thread");

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// Arrival of a block on the cluster barrier that orders the block's reads before it.  A release by every warp costs
// each of them a fence (256 x 256: 55 us a factor); here the work warps arrive on a block barrier, which
// orders their reads before the inversion warp's part of it, and relaxed on the cluster barrier, and the
// inversion warp, which has nothing else to do then, releases for all.
__device__ __forceinline__ void cluster_arrive(bool work) {
  if (work) {
    asm volatile("bar.arrive 2, 160;" ::: "memory");
    asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
  } else {
    asm volatile("bar.sync 2, 160;" ::: "memory");
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  }
}
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// mapa: the shared::cluster address of `local` in block `rank` of this cluster
__device__ __forceinline__ uint32_t peer_addr(const void* local, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem_addr(local)), "r"(rank));
  return r;
}
__device__ __forceinline__ uint32_t peer_addr32(uint32_t local, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(local), "r"(rank));
  return r;
}
// arrive on a peer block's mbarrier; release at cluster scope orders this block's earlier writes
__device__ __forceinline__ void arrive_peer(uint32_t bar_cluster_addr) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar_cluster_addr) : "memory");
}
// asynchronous 16-byte store to a block of the cluster, counted in bytes on that block's mbarrier
__device__ __forceinline__ void st_async16(uint32_t addr, uint4 v, uint32_t bar) {
  asm volatile(
      "st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(addr),
      "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w), "r"(bar)
      : "memory");
}
__device__ __forceinline__ void work_sync() { asm volatile("bar.sync 1, 128;" ::: "memory"); }  // the row-work warps
// bounded wait for phase `parity` of a local mbarrier, acquire at cluster scope
__device__ __forceinline__ bool wait_cluster_bounded(uint64_t* bar, unsigned parity, unsigned* status) {
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
    if ((++k & 255u) == 0 && globaltimer_ns() - t0 > wait_limit(status)) {
      set_status(status, XBAR_DEV_TIMEOUT);
      return false;
    }
  }
  return true;
}
// sums of NS values (a power of two <= 32) over the 32 lanes; lane l then holds sum l / (32 / NS) in v[0]
template <int NS>
__device__ __forceinline__ void warp_sums_f(float (&v)[NS], int lane) {
  int n = NS;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    if (n > 1) {
      const bool up = (lane & o) != 0;
#pragma unroll
      for (int q = 0; q < NS / 2; ++q)
        if (q < n / 2) {
          const float send = up ? v[q] : v[q + n / 2], keep = up ? v[q + n / 2] : v[q];
          v[q] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
      n >>= 1;
    } else {
      v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
    }
  }
}

}  // namespace

// dynamic shared memory: mbarriers [16 rows + 16 inverses + 16 W' + 2 staging]; floats: W = -W'^T [R][R] of the
// panel being applied, Bp [R][R] next pivot block, DmT [R][R] transpose of this block's inverse, Dall
// [16][R][R] inverse pivot blocks by panel (own and received), Wall [16][R][R] the owners' -W'^T by panel, rw
// [2][2][R] the inversion's pivot rows, pa, pb, xs [R][R+1] own rows in the columns of this panel and of the
// next, R_p in those of the next, reductions [4][32] and [4][16], row sums [2][R], scale and coupling of the
// right neighbour (meeting column) [2][Mp]; then two staging buffers of a column step's inputs: h_j own
// rows [R] in FP64, C_j own rows [R][Mp], s_j, s of the previous column and the coupling to it [Mp] each
constexpr int kPitch = kRows + 1;
constexpr int kBars = 50;
constexpr int kSmFloats = 3 * kRows * kPitch + (3 + 32) * kRows * kRows + 4 * kRows + 4 * 32 + 4 * 16 + 2 * kRows;
static_assert(kSmFloats % 4 == 0, "16-byte aligned vectors after the fixed part");
__host__ __device__ constexpr size_t stage_bytes(int Mp) {
  return kRows * sizeof(double) + ((size_t)kRows * Mp + 3 * (size_t)Mp) * sizeof(float);
}
size_t factor_cluster_smem_bytes(int Mp) {
  return kBars * sizeof(uint64_t) + ((size_t)kSmFloats + 2 * (size_t)Mp) * sizeof(float) + 2 * stage_bytes(Mp);
}

// global panel slots, one per block of each chain's cluster: R_p [R][Mp]
size_t factor_cluster_pbuf_floats(int Mp) {
  const size_t C = (size_t)Mp / kRows;
  return 2 * C * (size_t)kRows * Mp;
}

// acc[c][r] += sum_m coefT[m*16 + r] * x[c][m] (r, m < 16, two columns c): two rows per packed multiply-add,
// coefficients read as 16-byte broadcasts
__device__ __forceinline__ void fma2(float& a0, float& a1, float w0, float w1, float x) {
  asm("{\n\t.reg .b64 A, W, X;\n\tmov.b64 A, {%0, %1};\n\tmov.b64 W, {%2, %3};\n\tmov.b64 X, {%4, %4};\n\t"
      "fma.rn.f32x2 A, W, X, A;\n\tmov.b64 {%0, %1}, A;\n\t}"
      : "+f"(a0), "+f"(a1)
      : "f"(w0), "f"(w1), "f"(x));
}
__device__ __forceinline__ void rank16_update(float (&acc)[2][16], const float* __restrict__ coefT,
                                              const float (&x)[2][16]) {
#pragma unroll
  for (int m = 0; m < 16; ++m) {
    const float4* c4 = reinterpret_cast<const float4*>(coefT + m * 16);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float4 w = c4[q];
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        fma2(acc[c][4 * q], acc[c][4 * q + 1], w.x, w.y, x[c][m]);
        fma2(acc[c][4 * q + 2], acc[c][4 * q + 3], w.z, w.w, x[c][m]);
      }
    }
  }
}

// Cluster c of the grid walks chain chain0 + c; kMeet: one cluster, the meeting column.
template <bool kMeet>
__global__ void __launch_bounds__(kThreads, 1)
    factor_cluster_kernel(const FactorParams<float>* __restrict__ params, int C, int chain0, unsigned* status) {
  constexpr int R = kRows;  // rows per block = panel width
  const FactorParams<float> p = *params;
  const uint32_t g = cluster_rank();
  const int M = p.M, Mp = p.Mp, N = p.N, m = p.meet;
  const int chain = kMeet ? 0 : chain0 + (int)blockIdx.x / C;
  const int nsteps = kMeet ? 1 : (chain == 0 ? m : N - 1 - m);
  auto col_of = [&](int s) { return kMeet ? m : (chain == 0 ? s : N - 1 - s); };
  const bool left = kMeet && m > 0, right = kMeet && m + 1 < N;  // chains that end at the meeting column
  float* sig = p.sig + (size_t)chain * 2 * Mp;
  const int r0 = (int)g * R;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint64_t wlim = wait_limit(status);

  extern __shared__ __align__(16) unsigned char smraw[];
  uint64_t* bars = reinterpret_cast<uint64_t*>(smraw);  // [16]: the rows of panel p are in its slot
  uint64_t* dbars = bars + 16;                           // [16]: D_p^-1 is in Dall
  uint64_t* wbars = bars + 32;                           // [16]: the owner's W' for panel p-1 is in Wall
  uint64_t* pbar = bars + 48;                            // [2]: staging buffer b has landed
  float* W = reinterpret_cast<float*>(smraw + kBars * sizeof(uint64_t));  // (vectors read by float4 first)
  float* Bp = W + R * R;
  float* DmT = Bp + R * R;
  float* Dall = DmT + R * R;
  float* Wall = Dall + 16 * R * R;
  float* rw = Wall + 16 * R * R;
  float* pa = rw + 4 * R;
  float* pb = pa + R * kPitch;
  float* xs = pb + R * kPitch;
  float* red = xs + R * kPitch;
  float* Dm = Dall + (size_t)g * R * R;  // this block's own
  float* red2 = red + 4 * 32;
  float* sgs = red2 + 4 * 16;
  float* abss = sgs + R;
  float* s2v = abss + R;
  float* e2v = s2v + Mp;
  unsigned char* stg = reinterpret_cast<unsigned char*>(e2v + Mp);

  if (Mp != C * R || C > 16 || (int)blockDim.x != kThreads) {
    if (tid == 0) set_status(status, XBAR_DEV_BADLAUNCH);
    return;  // uniform across the cluster: every block sees the same arguments
  }
  const float gw = (float)p.gw;
  if (tid < C) {
    mbar_init(&bars[tid], 1);
    mbar_init(&dbars[tid], 1);
    mbar_init(&wbars[tid], 1);
  }
  if (tid == 0) {
    mbar_init(&pbar[0], 1);
    mbar_init(&pbar[1], 1);
  }
  fence_mbar_init();
  cluster_sync();  // every block's mbarriers are initialised before any peer arrives on them
  // step ss's inputs -> staging buffer ss & 1 by bulk copies, one step ahead (thread 0)
  auto stage_inputs = [&](int ss) {
    unsigned char* buf = stg + (size_t)(ss & 1) * stage_bytes(Mp);
    float* bc = reinterpret_cast<float*>(buf + R * sizeof(double));
    float* bf = bc + (size_t)R * Mp;
    uint64_t* bar = &pbar[ss & 1];
    const int jj = col_of(ss), jp = chain == 0 ? jj - 1 : jj + 1;
    const unsigned cb = (unsigned)(R * Mp * sizeof(float)), vb = (unsigned)(Mp * sizeof(float));
    const unsigned hb = (unsigned)(R * sizeof(double));
    mbar_arrive_expect_tx(bar, cb + hb + vb + (ss > 0 ? 2 * vb : 0));
    bulk_g2s(bc, p.Coff + ((size_t)jj * Mp + r0) * Mp, cb, bar);
    bulk_g2s(buf, p.h + (size_t)jj * Mp + r0, hb, bar);
    bulk_g2s(bf, p.s32 + (size_t)jj * Mp, vb, bar);
    if (ss > 0) {
      bulk_g2s(bf + Mp, p.s32 + (size_t)jp * Mp, vb, bar);
      bulk_g2s(bf + 2 * Mp, p.e32 + (size_t)min(jj, jp) * Mp, vb, bar);
    }
  };
  if (tid == 0) stage_inputs(0);
  const size_t slot = (size_t)R * Mp;  // floats per panel slot
  __shared__ unsigned failed;                  // a wait of this block expired: stop waiting
  if (tid == 0) failed = 0;
  __syncthreads();

  // Two neighbouring columns per thread: the coefficients of an update reach every lane through shared
  // memory's 128 bytes a cycle (a 16-byte broadcast fills 512), which bounds it, and serve both.
  const bool colt = tid < Mp / 2;  // threads with columns
  const int kc[2] = {2 * tid, 2 * tid + 1};
  float a[2][R], x2[2][kMeet ? R : 1];
#pragma unroll
  for (int c = 0; c < 2; ++c)
#pragma unroll
    for (int r = 0; r < R; ++r) a[c][r] = 0.0f;
  if (kMeet) {  // own rows of both neighbours' inverses
#pragma unroll
    for (int c = 0; c < 2; ++c)
#pragma unroll
      for (int r = 0; r < R; ++r) {
        a[c][r] = left && colt ? p.X[((size_t)(m - 1) * Mp + r0 + r) * Mp + kc[c]] : 0.0f;
        x2[c][r] = right && colt ? p.X[((size_t)(m + 1) * Mp + r0 + r) * Mp + kc[c]] : 0.0f;
      }
  }

  float sg_prev[2] = {0.0f, 0.0f};  // sigma of this thread's columns, previous column step
  for (int s = 0; s < nsteps; ++s) {
    const int j = col_of(s), jp = chain == 0 ? j - 1 : j + 1;
    const bool has_prev = s > 0;
    // this step's inputs from the staging buffer (the next step's copies overlap this step)
    const double* hj = reinterpret_cast<const double*>(stg + (size_t)(s & 1) * stage_bytes(Mp));  // h_j of own rows
    float* Cj = reinterpret_cast<float*>(stg + (size_t)(s & 1) * stage_bytes(Mp) + R * sizeof(double));  // of C_j
    float* sj = Cj + (size_t)R * Mp;                                                    // s_j
    float* sp = sj + Mp;                                                                // s of the previous column
    float* ep = sp + Mp;                                                                // coupling to it
    if (tid < C && tid != (int)g && !*(volatile unsigned*)&failed) {
      mbar_arrive_expect_tx(&dbars[tid], R * R * sizeof(float));
      if (tid > 0) mbar_arrive_expect_tx(&wbars[tid], R * R * sizeof(float));  // panel 0 has none before it
    }
    if (tid == 0) {
      if (!failed && !mbar_wait_bounded(&pbar[s & 1], (unsigned)((s >> 1) & 1), status, wlim))
        failed = 1;
    }
    if (kMeet) {  // both neighbours' scales and couplings
      for (int t = tid; t < Mp; t += kThreads) {
        sp[t] = left ? p.s32[(size_t)(m - 1) * Mp + t] : 0.0f;
        ep[t] = left ? p.e32[(size_t)(m - 1) * Mp + t] : 0.0f;
        s2v[t] = right ? p.s32[(size_t)(m + 1) * Mp + t] : 0.0f;
        e2v[t] = right ? p.e32[(size_t)m * Mp + t] : 0.0f;
      }
    }
    __syncthreads();

    // Z^_j of own rows: X^_prev (in the registers) goes to the output and is replaced by the off-diagonal
    // part; per row the sums of  X^_prev S sigma_prev  and of |Z^_ik| / s_k, for
    //   sigma_j = h_j (+ g_s in column 0) + g_w S X^_prev S sigma_prev  (from both sides in the meeting column)
    // and the subtraction-free diagonal
    const bool use = has_prev || kMeet;
    // (the buffer's last readers passed this step's first barrier)
    if (tid == 32 * kInvWarp && s + 1 < nsteps) stage_inputs(s + 1);
    if (warp < kInvWarp) {
      float v[2 * R], v2[kMeet ? R : 1];
#pragma unroll
      for (int r = 0; r < 2 * R; ++r) v[r] = 0.0f;
      if (kMeet)
#pragma unroll
        for (int r = 0; r < R; ++r) v2[r] = 0.0f;
      if (colt) {
        const int k = kc[0];  // and k + 1
        const float2 sk = *reinterpret_cast<const float2*>(sj + k);
        float2 ek = make_float2(0.0f, 0.0f), spk = ek, sg2 = ek, e2k = ek;
        if (use) {
          ek = *reinterpret_cast<const float2*>(ep + k);
          spk = *reinterpret_cast<const float2*>(sp + k);
        }
        if (kMeet) {
          sg_prev[0] = left ? __ldcg(p.sig + (size_t)((m - 1) & 1) * Mp + k) : 0.0f;
          sg_prev[1] = left ? __ldcg(p.sig + (size_t)((m - 1) & 1) * Mp + k + 1) : 0.0f;
          const float* sr = p.sig + (size_t)(2 + ((N - 2 - m) & 1)) * Mp + k;
          sg2 = right ? make_float2(__ldcg(sr) * s2v[k], __ldcg(sr + 1) * s2v[k + 1]) : sg2;
          e2k = *reinterpret_cast<const float2*>(e2v + k);
        }
        const float g0 = sg_prev[0] * spk.x, g1 = sg_prev[1] * spk.y;
        const float rs0 = 1.0f / sk.x, rs1 = 1.0f / sk.y;
        float* Xo = p.X + ((size_t)jp * Mp + r0) * Mp + k;
#pragma unroll
        for (int r = 0; r < R; ++r) {
          const int i = r0 + r;
          const float x0 = a[0][r], x1 = a[1][r];
          if (has_prev) *reinterpret_cast<float2*>(Xo + (size_t)r * Mp) = make_float2(x0, x1);
          v[r] = fmaf(x1, g1, x0 * g0);
          const float2 c2 = *reinterpret_cast<const float2*>(Cj + (size_t)r * Mp + k);
          const float si = sj[i];
          float z0 = si * sk.x * c2.x, z1 = si * sk.y * c2.y;
          if (use) {
            const float ei = ep[i];
            z0 -= ei * ek.x * x0;
            z1 -= ei * ek.y * x1;
          }
          if (kMeet) {
            const float e2 = e2v[i];
            z0 -= e2 * e2k.x * x2[0][r];
            z1 -= e2 * e2k.y * x2[1][r];
            v2[r] = fmaf(x2[1][r], sg2.y, x2[0][r] * sg2.x);
          }
          a[0][r] = (i < M && k < M && k != i) ? z0 : 0.0f;
          a[1][r] = (i < M && k + 1 < M && k + 1 != i) ? z1 : 0.0f;
          v[R + r] = fmaf(fabsf(a[1][r]), rs1, fabsf(a[0][r]) * rs0);
        }
      }
      warp_sums_f<2 * R>(v, lane);
      red[warp * 32 + lane] = v[0];
      if constexpr (kMeet) {
        warp_sums_f<R>(v2, lane);
        if ((lane & 1) == 0) red2[warp * 16 + (lane >> 1)] = v2[0];
      }
    }
    __syncthreads();
    if (tid < 2 * R) {
      float t = 0.0f;
#pragma unroll
      for (int w = 0; w < kInvWarp; ++w) t += red[w * 32 + tid];
      if (tid < R) {
        const int i = r0 + tid;
        float sg = 0.0f;
        if (i < M) {
          sg = (float)(hj[tid] + (j == 0 ? p.gsrc : 0.0));
          if (use) sg += gw * sp[i] * t;
          if (kMeet) {
            float t2 = 0.0f;
#pragma unroll
            for (int w = 0; w < kInvWarp; ++w) t2 += red2[w * 16 + tid];
            sg += gw * s2v[i] * t2;
          }
        }
        sgs[tid] = sg;
        if (!kMeet) sig[(size_t)(s & 1) * Mp + i] = sg;
      } else {
        abss[tid - R] = t;
      }
    }
    __syncthreads();
    if (colt)
#pragma unroll
      for (int c = 0; c < 2; ++c)
#pragma unroll
        for (int r = 0; r < R; ++r)
          if (kc[c] == r0 + r) {
            const float si = sj[kc[c]];
            a[c][r] = kc[c] < M ? si * si * (sgs[r] + (kMeet ? 0.0f : gw)) + si * abss[r] : 1.0f;
          }

    if (has_prev) cluster_wait();  // the previous step's arrivals

    // (4) blocked Gauss-Jordan inversion; panel p = rows of block p.
    // Pivot blocks are inverted in one warp's registers (Gauss-Jordan, no pivoting: the block is
    // symmetric positive definite), two pivots at a time: one exchange for both, on the chain from panel to
    // panel, and each pivot with its own reciprocal, the second one that of the Schur complement (solving
    // for both rows by the 2 x 2 determinant needs one reciprocal, but rounds once more: 4.1e-8 instead of
    // 1.7e-8 for the inverse of a 128-row block).  Lane l holds column l % 16 of rows 8 (l / 16) .. + 7.  The two
    // pivot rows go through shared memory and stand for the pivot columns too (the swept part is antisymmetric
    // to the rest): eight loads a step against 22 shuffles, which the one warp issues no faster than one per
    // eight cycles.
    static_assert(R == 16, "register layout assumes 16 x 16 pivot blocks");
    const int ib = lane & 15, pa0 = (lane >> 4) * 8;
    float* slots = p.pbuf + (size_t)chain * C * slot;
    float* myslot = slots + (size_t)g * slot;  // R_g
    // one warp: a 1 KB block of this block's shared memory to the same place in every peer's, the next
    // owner first
    auto send_block = [&](const float* blk, uint64_t* mbar) {
      const uint4 v0 = reinterpret_cast<const uint4*>(blk)[lane], v1 = reinterpret_cast<const uint4*>(blk)[32 + lane];
      const uint32_t dst = smem_addr(blk) + 16u * lane, bar = smem_addr(mbar);
      for (int q = 1; q < C; ++q) {
        int peer = (int)g + q;
        if (peer >= C) peer -= C;
        const uint32_t pd = peer_addr32(dst, (uint32_t)peer), pbr = peer_addr32(bar, (uint32_t)peer);
        st_async16(pd, v0, pbr);
        st_async16(pd + 512u, v1, pbr);
      }
    };
    auto invert_send = [&]() {  // warp kInvWarp: Bp -> D^-1 in Dm and in every peer's Dall
      float d[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) d[e] = Bp[(pa0 + e) * R + ib];
      if (pa0 == 0) {
        rw[ib] = d[0];
        rw[R + ib] = d[1];
      }
#pragma unroll
      for (int q = 0; q < R; q += 2) {
        const float* rq = rw + (q & 2) * R;  // rows q, q + 1
        __syncwarp();
        const float2 pt = *reinterpret_cast<const float2*>(rq + q), pu = *reinterpret_cast<const float2*>(rq + R + q);
        const float p00 = pt.x, p01 = pt.y, p10 = pu.x, p11 = pu.y;
        float r0 = rq[ib], r1 = rq[R + ib];
        float c0[8], c1[8];  // D[a0 + e][q], D[a0 + e][q + 1] from the rows, by symmetry
        *reinterpret_cast<float4*>(c0) = *reinterpret_cast<const float4*>(rq + pa0);
        *reinterpret_cast<float4*>(c0 + 4) = *reinterpret_cast<const float4*>(rq + pa0 + 4);
        *reinterpret_cast<float4*>(c1) = *reinterpret_cast<const float4*>(rq + R + pa0);
        *reinterpret_cast<float4*>(c1 + 4) = *reinterpret_cast<const float4*>(rq + R + pa0 + 4);
        const float i0 = __fdividef(1.0f, p00), t = p01 * i0, i1 = __fdividef(1.0f, fmaf(-p10, t, p11));
        // rows q, q+1 become P^-1 [r0; r1] (P^-1 itself in the pivot columns); all other rows lose their
        // pivot-column entries times those
        const bool in0 = ib == q, in1 = ib == q + 1;
        r0 = in0 ? 1.0f : in1 ? 0.0f : r0;
        r1 = in1 ? 1.0f : in0 ? 0.0f : r1;
        const float h0 = r0 * i0, f1 = fmaf(-p10, h0, r1) * i1, f0 = fmaf(-t, f1, h0);
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          const float sgn = pa0 + e < q ? 1.0f : -1.0f;  // rows already swept: the column is minus the row
          const float v = fmaf(sgn * c1[e], f1, fmaf(sgn * c0[e], f0, in0 || in1 ? 0.0f : d[e]));
          d[e] = pa0 + e == q ? f0 : pa0 + e == q + 1 ? f1 : v;
        }
        if (q + 2 < R && pa0 == ((q + 2) & 8)) {
          float* nx = rw + ((q + 2) & 2) * R;
          nx[ib] = d[(q + 2) & 7];
          nx[R + ib] = d[(q + 3) & 7];
        }
      }
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        Dm[(pa0 + e) * R + ib] = d[e];
        DmT[ib * R + pa0 + e] = d[e];
      }
      __syncwarp();
      send_block(Dm, &dbars[g]);
    };
    auto signal_rows = [&]() {  // after a work_sync that follows every write of the slot
      if (tid < C && tid != (int)g) arrive_peer(peer_addr(&bars[g], (uint32_t)tid));
    };
    const int ar = tid >> 4, bc = tid & 15;  // this thread's elements of the 16 x 16 products: rows ar, ar + 8
    if (warp == kInvWarp) {
      __syncthreads();  // Bp is written
      invert_send();
      __syncthreads();  // Dm is written
    } else {
      // wait on an mbarrier of this column step (one lane per warp; the acquire orders the warp's reads)
      auto await = [&](uint64_t* bar) {
        if (lane == 0 && !*(volatile unsigned*)&failed && !wait_cluster_bounded(bar, (unsigned)(s & 1), status))
          failed = 1;
        __syncwarp();
      };
      auto publish_rows = [&]() {
        if (colt)
#pragma unroll
          for (int r = 0; r < R; ++r)
            *reinterpret_cast<float2*>(myslot + (size_t)r * Mp + kc[0]) = make_float2(a[0][r], a[1][r]);
        work_sync();
        signal_rows();
      };
      // this thread's entries of `v` in the columns [c0, c0 + R) to dst (row pitch dp)
      auto put_cols = [&](float* dst, int dp, const float (&v)[2][R], int c0) {
        if (colt)
#pragma unroll
          for (int c = 0; c < 2; ++c) {
            const unsigned kk = (unsigned)(kc[c] - c0);
            if (kk < (unsigned)R)
#pragma unroll
              for (int r = 0; r < R; ++r) dst[r * dp + kk] = v[c][r];
          }
      };
      // the pivot columns [c0, c0 + R) of v become wt's rows (wt[kk][r])
      auto set_cols = [&](float (&v)[2][R], const float* wt, int c0) {
        if (colt)
#pragma unroll
          for (int c = 0; c < 2; ++c) {
            const unsigned kk = (unsigned)(kc[c] - c0);
            if (kk < (unsigned)R)
#pragma unroll
              for (int r = 0; r < R; ++r) v[c][r] = wt[kk * R + r];
          }
      };
      if ((int)g == 0) {
        put_cols(Bp, R, a, 0);
        __syncthreads();  // to the inversion warp
      }
      if ((int)g <= 1) publish_rows();
      float x[2][R];   // this thread's columns of R_pp (and, on entry to a panel, of the panel before)
      float xn[2][R];  // its columns of the next owner's rows, loaded one panel ahead
      auto load_rows = [&](int q) {
        if (q >= C || q == (int)g) return;
        await(&bars[q]);
        const float* src = slots + (size_t)q * slot + kc[0];
        if (colt)
#pragma unroll
          for (int u = 0; u < R; ++u) {
            const float2 t = __ldcg(reinterpret_cast<const float2*>(src + (size_t)u * Mp));
            xn[0][u] = t.x;
            xn[1][u] = t.y;
          }
      };
      load_rows(0);
      for (int pp = 0; pp < C; ++pp) {
        const int P0 = pp * R, P1 = P0 + R;
        if ((int)g == pp) {
          load_rows(pp + 1);
          __syncthreads();  // the inversion warp has written Dm
          // own rows become the panel rows: D^-1 R outside the pivot columns, D^-1 inside
          if (colt) {
            float acc[2][R];
#pragma unroll
            for (int c = 0; c < 2; ++c)
#pragma unroll
              for (int r = 0; r < R; ++r) acc[c][r] = 0.0f;
            rank16_update(acc, DmT, a);
#pragma unroll
            for (int c = 0; c < 2; ++c)
#pragma unroll
              for (int r = 0; r < R; ++r) {
                x[c][r] = a[c][r];
                a[c][r] = acc[c][r];
              }
          }
          set_cols(a, DmT, P0);  // (DmT[kk][r] = D^-1[r][kk])
          continue;
        }
        const bool ahead = (int)g == pp + 1;  // owner of the next panel
        put_cols(pa, kPitch, a, P0);
        if (ahead) put_cols(pb, kPitch, a, P1);
        // R_pp: the owner's rows before panel pp-1 (in xn), then that panel applied
        if (pp > 0) {
          await(&wbars[pp]);
          const float* Wp = Wall + (size_t)pp * R * R;
          if (colt) rank16_update(xn, Wp, x);
          set_cols(xn, Wp, P0 - R);  // its pivot columns hold -W'
        }
#pragma unroll
        for (int c = 0; c < 2; ++c)
#pragma unroll
          for (int u = 0; u < R; ++u) x[c][u] = xn[c][u];
        if (ahead) put_cols(xs, kPitch, x, P1);
        work_sync();  // pa, pb, xs
        await(&dbars[pp]);
        float* Wt = ahead ? Wall + (size_t)g * R * R : W;
        {  // -W' = -own rows[P] D_pp^-1, two elements per thread, stored transposed
          const float* Dp = Dall + (size_t)pp * R * R;
          float w0 = 0.0f, w1 = 0.0f;
#pragma unroll
          for (int u = 0; u < R; ++u) {
            const float d = Dp[u * R + bc];
            w0 = fmaf(pa[ar * kPitch + u], d, w0);
            w1 = fmaf(pa[(ar + 8) * kPitch + u], d, w1);
          }
          Wt[bc * R + ar] = -w0;
          Wt[bc * R + ar + 8] = -w1;
        }
        work_sync();
        if (ahead) {  // its pivot block after this panel, same operation order as the update below
          float v0 = pb[ar * kPitch + bc], v1 = pb[(ar + 8) * kPitch + bc];
#pragma unroll
          for (int u = 0; u < R; ++u) {
            const float d = xs[u * kPitch + bc];
            v0 = fmaf(Wt[u * R + ar], d, v0);
            v1 = fmaf(Wt[u * R + ar + 8], d, v1);
          }
          Bp[ar * R + bc] = v0;
          Bp[(ar + 8) * R + bc] = v1;
          __syncthreads();  // to the inversion warp
          if (warp == kInvWarp - 1) send_block(Wt, &wbars[g]);
        }
        load_rows(pp + 1);  // in flight during the update
        //   row <- row - W' R_pp outside the pivot columns, -W' inside
        if (colt) rank16_update(a, Wt, x);
        set_cols(a, Wt, P0);  // R_pp holds D there, not D^-1
        if ((int)g == pp + 2) publish_rows();
      }
    }
    // every block has published its sigma before its rows, which this one has waited for
    if (!kMeet && colt)
#pragma unroll
      for (int c = 0; c < 2; ++c) sg_prev[c] = __ldcg(sig + (size_t)(s & 1) * Mp + kc[c]);
    // every block's reads of this step's slots and blocks come before the next step's first hand-over: arrive
    // here, wait there, with the next column's formation in between
    cluster_arrive(warp < kInvWarp);
  }
  {
    if (colt)
#pragma unroll
      for (int r = 0; r < R; ++r)
        *reinterpret_cast<float2*>(p.X + ((size_t)col_of(nsteps - 1) * Mp + r0 + r) * Mp + kc[0]) =
            make_float2(a[0][r], a[1][r]);
  }
  cluster_wait();
  // No block leaves while a peer's store may still arrive in its shared memory: a block that has waited
  // for everything has received everything; after a wait that ran out, a pause on either side of the
  // barrier lets land what nobody waits for.
  auto pause = [&]() {
    if (!*(volatile unsigned*)&failed) return;
    const uint64_t t0 = globaltimer_ns();
    while (globaltimer_ns() - t0 < 200000) __nanosleep(1000);
  };
  pause();
  cluster_sync();
  pause();
}

bool factor_cluster_supported(int Mp) { return Mp >= 2 * kRows && Mp <= 16 * kRows && Mp % kRows == 0; }

int factor_cluster_launches(int N) { return N > 1 ? 2 : 1; }

template <bool kMeet>
static cudaError_t launch_clusters(const FactorParams<float>* params, int C, int clusters, int chain0, size_t smem,
                                   unsigned* status, cudaStream_t st) {
  cudaError_t err = cudaFuncSetAttribute(factor_cluster_kernel<kMeet>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)smem);
  if (err == cudaSuccess && C > 8)
    err = cudaFuncSetAttribute(factor_cluster_kernel<kMeet>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (err != cudaSuccess) return err;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(clusters * C);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = C;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, factor_cluster_kernel<kMeet>, params, C, chain0, status);
}

// the chains (those that have columns), then the meeting column; the launch boundary is what the
// second waits for, so no cluster waits for another
cudaError_t launch_factor_cluster(const FactorParams<float>* params_dev, int Mp, int N, int meet, unsigned* status,
                                  cudaStream_t st) {
  if (meet < 0 || meet >= N) return cudaErrorInvalidValue;
  const int C = Mp / kRows;
  const size_t smem = factor_cluster_smem_bytes(Mp);
  const bool left = meet > 0, right = meet < N - 1;
  if (left || right) {
    const cudaError_t err = launch_clusters<false>(params_dev, C, (left ? 1 : 0) + (right ? 1 : 0), left ? 0 : 1, smem,
                                                   status, st);
    if (err != cudaSuccess) return err;
  }
  return launch_clusters<true>(params_dev, C, 1, 0, smem, status, st);
}

}  // namespace xbar
