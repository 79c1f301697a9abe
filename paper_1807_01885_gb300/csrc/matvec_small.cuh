// The float product on small grids (16 <= N <= 64, radix 8) in one launch.
//
// At these sizes the three passes are three launches of a few small blocks each, and a call
// of bem_matvec costs the host three launches.  Here one block (N <= 32) or a cluster of
// four holds the whole product: each block transforms its share of the rows, sends every
// frequency pair to the block that owns its columns (distributed shared memory),
// transforms its columns in place, and gathers its rows back.  The transforms and tables
// are those of the passes (results agree to rounding: the compiler contracts products and
// sums by context).  Solves keep the passes, which their captured and plain iterations
// share bit for bit.  N = 128 stays with them: 11.0 us on eight SMs against 6.4.
// Measured on GB300, three passes / one launch: calls back to back N = 32 11.6 / 6.7 us,
// 64 11.6 / 6.9; a product in a chain on the device N = 16 4.7 / 4.2 us, 32 4.7 / 4.8,
// 64 5.9 / 6.5 (eight blocks 6.9, two 8.1, one 10.4).
#pragma once

#include <cooperative_groups.h>

#include "matvec_reg.cuh"

namespace bem {

template <int LOGN>
struct Small {
  static constexpr int CTAS = LOGN <= 5 ? 1 : 4;
  static constexpr int N = 1 << LOGN, RB = N / CTAS, TR = Plan<LOGN, 3>::T, TC = Plan<LOGN + 1, 3>::T;
  static constexpr int NP = N / 2 + 1, PC = (NP + CTAS - 1) / CTAS;   // pairs in all and per block
  static constexpr int WANT = RB * TR > PC * TC ? RB * TR : PC * TC, T = (WANT + 31) / 32 * 32;
  static constexpr int GR = T / TR, GC = T / TC;   // transforms that the threads make up (some idle)
  static constexpr int ROW = row_sh<LOGN, 3>(), COL = Plan<LOGN + 1, 3>::PADL + 8;
  static constexpr size_t EX_R = (size_t)GR * ROW * sizeof(float2), EX_C = (size_t)GC * COL * sizeof(pr::CP);
  static constexpr size_t SMEM = (size_t)PC * N * sizeof(float4) + (EX_R > EX_C ? EX_R : EX_C);
};

// A block's shared memory may be written by its peers only once it has started: every
// thread of the cluster arrives on entry, and waits before the first remote store.  The
// arrival publishes nothing (relaxed); the wait hides behind the row transform.
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.relaxed.aligned;\n" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;\n" ::: "memory"); }

template <int LOGN>
__global__ void __cluster_dims__(Small<LOGN>::CTAS, 1, 1) __launch_bounds__(Small<LOGN>::T)
k_product_small(const float* __restrict__ p, float* __restrict__ u, const float2* __restrict__ tab2,
                const float2* __restrict__ twr, const float4* __restrict__ twp, const float2* __restrict__ tw) {
  using Z = Small<LOGN>;
  using C = float2;
  constexpr int N = Z::N, M = 2 * N, R = 8, TR = Z::TR, TC = Z::TC;
  if constexpr (Z::CTAS > 1) cluster_arrive();
  pdl_enter();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float4* const colb = reinterpret_cast<float4*>(smem_raw);            // [PC][N]: this block's columns
  unsigned char* const ex = smem_raw + (size_t)Z::PC * N * sizeof(float4);
  auto cluster = cooperative_groups::this_cluster();
  const int rank = (int)cluster.block_rank();
  const int rl = threadIdx.x / TR, t = threadIdx.x - rl * TR;
  const int row = rank * Z::RB + rl;
  const bool on = rl < Z::RB;
  C* const sh = reinterpret_cast<C*>(ex) + rl * Z::ROW;
  {
    // rows forward (k_row_fwd_r)
    C v[R];
    const C* prow = reinterpret_cast<const C*>(p + (size_t)(on ? row : 0) * N);
#pragma unroll
    for (int q = 0; q < R / 2; ++q) v[q] = on ? prow[t + TR * q] : mk(0.f, 0.f);
#pragma unroll
    for (int q = R / 2; q < R; ++q) v[q] = mk(0.f, 0.f);
    reg_fft<LOGN, 3, false, true, float, Z::GR>(v, sh, twr, t, rl);
#pragma unroll
    for (int q = 0; q < R; ++q) sh[padi<3>(t + TR * q)] = v[q];
    GroupSync<TR, Z::GR>::sync(rl);
    if constexpr (Z::CTAS > 1) cluster_wait();
    if (on) {
      const C wa = tw[2 * t], wb = tw[2 * t + 1];
      auto put = [&](int jp, float4 x) { cluster.map_shared_rank(colb, jp / Z::PC)[(jp % Z::PC) * N + row] = x; };
#pragma unroll
      for (int k = 0; k < R; k += 2) {
        const int j = 2 * t + TR * k;
        C X2[2];
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const int jj = j + e;
          const C za = sh[padi<3>(jj)];
          const C zb = cconj(sh[padi<3>((N - jj) & (N - 1))]);
          const C E = cscale(cadd(za, zb), 0.5f);
          const C O = cscale(cmul_mi(csub(za, zb)), 0.5f);
          X2[e] = cadd(E, cmul(O, recomb_tw<float, R>(tw, e ? wb : wa, jj, k)));
        }
        put(j / 2, make_float4(X2[0].x, X2[1].x, X2[0].y, X2[1].y));
      }
      if (t == 0) {
        const C z0 = sh[0];
        put(N / 2, make_float4(z0.x - z0.y, 0.f, 0.f, 0.f));
      }
    }
  }
  cluster.sync();
  {
    // columns in place (k_col_p)
    using pr::CP;
    const int c = threadIdx.x / TC, tc = threadIdx.x - c * TC, pair = rank * Z::PC + c;
    const bool active = c < Z::PC && pair < Z::NP;
    CP* const shc = reinterpret_cast<CP*>(ex) + c * Z::COL;
    float4* const col = colb + (active ? c : 0) * N;
    CP v[R];
#pragma unroll
    for (int q = 0; q < R / 2; ++q) v[q] = active ? pr::cp_load(col + tc + TC * q) : pr::cp_zero();
#pragma unroll
    for (int q = R / 2; q < R; ++q) v[q] = pr::cp_zero();
    float2 kv[R];
    const float2* kt = tab2 + (size_t)(active ? pair : 0) * (N + 1);
#pragma unroll
    for (int q = 0; q < R; ++q) {
      const int i = tc + TC * q;
      kv[q] = active ? kt[q < R / 2 ? i : M - i] : make_float2(0.f, 0.f);
    }
    pr::pair_fft<LOGN + 1, 3, false, true, Z::GC>(v, shc, twp, tc, c);
#pragma unroll
    for (int q = 0; q < R; ++q) v[q] = pr::cscale2(v[q], pr::pk2(kv[q].x, kv[q].y));
    pr::pair_fft<LOGN + 1, 3, true, false, Z::GC>(v, shc, twp, tc, c);
    if (active) {
#pragma unroll
      for (int q = 0; q < R / 2; ++q) pr::cp_store(col + tc + TC * q, v[q]);
    }
  }
  cluster.sync();
  {
    // rows inverse (k_row_inv_r)
    C v[R];
    const C wt = tw[t];
    auto get = [&](int j) {
      const int jp = j >> 1;
      const float* b = reinterpret_cast<const float*>(cluster.map_shared_rank(colb, jp / Z::PC) + (jp % Z::PC) * N + row) +
                       (j & 1);
      return mk(b[0], b[2]);
    };
#pragma unroll
    for (int q = 0; q < R; ++q) {
      const int j = t + TR * q;
      C y1 = mk(0.f, 0.f), y2 = mk(0.f, 0.f);
      if (on) {
        y1 = get(j);
        y2 = cconj(get(N - j));
      }
      const C e = cadd(y1, y2);
      const C o = cmul_pi(cmulc(csub(y1, y2), recomb_tw<float, R>(tw, wt, j, q)));
      v[q] = cadd(e, o);
    }
    reg_fft<LOGN, 3, true, false, float, Z::GR>(v, sh, twr, t, rl);
    if (on) {
      C* urow = reinterpret_cast<C*>(u + (size_t)row * N);
#pragma unroll
      for (int q = 0; q < R / 2; ++q) urow[t + TR * q] = v[q];
    }
  }
  cluster.sync();   // no block leaves while another reads its columns
}

template <int LOGN>
struct SmallLaunch {
  static void prepare() {
    static std::atomic<unsigned long long> attr{0};
    if (first_on_device(attr))
      cudaFuncSetAttribute(k_product_small<LOGN>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Small<LOGN>::SMEM);
  }
  static void run(const bem_kernel_s* k, const float* p, float* u, cudaStream_t s) {
    prepare();
    launch_pdl(k_product_small<LOGN>, Small<LOGN>::CTAS, Small<LOGN>::T, Small<LOGN>::SMEM, s, p, u, (const float2*)k->ws.table,
               (const float2*)small_twr(k), (const float4*)small_twp(k), (const float2*)k->ws.tw);
  }
};

template <typename F>
void small_logn(int logn, F&& f) {
  switch (logn) {
    case 4: f(SmallLaunch<4>{}); break;
    case 5: f(SmallLaunch<5>{}); break;
    case 6: f(SmallLaunch<6>{}); break;
    default: break;
  }
}

}  // namespace bem
