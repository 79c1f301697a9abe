// The product u = K p of bem_matvec in double (N >= 16) on 64-bit fixed-point transforms
// (fft_fix.cuh); the passes, the pruning of the zero half and the order of the spectrum
// (column-major, spec[j N + r]) are those of matvec_reg.cuh.
//
// Every transform has its own scale, so no value has to share one with a transform of
// another size: the row pass leaves the exponent of each row's spectrum in fexp[r], the
// column pass aligns its N values to the exponent of the column's own sum, multiplies by
// K^ (a 53-bit significand and an exponent per entry), scales again by the sum of the
// products (K^ falls like 1/k, so a few low wave numbers may carry the column) and leaves
// the exponent in fexp[N + j]; the row inverse does the same over the columns.  A value
// that is not finite marks its row, every column and so every output, as it spreads over
// a double transform.
//
// The solves keep the passes on the FP64 pipe: their conjugate gradients on a symmetric
// problem (sphere, punch) turn a change in the last place of a product into one of the
// size of the tolerance (1e-9 of the pressure at tol = 1e-10, and a step more or less),
// so a solve would no longer return the pressures it did.
//
// What bounds the passes: the integer multiply-adds (three per real product); at small
// and middle grids the latency of the stages and of the two reductions per transform.
// Product in a chain of products on GB300, FP64 pipe / fixed point: N = 64 29 / 22 us,
// 256 38 / 31, 512 156 / 40, 1024 440 / 111, 2048 1910 / 533.  Relative error against
// quadruple precision, FP64 pipe / fixed point: a contact pressure (positive part of
// white noise) N = 512 3.7e-16 / 0.5e-16, 1024 3.1e-16 / 0.5e-16, 2048 2.6e-16 / 0.6e-16;
// white noise 3.1e-16 / 1.0e-16, 3.5e-16 / 1.2e-16, 3.9e-16 / 2.1e-16.
#include "bem_internal.cuh"
#include "fft_fix.cuh"

namespace bem {
namespace fx {

// rows and columns per block: two rows whose records of one frequency fill a 32-byte
// sector, one column, at least a warp
__host__ __device__ constexpr int per_warp(int want, int t) { return want * t < 32 ? 32 / t : want; }
template <int LOGN>
__host__ __device__ constexpr int fix_rows() {
  constexpr int r = per_warp(2, Plan<LOGN, 3>::T);
  return r > (1 << LOGN) ? (1 << LOGN) : r;
}
template <int LOGM>
__host__ __device__ constexpr int fix_cols() { return per_warp(1, Plan<LOGM, 3>::T); }
// complex slots of one transform's exchange buffer (even, so that every one starts on a
// 32-byte boundary), and words for its reductions
template <int LOGL>
__host__ __device__ constexpr int fix_sh() { return Plan<LOGL, 3>::PADL + 8; }
constexpr int kRedWords = 16;

template <int LOGN>
__global__ void __launch_bounds__((fix_rows<LOGN>() * Plan<LOGN, 3>::T))
k_row_fwd_x(const double* __restrict__ p, I2* __restrict__ spec, int* __restrict__ fexp, const int4* __restrict__ twr,
            const int4* __restrict__ tw) {
  using P = Plan<LOGN, 3>;
  constexpr int N = 1 << LOGN, TT = P::T, SH = fix_sh<LOGN>(), R = P::R, RPB = fix_rows<LOGN>();
  pdl_enter();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int red[RPB][kRedWords];
  I2* const sh0 = reinterpret_cast<I2*>(smem_raw);
  const int rl = threadIdx.x / TT, t = threadIdx.x - rl * TT;
  const int r0 = blockIdx.x * RPB;
  I2* sh = sh0 + rl * SH;
  const double2* prow = reinterpret_cast<const double2*>(p + (size_t)(r0 + rl) * N);
  double2 z[R / 2];
#pragma unroll
  for (int q = 0; q < R / 2; ++q) z[q] = prow[t + TT * q];
  unsigned a[R];
  int e[R];
#pragma unroll
  for (int q = 0; q < R / 2; ++q) {
    term_of(z[q].x, a[2 * q], e[2 * q]);
    term_of(z[q].y, a[2 * q + 1], e[2 * q + 1]);
  }
  Bound b = l1_exponent<TT, RPB>(a, e, red[rl], t, rl);
  b.max += 1;   // the terms are real and imaginary parts
  const int E0 = stage_exponent<LOGN, true>(b, 0);
  I2 v[R];
#pragma unroll
  for (int q = 0; q < R / 2; ++q) v[q] = I2{to_fix(z[q].x, E0), to_fix(z[q].y, E0)};
#pragma unroll
  for (int q = R / 2; q < R; ++q) v[q] = I2{0, 0};
  fix_fft<LOGN, false, true, RPB>(v, b, sh, twr, t, rl);
#pragma unroll
  for (int q = 0; q < R; ++q) sh[padi<3>(t + TT * q)] = v[q];
  if (t == 0) fexp[r0 + rl] = b.sum;
  __syncthreads();
  // X[j] = (Z[j] + Z*[N-j])/2 - (i/2) e^{-i pi j/N} (Z[j] - Z*[N-j]); thread (j0, rr)
  // forms X[j0 + TT k] of row r0 + rr, so that the block's rows go out side by side
  const int j0 = threadIdx.x / RPB, rr = threadIdx.x - j0 * RPB;
  const I2* shr = sh0 + rr * SH;
  I2* out = spec + r0 + rr;
#pragma unroll
  for (int k = 0; k < R; ++k) {
    const int j = j0 + TT * k;
    const I2 za = shr[padi<3>(j)], zb = shr[padi<3>((N - j) & (N - 1))];
    const I2 Ev = I2{mean(za.x, zb.x), mean(za.y, -zb.y)};
    const I2 Od = I2{mean(za.y, zb.y), mean(zb.x, -za.x)};   // -i (za - zb*) / 2
    out[(size_t)j * N] = cadd(Ev, twmul<false>(Od, tw[j]));
  }
  if (j0 == 0) {
    const I2 z0 = shr[0];
    out[(size_t)N * N] = I2{z0.x - z0.y, 0};
  }
}

template <int LOGM>
__global__ void __launch_bounds__((fix_cols<LOGM>() * Plan<LOGM, 3>::T))
k_col_x(I2* __restrict__ spec, int* __restrict__ fexp, const double* __restrict__ table, const int4* __restrict__ twc,
        int nslots) {
  using P = Plan<LOGM, 3>;
  constexpr int M = 1 << LOGM, N = M / 2, TT = P::T, SH = fix_sh<LOGM>(), R = P::R, CPB = fix_cols<LOGM>();
  pdl_enter();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int red[CPB][kRedWords];
  const int c = threadIdx.x / TT, t = threadIdx.x - c * TT;
  const int slot = blockIdx.x * CPB + c;   // frequency column j
  const bool active = slot < nslots;
  I2* sh = reinterpret_cast<I2*>(smem_raw) + c * SH;
  I2* col = spec + (size_t)slot * N;
  I2 v[R];
  Bound b;
  {
    unsigned a[R / 2];
    int e[R / 2];
#pragma unroll
    for (int q = 0; q < R / 2; ++q) {
      v[q] = active ? col[t + TT * q] : I2{0, 0};
      e[q] = active ? fexp[t + TT * q] : 0;
      a[q] = nonzero(v[q]) || is_nan_exp(e[q]) ? mag(v[q]) : 0u;
    }
    // units of mag are 2^32 of v's last place, which is 2^(e - 62)
    b = l1_exponent<TT, CPB>(a, e, red[c], t, c);
    b = Bound{b.max - 30, b.sum - 30};
    const int E0 = stage_exponent<LOGM, true>(b, 0);
#pragma unroll
    for (int q = 0; q < R / 2; ++q) v[q] = I2{shift(v[q].x, e[q] - E0), shift(v[q].y, e[q] - E0)};
  }
#pragma unroll
  for (int q = R / 2; q < R; ++q) v[q] = I2{0, 0};
  fix_fft<LOGM, false, true, CPB>(v, b, sh, twc, t, c);
  {
    const double* kt = table + (size_t)slot * (N + 4);   // row j = slot of the square table (stride N + 4)
    unsigned a[R];
    int e[R];
#pragma unroll
    for (int q = 0; q < R; ++q) {
      const int i = t + TT * q;
      const int f = (q < R / 2) ? i : M - i;
      // K^ = +-m 2^(x - 62), m in [2^61, 2^62) (a subnormal or zero entry: smaller)
      const double kv = active ? kt[f] : 0.0;
      const unsigned hi = (unsigned)__double2hiint(kv);
      const int x = (int)((hi >> 20) & 0x7ffu);
      i64 m = (((i64)((hi & 0xfffffu) | (x != 0 ? 0x100000u : 0u)) << 32) | (unsigned)__double2loint(kv)) << 9;
      if ((int)hi < 0) m = -m;
      int wh, wl;
      halves(m, wh, wl);
      v[q] = I2{mulr(v[q].x, wh, wl), mulr(v[q].y, wh, wl)};
      e[q] = (x == 2047 ? kNanExp : (x != 0 ? x : 1) - 1022) + b.sum;
      a[q] = nonzero(v[q]) || is_nan_exp(e[q]) ? mag(v[q]) : 0u;
    }
    b = l1_exponent<TT, CPB>(a, e, red[c], t, c);
    b = Bound{b.max - 30, b.sum - 30};
    const int E0 = stage_exponent<LOGM, false>(b, 0);
#pragma unroll
    for (int q = 0; q < R; ++q) v[q] = I2{shift(v[q].x, e[q] - E0), shift(v[q].y, e[q] - E0)};
  }
  fix_fft<LOGM, true, false, CPB>(v, b, sh, twc, t, c);
  if (active) {
#pragma unroll
    for (int q = 0; q < R / 2; ++q) col[t + TT * q] = v[q];
    if (t == 0) fexp[N + slot] = b.sum;
  }
}

__device__ __forceinline__ void cp_async_rec(I2* smem, const I2* gmem) {
  const unsigned a = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(a), "l"(gmem) : "memory");
}

template <int LOGN>
__global__ void __launch_bounds__((fix_rows<LOGN>() * Plan<LOGN, 3>::T))
k_row_inv_x(const I2* __restrict__ spec, const int* __restrict__ fexp, double* __restrict__ u,
            const int4* __restrict__ twr, const int4* __restrict__ tw) {
  using P = Plan<LOGN, 3>;
  constexpr int N = 1 << LOGN, TT = P::T, SH = fix_sh<LOGN>(), R = P::R, RPB = fix_rows<LOGN>(), NT = RPB * TT;
  pdl_enter();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int red[RPB][kRedWords];
  I2* const sh0 = reinterpret_cast<I2*>(smem_raw);
  const int rl = threadIdx.x / TT, t = threadIdx.x - rl * TT;
  const int r0 = blockIdx.x * RPB;
  I2* sh = sh0 + rl * SH;
  const I2* in = spec + r0;
#pragma unroll
  for (int k = 0; k < (RPB * (N + 1) + NT - 1) / NT; ++k) {
    const int e = threadIdx.x + NT * k;
    if (e < RPB * (N + 1)) {
      const int j = e / RPB, rr = e - j * RPB;
      cp_async_rec(sh0 + rr * SH + j, in + (size_t)j * N + rr);
    }
  }
  const int* ce = fexp + N;
  int e[2 * R];
#pragma unroll
  for (int q = 0; q < R; ++q) {
    e[2 * q] = ce[t + TT * q];
    e[2 * q + 1] = ce[N - (t + TT * q)];
  }
  asm volatile("cp.async.wait_all;\n" ::: "memory");
  __syncthreads();
  // Zi[j] = (Y[j] + Y*[N-j]) + i e^{+i pi j/N} (Y[j] - Y*[N-j]): at most twice the moduli
  unsigned a[2 * R];
#pragma unroll
  for (int q = 0; q < R; ++q) {
    const I2 y1 = sh[t + TT * q], y2 = sh[N - (t + TT * q)];
    a[2 * q] = nonzero(y1) || is_nan_exp(e[2 * q]) ? mag(y1) : 0u;
    a[2 * q + 1] = nonzero(y2) || is_nan_exp(e[2 * q + 1]) ? mag(y2) : 0u;
  }
  Bound b = l1_exponent<TT, RPB>(a, e, red[rl], t, rl);
  b = Bound{b.max - 30 + 2, b.sum - 30 + 1};   // |Zi| <= 2 (|y1| + |y2|)
  const int E0 = stage_exponent<LOGN, false>(b, 0), E = b.sum;
  I2 v[R];
#pragma unroll
  for (int q = 0; q < R; ++q) {
    const int j = t + TT * q;
    I2 y1 = sh[j], y2 = sh[N - j];
    y1 = I2{shift(y1.x, e[2 * q] - E0), shift(y1.y, e[2 * q] - E0)};
    y2 = I2{shift(y2.x, e[2 * q + 1] - E0), shift(y2.y, e[2 * q + 1] - E0)};
    const I2 d = twmul<true>(I2{y1.x - y2.x, y1.y + y2.y}, tw[j]);
    v[q] = I2{y1.x + y2.x - d.y, y1.y - y2.y + d.x};
  }
  __syncthreads();
  fix_fft<LOGN, true, false, RPB>(v, b, sh, twr, t, rl);
  double2* urow = reinterpret_cast<double2*>(u + (size_t)(r0 + rl) * N);
  const double bad = __hiloint2double(0x7ff80000, 0);
  const bool nan = is_nan_exp(E);
#pragma unroll
  for (int q = 0; q < R / 2; ++q)
    urow[t + TT * q] = nan ? make_double2(bad, bad) : make_double2(from_fix(v[q].x, E), from_fix(v[q].y, E));
}

// All twiddles of a handle in one launch, one per thread (the Taylor sums are chains of FP64
// operations, so blocks of one warp spread them over the SMs): tw[j] = e^{-2 pi i j / M},
// j < M = 2N, then the stage tables of the lengths N and M, L - 8 records each.
__global__ void __launch_bounds__(32) k_twiddles_fix(int4* __restrict__ tw, int4* __restrict__ twr, int4* __restrict__ twc,
                                                     int logn) {
  const int N = 1 << logn, M = 2 * N;
  int i = blockIdx.x * 32 + threadIdx.x;
  if (i < M) {
    tw[i] = fix_twiddle(i, M);
    return;
  }
  i -= M;
  const bool rows = i < N - 8;
  if (!rows) i -= N - 8;
  if (i >= M - 8) return;
  int4* out = (rows ? twr : twc) + i;
  const int logl = rows ? logn : logn + 1;
  int ns = 8, s = 1;   // stage s: planes r = 1 .. Q - 1 of ns records
  for (;; ++s) {
    const int Q = s < logl / 3 ? 8 : 1 << (logl % 3);
    if (i < (Q - 1) * ns) {
      *out = fix_twiddle((i % ns) * (i / ns + 1), ns * Q);
      return;
    }
    i -= (Q - 1) * ns;
    ns *= Q;
  }
}

template <int LOGN>
struct Fix {
  static constexpr int N = 1 << LOGN, rpb = fix_rows<LOGN>(), cpb = fix_cols<LOGN + 1>();
  static constexpr size_t row_smem = (size_t)rpb * fix_sh<LOGN>() * sizeof(I2);
  static constexpr size_t col_smem = (size_t)cpb * fix_sh<LOGN + 1>() * sizeof(I2);
  static void prepare() {
    static std::atomic<unsigned long long> attr{0};
    if (first_on_device(attr)) {
      cudaFuncSetAttribute(k_row_fwd_x<LOGN>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)row_smem);
      cudaFuncSetAttribute(k_row_inv_x<LOGN>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)row_smem);
      cudaFuncSetAttribute(k_col_x<LOGN + 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)col_smem);
    }
  }
  static void pass(const bem_kernel_s* k, int which, const double* p, double* u, cudaStream_t s) {
    prepare();
    I2* spec = (I2*)k->ws.spec;
    const int4 *tw = (const int4*)k->ws.twf, *twr = tw + k->M, *twc = twr + stage_tw_count(LOGN);
    constexpr int rt = rpb * Plan<LOGN, 3>::T, ct = cpb * Plan<LOGN + 1, 3>::T;
    if (which == 0)
      launch_pdl(k_row_fwd_x<LOGN>, N / rpb, rt, row_smem, s, p, spec, k->ws.fexp, twr, tw);
    else if (which == 1)
      launch_pdl(k_col_x<LOGN + 1>, (N + cpb) / cpb, ct, col_smem, s, spec, k->ws.fexp, (const double*)k->ws.table, twc,
                 N + 1);
    else
      launch_pdl(k_row_inv_x<LOGN>, N / rpb, rt, row_smem, s, (const I2*)spec, (const int*)k->ws.fexp, u, twr, tw);
  }
};

template <typename F>
void with_logn(int logn, F&& f) {
  switch (logn) {
    case 4: f(Fix<4>{}); break;
    case 5: f(Fix<5>{}); break;
    case 6: f(Fix<6>{}); break;
    case 7: f(Fix<7>{}); break;
    case 8: f(Fix<8>{}); break;
    case 9: f(Fix<9>{}); break;
    case 10: f(Fix<10>{}); break;
    case 11: f(Fix<11>{}); break;
    default: break;
  }
}

}  // namespace fx

void fix_pass(const bem_kernel_s* k, int which, const double* p, double* u, cudaStream_t s) {
  fx::with_logn(k->logN, [&](auto f) { f.pass(k, which, p, u, s); });
}

size_t fix_tw_bytes(const bem_kernel_s* k) {
  return ((size_t)k->M + stage_tw_count(k->logN) + stage_tw_count(k->logN + 1)) * sizeof(int4);
}

// twiddles of the recombination and of the stages of both lengths: they depend on N only
void fix_twiddles(const bem_kernel_s* k, cudaStream_t s) {
  int4 *tw = (int4*)k->ws.twf, *twr = tw + k->M, *twc = twr + stage_tw_count(k->logN);
  fx::k_twiddles_fix<<<(2 * k->M + k->N + 31) / 32, 32, 0, s>>>(tw, twr, twc, k->logN);
  note_launches(1);
}
}  // namespace bem
