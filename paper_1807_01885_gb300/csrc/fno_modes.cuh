// The spectral branch along x: truncated transforms along x of the rows' modes (included by
// fno.cu, inside its anonymous namespace; the kernels of fno.cu for any number of modes
// give the same results).  tw[k] = e^{-2 pi i k / N}; the kept wave numbers are kx = 0 .. m-1 (index
// kx) and kx = -m .. -1 (index 2m + kx).
//
// Both transforms are sums over x (or kx) of O(m^2 N) complex products per channel, so
// the arithmetic is small and the work is in feeding it: rows and twiddles are staged in
// shared memory and each thread keeps a register tile (2 ky x 4 pairs +-k, or 2 ky x 4 x).
// The twiddles come from a table in the order of use, twx[x][k] = tw[k x mod N] for k in
// [0, m] (rows of dft_x_kt(m), the rest 0), so that staging them is a plain copy.
// Every sum keeps one fixed order and form: the forward one adds the products of the rows
// x = sl, sl + S, ... of each of S = 256 / m slices and then the slices in order, the
// inverse one the kept wave numbers in the order of their index.  (Sharing the products
// with cos and sin between the sums of +k and -k needs 40 % of the multiply-adds, but
// rounds differently, and a network's output can be a small difference of its hidden
// values: a pressure cut at zero then moved by up to 1e-3 of its rms.)
// Measured on GB300, 512 channels of N = 256, m = 16, one thread per output with a twiddle
// load per product / tiled: forward 80 / 43 us, inverse 60 / 22 us (1024 channels, tiled:
// 75 and 38).
#pragma once

constexpr int kXRows = 64;        // rows x per block of the inverse
constexpr int kXSmem = 36864;     // bytes of shared memory of the forward transform (128 rows at 16 modes)
constexpr int kXModes = 32;       // most modes per axis that the tiled kernels take

// row length of the twiddle table: k in [0, m], rounded up to groups of four
__host__ __device__ inline int dft_x_kt(int m) { return 4 * ((m + 4) / 4); }

__global__ void k_twiddle_x(const float2* __restrict__ tw, float2* __restrict__ twx, int N, int m) {
  const int kt = dft_x_kt(m);
  FOR_N(i, (size_t)N * kt) {
    const unsigned k = (unsigned)(i % kt);
    const size_t x = i / kt;
    twx[i] = (int)k <= m ? tw[(k * x) % (size_t)N] : make_float2(0.f, 0.f);
  }
}

// Forward transform's shape for m modes: items = register tiles, S slices of the rows, SB of
// them at a time per block (SB items threads, at most 384), I rows of each slice staged
struct DftX {
  int ky2, kt, items, S, SB, I;
  __host__ __device__ explicit DftX(int m) {
    ky2 = (m + 1) / 2;
    kt = dft_x_kt(m);
    items = ky2 * (kt / 4);
    S = 256 / m;
    const int most = 384 / items, g = (S + most - 1) / most;
    SB = (S + g - 1) / g;
    const int rows = kXSmem / (8 * (2 * ky2 + kt));
    I = rows / SB < 1 ? 1 : (rows / SB > 32 ? 32 : rows / SB);
  }
  __host__ __device__ int groups() const { return (S + SB - 1) / SB; }
};
// Where the tiled kernels are the faster ones.  Forward: a block per channel has to fill the
// GPU and the modes its threads (m = 16, N = 256, 512 channels: 80 -> 43 us; predictions of
// one sample of N = 164, m = 8, were 30 % slower with it, 32 channels of N = 2048 5 %).
// Inverse: the same for blocks of 64 rows.
inline bool dft_x_tiled(size_t bc, int m) { return m >= 12 && m <= kXModes && bc >= 304; }
inline bool idft_x_tiled(size_t bc, int m, int N) {
  return m >= 12 && m <= kXModes && bc * ((N + kXRows - 1) / kXRows) >= 304;
}

// X[q][kxi][ky] = wky[ky] sum_x A[q][x][ky] e^{-2 pi i kx x / N}: a block per channel
__global__ void __launch_bounds__(384, 2) k_dft_x(const float2* __restrict__ A, float2* __restrict__ X,
                                               const float2* __restrict__ twx, const float* __restrict__ wky, int N,
                                               int m) {
  __shared__ __align__(16) unsigned char smem[kXSmem];
  const DftX d(m);
  const int rows = d.SB * d.I, kt = d.kt, ky2 = d.ky2, items = d.items;
  float2* const sA = reinterpret_cast<float2*>(smem);     // [I][SB][2 ky2]
  float2* const sT = sA + rows * 2 * ky2;                 // [I][SB][kt]
  float2* const red = reinterpret_cast<float2*>(smem);    // [SB][8][items] of one pair sign
  const size_t q = blockIdx.x, nm = 2 * (size_t)m * m;
  const int tid = threadIdx.x, sl = tid / items, item = tid - sl * items;
  const int kyp = item % ky2, k0 = 4 * (item / ky2);
  const int steps = (N + d.S - 1) / d.S;
  const int ca = tid % ky2, step_a = blockDim.x / ky2, ct = tid % (kt / 2), step_t = blockDim.x / (kt / 2);
  const unsigned magic = ((1u << 20) + d.SB - 1) / d.SB;   // r / SB = r magic 2^-20 for the rows staged
  const int groups = d.groups();
  const int nout = items * 8;
  float2 tot[2][4];
  for (int gr = 0; gr < groups; ++gr) {
    const int s0 = gr * d.SB, ns = min(d.SB, d.S - s0);
    float2 ap[4][2] = {}, an[4][2] = {};   // sums for +k and -k
    for (int i0 = 0; i0 < steps; i0 += d.I) {
      const int ni = min(d.I, steps - i0);
      __syncthreads();
      // a record of two ky, or two twiddles, per thread and row (threads past the last whole
      // row stage nothing)
      if (tid < step_a * ky2) {
        for (int r = tid / ky2; r < ni * d.SB; r += step_a) {
          const int i = (int)(((unsigned)r * magic) >> 20), c = r - i * d.SB, x = (i0 + i) * d.S + s0 + c;
          float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
          if (x < N && c < ns) {
            const float2* a = A + (q * N + x) * m + 2 * ca;
            if (m % 2 == 0) {
              v = *reinterpret_cast<const float4*>(a);
            } else {
              v.x = a[0].x; v.y = a[0].y;
              if (2 * ca + 1 < m) { v.z = a[1].x; v.w = a[1].y; }
            }
          }
          reinterpret_cast<float4*>(sA)[r * ky2 + ca] = v;
        }
      }
      if (tid < step_t * (kt / 2)) {
        for (int r = tid / (kt / 2); r < ni * d.SB; r += step_t) {
          const int i = (int)(((unsigned)r * magic) >> 20), c = r - i * d.SB, x = (i0 + i) * d.S + s0 + c;
          if (x < N && c < ns)
            reinterpret_cast<float4*>(sT)[r * (kt / 2) + ct] = reinterpret_cast<const float4*>(twx + (size_t)x * kt)[ct];
        }
      }
      __syncthreads();
      if (sl < ns) {
        for (int i = 0; i < ni; ++i) {
          if ((i0 + i) * d.S + s0 + sl >= N) break;
          const int r = i * d.SB + sl;
          const float4 v = *reinterpret_cast<const float4*>(sA + r * 2 * ky2 + 2 * kyp);
          const float4* tp = reinterpret_cast<const float4*>(sT + r * kt + k0);
          const float4 wa = tp[0], wb = tp[1];
          const float wx[4] = {wa.x, wa.z, wb.x, wb.z}, wy[4] = {wa.y, wa.w, wb.y, wb.w};
#pragma unroll
          for (int k = 0; k < 4; ++k)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              const float vx = h ? v.z : v.x, vy = h ? v.w : v.y;
              ap[k][h].x += vx * wx[k] - vy * wy[k];
              ap[k][h].y += vx * wy[k] + vy * wx[k];
              an[k][h].x += vx * wx[k] - vy * -wy[k];
              an[k][h].y += vx * -wy[k] + vy * wx[k];
            }
        }
      }
    }
    // the slices' sums, added in slice order
#pragma unroll
    for (int sign = 0; sign < 2; ++sign) {
      __syncthreads();
      if (sl < ns) {
#pragma unroll
        for (int k = 0; k < 4; ++k)
#pragma unroll
          for (int h = 0; h < 2; ++h) red[(sl * 8 + k * 2 + h) * items + item] = sign ? an[k][h] : ap[k][h];
      }
      __syncthreads();
      // output o: tile it, pair and ky kh; false where there is none
      auto place = [&](int o, size_t& at, int& ky) {
        const int it = o % items, kh = o / items, k = 4 * (it / ky2) + kh / 2;
        ky = 2 * (it % ky2) + (kh & 1);
        at = q * nm + (size_t)(sign ? 2 * m - k : k) * m + ky;
        return ky < m && (sign ? (k >= 1 && k <= m) : k < m);
      };
      size_t at;
      int ky;
#pragma unroll
      for (int o4 = 0; o4 < 4; ++o4) {   // (at most 4 outputs per thread and sign)
        const int o = tid + o4 * blockDim.x;
        if (o >= nout) break;
        if (!place(o, at, ky)) continue;
        float2 t = gr > 0 ? tot[sign][o4] : red[o];
        for (int c = gr > 0 ? 0 : 1; c < ns; ++c) {
          const float2 u = red[c * nout + o];
          t = make_float2(t.x + u.x, t.y + u.y);
        }
        tot[sign][o4] = t;
        if (gr + 1 == groups) {
          const float sc = wky != nullptr ? wky[ky] : 1.f;
          X[at] = make_float2(t.x * sc, t.y * sc);
        }
      }
    }
  }
}

// A[q][x][ky] = sum_kxi Y[q][kxi][ky] e^{+2 pi i kx x / N}: block (channel, kXRows rows)
inline size_t idft_x_smem(int m) {
  return (size_t)2 * m * ((m + 1) / 2) * sizeof(float4) + (size_t)kXRows * dft_x_kt(m) * sizeof(float2);
}
__global__ void __launch_bounds__(256) k_idft_x(const float2* __restrict__ Y, float2* __restrict__ A,
                                                const float2* __restrict__ twx, int N, int m) {
  extern __shared__ __align__(16) float4 sY[];                        // [2m][ky2]: two ky per record
  const size_t q = blockIdx.x;
  const int x0 = blockIdx.y * kXRows, nx = min(kXRows, N - x0);
  const int ky2 = (m + 1) / 2, kt = dft_x_kt(m);
  float2* const sT = reinterpret_cast<float2*>(sY + 2 * m * ky2);     // [x][kt]
  const float2* y = Y + q * 2 * m * m;
  for (int e = threadIdx.x; e < 2 * m * ky2; e += blockDim.x) {
    const int k = e / ky2, ky = 2 * (e - k * ky2);
    const float2 a = y[k * m + ky], b = ky + 1 < m ? y[k * m + ky + 1] : make_float2(0.f, 0.f);
    sY[e] = make_float4(a.x, a.y, b.x, b.y);
  }
  for (int e = threadIdx.x; e < nx * kt / 2; e += blockDim.x)
    reinterpret_cast<float4*>(sT)[e] = reinterpret_cast<const float4*>(twx + (size_t)x0 * kt)[e];
  __syncthreads();
  for (int it = threadIdx.x; it < ky2 * (kXRows / 4); it += blockDim.x) {
    const int kyp = it % ky2, xl = 4 * (it / ky2);
    if (xl >= nx) continue;
    float o[4][4] = {};
    auto add = [&](int kxi, int k, bool neg) {
      const float4 v = sY[kxi * ky2 + kyp];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        float2 w = sT[min(xl + e, nx - 1) * kt + k];
        if (neg) w.y = -w.y;
        o[e][0] += v.x * w.x + v.y * w.y;
        o[e][1] += v.y * w.x - v.x * w.y;
        o[e][2] += v.z * w.x + v.w * w.y;
        o[e][3] += v.w * w.x - v.z * w.y;
      }
    };
#pragma unroll 4
    for (int k = 0; k < m; ++k) add(k, k, false);
#pragma unroll 4
    for (int k = m; k > 0; --k) add(2 * m - k, k, true);
    float2* a = A + (q * N + x0 + xl) * m + 2 * kyp;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      if (xl + e >= nx) break;
      if (m % 2 == 0) {
        *reinterpret_cast<float4*>(a + (size_t)e * m) = make_float4(o[e][0], o[e][1], o[e][2], o[e][3]);
      } else {
        a[(size_t)e * m] = make_float2(o[e][0], o[e][1]);
        if (2 * kyp + 1 < m) a[(size_t)e * m + 1] = make_float2(o[e][2], o[e][3]);
      }
    }
  }
}
