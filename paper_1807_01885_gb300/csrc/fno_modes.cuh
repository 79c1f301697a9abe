// The spectral branch along x and over the channels: truncated transforms along x of the
// rows' modes and the per-mode channel mixing (included by fno.cu, inside its anonymous
// namespace).  tw[k] = e^{-2 pi i k / N}; the kept wave numbers are kx = 0 .. m-1 (index
// kx) and kx = -m .. -1 (index 2m + kx).
//
// Both transforms are sums over x (or kx) of O(m^2 N) complex products per channel, so
// the arithmetic is small and the work is in feeding it.  Wave numbers come in pairs
// +-k that share their products with cos and sin, which halves the multiply-adds, and
// each thread keeps a register tile (2 ky x 4 k, or 2 ky x 4 x), so that one 16-byte and
// four 8-byte shared-memory reads serve 32 multiply-adds.
// The twiddles come from a table in the order of use, twx[x][k] = tw[k x mod N] for k in
// [0, m] (rows of dft_x_kt(m), the rest 0), so that staging them is a plain copy.
// (One thread per output and a twiddle load per product took 80 and 60 us for 512 channels
// of N = 256, m = 16; twiddles gathered by every block 28 and 20 us.)
#pragma once

constexpr int kXRows = 64;        // rows x per block of the inverse
// rows x that the forward transform stages at a time: few modes leave room for more, and
// their many slices want them (m = 4 with 64 rows was no faster than the gathered form)
__host__ __device__ inline int dft_x_rows(int m) { return m <= 4 ? 256 : (m <= 12 ? 128 : 64); }
constexpr int kXModes = 32;       // most modes per axis that the tiled kernels take
constexpr int kXBlocks = 912;     // blocks that fill the GPU (six per SM)

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

// blocks per channel along x of k_dft_x (each adds its share of the rows)
inline int dft_x_chunks(size_t bc, int N, int m) {
  const size_t tiles = (N + dft_x_rows(m) - 1) / dft_x_rows(m), want = (kXBlocks + bc - 1) / bc;
  return (int)std::min(tiles, std::max<size_t>(want, 1));
}

// Xp[chunk][q][kxi][ky] = wky[ky] sum over the chunk's rows x of A[q][x][ky] e^{-2 pi i kx x / N}
__global__ void __launch_bounds__(256) k_dft_x(const float2* __restrict__ A, float2* __restrict__ Xp,
                                               const float2* __restrict__ twx, const float* __restrict__ wky, int N,
                                               int m) {
  __shared__ __align__(16) float smem[64 * (kXModes * 2 + 36 * 2)];   // rows (2 ky2 + kt) float2 at every m, and 256 x 32
  const int rows = dft_x_rows(m);
  const int ky2 = (m + 1) / 2, kg = (m + 4) / 4, kt = dft_x_kt(m), items = ky2 * kg, S = 256 / items;
  float2* const sA = reinterpret_cast<float2*>(smem);                  // [rows][2 ky2]
  float2* const sT = sA + rows * 2 * ky2;                              // [rows][kt]
  const size_t q = blockIdx.x;
  const int tid = threadIdx.x, slice = tid / items, item = tid - slice * items;
  const int kyp = item % ky2, k0 = 4 * (item / ky2);
  const int tiles = (N + rows - 1) / rows;
  const int t0 = (int)((long long)tiles * blockIdx.y / gridDim.y), t1 = (int)((long long)tiles * (blockIdx.y + 1) / gridDim.y);
  // sums of re wx, im wy, re wy, im wx for 4 k and 2 ky
  float acc[4][2][4] = {};
  for (int tile = t0; tile < t1; ++tile) {
    const int x0 = tile * rows, nx = min(rows, N - x0);
    __syncthreads();
    if (m % 2 == 0) {
      const float4* a = reinterpret_cast<const float4*>(A + (q * N + x0) * m);
      for (int e = tid; e < nx * ky2; e += 256) reinterpret_cast<float4*>(sA)[e] = a[e];
    } else {
      for (int e = tid; e < nx * 2 * ky2; e += 256) {
        const int x = e / (2 * ky2), ky = e - x * 2 * ky2;
        sA[e] = ky < m ? A[(q * N + x0 + x) * m + ky] : make_float2(0.f, 0.f);
      }
    }
    for (int e = tid; e < nx * kt / 2; e += 256)
      reinterpret_cast<float4*>(sT)[e] = reinterpret_cast<const float4*>(twx + (size_t)x0 * kt)[e];
    __syncthreads();
    if (slice < S) {
      for (int x = slice; x < nx; x += S) {
        const float4 v = *reinterpret_cast<const float4*>(sA + x * 2 * ky2 + 2 * kyp);
        const float4* tp = reinterpret_cast<const float4*>(sT + x * kt + k0);
        const float4 wa = tp[0], wb = tp[1];
        const float wx[4] = {wa.x, wa.z, wb.x, wb.z}, wy[4] = {wa.y, wa.w, wb.y, wb.w};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          acc[k][0][0] = fmaf(v.x, wx[k], acc[k][0][0]);
          acc[k][0][1] = fmaf(v.y, wy[k], acc[k][0][1]);
          acc[k][0][2] = fmaf(v.x, wy[k], acc[k][0][2]);
          acc[k][0][3] = fmaf(v.y, wx[k], acc[k][0][3]);
          acc[k][1][0] = fmaf(v.z, wx[k], acc[k][1][0]);
          acc[k][1][1] = fmaf(v.w, wy[k], acc[k][1][1]);
          acc[k][1][2] = fmaf(v.z, wy[k], acc[k][1][2]);
          acc[k][1][3] = fmaf(v.w, wx[k], acc[k][1][3]);
        }
      }
    }
  }
  // the slices' sums, added in slice order; red[(slice 32 + j) items + item]
  __syncthreads();
  float* const red = smem;
  if (slice < S) {
#pragma unroll
    for (int k = 0; k < 4; ++k)
#pragma unroll
      for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int e = 0; e < 4; ++e) red[(slice * 32 + (k * 2 + h) * 4 + e) * items + item] = acc[k][h][e];
  }
  __syncthreads();
  for (int o = tid; o < items * 32; o += 256) {
    float s = red[o];
    for (int sl = 1; sl < S; ++sl) s += red[sl * 32 * items + o];
    red[o] = s;
  }
  __syncthreads();
  float2* out = Xp + ((size_t)blockIdx.y * gridDim.x + q) * 2 * m * m;
  for (int o = tid; o < items * 8; o += 256) {
    const int it = o % items, kh = o / items;
    const int k = 4 * (it / ky2) + kh / 2, ky = 2 * (it % ky2) + (kh & 1);
    if (k > m || ky >= m) continue;
    const float* s = red + kh * 4 * items + it;
    const float sc = wky != nullptr ? wky[ky] : 1.f;
    if (k < m) out[k * m + ky] = make_float2((s[0] - s[items]) * sc, (s[2 * items] + s[3 * items]) * sc);
    if (k > 0) out[(2 * m - k) * m + ky] = make_float2((s[0] + s[items]) * sc, (s[3 * items] - s[2 * items]) * sc);
  }
}

// A[q][x][ky] = sum_kxi Y[q][kxi][ky] e^{+2 pi i kx x / N}: block (channel, kXRows rows)
inline size_t idft_x_smem(int m) {
  return (size_t)(m + 1) * (2 * ((m + 1) / 2)) * sizeof(float4) + (size_t)kXRows * dft_x_kt(m) * sizeof(float2);
}
__global__ void __launch_bounds__(256) k_idft_x(const float2* __restrict__ Y, float2* __restrict__ A,
                                                const float2* __restrict__ twx, int N, int m) {
  extern __shared__ __align__(16) float4 sY[];                    // [m + 1][2 ky2]: Y+ + Y-, Y+ - Y-
  const size_t q = blockIdx.x;
  const int x0 = blockIdx.y * kXRows, nx = min(kXRows, N - x0);
  const int ky2 = (m + 1) / 2, row = 2 * ky2, kt = dft_x_kt(m);
  float2* const sT = reinterpret_cast<float2*>(sY + (m + 1) * row);   // [x][kt]
  const float2* y = Y + q * 2 * m * m;
  for (int e = threadIdx.x; e < (m + 1) * row; e += blockDim.x) {
    const int k = e / row, ky = e - k * row;
    const float2 a = (k < m && ky < m) ? y[k * m + ky] : make_float2(0.f, 0.f);
    const float2 b = (k > 0 && ky < m) ? y[(2 * m - k) * m + ky] : make_float2(0.f, 0.f);
    sY[e] = make_float4(a.x + b.x, a.y + b.y, a.x - b.x, a.y - b.y);
  }
  for (int e = threadIdx.x; e < nx * kt / 2; e += blockDim.x)
    reinterpret_cast<float4*>(sT)[e] = reinterpret_cast<const float4*>(twx + (size_t)x0 * kt)[e];
  __syncthreads();
  for (int it = threadIdx.x; it < ky2 * (kXRows / 4); it += blockDim.x) {
    const int kyp = it % ky2, xl = 4 * (it / ky2);
    if (xl >= nx) continue;
    float o[4][4] = {};
    for (int k = 0; k <= m; ++k) {
      const float4 y0 = sY[k * row + 2 * kyp], y1 = sY[k * row + 2 * kyp + 1];
      float wx[4], wy[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const float2 w = sT[min(xl + e, nx - 1) * kt + k];
        wx[e] = w.x;
        wy[e] = w.y;
      }
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        o[e][0] = fmaf(y0.w, wy[e], fmaf(y0.x, wx[e], o[e][0]));
        o[e][1] = fmaf(-y0.z, wy[e], fmaf(y0.y, wx[e], o[e][1]));
        o[e][2] = fmaf(y1.w, wy[e], fmaf(y1.x, wx[e], o[e][2]));
        o[e][3] = fmaf(-y1.z, wy[e], fmaf(y1.y, wx[e], o[e][3]));
      }
    }
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

// Per-mode channel mixing of 32 modes and kMixB samples per block, the samples' modes in
// shared memory (the chunks of k_dft_x are added on the way in, and kept in Xh when
// there is more than one):  CONJ false: Y[b][o] = sum_i X[b][i] R[i][o];  CONJ true, the
// data gradient: Y[b][i] = sum_o X[b][o] conj(R[i][o]).  A warp forms OPW outputs.
constexpr int kMixB = 2;
template <int OPW, bool CONJ>
__global__ void __launch_bounds__(256) k_mix(const float2* __restrict__ Xp, int chunks, float2* __restrict__ Xh,
                                             const bf16* __restrict__ Rre, const bf16* __restrict__ Rim,
                                             float2* __restrict__ Y, int W, int nm, int B) {
  __shared__ float2 xs[kMixB][64][32];
  const int lane = threadIdx.x % 32, wid = threadIdx.x / 32;
  const int mode = blockIdx.x * 32 + lane, b0 = blockIdx.y * kMixB;
  const bool on = mode < nm;
  const size_t all = (size_t)B * W * nm;
  for (int r = wid; r < kMixB * W; r += 8) {
    const int bb = r / W, c = r - bb * W;
    float2 v = make_float2(0.f, 0.f);
    if (on && b0 + bb < B) {
      const size_t at = ((size_t)(b0 + bb) * W + c) * nm + mode;
      v = Xp[at];
      for (int k = 1; k < chunks; ++k) {
        const float2 u = Xp[k * all + at];
        v.x += u.x;
        v.y += u.y;
      }
      if (chunks > 1 && Xh != nullptr && blockIdx.z == 0) Xh[at] = v;
    }
    xs[bb][c][lane] = v;
  }
  __syncthreads();
  if (!on) return;
  const int o0 = (blockIdx.z * 8 + wid) * OPW;
  if (o0 >= W) return;
  float2 acc[kMixB][OPW] = {};
#pragma unroll 4
  for (int c = 0; c < W; ++c) {
#pragma unroll
    for (int j = 0; j < OPW; ++j) {
      const int o = min(o0 + j, W - 1);
      const size_t r = (CONJ ? (size_t)o * W + c : (size_t)c * W + o) * nm + mode;
      const float rr = b2f(Rre[r]), ri = CONJ ? -b2f(Rim[r]) : b2f(Rim[r]);
#pragma unroll
      for (int bb = 0; bb < kMixB; ++bb) {
        const float2 x = xs[bb][c][lane];
        acc[bb][j].x += x.x * rr - x.y * ri;
        acc[bb][j].y += x.x * ri + x.y * rr;
      }
    }
  }
#pragma unroll
  for (int bb = 0; bb < kMixB; ++bb)
#pragma unroll
    for (int j = 0; j < OPW; ++j)
      if (b0 + bb < B && o0 + j < W) Y[((size_t)(b0 + bb) * W + o0 + j) * nm + mode] = acc[bb][j];
}

template <bool CONJ>
void mix(const float2* Xp, int chunks, float2* Xh, const bf16* Rre, const bf16* Rim, float2* Y, int W, int nm, int B,
         cudaStream_t s) {
  // two outputs per warp; one where that leaves the GPU with few blocks
  const dim3 g((nm + 31) / 32, (B + kMixB - 1) / kMixB);
  if (g.x * g.y >= 128) k_mix<2, CONJ><<<dim3(g.x, g.y, (W + 15) / 16), 256, 0, s>>>(Xp, chunks, Xh, Rre, Rim, Y, W, nm, B);
  else k_mix<1, CONJ><<<dim3(g.x, g.y, (W + 7) / 8), 256, 0, s>>>(Xp, chunks, Xh, Rre, Rim, Y, W, nm, B);
}
