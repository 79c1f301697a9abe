// Backward pass of the projection out = Q2 gelu(Q1 v + q1) + q2 in one kernel (included by
// fno.cu, inside its anonymous namespace).
#pragma once

// From v and dout: dv = Q1^T da, and this block's share of dQ1 = da v^T, dq1 = sum da,
// dQ2 = sum dout h, dq2 = sum dout, where a = Q1 v + q1, h = gelu(a), da = dout Q2 gelu'(a).
// The hidden layer (H values per pixel, twice v) is formed again from v instead of being
// stored by the forward pass and read back four times.
//
// A warp takes 16 pixels at a time and keeps hidden units as rows and pixels as columns:
//   a (H x 16)  = Q1 (rows of weights as stored) x v (split hi/lo),
//   dQ1 (H x W) = da (the accumulator layout is the operand layout) x v^T, both in three
//                 parts (24 bits; six products of parts),
//   dv (W x 16) = Q1^T x da.
// v is loaded once in the order of the second product; the first and third need 8 x 8
// blocks transposed, which movmatrix does on the packed bf16 parts.  dQ1 stays in
// registers over all of a warp's tiles (each tile's product is added in float, since the
// unit's accumulators truncate).  With two parts (16 bits) the products' rounding showed in
// dQ1 on small grids, where the sum is short and its terms cancel: error up to 1.17 times
// that of float products at 64 x 64 pixels (geometric mean of 36 networks of up to 16384
// pixels 1.03; with three parts 1.007, gradient pass of 16 x 256 x 256 2.72 -> 2.75 ms).
// Measured (GB300, 16 samples of 256 x 256, W = 32, H = 64): this kernel 244 us (218 with
// two parts); the gradient pass 3.10 -> 2.52 ms, with two parts, against the separate kernels (two layers forward,
// gelu', two data and two weight gradients).
constexpr int kProjBlocks = 304;   // two per SM; one partial of every gradient each

__device__ __forceinline__ unsigned trans8(unsigned x) {   // 8 x 8 b16 block, rows <-> columns
  unsigned d;
  asm("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(d) : "r"(x));
  return d;
}

// x = hi + lo + m in three bf16 parts (24 bits), pairs packed
__device__ __forceinline__ void split3(float x0, float x1, unsigned& hi, unsigned& lo, unsigned& m) {
  split2(x0, x1, hi, lo);
  const float r0 = (x0 - __uint_as_float(hi << 16)) - __uint_as_float(lo << 16);
  const float r1 = (x1 - __uint_as_float(hi & 0xffff0000u)) - __uint_as_float(lo & 0xffff0000u);
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(m) : "f"(r1), "f"(r0));
}

template <int KT, int MH>
__global__ void __launch_bounds__(128, 2)
k_proj_bwd(const float* __restrict__ V, const float* __restrict__ dout, const bf16* __restrict__ Q1,
           const bf16* __restrict__ q1, const bf16* __restrict__ Q2, float* __restrict__ dV, float* __restrict__ part1,
           float* __restrict__ part2, int W, int H, unsigned P, unsigned tiles_per_sample, unsigned tiles) {
  constexpr int NT = 2 * KT;
  __shared__ __align__(16) uint4 sQ[MH][KT][32], sQT[MH][KT][32];
  __shared__ float red[4][16 * MH * 16 * KT];
  __shared__ float red2[4][2][16 * MH];
  __shared__ float redb[4];
  __shared__ float2 sqw[16 * MH];   // (q1, Q2) of hidden unit j
  const int lane = threadIdx.x % 32, g = lane / 4, t = lane % 4, wid = threadIdx.x / 32;
  // operand fragments of Q1 (rows j, k = c) and Q1^T (rows c, k = j)
  auto bits = [&](int j, int c) -> unsigned {
    return (j < H && c < W) ? (unsigned)__bfloat16_as_ushort(Q1[j * W + c]) : 0u;
  };
  for (int i = wid; i < MH * KT; i += 4) {
    const int mt = i / KT, kb = i % KT;
    unsigned a[4], b[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int r = g + 8 * (e & 1), k = 2 * t + 8 * (e >> 1);
      a[e] = bits(16 * mt + r, 16 * kb + k) | (bits(16 * mt + r, 16 * kb + k + 1) << 16);
      b[e] = bits(16 * mt + k, 16 * kb + r) | (bits(16 * mt + k + 1, 16 * kb + r) << 16);
    }
    sQ[mt][kb][lane] = make_uint4(a[0], a[1], a[2], a[3]);
    sQT[mt][kb][lane] = make_uint4(b[0], b[1], b[2], b[3]);
  }
  for (int j = threadIdx.x; j < 16 * MH; j += 128)
    sqw[j] = j < H ? make_float2(b2f(q1[j]), b2f(Q2[j])) : make_float2(0.f, 0.f);
  __syncthreads();
  float dq1[MH][NT][4] = {}, gq1[MH][2] = {}, gq2[MH][2] = {}, gb2 = 0.f;
  for (unsigned tile = blockIdx.x * 4 + wid; tile < tiles; tile += gridDim.x * 4) {
    const unsigned b = tile / tiles_per_sample, p0 = (tile - b * tiles_per_sample) * 16;
    const float* vb = V + (size_t)b * W * P;
    float* db = dV + (size_t)b * W * P;
    // v: packed pairs of pixels 2t, 2t + 1 of rows c = 8 nt + g, in three parts
    unsigned vh[NT][2], vl[NT][2], vm[NT][2];
    float2 go[2];
#pragma unroll
    for (int pt = 0; pt < 2; ++pt) {
      const unsigned p = p0 + 8 * pt + 2 * t;
      go[pt] = p < P ? *reinterpret_cast<const float2*>(dout + (size_t)b * P + p) : make_float2(0.f, 0.f);
      if (g == 0) gb2 += go[pt].x + go[pt].y;
#pragma unroll
      for (int nt = 0; nt < NT; ++nt) {
        const int c = 8 * nt + g;
        const float2 x = (c < W && p < P) ? *reinterpret_cast<const float2*>(vb + (unsigned)c * P + p)
                                          : make_float2(0.f, 0.f);
        split3(x.x, x.y, vh[nt][pt], vl[nt][pt], vm[nt][pt]);
      }
    }
    unsigned th[NT][2], tl[NT][2];   // the same transposed: pixel rows, channel pairs
#pragma unroll
    for (int nt = 0; nt < NT; ++nt)
#pragma unroll
      for (int pt = 0; pt < 2; ++pt) {
        th[nt][pt] = trans8(vh[nt][pt]);
        tl[nt][pt] = trans8(vl[nt][pt]);
      }
    float dv[KT][2][4] = {};
#pragma unroll
    for (int mt = 0; mt < MH; ++mt) {
      unsigned ah[4], al[4], am[4];   // da of rows 16 mt + g (+ 8), pixels 2t, 2t + 1 (+ 8): e = row half + 2 pt
#pragma unroll
      for (int pt = 0; pt < 2; ++pt) {
        float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int kb = 0; kb < KT; ++kb) {
          const uint4 q = sQ[mt][kb][lane];
          const unsigned qa[4] = {q.x, q.y, q.z, q.w};
          mma_bf16(acc, qa, tl[2 * kb][pt], tl[2 * kb + 1][pt]);
          mma_bf16(acc, qa, th[2 * kb][pt], th[2 * kb + 1][pt]);
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const float2 q = sqw[16 * mt + 8 * h + g];
          float h0, h1, d0, d1;
          gelu_both2(acc[2 * h] + q.x, acc[2 * h + 1] + q.x, h0, h1, d0, d1);
          gq2[mt][h] += go[pt].x * h0 + go[pt].y * h1;
          d0 *= go[pt].x * q.y;
          d1 *= go[pt].y * q.y;
          gq1[mt][h] += d0 + d1;
          split3(d0, d1, ah[h + 2 * pt], al[h + 2 * pt], am[h + 2 * pt]);
        }
      }
#pragma unroll
      for (int nt = 0; nt < NT; ++nt) {
        float d[4] = {0.f, 0.f, 0.f, 0.f};
        mma_bf16(d, ah, vm[nt][0], vm[nt][1]);
        mma_bf16(d, am, vh[nt][0], vh[nt][1]);
        mma_bf16(d, al, vl[nt][0], vl[nt][1]);
        mma_bf16(d, ah, vl[nt][0], vl[nt][1]);
        mma_bf16(d, al, vh[nt][0], vh[nt][1]);
        mma_bf16(d, ah, vh[nt][0], vh[nt][1]);
#pragma unroll
        for (int e = 0; e < 4; ++e) dq1[mt][nt][e] += d[e];
      }
#pragma unroll
      for (int pt = 0; pt < 2; ++pt) {
        const unsigned bh0 = trans8(ah[2 * pt]), bh1 = trans8(ah[2 * pt + 1]);
        const unsigned bl0 = trans8(al[2 * pt]), bl1 = trans8(al[2 * pt + 1]);
#pragma unroll
        for (int ct = 0; ct < KT; ++ct) {
          const uint4 q = sQT[mt][ct][lane];
          const unsigned qa[4] = {q.x, q.y, q.z, q.w};
          mma_bf16(dv[ct][pt], qa, bl0, bl1);
          mma_bf16(dv[ct][pt], qa, bh0, bh1);
        }
      }
    }
#pragma unroll
    for (int ct = 0; ct < KT; ++ct)
#pragma unroll
      for (int pt = 0; pt < 2; ++pt)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int c = 16 * ct + 8 * h + g;
          const unsigned p = p0 + 8 * pt + 2 * t;
          if (c < W && p < P)
            *reinterpret_cast<float2*>(db + (unsigned)c * P + p) = make_float2(dv[ct][pt][2 * h], dv[ct][pt][2 * h + 1]);
        }
  }
  // the four warps' sums, added in warp order
  constexpr int WP = 16 * KT;
#pragma unroll
  for (int mt = 0; mt < MH; ++mt) {
#pragma unroll
    for (int nt = 0; nt < NT; ++nt)
#pragma unroll
      for (int e = 0; e < 4; ++e)
        red[wid][(16 * mt + g + 8 * (e >> 1)) * WP + 8 * nt + 2 * t + (e & 1)] = dq1[mt][nt][e];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      float a = gq1[mt][h], c = gq2[mt][h];
#pragma unroll
      for (int o = 1; o <= 2; o <<= 1) {
        a += __shfl_xor_sync(0xffffffffu, a, o);
        c += __shfl_xor_sync(0xffffffffu, c, o);
      }
      if (t == 0) {
        red2[wid][0][16 * mt + 8 * h + g] = a;
        red2[wid][1][16 * mt + 8 * h + g] = c;
      }
    }
  }
  gb2 += __shfl_xor_sync(0xffffffffu, gb2, 1);
  gb2 += __shfl_xor_sync(0xffffffffu, gb2, 2);
  if (lane == 0) redb[wid] = gb2;
  __syncthreads();
  float* o1 = part1 + (size_t)blockIdx.x * (H * W + H);
  float* o2 = part2 + (size_t)blockIdx.x * (H + 1);
  for (int e = threadIdx.x; e < H * W; e += 128) {
    const int i = (e / W) * WP + e % W;
    o1[e] = (red[0][i] + red[1][i]) + (red[2][i] + red[3][i]);
  }
  for (int j = threadIdx.x; j < H; j += 128) {
    o1[H * W + j] = (red2[0][0][j] + red2[1][0][j]) + (red2[2][0][j] + red2[3][0][j]);
    o2[j] = (red2[0][1][j] + red2[1][1][j]) + (red2[2][1][j] + red2[3][1][j]);
  }
  if (threadIdx.x == 0) o2[H] = (redb[0] + redb[1]) + (redb[2] + redb[3]);
}
