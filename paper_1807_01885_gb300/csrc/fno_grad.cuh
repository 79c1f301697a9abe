// Weight gradients of the pointwise layers on the tensor cores (included by fno.cu,
// inside its anonymous namespace).
#pragma once

// gw[o][c] = sum over samples and pixels of dY[b][o][p] X[b][c][p], gb[o] = sum dY[b][o][p].
//
// A contraction over the pixels with at most 64 x 64 outputs: what it cannot do without
// is one read of both arrays, so the kernel is made to stream.  Each warp takes groups of
// 32 consecutive pixels; lane (g, t) loads 8 consecutive pixels (two 16-byte loads) of
// every row it holds, which are at once the fragments of four mma.sync m16n8k8 steps: the
// order of the pixels inside a sum is free, so step s takes elements 2s and 2s + 1 of
// each lane as k = t and k = t + 4, and neither operand needs a transposition.
// Precision: a float is split into two tf32 parts (hi and lo of 11 bits each, rounded:
// 2^-23 of the value is lost) and a product takes hi.hi + hi.lo + lo.hi.  The unit's
// accumulators truncate, so every hi.hi step is added to a float register instead of to
// the next step; the small terms keep an accumulator over the group.  With one
// accumulator for all three, twelve steps long, sums came out about 5e-7 too small.
// Measured (GB300, 16 samples of 256 x 256, 32 x 32 channels): 885 us for the float
// kernel that staged 256 pixels in shared memory and 540 us for the sum of its 4096
// partials, which ran as one chain of loads per output.
constexpr int kWgMT = 2, kWgNT = 4;        // 32 x 32 outputs per block; blockIdx.z walks over larger layers
constexpr int kWgBlocks = 456;             // blocks per 32 x 32 outputs (three per SM): partials to add

// The integer rounding of hi turns 0x7fffffff, the NaN of float instructions, into -0; lo
// is then that NaN, and its conversion keeps it one (an integer add would lose it too), so a
// product with a value that is not finite is NaN.  Gradient pass of 16 x 256 x 256: 2.71 ms,
// 2.74 with the conversion for both parts.
__device__ __forceinline__ void split_tf32(float x, unsigned& hi, unsigned& lo) {
  hi = (__float_as_uint(x) + 0x1000u) & 0xffffe000u;
  asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(lo) : "f"(x - __uint_as_float(hi)));   // (the unit drops the low 13 bits)
}
__device__ __forceinline__ void mma_tf32(float (&d)[4], const unsigned (&a)[4], unsigned b0, unsigned b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
      "{%0, %1, %2, %3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// eight consecutive values from p (n of them exist); VEC: p is 16-byte aligned
template <bool VEC>
__device__ __forceinline__ void load8(const float* p, int n, float (&o)[8]) {
  if (VEC && n >= 8) {
    const float4 a = reinterpret_cast<const float4*>(p)[0], b = reinterpret_cast<const float4*>(p)[1];
    o[0] = a.x; o[1] = a.y; o[2] = a.z; o[3] = a.w;
    o[4] = b.x; o[5] = b.y; o[6] = b.z; o[7] = b.w;
  } else {
#pragma unroll
    for (int e = 0; e < 8; ++e) o[e] = e < n ? p[e] : 0.f;
  }
}

// part[block][cout * cin + cout]: this block's share of the sums (blockIdx.z: its 32 x 32
// outputs; every entry is written by exactly one z)
template <bool VEC>
__global__ void __launch_bounds__(128, 3) k_pw_wgrad_tc(const float* __restrict__ dY, const float* __restrict__ X,
                                                        float* __restrict__ part, int cout, int cin, unsigned P,
                                                        unsigned groups_per_sample, unsigned groups) {
  const int lane = threadIdx.x % 32, g = lane / 4, t = lane % 4, wid = threadIdx.x / 32;
  const int ng = (cin + 31) / 32;
  const int o0 = 32 * (blockIdx.z / ng), c0 = 32 * (blockIdx.z % ng);
  float acc[kWgMT][kWgNT][4], bsum[kWgMT][2];
#pragma unroll
  for (int mt = 0; mt < kWgMT; ++mt) {
    bsum[mt][0] = bsum[mt][1] = 0.f;
#pragma unroll
    for (int nt = 0; nt < kWgNT; ++nt)
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[mt][nt][e] = 0.f;
  }
  for (unsigned gr = blockIdx.x * 4 + wid; gr < groups; gr += gridDim.x * 4) {
    const unsigned b = gr / groups_per_sample;
    const unsigned p = (gr - b * groups_per_sample) * 32 + 8 * t;   // this lane's first pixel
    const int n = p < P ? (int)min(8u, P - p) : 0;
    float xb[kWgNT][8];
#pragma unroll
    for (int nt = 0; nt < kWgNT; ++nt) {
      const int c = c0 + 8 * nt + g;
      load8<VEC>(X + ((size_t)b * cin + (c < cin ? c : 0)) * P + p, c < cin ? n : 0, xb[nt]);
    }
    float ya[kWgMT][2][8];
#pragma unroll
    for (int mt = 0; mt < kWgMT; ++mt)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int o = o0 + 16 * mt + 8 * h + g;
        load8<VEC>(dY + ((size_t)b * cout + (o < cout ? o : 0)) * P + p, o < cout ? n : 0, ya[mt][h]);
        bsum[mt][h] += ((ya[mt][h][0] + ya[mt][h][1]) + (ya[mt][h][2] + ya[mt][h][3])) +
                       ((ya[mt][h][4] + ya[mt][h][5]) + (ya[mt][h][6] + ya[mt][h][7]));
      }
    unsigned ah[4][kWgMT][4], al[4][kWgMT][4];
#pragma unroll
    for (int s = 0; s < 4; ++s)
#pragma unroll
      for (int mt = 0; mt < kWgMT; ++mt)
#pragma unroll
        for (int e = 0; e < 4; ++e) split_tf32(ya[mt][e & 1][2 * s + (e >> 1)], ah[s][mt][e], al[s][mt][e]);
#pragma unroll
    for (int nt = 0; nt < kWgNT; ++nt) {
      float r[kWgMT][4] = {};   // the two small terms of the group
#pragma unroll
      for (int s = 0; s < 4; ++s) {
        unsigned bh[2], bl[2];
        split_tf32(xb[nt][2 * s], bh[0], bl[0]);
        split_tf32(xb[nt][2 * s + 1], bh[1], bl[1]);
#pragma unroll
        for (int mt = 0; mt < kWgMT; ++mt) {
          float d[4] = {};
          mma_tf32(d, ah[s][mt], bh[0], bh[1]);
          mma_tf32(r[mt], ah[s][mt], bl[0], bl[1]);
          mma_tf32(r[mt], al[s][mt], bh[0], bh[1]);
#pragma unroll
          for (int e = 0; e < 4; ++e) acc[mt][nt][e] += d[e];
        }
      }
#pragma unroll
      for (int mt = 0; mt < kWgMT; ++mt)
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[mt][nt][e] += r[mt][e];
    }
  }
  // the four warps' sums, added in warp order
  __shared__ float sh[4][32 * 33 + 32];
#pragma unroll
  for (int mt = 0; mt < kWgMT; ++mt) {
#pragma unroll
    for (int nt = 0; nt < kWgNT; ++nt)
#pragma unroll
      for (int e = 0; e < 4; ++e)
        sh[wid][(16 * mt + g + 8 * (e >> 1)) * 33 + 8 * nt + 2 * t + (e & 1)] = acc[mt][nt][e];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      float s = bsum[mt][h];
      s += __shfl_xor_sync(0xffffffffu, s, 1);
      s += __shfl_xor_sync(0xffffffffu, s, 2);
      if (t == 0) sh[wid][32 * 33 + 16 * mt + 8 * h + g] = s;
    }
  }
  __syncthreads();
  float* out = part + (size_t)blockIdx.x * (cout * cin + cout);
  for (int e = threadIdx.x; e < 32 * 32; e += 128) {
    const int o = e / 32, c = e % 32, i = o * 33 + c;
    if (o0 + o < cout && c0 + c < cin)
      out[(o0 + o) * cin + c0 + c] = (sh[0][i] + sh[1][i]) + (sh[2][i] + sh[3][i]);
  }
  if (c0 == 0 && threadIdx.x < 32 && o0 + (int)threadIdx.x < cout) {
    const int i = 32 * 33 + threadIdx.x;
    out[cout * cin + o0 + threadIdx.x] = (sh[0][i] + sh[1][i]) + (sh[2][i] + sh[3][i]);
  }
}

// gw, gb = the blocks' partials added: 32 outputs per block, 8 threads per output, each
// over every eighth block, then in thread order
__global__ void __launch_bounds__(256) k_pw_wgrad_sum(const float* __restrict__ part, int nblk, int nw, int nout,
                                                      float* __restrict__ gw, float* __restrict__ gb) {
  __shared__ float sh[8][32];
  const int e = blockIdx.x * 32 + threadIdx.x % 32, sl = threadIdx.x / 32;
  float s = 0.f;
  if (e < nout) {
#pragma unroll 8
    for (int k = sl; k < nblk; k += 8) s += part[(size_t)k * nout + e];
  }
  sh[sl][threadIdx.x % 32] = s;
  __syncthreads();
  if (sl == 0 && e < nout) {
#pragma unroll
    for (int k = 1; k < 8; ++k) s += sh[k][threadIdx.x];
    if (e < nw) gw[e] = s;
    else gb[e - nw] = s;
  }
}
