// The network's inference in one pass over the pixels per layer (included by fno.cu, inside
// its anonymous namespace).
//
// Between layers the activations are kept as their two bf16 parts, hi and lo, of pairs of
// channels: records (hi_c, hi_c+1 | lo_c, lo_c+1) of 8 bytes, [b][W/2][N N], the same four
// bytes per value as floats.  The only readers are products that split a float into just
// these parts, so nothing is rounded that was not, and a record is an operand register
// pair as it is: the reading kernel converts nothing, and the writing one has the pair in
// its accumulator layout.  Each kernel also forms the truncated transform along y of the
// rows it produces (the next layer's spectral input) from the parts it just made, and the
// last layer goes straight through the projection, so per layer the activations are read
// once and written once and the last ones never leave the SM.
// Measured on GB300 (32 channels, 16 modes, 4 layers, one sample of N = 2048): forward 3.02
// -> 1.87 ms; a layer 338 us (1.07 GB) where layer and transform took 520; three blocks of
// 168 registers per SM against four of 128 1.81 / 1.93 ms, two 1.88.
#pragma once

constexpr int kInfRow = 20;          // records per staged row of 16 pixels (160 bytes: conflict-free operand reads)
constexpr int kInfMaxN = 2048;       // at most four chunks of 32 tiles per row, one per warp of a block

// chunks of a row of YT tiles: 1, 2 or 4, so that a block's four warps hold whole rows
inline int infer_chunks(int YT) { return YT <= 32 ? 1 : (YT <= 64 ? 2 : 4); }

// the transform's operand fragments of tile yt (nm column blocks of them)
template <int NM>
__device__ __forceinline__ void load_dft(uint4 (&b)[NM], const uint4* __restrict__ TfB, int yt, int nm, int lane) {
#pragma unroll
  for (int j = 0; j < NM; ++j) b[j] = j < nm ? __ldg(TfB + ((size_t)yt * nm + j) * 32 + lane) : make_uint4(0, 0, 0, 0);
}

// transforms along y of a tile's 16 pixels x W channels, added to acc: hp / lp [nt][h] are
// the packed channel pairs 8 nt + 2t, + 1 of pixel g + 8 h; b from load_dft
template <int NT, int NM>
__device__ __forceinline__ void tile_dft(float (&acc)[(NT + 1) / 2][NM][4], const unsigned (&hp)[NT][2],
                                         const unsigned (&lp)[NT][2], const uint4 (&b)[NM], int nm) {
#pragma unroll
  for (int mt = 0; mt < (NT + 1) / 2; ++mt) {
    // rows = channels 16 mt + g (+ 8), k = pixels: the 8 x 8 blocks transposed
    unsigned ah[4], al[4];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      ah[2 * h] = trans8(hp[2 * mt][h]);
      al[2 * h] = trans8(lp[2 * mt][h]);
      if (2 * mt + 1 < NT) {
        ah[2 * h + 1] = trans8(hp[2 * mt + 1 < NT ? 2 * mt + 1 : 0][h]);
        al[2 * h + 1] = trans8(lp[2 * mt + 1 < NT ? 2 * mt + 1 : 0][h]);
      } else {
        ah[2 * h + 1] = al[2 * h + 1] = 0u;
      }
    }
#pragma unroll
    for (int j = 0; j < NM; ++j) {
      if (j < nm) mma3(acc[mt][j], ah, al, b[j]);
    }
  }
}

// adds the chunks' transforms of the block's rows (in chunk order) and writes them:
// A[((b W + o) N + x) n2m + k]; red: 4 x 16 MT x 8 NM floats
template <int NT, int NM, int CH>
__device__ __forceinline__ void store_dft(const float (&acc)[(NT + 1) / 2][NM][4], float* red, float* __restrict__ A,
                                          size_t row, size_t rows, int N, int n2m, int lane, int wid) {
  constexpr int W = 8 * NT, K = 8 * NM;
  const int g = lane / 4, t = lane % 4;
  __syncthreads();   // the staging buffers that red overlays have been read
  float* mine = red + wid * W * K;
#pragma unroll
  for (int mt = 0; mt < (NT + 1) / 2; ++mt)
#pragma unroll
    for (int j = 0; j < NM; ++j)
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int o = 16 * mt + g + 8 * (e >> 1);
        if (o < W) mine[o * K + 8 * j + 2 * t + (e & 1)] = acc[mt][j][e];
      }
  __syncthreads();
  if (row >= rows) return;
  const int chunk = wid % CH;
  const size_t b = row / N;
  const int x = (int)(row % N);
  const float* first = red + (wid - chunk) * W * K;
  // the row's warps share the outputs
  for (int i = chunk * 32 + lane; i < W * K; i += CH * 32) {
    const int o = i / K, k = i % K;
    if (k >= n2m) continue;
    float s = first[i];
    for (int c = 1; c < CH; ++c) s += first[c * W * K + i];
    A[((b * W + o) * N + x) * n2m + k] = s;
  }
}

// v0 = P x + p in records, and its transform along y
template <int NT, int NM, int CH>
__global__ void __launch_bounds__(128, 4) k_lift_inf(const float* __restrict__ X, const bf16* __restrict__ Pw,
                                                     const bf16* __restrict__ Pb, const uint4* __restrict__ TfB,
                                                     uint2* __restrict__ V, float* __restrict__ A, int N, int n2m,
                                                     size_t rows) {
  constexpr int W = 8 * NT, MT = (NT + 1) / 2;
  __shared__ float red[4 * W * 8 * NM];
  const int lane = threadIdx.x % 32, g = lane / 4, t = lane % 4, wid = threadIdx.x / 32;
  const int YT = N / 16, tpw = (YT + CH - 1) / CH;
  const size_t row = ((size_t)blockIdx.x * 4 + wid) / CH;
  const int chunk = wid % CH;
  float dacc[MT][NM][4] = {};
  if (row < rows) {
    const size_t b = row / N, P = (size_t)N * N, base = (row % N) * (size_t)N;
    unsigned wf[NT];
    float bv[NT][2];
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) {
      const int o = 8 * nt + g, c = 2 * t;
      wf[nt] = (unsigned)__bfloat16_as_ushort(Pw[o * 7 + c]) |
               (c + 1 < 7 ? (unsigned)__bfloat16_as_ushort(Pw[o * 7 + c + 1]) << 16 : 0u);
#pragma unroll
      for (int e = 0; e < 2; ++e) bv[nt][e] = b2f(Pb[8 * nt + 2 * t + e]);
    }
    const float* xc = X + (b * 7 + 2 * t) * P + base + g;
    uint2* vp = V + (b * (W / 2) + t) * P + base + g;
    const int yt0 = chunk * tpw, yt1 = min(YT, yt0 + tpw);
    float cur[4], nxt[4];
    auto load = [&](int yt, float (&x)[4]) {
      const float* q = xc + 16 * yt;
      x[0] = q[0];
      x[2] = q[8];
      x[1] = t < 3 ? q[P] : 0.f;
      x[3] = t < 3 ? q[P + 8] : 0.f;
    };
    if (yt0 < yt1) load(yt0, cur);
    for (int yt = yt0; yt < yt1; ++yt) {
      if (yt + 1 < yt1) load(yt + 1, nxt);
      uint4 tb[NM];
      load_dft<NM>(tb, TfB, yt, (n2m + 7) / 8, lane);
      unsigned ah[4] = {0u, 0u, 0u, 0u}, al[4] = {0u, 0u, 0u, 0u};
      split2(cur[0], cur[1], ah[0], al[0]);
      split2(cur[2], cur[3], ah[1], al[1]);
      unsigned hp[NT][2], lp[NT][2];
#pragma unroll
      for (int nt = 0; nt < NT; ++nt) {
        float acc[4] = {0.f, 0.f, 0.f, 0.f};
        mma_bf16(acc, ah, wf[nt], 0u);
        mma_bf16(acc, al, wf[nt], 0u);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          split2(acc[2 * h] + bv[nt][0], acc[2 * h + 1] + bv[nt][1], hp[nt][h], lp[nt][h]);
          vp[(size_t)(4 * nt) * P + 16 * yt + 8 * h] = make_uint2(hp[nt][h], lp[nt][h]);
        }
      }
      tile_dft<NT, NM>(dacc, hp, lp, tb, (n2m + 7) / 8);
#pragma unroll
      for (int e = 0; e < 4; ++e) cur[e] = nxt[e];
    }
  }
  store_dft<NT, NM, CH>(dacc, red, A, row, rows, N, n2m, lane, wid);
}

// One Fourier layer on records (the arithmetic of k_layer_tc).  LAST false: v' = gelu(z)
// in records and its transform along y; LAST true: z through the projection (the
// arithmetic of k_proj_tc) into out.
template <int KT, int NT, int KS, bool LAST, int CH>
__global__ void __launch_bounds__(128, 3)
k_layer_inf(const uint2* __restrict__ V, const bf16* __restrict__ Ww, const bf16* __restrict__ Wb, float* A,
            const float* __restrict__ cs, const uint4* __restrict__ TfA, const uint4* __restrict__ TfB,
            uint2* __restrict__ Vout, const bf16* __restrict__ Q1, const bf16* __restrict__ q1,
            const bf16* __restrict__ Q2, const bf16* __restrict__ q2, int H, float* __restrict__ out, int N, int n2m,
            size_t rows) {
  constexpr int W = 8 * NT, NP = 4 * NT, MT = (NT + 1) / 2, NM = 2 * KS, STAGE = NP * kInfRow;
  constexpr int kStageBytes = 4 * 2 * STAGE * (int)sizeof(uint2), kRedBytes = 4 * W * 8 * NM * 4;
  __shared__ __align__(16) unsigned char raw[LAST || kStageBytes > kRedBytes ? kStageBytes : kRedBytes];
  __shared__ __align__(16) uint4 sf[4][KS][NT][32];          // the row's mode coefficients, split: h0 h1 l0 l1
  __shared__ uint2 sq[LAST ? KT * 8 * 32 : 1];               // Q1 fragments
  __shared__ float2 sqb[LAST ? 8 * 4 : 1], sqw[LAST ? 8 * 4 : 1];
  uint2(*stage)[2][STAGE] = reinterpret_cast<uint2(*)[2][STAGE]>(raw);
  const int lane = threadIdx.x % 32, g = lane / 4, t = lane % 4, wid = threadIdx.x / 32;
  const int YT = N / 16, tpw = (YT + CH - 1) / CH;
  const size_t row = ((size_t)blockIdx.x * 4 + wid) / CH;
  const int chunk = wid % CH;
  const int nh = (H + 7) / 8;
  if constexpr (LAST) {
    for (int i = threadIdx.x; i < KT * nh * 32; i += 128) {
      const int ln = i % 32, j = 8 * ((i / 32) % nh) + ln / 4, kb = i / (32 * nh);
      unsigned w[2];
#pragma unroll
      for (int hh = 0; hh < 2; ++hh) {
        const int c = 16 * kb + 2 * (ln % 4) + 8 * hh;
        w[hh] = (j < H && c < W) ? (unsigned)__bfloat16_as_ushort(Q1[j * W + c]) |
                                       ((unsigned)__bfloat16_as_ushort(Q1[j * W + c + 1]) << 16)
                                 : 0u;
      }
      sq[i] = make_uint2(w[0], w[1]);
    }
    for (int i = threadIdx.x; i < nh * 4; i += 128) {
      const int j = 2 * i;
      sqb[i] = make_float2(j < H ? b2f(q1[j]) : 0.f, j + 1 < H ? b2f(q1[j + 1]) : 0.f);
      sqw[i] = make_float2(j < H ? b2f(Q2[j]) : 0.f, j + 1 < H ? b2f(Q2[j + 1]) : 0.f);
    }
    __syncthreads();
  }
  float dacc[LAST ? 1 : MT][LAST ? 1 : NM][4] = {};
  if (row < rows) {
    const size_t b = row / N, P = (size_t)N * N, base = (row % N) * (size_t)N;
    const int x = (int)(row % N);
    unsigned wf[KT][NT][2];
#pragma unroll
    for (int kb = 0; kb < KT; ++kb)
#pragma unroll
      for (int nt = 0; nt < NT; ++nt) {
        const int o = 8 * nt + g;
#pragma unroll
        for (int hh = 0; hh < 2; ++hh) {
          const int c = 16 * kb + 2 * t + 8 * hh;
          const bool cv = 16 * kb + 8 * hh < W;
          wf[kb][nt][hh] = cv ? (unsigned)__bfloat16_as_ushort(Ww[o * W + c]) |
                                    ((unsigned)__bfloat16_as_ushort(Ww[o * W + c + 1]) << 16)
                              : 0u;
        }
      }
#pragma unroll
    for (int ks = 0; ks < KS; ++ks)
#pragma unroll
      for (int nt = 0; nt < NT; ++nt) {
        const float* ar = A + ((b * W + 8 * nt + g) * N + x) * n2m;
        uint4 s;
        auto co = [&](int k) { return k < n2m ? ar[k] * cs[k / 2] : 0.f; };
        const int k = 16 * ks + 2 * t;
        split2(co(k), co(k + 1), s.x, s.z);
        split2(co(k + 8), co(k + 9), s.y, s.w);
        sf[wid][ks][nt][lane] = s;
      }
    float bv[NT][2];
#pragma unroll
    for (int nt = 0; nt < NT; ++nt)
#pragma unroll
      for (int e = 0; e < 2; ++e) bv[nt][e] = b2f(Wb[8 * nt + 2 * t + e]);
    const uint2* vb = V + b * NP * P + base;
    uint2* vo = LAST ? nullptr : Vout + (b * NP + t) * P + base + g;
    float* ob = LAST ? out + b * P + base : nullptr;
    const float bias2 = LAST ? b2f(q2[0]) : 0.f;
    auto prefetch = [&](int yt, int st) {   // NP rows of 128 bytes
#pragma unroll
      for (int j = lane; j < 8 * NP; j += 32) {
        const int c = j >> 3, part = j & 7;
        cp_async16(&stage[wid][st][c * kInfRow + 2 * part], vb + (size_t)c * P + 16 * yt + 2 * part);
      }
      cp_async_commit();
    };
    const int yt0 = chunk * tpw, yt1 = min(YT, yt0 + tpw);
    // the inverse transform's pixel operand, loaded a tile ahead (the unit's waits for these
    // loads were the kernel's largest stall)
    unsigned th[KS][4], tl[KS][4];
    auto load_inv = [&](int yt) {
#pragma unroll
      for (int ks = 0; ks < KS; ++ks) {
        const uint4* tp = TfA + (((size_t)yt * KS + ks) * 32 + lane) * 2;
        const uint4 h4 = __ldg(tp), l4 = __ldg(tp + 1);
        th[ks][0] = h4.x; th[ks][1] = h4.y; th[ks][2] = h4.z; th[ks][3] = h4.w;
        tl[ks][0] = l4.x; tl[ks][1] = l4.y; tl[ks][2] = l4.z; tl[ks][3] = l4.w;
      }
    };
    if (yt0 < yt1) {
      prefetch(yt0, 0);
      load_inv(yt0);
    }
    for (int yt = yt0; yt < yt1; ++yt) {
      const int i = yt - yt0;
      [[maybe_unused]] uint4 tb[LAST ? 1 : NM];
      if constexpr (!LAST) load_dft<NM>(tb, TfB, yt, (n2m + 7) / 8, lane);
      if (yt + 1 < yt1) prefetch(yt + 1, (i + 1) & 1);
      else cp_async_commit();
      cp_async_wait<1>();
      __syncwarp();
      const uint2* sb = stage[wid][i & 1];
      unsigned ah[KT][4], al[KT][4];
#pragma unroll
      for (int kb = 0; kb < KT; ++kb)
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          // registers (pixel g, channels 2t), (pixel g + 8, .), (g, channels + 8), (g + 8, .)
          const bool cv = 16 * kb + 8 * (e >> 1) < W;
          const uint2 r = cv ? sb[(8 * kb + 4 * (e >> 1) + t) * kInfRow + g + 8 * (e & 1)] : make_uint2(0u, 0u);
          ah[kb][e] = r.x;
          al[kb][e] = r.y;
        }
      __syncwarp();   // every lane has read the stage before it is refilled
      unsigned hp[NT][2], lp[NT][2];
#pragma unroll
      for (int nt = 0; nt < NT; ++nt) {
        float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int kb = 0; kb < KT; ++kb) {
          mma_bf16(acc, ah[kb], wf[kb][nt][0], wf[kb][nt][1]);
          mma_bf16(acc, al[kb], wf[kb][nt][0], wf[kb][nt][1]);
        }
#pragma unroll
        for (int ks = 0; ks < KS; ++ks) {
          const uint4 s = sf[wid][ks][nt][lane];
          mma_bf16(acc, th[ks], s.x, s.y);
          mma_bf16(acc, th[ks], s.z, s.w);
          mma_bf16(acc, tl[ks], s.x, s.y);
        }
        float va[2] = {acc[0] + bv[nt][0], acc[1] + bv[nt][1]}, vb2[2] = {acc[2] + bv[nt][0], acc[3] + bv[nt][1]};
        if constexpr (!LAST) {
          gelu2(va[0], vb2[0]);
          gelu2(va[1], vb2[1]);
        }
        split2(va[0], va[1], hp[nt][0], lp[nt][0]);
        split2(vb2[0], vb2[1], hp[nt][1], lp[nt][1]);
        if constexpr (!LAST) {
#pragma unroll
          for (int h = 0; h < 2; ++h)
            vo[(size_t)(4 * nt) * P + 16 * yt + 8 * h] = make_uint2(hp[nt][h], lp[nt][h]);
        }
      }
      if (yt + 1 < yt1) load_inv(yt + 1);
      if constexpr (!LAST) {
        tile_dft<NT, NM>(dacc, hp, lp, tb, (n2m + 7) / 8);
      } else {
        float sa = 0.f, sb2 = 0.f;
        for (int j = 0; j < nh; ++j) {
          float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
          for (int kb = 0; kb < KT; ++kb) {
            const uint2 w = sq[(kb * nh + j) * 32 + lane];
            unsigned zh[4], zl[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              const int nt = 2 * kb + (e >> 1);
              zh[e] = nt < NT ? hp[nt < NT ? nt : 0][e & 1] : 0u;
              zl[e] = nt < NT ? lp[nt < NT ? nt : 0][e & 1] : 0u;
            }
            mma_bf16(acc, zh, w.x, w.y);
            mma_bf16(acc, zl, w.x, w.y);
          }
          const float2 qb = sqb[j * 4 + t], qw = sqw[j * 4 + t];
          float h0 = acc[0] + qb.x, h1 = acc[1] + qb.y, h2 = acc[2] + qb.x, h3 = acc[3] + qb.y;
          gelu2_proj(h0, h1);
          gelu2_proj(h2, h3);
          sa += qw.x * h0 + qw.y * h1;
          sb2 += qw.x * h2 + qw.y * h3;
        }
        sa += __shfl_xor_sync(0xffffffffu, sa, 1);
        sa += __shfl_xor_sync(0xffffffffu, sa, 2);
        sb2 += __shfl_xor_sync(0xffffffffu, sb2, 1);
        sb2 += __shfl_xor_sync(0xffffffffu, sb2, 2);
        if (t == 0) {
          ob[16 * yt + g] = sa + bias2;
          ob[16 * yt + g + 8] = sb2 + bias2;
        }
      }
    }
    cp_async_wait<0>();
  }
  if constexpr (!LAST)
    store_dft<NT, NM, CH>(dacc, reinterpret_cast<float*>(raw), A, row, rows, N, n2m, lane, wid);
}
