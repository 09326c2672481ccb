// Learned refinement proposal (2D): a small per-block CNN predicts whether the
// safety refinement of a block (Sec. 2.1 step 1) will be kept after the step.
// Exact detail thresholding stays the fallback (a block whose own details are
// >= eps is always refined) and the miss check (misses are counted after the step).
//
// Network on x[2][T][T] (T = Bs + 2 ng, the synchronised tile):
//   h1 = relu(conv3x3 s1 (2 -> 16)), h2 = relu(conv3x3 s2 (16 -> 16)),
//   h3 = relu(conv3x3 s2 (16 -> 16)), z = global max of h3, p = sigmoid(wl.z + bl).
// Parameters packed W1 b1 W2 b2 W3 b3 wl bl (4961 values).  Training keeps FP32
// master weights (Adam); inference uses BF16-rounded weights, FP32 accumulation.
// Input channels: 0 = field variable 0 minus its tile-centre value, divided by
// the largest such difference on the tile; 1 = log10(1e-3 + |d|/(s_v eps)) of
// the block's details (max over variables) at interior nodes, -3 elsewhere.
#include <cooperative_groups.h>
#include <cuda_bf16.h>

#include <algorithm>

#include "mr_device.cuh"
#include "mr_cnn.h"

namespace mr {

constexpr int kC = 16;
constexpr int kW1 = 0, kB1 = kW1 + kC * 2 * 9, kW2 = kB1 + kC, kB2 = kW2 + kC * kC * 9,
              kW3 = kB2 + kC, kB3 = kW3 + kC * kC * 9, kWL = kB3 + kC, kBL = kWL + kC;
static_assert(kBL + 1 == kCnnParams, "parameter count");

template <int T>
struct CnnGeo {
  static constexpr int T2 = (T - 1) / 2 + 1;
  static constexpr int T3 = (T2 - 1) / 2 + 1;
  static constexpr int NX = 2 * T * T;
  static constexpr int N1 = kC * T * T;
  static constexpr int N2 = kC * T2 * T2;
  static constexpr int N3 = kC * T3 * T3;
};

// ------------------------------------------------------------- features ------
// Input tile of the network for every active block: channel 0 = variable 0
// minus its centre value over its largest deviation; channel 1 =
// log10(1e-3 + |d| / (s_v eps)) at the odd interior nodes (largest over the
// variables), -3 elsewhere.  FP32 throughout (a feature, not a decision; FP64
// runs at a small fraction of the FP32 rate here); the details come from the
// separable 4-point prediction, x on coarse rows then y.
template <int B>
struct FeatGeo {
  using Gm = Geo<2, B>;
  using Bx = Box<2, B, kG>;
  static constexpr int NC = (B + 1) / 2 + 2;  // coarse rows -1 .. (B+1)/2
  static constexpr int NX = NC * B;
  static size_t smem(int nv) {
    return kRingBytesD<2> + sizeof(float) * ((size_t)nv * (Gm::TILE + Bx::CBOX + Bx::SCR) + NX + Gm::NI);
  }
};

template <int B, typename TS>
__global__ void __launch_bounds__(256) k_features(PoolView pv, const TS* __restrict__ y,
                                                  float* __restrict__ feat, float* __restrict__ mpre,
                                                  int64_t base) {
  pdl_enter();
  using Gm = Geo<2, B>;
  using Bx = Box<2, B, kG>;
  using FG = FeatGeo<B>;
  constexpr int T = Gm::T;
  const int nv = pv.nvar;
  RingD<2>& R = *smem_as<RingD<2>>(0);
  __shared__ float red[2][32];
  float* tile = smem_as<float>(kRingBytesD<2>);
  float* cbox = tile + nv * Gm::TILE;
  float* scr = cbox + nv * Bx::CBOX;
  float* X = scr + nv * Bx::SCR;
  float* dmap = X + FG::NX;
  const int nact = pv.cnt->n_act;
  for (int p = blockIdx.x; p < nact; p += gridDim.x) {
    const BlockInfo b = load_block(pv, pv.act[p]);
    const TreeDev& td = pv.trees[b.tree];
    float* out = feat + (base + p) * (int64_t)(2 * T * T);
    build_ring<2, B>(pv, td, b, R);
    __syncthreads();
    fill_tile<2, B, TS, float>(pv, b, y, (TS*)y, tile, false, R, cbox, scr);
    for (int q = threadIdx.x; q < Gm::NI; q += blockDim.x) dmap[q] = 0.f;
    __syncthreads();
    const float centre = tile[Gm::tix((B - 1) / 2, (B - 1) / 2, 0)];
    float mx = 0.f;
    for (int idx = threadIdx.x; idx < Gm::TILE; idx += blockDim.x) mx = fmaxf(mx, fabsf(tile[idx] - centre));
    for (int s = 16; s > 0; s >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, s));
    if ((threadIdx.x & 31) == 0) red[0][threadIdx.x >> 5] = mx;
    __syncthreads();
    mx = 0.f;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) mx = fmaxf(mx, red[0][w]);
    const float inv = mx > 0.f ? 1.f / mx : 0.f;
    for (int v = 0; v < nv; ++v) {
      const float* tv = tile + v * Gm::TILE;
      double svd = pv.norm_kind == 1 ? pv.svar[b.tree * nv + v] : 1.0;
      const float sv = svd == 0.0 ? 1.f : (float)svd;
      for (int idx = threadIdx.x; idx < FG::NX; idx += blockDim.x) {  // x pass on coarse rows
        const int x = idx % B, yy = 2 * (idx / B - 1);
        X[idx] = (x & 1) ? dd4(tv[Gm::tix(x - 3, yy, 0)], tv[Gm::tix(x - 1, yy, 0)], tv[Gm::tix(x + 1, yy, 0)],
                               tv[Gm::tix(x + 3, yy, 0)])
                         : tv[Gm::tix(x, yy, 0)];
      }
      __syncthreads();
      for (int q = threadIdx.x; q < Gm::NI; q += blockDim.x) {
        const int i = q % B, j = q / B;
        if (((i | j) & 1) == 0) continue;
        float pr;
        if ((j & 1) == 0) {
          pr = X[(j / 2 + 1) * B + i];
        } else {
          const int m0 = (j - 1) / 2;
          pr = dd4(X[m0 * B + i], X[(m0 + 1) * B + i], X[(m0 + 2) * B + i], X[(m0 + 3) * B + i]);
        }
        dmap[q] = fmaxf(dmap[q], fabsf(tv[Gm::tix(i, j, 0)] - pr) / sv);
      }
      __syncthreads();
    }
    float md = 0.f;
    const float ieps = (float)(1.0 / td.eps);
    for (int idx = threadIdx.x; idx < Gm::TILE; idx += blockDim.x) {
      const int i = idx % T - Gm::G, j = idx / T - Gm::G;
      out[idx] = (tile[idx] - centre) * inv;
      float dv = -3.f;
      if (i >= 0 && i < B && j >= 0 && j < B && ((i | j) & 1)) {
        const float dm = dmap[j * B + i];
        md = fmaxf(md, dm);
        dv = log10f(1e-3f + dm * ieps);
      }
      out[T * T + idx] = dv;
    }
    for (int s = 16; s > 0; s >>= 1) md = fmaxf(md, __shfl_xor_sync(0xffffffffu, md, s));
    if ((threadIdx.x & 31) == 0) red[1][threadIdx.x >> 5] = md;
    __syncthreads();
    if (threadIdx.x == 0) {
      for (int w = 1; w < (int)(blockDim.x >> 5); ++w) md = fmaxf(md, red[1][w]);
      if (mpre) mpre[p] = md;
    }
    __syncthreads();
  }
}

// ----------------------------------------------------------- inference -------
// Inference: p for every active block below Jmax (others get 0).  The
// weights are staged once per CTA in shared memory as floats, transposed so
// that the 16 output channels of a tap are contiguous; each thread computes
// all 16 output channels of one pixel (one input load feeds 16 FMAs, the 16
// weights come as four broadcast 16-byte loads).  Per output the sum runs over
// bias, then input channel, row, column.
template <int T>
struct InferGeo {
  using CG = CnnGeo<T>;
  // transposed weights: layer l, input channel c, tap t -> 16 floats (o)
  static constexpr int WT1 = 0, WT2 = WT1 + 2 * 9 * kC, WT3 = WT2 + kC * 9 * kC, WTE = WT3 + kC * 9 * kC;
  static constexpr int NW = WTE + 4 * kC + 1;  // + b1, b2, b3, wl, bl
  static constexpr int X0 = (NW + 3) / 4 * 4;  // activations after the weights
  static constexpr size_t SMEM = sizeof(float) * (X0 + CG::NX + CG::N1 + CG::N2 + CG::N3);
};

template <int T, int CIN, int S>
__device__ __forceinline__ void conv_all_o(const float* __restrict__ in, int Tin, const float* __restrict__ wt,
                                           const float* __restrict__ bias, float* __restrict__ out, int Tout) {
  for (int pix = threadIdx.x; pix < Tout * Tout; pix += blockDim.x) {
    const int i = pix / Tout, j = pix % Tout;
    float acc[kC];
#pragma unroll
    for (int o = 0; o < kC; ++o) acc[o] = bias[o];
    for (int c = 0; c < CIN; ++c) {
#pragma unroll
      for (int di = 0; di < 3; ++di) {
        const int ii = S * i + di - 1;
        if (ii < 0 || ii >= Tin) continue;
#pragma unroll
        for (int dj = 0; dj < 3; ++dj) {
          const int jj = S * j + dj - 1;
          if (jj < 0 || jj >= Tin) continue;
          const float xv = in[c * Tin * Tin + ii * Tin + jj];
          const float4* w4 = reinterpret_cast<const float4*>(wt + ((c * 3 + di) * 3 + dj) * kC);
#pragma unroll
          for (int o4 = 0; o4 < kC / 4; ++o4) {
            const float4 wv = w4[o4];
            acc[4 * o4 + 0] += wv.x * xv;
            acc[4 * o4 + 1] += wv.y * xv;
            acc[4 * o4 + 2] += wv.z * xv;
            acc[4 * o4 + 3] += wv.w * xv;
          }
        }
      }
    }
#pragma unroll
    for (int o = 0; o < kC; ++o) out[o * Tout * Tout + pix] = fmaxf(acc[o], 0.f);
  }
}

template <int T>
__global__ void __launch_bounds__(256) k_cnn_infer(PoolView pv, const float* __restrict__ feat,
                                                   const __nv_bfloat16* __restrict__ wb,
                                                   float* __restrict__ prob, int64_t n_explicit) {
  pdl_enter();
  using CG = CnnGeo<T>;
  using IG = InferGeo<T>;
  float* ws = smem_as<float>(0);
  float* x = ws + IG::X0;
  float* h1 = x + CG::NX;
  float* h2 = h1 + CG::N1;
  float* h3 = h2 + CG::N2;
  __shared__ float z[kC];
  // stage the weights, transposed to [c][tap][o]
  for (int q = threadIdx.x; q < kC * 2 * 9; q += blockDim.x) {
    const int o = q / 18, c = (q / 9) % 2, t = q % 9;
    ws[IG::WT1 + (c * 9 + t) * kC + o] = __bfloat162float(wb[kW1 + q]);
  }
  for (int q = threadIdx.x; q < kC * kC * 9; q += blockDim.x) {
    const int o = q / (kC * 9), c = (q / 9) % kC, t = q % 9;
    ws[IG::WT2 + (c * 9 + t) * kC + o] = __bfloat162float(wb[kW2 + q]);
    ws[IG::WT3 + (c * 9 + t) * kC + o] = __bfloat162float(wb[kW3 + q]);
  }
  if (threadIdx.x < kC) {
    ws[IG::WTE + threadIdx.x] = __bfloat162float(wb[kB1 + threadIdx.x]);
    ws[IG::WTE + kC + threadIdx.x] = __bfloat162float(wb[kB2 + threadIdx.x]);
    ws[IG::WTE + 2 * kC + threadIdx.x] = __bfloat162float(wb[kB3 + threadIdx.x]);
    ws[IG::WTE + 3 * kC + threadIdx.x] = __bfloat162float(wb[kWL + threadIdx.x]);
  }
  if (threadIdx.x == 0) ws[IG::WTE + 4 * kC] = __bfloat162float(wb[kBL]);
  __syncthreads();
  const int64_t n = n_explicit >= 0 ? n_explicit : (int64_t)pv.cnt->n_act;
  for (int64_t p = blockIdx.x; p < n; p += gridDim.x) {
    if (n_explicit < 0) {
      const int s = pv.act[p];
      if (pv.lvl[s] >= pv.trees[pv.tree[s]].Jmax) {
        if (threadIdx.x == 0) prob[p] = 0.f;
        continue;
      }
    }
    for (int idx = threadIdx.x; idx < CG::NX; idx += blockDim.x) x[idx] = feat[p * CG::NX + idx];
    __syncthreads();
    conv_all_o<T, 2, 1>(x, T, ws + IG::WT1, ws + IG::WTE, h1, T);
    __syncthreads();
    conv_all_o<T, kC, 2>(h1, T, ws + IG::WT2, ws + IG::WTE + kC, h2, CG::T2);
    __syncthreads();
    conv_all_o<T, kC, 2>(h2, CG::T2, ws + IG::WT3, ws + IG::WTE + 2 * kC, h3, CG::T3);
    __syncthreads();
    if (threadIdx.x < kC) {
      float m = h3[threadIdx.x * CG::T3 * CG::T3];
      for (int q = 1; q < CG::T3 * CG::T3; ++q) m = fmaxf(m, h3[threadIdx.x * CG::T3 * CG::T3 + q]);
      z[threadIdx.x] = m;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      float logit = ws[IG::WTE + 4 * kC];
      for (int o = 0; o < kC; ++o) logit += ws[IG::WTE + 3 * kC + o] * z[o];
      prob[p] = 1.f / (1.f + expf(-logit));
    }
    __syncthreads();
  }
}

// ---------------------------------------------------- training (fwd + bwd) ---
// Samples [s0, s0 + nb) of the dataset (index list idx), mean weighted BCE, one
// sample at a time per CTA.  FP32 throughout (1.6 M multiply-adds per sample of
// 25^2).  Shared-memory reads bound the kernel (a load writes a register per lane,
// a broadcast one too, so every loaded value has to meet several others), and
// every pass is tiled in registers:
//   conv1: 16 channels of a pixel per thread; conv2: 4 channels of two pixels, one
//   above the other; conv3: 4 channels of a pixel (weights transposed to
//   [channel][tap][16]);
//   conv2 weight gradient: 4 outputs x 3 taps of a row per thread, conv1: 2 outputs x
//   2 channels x 3, conv3 (nonzero only at each channel's maximum): the 9 taps of an
//   (o, c) pair -- all kept in registers over the CTA's samples, to which the sums of
//   one sample are added: with every pixel added to the running sum, the summation
//   alone lost 4 to 7 times more of conv2's gradient (1024 samples of 25^2 per CTA:
//   1.8e-6 of its norm, now 3.0e-7; in a call of 90000 samples 2.1e-7 and 1.8e-7),
//   at the same time per call;
//   da1: a 2 x 2 pixel block (its 9 taps meet 4 output pixels) of 2 channels.
// Activations are padded by one node, so no tap tests its bounds, and the rows of
// h1 hold their even columns, then the odd ones: the stride-2 convolution reads
// consecutive words.  Products with a zero gradient are left out (a non-finite
// input under an inactive unit has no gradient).
// 3000 samples of 25^2: 5890 us with one output value per thread and loop, now
// 510 us (shared-memory pipe near 90 % of peak).  Larger tiles (two pixels in conv1, four
// in conv2, two blocks in da1) read less but leave threads idle: 490-510 us.
// a + w x, product and sum each rounded: the forward pass rounds as k_cnn_infer does,
// term by term (padding adds exact zeros), so both take the same maxima and ReLU
// branches, whatever the tiling; a different rounding would move gradients between
// nearly equal maxima.
__device__ __forceinline__ float mul_add(float w, float x, float a) { return __fadd_rn(a, __fmul_rn(w, x)); }

template <int T>
struct TrainGeo {
  using CG = CnnGeo<T>;
  // 25^2: two CTAs of 12 warps per SM; 41^2: one of 24 (its activations fill the shared memory)
  static constexpr int NT = T == 25 ? 384 : 768;
  static constexpr int T2 = CG::T2, T3 = CG::T3;
  static constexpr int P = T + 2, H = (P + 1) / 2;  // padded width; even columns of a row
  static constexpr int P2 = T2 + 2;
  static constexpr int DP = 20;                     // pitch of a pixel's 16 gradients
  // offsets (floats)
  static constexpr int W1 = 0, W2 = W1 + 18 * kC, W3 = W2 + 144 * kC, WS = W3 + 144 * kC;  // WS: b1 b2 b3 wl bl
  static constexpr int D2 = (WS + 4 * kC + 1 + 3) / 4 * 4;
  static constexpr int X = D2 + T2 * T2 * DP;
  static constexpr int H1 = X + 2 * P * P;
  static constexpr int H2 = H1 + kC * P * P;
  static constexpr int H3 = H2 + kC * P2 * P2;
  static constexpr int END = H3 + kC * T3 * T3;
  static constexpr size_t SMEM = sizeof(float) * END;
  static constexpr int MINB = SMEM <= 112 * 1024 ? 2 : 1;
  static_assert(kC * P * P >= kCnnParams, "the gradients are summed over h1 at the end");
  // node (r, c) of a padded h1 plane
  __device__ static __forceinline__ int h1at(int o, int r, int c) { return (o * P + r) * P + (c & 1) * H + (c >> 1); }
};

template <int T>
__global__ void __launch_bounds__(TrainGeo<T>::NT, TrainGeo<T>::MINB)
    k_cnn_train(const float* __restrict__ feat, const float* __restrict__ label, const int32_t* __restrict__ idx,
                int64_t s0, int nb, const float* __restrict__ w, float w_pos, float* __restrict__ grad,
                float* __restrict__ loss, float* __restrict__ prob_out) {
  pdl_enter();
  using G = TrainGeo<T>;
  constexpr int NT = G::NT, T2 = G::T2, T3 = G::T3, P = G::P, H = G::H, P2 = G::P2, DP = G::DP;
  float* sm = smem_as<float>(0);
  const float4* w1 = reinterpret_cast<const float4*>(sm + G::W1);
  const float4* w2 = reinterpret_cast<const float4*>(sm + G::W2);
  const float4* w3 = reinterpret_cast<const float4*>(sm + G::W3);
  const float *b1 = sm + G::WS, *b2 = b1 + kC, *b3 = b2 + kC, *wl = b3 + kC, *bl = wl + kC;
  float *d2 = sm + G::D2, *x = sm + G::X, *h1 = sm + G::H1, *h2 = sm + G::H2, *h3 = sm + G::H3;
  __shared__ float z[kC];
  __shared__ int arg[kC];
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  for (int q = t; q < G::END; q += NT) sm[q] = 0.f;  // the padding stays zero
  __syncthreads();
  for (int q = t; q < kC * 18; q += NT) sm[G::W1 + (q % 18) * kC + q / 18] = w[kW1 + q];
  for (int q = t; q < kC * 144; q += NT) {
    sm[G::W2 + (q % 144) * kC + q / 144] = w[kW2 + q];
    sm[G::W3 + (q % 144) * kC + q / 144] = w[kW3 + q];
  }
  if (t < kC) {
    sm[G::WS + t] = w[kB1 + t];
    sm[G::WS + kC + t] = w[kB2 + t];
    sm[G::WS + 2 * kC + t] = w[kB3 + t];
    sm[G::WS + 3 * kC + t] = w[kWL + t];
  }
  if (t == 0) sm[G::WS + 4 * kC] = w[kBL];
  float lsum = 0.f;
  // gradients of this thread, over the CTA's samples
  const int o3 = t >> 4, c3 = t & 15;                                  // conv3: pair (o, c), t < 256
  const int og2 = t & 3, cd2 = (t >> 2) % 48, part2 = t / 192;         // conv2: 4 outputs, channel and row tap
  const int c2 = cd2 / 3, di2 = cd2 % 3;
  const int cb1 = t % 24, part1 = t / 24, op1 = cb1 / 3, di1 = cb1 % 3;  // conv1: 2 outputs, row tap
  float g3[9] = {}, g2[4][3] = {}, g1[2][2][3] = {};
  float gb1[2] = {}, gb2 = 0.f, gb3 = 0.f, gwl = 0.f, gbl = 0.f;
  for (int sb = blockIdx.x; sb < nb; sb += gridDim.x) {
    __syncthreads();
    const int64_t sidx = idx ? (int64_t)idx[s0 + sb] : s0 + sb;
    const float* in = feat + sidx * (2 * T * T);
    for (int q = t; q < 2 * T * T; q += NT) {
      const int c = q / (T * T), r = q % (T * T);
      x[(c * P + r / T + 1) * P + r % T + 1] = in[q];
    }
    for (int q = t; q < T2 * T2 * DP; q += NT) d2[q] = 0.f;
    const float yv = label[sidx];
    __syncthreads();
    // conv1
    for (int pix = t; pix < T * T; pix += NT) {
      const int i = pix / T, j = pix % T;
      float a[kC];
#pragma unroll
      for (int o = 0; o < kC; ++o) a[o] = b1[o];
#pragma unroll 1
      for (int kd = 0; kd < 6; ++kd)  // channel and row of the tap
#pragma unroll
        for (int dj = 0; dj < 3; ++dj) {
          const float xv = x[((kd / 3) * P + i + kd % 3) * P + j + dj];
          const float4* wp = w1 + (kd * 3 + dj) * 4;
#pragma unroll
          for (int o4 = 0; o4 < 4; ++o4) {
            const float4 wv = wp[o4];
            a[4 * o4] = mul_add(wv.x, xv, a[4 * o4]);
            a[4 * o4 + 1] = mul_add(wv.y, xv, a[4 * o4 + 1]);
            a[4 * o4 + 2] = mul_add(wv.z, xv, a[4 * o4 + 2]);
            a[4 * o4 + 3] = mul_add(wv.w, xv, a[4 * o4 + 3]);
          }
        }
      const int at = G::h1at(0, i + 1, j + 1);
#pragma unroll
      for (int o = 0; o < kC; ++o) h1[at + o * P * P] = fmaxf(a[o], 0.f);
    }
    __syncthreads();
    // conv2: pixels (2 ip, j) and (2 ip + 1, j), 4 channels
    constexpr int NP = (T2 + 1) / 2;
    for (int q = t; q < NP * T2 * 4; q += NT) {
      const int og = q / (NP * T2), r = q % (NP * T2), ip = r / T2, j = r % T2;
      float a[2][4];
#pragma unroll
      for (int m = 0; m < 2; ++m)
#pragma unroll
        for (int o = 0; o < 4; ++o) a[m][o] = b2[4 * og + o];
      const float* hp = h1 + 4 * ip * P + j;
      const int down = 2 * ip + 1 < T2 ? P : 0;  // rows 3 and 4 repeat row 2 where the second pixel lies outside
#pragma unroll 1
      for (int c = 0; c < kC; ++c, hp += P * P) {
        float v[5][3];
#pragma unroll
        for (int k = 0; k < 5; ++k) {
          const float* h = hp + (k < 3 ? k * P : 2 * P + (k - 2) * down);
          v[k][0] = h[0];
          v[k][1] = h[H];
          v[k][2] = h[1];
        }
#pragma unroll
        for (int tap = 0; tap < 9; ++tap) {
          const float4 wv = w2[(c * 9 + tap) * 4 + og];
#pragma unroll
          for (int m = 0; m < 2; ++m) {
            const float hv = v[2 * m + tap / 3][tap % 3];
            a[m][0] = mul_add(wv.x, hv, a[m][0]);
            a[m][1] = mul_add(wv.y, hv, a[m][1]);
            a[m][2] = mul_add(wv.z, hv, a[m][2]);
            a[m][3] = mul_add(wv.w, hv, a[m][3]);
          }
        }
      }
#pragma unroll
      for (int m = 0; m < 2; ++m)
        if (2 * ip + m < T2)
#pragma unroll
          for (int o = 0; o < 4; ++o) h2[((4 * og + o) * P2 + 2 * ip + m + 1) * P2 + j + 1] = fmaxf(a[m][o], 0.f);
    }
    __syncthreads();
    // conv3
    for (int q = t; q < T3 * T3 * 4; q += NT) {
      const int og = q / (T3 * T3), pix = q % (T3 * T3), i = pix / T3, j = pix % T3;
      float a[4];
#pragma unroll
      for (int o = 0; o < 4; ++o) a[o] = b3[4 * og + o];
      const float* hp = h2 + 2 * i * P2 + 2 * j;
#pragma unroll 1
      for (int c = 0; c < kC; ++c)
#pragma unroll
        for (int tap = 0; tap < 9; ++tap) {
          const float hv = hp[(c * P2 + tap / 3) * P2 + tap % 3];
          const float4 wv = w3[(c * 9 + tap) * 4 + og];
          a[0] = mul_add(wv.x, hv, a[0]);
          a[1] = mul_add(wv.y, hv, a[1]);
          a[2] = mul_add(wv.z, hv, a[2]);
          a[3] = mul_add(wv.w, hv, a[3]);
        }
#pragma unroll
      for (int o = 0; o < 4; ++o) h3[(4 * og + o) * T3 * T3 + pix] = fmaxf(a[o], 0.f);
    }
    __syncthreads();
    // global maximum of each channel and its first pixel
    for (int c = warp; c < kC; c += NT / 32) {
      float m = -1.f;
      int a = 1 << 20;
      for (int q = lane; q < T3 * T3; q += 32) {
        const float v = h3[c * T3 * T3 + q];
        if (v > m) { m = v; a = q; }
      }
      for (int s = 16; s > 0; s >>= 1) {
        const float om = __shfl_xor_sync(0xffffffffu, m, s);
        const int oa = __shfl_xor_sync(0xffffffffu, a, s);
        if (om > m || (om == m && oa < a)) { m = om; a = oa; }
      }
      if (lane == 0) { z[c] = m; arg[c] = a; }
    }
    __syncthreads();
    float logit = *bl;
#pragma unroll
    for (int o = 0; o < kC; ++o) logit = mul_add(wl[o], z[o], logit);
    const float p = 1.f / (1.f + expf(-logit));
    const float dl = (yv * w_pos * (p - 1.f) + (1.f - yv) * p) / nb;
    if (t == 0) {
      const float pc = fminf(fmaxf(p, 1e-7f), 1.f - 1e-7f);
      lsum += -(w_pos * yv * logf(pc) + (1.f - yv) * logf(1.f - pc)) / nb;
      if (prob_out) prob_out[s0 + sb] = p;
      gbl += dl;
    }
    if (t < kC) {
      gwl = fmaf(dl, z[t], gwl);
      if (z[t] > 0.f) gb3 = fmaf(dl, wl[t], gb3);
    }
    // conv3: da3 is nonzero only at each channel's (first) maximum, if positive
    if (t < 256) {
      const float da = z[o3] > 0.f ? dl * wl[o3] : 0.f;
      if (da != 0.f) {
        const float* hp = h2 + (c3 * P2 + 2 * (arg[o3] / T3)) * P2 + 2 * (arg[o3] % T3);
#pragma unroll
        for (int tap = 0; tap < 9; ++tap) g3[tap] = fmaf(da, hp[(tap / 3) * P2 + tap % 3], g3[tap]);
      }
    }
    if (warp >= 6) {
      // gradient of h2, added output by output: a warp holds the 9 taps of 3 channels
      const int c = (warp - 6) * 3 + lane / 9, tap = lane % 9;
      for (int o = 0; o < kC; ++o) {
        const float da = z[o] > 0.f ? dl * wl[o] : 0.f;
        const int ii = 2 * (arg[o] / T3) + tap / 3 - 1, jj = 2 * (arg[o] % T3) + tap % 3 - 1;
        if (lane < 27 && c < kC && da != 0.f && ii >= 0 && ii < T2 && jj >= 0 && jj < T2) {
          float* d = d2 + (ii * T2 + jj) * DP + c;
          *d = fmaf(da, sm[G::W3 + (c * 9 + tap) * kC + o], *d);
        }
        __syncwarp();
      }
    }
    __syncthreads();
    for (int q = t; q < T2 * T2 * kC; q += NT) {  // da2 = dh2 * relu'(a2)
      const int pix = q >> 4, o = q & 15;
      if (!(h2[(o * P2 + pix / T2 + 1) * P2 + pix % T2 + 1] > 0.f)) d2[pix * DP + o] = 0.f;
    }
    __syncthreads();
    // conv2 weights: dW2[o][c][di][dj] = sum_pix da2[o][pix] h1[c][2i+di-1][2j+dj-1]
    float s2[4][3] = {};
    for (int i = part2; i < T2; i += NT / 192) {
      const float* hr = h1 + (c2 * P + 2 * i + di2) * P;
      const float4* dr = reinterpret_cast<const float4*>(d2 + i * T2 * DP) + og2;
      float e0 = hr[0];
      for (int j = 0; j < T2; ++j) {
        const float4 d = dr[j * (DP / 4)];
        const float od = hr[H + j], e1 = hr[j + 1];
        const float dv[4] = {d.x, d.y, d.z, d.w};
#pragma unroll
        for (int o = 0; o < 4; ++o)
          if (dv[o] != 0.f) {
            s2[o][0] = fmaf(dv[o], e0, s2[o][0]);
            s2[o][1] = fmaf(dv[o], od, s2[o][1]);
            s2[o][2] = fmaf(dv[o], e1, s2[o][2]);
          }
        e0 = e1;
      }
    }
#pragma unroll
    for (int o = 0; o < 4; ++o)
#pragma unroll
      for (int dj = 0; dj < 3; ++dj) g2[o][dj] += s2[o][dj];
    {  // bias: NT / 16 threads per channel
      const int o = t & 15;
      float sb2 = 0.f;
      for (int pix = t >> 4; pix < T2 * T2; pix += NT / 16) sb2 += d2[pix * DP + o];
      gb2 += sb2;
    }
    __syncthreads();
    // da1 = conv2^T(da2) * relu'(a1), written over h1: pixels (2a, 2b) .. (2a+1, 2b+1)
    for (int q = t; q < T2 * T2 * 8; q += NT) {
      const int cg = q / (T2 * T2), r = q % (T2 * T2), a = r / T2, b = r % T2;
      float s[2][2][2] = {};  // channel, row, column
      const bool ra = a + 1 < T2, rb = b + 1 < T2;
      const float4* dp = reinterpret_cast<const float4*>(d2 + r * DP);
#pragma unroll 1
      for (int o4 = 0; o4 < 4; ++o4) {
        const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
        float4 d[2][2];
        d[0][0] = dp[o4];
        d[0][1] = rb ? dp[o4 + DP / 4] : zero;
        d[1][0] = ra ? dp[o4 + T2 * (DP / 4)] : zero;
        d[1][1] = ra && rb ? dp[o4 + (T2 + 1) * (DP / 4)] : zero;
#pragma unroll
        for (int c = 0; c < 2; ++c)
#pragma unroll
          for (int tap = 0; tap < 9; ++tap) {
            const int di = tap / 3, dj = tap % 3;
            const float4 wv = w2[((2 * cg + c) * 9 + tap) * 4 + o4];
            const float4 dv = d[di == 0][dj == 0];
            float& u = s[c][di != 1][dj != 1];
            u = fmaf(wv.x, dv.x, u);
            u = fmaf(wv.y, dv.y, u);
            u = fmaf(wv.z, dv.z, u);
            u = fmaf(wv.w, dv.w, u);
          }
      }
#pragma unroll
      for (int c = 0; c < 2; ++c)
#pragma unroll
        for (int m = 0; m < 4; ++m) {
          const int i = 2 * a + m / 2, j = 2 * b + m % 2;
          if (i >= T || j >= T) continue;
          float* h = h1 + G::h1at(2 * cg + c, i + 1, j + 1);
          *h = *h > 0.f ? s[c][m / 2][m % 2] : 0.f;
        }
    }
    __syncthreads();
    // conv1 weights: dW1[o][k][di][dj] = sum_pix da1[o][pix] x[k][i+di-1][j+dj-1]
    float s1[2][2][3] = {}, sb1[2] = {};
    for (int i = part1; i < T; i += NT / 24) {
      const float* xr = x + (i + di1) * P;
      const float* ha = h1 + (2 * op1 * P + i + 1) * P;
      const float* hb = ha + P * P;
      float xv[2][3];
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        xv[k][0] = xr[k * P * P];
        xv[k][1] = xr[k * P * P + 1];
      }
      auto add = [&](float da, float db, int j) {
#pragma unroll
        for (int k = 0; k < 2; ++k) xv[k][2] = xr[k * P * P + j + 2];
        if (da != 0.f) {
#pragma unroll
          for (int k = 0; k < 2; ++k)
#pragma unroll
            for (int dj = 0; dj < 3; ++dj) s1[0][k][dj] = fmaf(da, xv[k][dj], s1[0][k][dj]);
        }
        if (db != 0.f) {
#pragma unroll
          for (int k = 0; k < 2; ++k)
#pragma unroll
            for (int dj = 0; dj < 3; ++dj) s1[1][k][dj] = fmaf(db, xv[k][dj], s1[1][k][dj]);
        }
        sb1[0] += da;
        sb1[1] += db;
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          xv[k][0] = xv[k][1];
          xv[k][1] = xv[k][2];
        }
      };
      // node j is padded column j + 1: odd columns of the row for even j
      for (int m = 0; m < T / 2; ++m) {
        add(ha[H + m], hb[H + m], 2 * m);
        add(ha[m + 1], hb[m + 1], 2 * m + 1);
      }
      add(ha[H + T / 2], hb[H + T / 2], T - 1);
    }
#pragma unroll
    for (int o = 0; o < 2; ++o) {
#pragma unroll
      for (int k = 0; k < 2; ++k)
#pragma unroll
        for (int dj = 0; dj < 3; ++dj) g1[o][k][dj] += s1[o][k][dj];
      gb1[o] += sb1[o];
    }
  }
  // sum of the CTA's threads in shared memory, then one addition per parameter
  __syncthreads();
  float* ga = h1;
  for (int q = t; q < kCnnParams; q += NT) ga[q] = 0.f;
  __syncthreads();
  if (t < 256)
#pragma unroll
    for (int tap = 0; tap < 9; ++tap) ga[kW3 + (o3 * kC + c3) * 9 + tap] = g3[tap];
#pragma unroll
  for (int o = 0; o < 4; ++o)
#pragma unroll
    for (int dj = 0; dj < 3; ++dj) atomicAdd(&ga[kW2 + ((4 * og2 + o) * kC + c2) * 9 + di2 * 3 + dj], g2[o][dj]);
#pragma unroll
  for (int o = 0; o < 2; ++o) {
#pragma unroll
    for (int k = 0; k < 2; ++k)
#pragma unroll
      for (int dj = 0; dj < 3; ++dj) atomicAdd(&ga[kW1 + ((2 * op1 + o) * 2 + k) * 9 + di1 * 3 + dj], g1[o][k][dj]);
    if (di1 == 0) atomicAdd(&ga[kB1 + 2 * op1 + o], gb1[o]);
  }
  atomicAdd(&ga[kB2 + (t & 15)], gb2);
  if (t < kC) {
    ga[kB3 + t] = gb3;
    ga[kWL + t] = gwl;
  }
  if (t == 0) ga[kBL] = gbl;
  // the CTAs of a cluster are added up first: with two CTAs per SM one addition per CTA
  // would lose more bits than one per SM (3000 samples of 25^2, gradient against FP64:
  // 2.7e-7 and 1.8e-7; clusters of four 1.3e-7, but 960 instead of 675 us per call)
  __shared__ float ls;
  if (t == 0) ls = lsum;
  namespace cg = cooperative_groups;
  const cg::cluster_group cl = cg::this_cluster();
  cl.sync();
  if (cl.block_rank() == 0) {
    const unsigned n = cl.num_blocks();
    for (int q = t; q < kCnnParams; q += NT) {
      float v = ga[q];
      for (unsigned r = 1; r < n; ++r) v += cl.map_shared_rank(ga, r)[q];
      if (v != 0.f) atomicAdd(&grad[q], v);
    }
    if (t == 0 && loss) {
      float v = ls;
      for (unsigned r = 1; r < n; ++r) v += *cl.map_shared_rank(&ls, r);
      atomicAdd(loss, v);
    }
  }
  cl.sync();  // until their sums have been read
}

__global__ void k_adam(float* w, float* m, float* v, float* g, int n, float lr, float b1, float b2,
                       float eps, int t, __nv_bfloat16* wb) {
  pdl_enter();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  // a non-finite gradient entry (seen once in a 64-tree training run, cause
  // not found) is skipped rather than allowed to poison the moments
  const float gi = isfinite(g[i]) ? g[i] : 0.f;
  const float mi = b1 * m[i] + (1.f - b1) * gi;
  const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
  m[i] = mi;
  v[i] = vi;
  const float mh = mi / (1.f - powf(b1, (float)t)), vh = vi / (1.f - powf(b2, (float)t));
  w[i] -= lr * mh / (sqrtf(vh) + eps);
  g[i] = 0.f;
  wb[i] = __float2bfloat16(w[i]);
}

__global__ void k_to_bf16(const float* w, __nv_bfloat16* wb, int n) {
  pdl_enter();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) wb[i] = __float2bfloat16(w[i]);
}

// ------------------------------------------------------ proposal at step -----
// flag = 1 (refine) if the block is below Jmax and (p >= tau or its own largest
// normalised detail >= eps); skip marks blocks left unrefined (for the miss check).
__global__ void k_propose(PoolView pv, const float* prob, const float* mpre, float tau, int8_t* skip,
                          int32_t* counts) {
  pdl_enter();
  const int nact = pv.cnt->n_act;
  for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < nact; p += gridDim.x * blockDim.x) {
    const int s = pv.act[p];
    const TreeDev& td = pv.trees[pv.tree[s]];
    const bool below = pv.lvl[s] < td.Jmax;
    const bool net = below && prob[p] >= tau;
    const bool fb = below && (double)mpre[p] >= td.eps;
    pv.flag[s] = (net || fb) ? 1 : 0;
    skip[s] = below && !(net || fb) ? 1 : 0;
    if (below) atomicAdd(&counts[0], 1);
    if (net) atomicAdd(&counts[1], 1);
    if (fb && !net) atomicAdd(&counts[2], 1);
  }
}

// Gradedness closure of +1 flags: a refined block forces the refinement of
// every touching leaf one level coarser (monotone 0 -> 1, order independent).
// The touching leaves are the level-(l-1) leaves covering the ring of
// level-(l+1) cells around the block.  skip (nullable) marks blocks left
// unrefined by a proposal.
template <int D>
__global__ void k_close(PoolView pv, int8_t* skip, int32_t* changed) {
  pdl_enter();
  const int nact = pv.cnt->n_act;
  constexpr int NR = D == 3 ? 64 : 16;
  for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < nact; p += gridDim.x * blockDim.x) {
    const int s = pv.act[p];
    if (pv.flag[s] != 1) continue;
    const BlockInfo b = load_block(pv, s);
    const TreeDev& td = pv.trees[b.tree];
    if (b.lvl >= td.Jmax || b.lvl - 1 < td.Jmin) continue;
    const int64_t nl1 = (int64_t)1 << (b.lvl + 1);
    for (int r = 0; r < NR; ++r) {
      const int q[3] = {r % 4 - 1, (r / 4) % 4 - 1, r / 16 - 1};
      bool inside = true;
      for (int a = 0; a < D; ++a) inside &= (q[a] == 0 || q[a] == 1);
      if (inside) continue;
      int64_t c2[3] = {0, 0, 0};
      for (int a = 0; a < D; ++a) c2[a] = ((2 * b.c[a] + q[a]) & (nl1 - 1)) >> 2;
      const int t = tab_get<D>(pv, td, b.lvl - 1, c2);
      if (t >= 0 && pv.flag[t] != 1) {
        pv.flag[t] = 1;
        if (skip) skip[t] = 0;
        atomicAdd(changed, 1);
      }
    }
  }
}

// Refinement indicators given by the caller: flag = +1 for a block below Jmax
// whose mask entry (canonical position) is positive, else 0.
__global__ void k_mask_flags(PoolView pv, const int8_t* mask) {
  pdl_enter();
  const int nact = pv.cnt->n_act;
  for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < nact; p += gridDim.x * blockDim.x) {
    const int s = pv.act[p];
    pv.flag[s] = (mask[p] > 0 && pv.lvl[s] < pv.trees[pv.tree[s]].Jmax) ? 1 : 0;
  }
}

// Miss check: a block left unrefined whose details after the step are >= eps.
__global__ void k_miss_check(PoolView pv, const int8_t* skip, const int32_t* skip_key, int32_t* counts) {
  pdl_enter();
  const int nact = pv.cnt->n_act;
  for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < nact; p += gridDim.x * blockDim.x) {
    const int s = pv.act[p];
    if (!skip[s]) continue;
    const int key = (pv.lvl[s] << 24) ^ (pv.crd[3 * s] << 12) ^ pv.crd[3 * s + 1];
    if (skip_key[s] != key) continue;  // the slot now holds another block
    if (pv.mdet[s] >= pv.trees[pv.tree[s]].eps) atomicAdd(&counts[3], 1);
  }
}

__global__ void k_skip_key(PoolView pv, const int8_t* skip, int32_t* skip_key) {
  pdl_enter();
  const int nact = pv.cnt->n_act;
  for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < nact; p += gridDim.x * blockDim.x) {
    const int s = pv.act[p];
    skip_key[s] = skip[s] ? ((pv.lvl[s] << 24) ^ (pv.crd[3 * s] << 12) ^ pv.crd[3 * s + 1]) : -1;
  }
}

// Labels of the samples recorded before a step: 1 iff the refinement was needed
// -- the block's region is subdivided after the step (its refinement was kept),
// or the block is a leaf again and its details reached eps (what the miss check
// counts as a miss when the block was left unrefined) -- 0 otherwise; -1 for
// blocks at Jmax.
// Samples whose own details were >= eps (mpre) are refined by the exact
// fallback whatever the network says; they get -1 too (not trained on).
__global__ void k_label(PoolView pv, const int32_t* key, const float* mpre, int64_t n, float* label) {
  pdl_enter();
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int tree = key[4 * i], l = key[4 * i + 1];
    const TreeDev& td = pv.trees[tree];
    if (l >= td.Jmax || (double)mpre[i] >= td.eps) { label[i] = -1.f; continue; }
    int64_t c[3] = {key[4 * i + 2], key[4 * i + 3], 0};
    const int self = tab_get<2>(pv, td, l, c);
    if (self >= 0) {  // merged back: positive iff its details reached eps (the miss check's event)
      label[i] = pv.mdet[self] >= td.eps ? 1.f : 0.f;
      continue;
    }
    bool above = false;
    for (int m = l - 1; m >= td.Jmin && !above; --m) {
      int64_t cm[3] = {c[0] >> (l - m), c[1] >> (l - m), 0};
      above = tab_get<2>(pv, td, m, cm) >= 0;
    }
    label[i] = above ? 0.f : 1.f;
  }
}

__global__ void k_sample_keys(PoolView pv, int32_t* key, int64_t base) {
  pdl_enter();
  const int nact = pv.cnt->n_act;
  for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < nact; p += gridDim.x * blockDim.x) {
    const int s = pv.act[p];
    int32_t* k = key + 4 * (base + p);
    k[0] = pv.tree[s];
    k[1] = pv.lvl[s];
    k[2] = pv.crd[3 * s];
    k[3] = pv.crd[3 * s + 1];
  }
}

// ------------------------------------------------------------- launchers -----
template <typename K>
static void prep(K kernel, size_t bytes) {
  if (bytes > 48 * 1024) cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

int cnn_tile(int Bs) { return Bs + 2 * kG; }

void launch_features(const PoolView& pv, const void* y, float* feat, float* mpre, int64_t base,
                     int num_sms, cudaStream_t st) {
  const bool d = pv.prec != MR_PREC_FP32;
  if (pv.Bs == 17) {
    const size_t smem = FeatGeo<17>::smem(pv.nvar);
    if (d) { auto k = k_features<17, double>; prep(k, smem); k<<<num_sms * 2, 256, smem, st>>>(pv, (const double*)y, feat, mpre, base); }
    else { auto k = k_features<17, float>; prep(k, smem); k<<<num_sms * 2, 256, smem, st>>>(pv, (const float*)y, feat, mpre, base); }
  } else {
    const size_t smem = FeatGeo<33>::smem(pv.nvar);
    if (d) { auto k = k_features<33, double>; prep(k, smem); k<<<num_sms * 2, 256, smem, st>>>(pv, (const double*)y, feat, mpre, base); }
    else { auto k = k_features<33, float>; prep(k, smem); k<<<num_sms * 2, 256, smem, st>>>(pv, (const float*)y, feat, mpre, base); }
  }
  count_launch();
}

template <int T>
static size_t infer_smem() {
  return InferGeo<T>::SMEM;
}
void launch_infer(const PoolView& pv, int Bs, const float* feat, const __nv_bfloat16* wb, float* prob,
                  int64_t n_explicit, int num_sms, cudaStream_t st) {
  if (Bs == 17) {
    auto k = k_cnn_infer<25>;
    prep(k, infer_smem<25>());
    k<<<num_sms * 4, 256, infer_smem<25>(), st>>>(pv, feat, wb, prob, n_explicit);
  } else {
    auto k = k_cnn_infer<41>;
    prep(k, infer_smem<41>());
    k<<<num_sms * 2, 256, infer_smem<41>(), st>>>(pv, feat, wb, prob, n_explicit);
  }
  count_launch();
}

void launch_train(int Bs, const float* feat, const float* label, const int32_t* idx, int64_t s0, int nb,
                  const float* w, float w_pos, float* grad, float* loss, float* prob_out, int num_sms,
                  cudaStream_t st) {
  auto go = [&](auto k, auto geo) {
    using G = decltype(geo);
    prep(k, G::SMEM);
    // clusters of two CTAs where two share an SM (a CTA beyond the samples adds zeros)
    const unsigned cs = G::MINB;
    cudaLaunchAttribute at = {};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = cs;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = ((unsigned)std::min(nb, num_sms * G::MINB) + cs - 1) / cs * cs;
    cfg.blockDim = G::NT;
    cfg.dynamicSmemBytes = G::SMEM;
    cfg.stream = st;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, k, feat, label, idx, s0, nb, w, w_pos, grad, loss, prob_out);
  };
  if (Bs == 17) go(k_cnn_train<25>, TrainGeo<25>{});
  else go(k_cnn_train<41>, TrainGeo<41>{});
  count_launch();
}

void launch_adam(float* w, float* m, float* v, float* g, float lr, int t, __nv_bfloat16* wb, cudaStream_t st) {
  k_adam<<<(kCnnParams + 255) / 256, 256, 0, st>>>(w, m, v, g, kCnnParams, lr, 0.9f, 0.999f, 1e-8f, t, wb);
  count_launch();
}
void launch_to_bf16(const float* w, __nv_bfloat16* wb, cudaStream_t st) {
  k_to_bf16<<<(kCnnParams + 255) / 256, 256, 0, st>>>(w, wb, kCnnParams);
  count_launch();
}
void launch_propose(const PoolView& pv, const float* prob, const float* mpre, float tau, int8_t* skip,
                    int32_t* counts, cudaStream_t st) {
  k_propose<<<256, 256, 0, st>>>(pv, prob, mpre, tau, skip, counts);
  count_launch();
}
void launch_close(const PoolView& pv, int8_t* skip, int32_t* changed, cudaStream_t st) {
  if (pv.dim == 3) k_close<3><<<256, 256, 0, st>>>(pv, skip, changed);
  else k_close<2><<<256, 256, 0, st>>>(pv, skip, changed);
  count_launch();
}
void launch_mask_flags(const PoolView& pv, const int8_t* mask, cudaStream_t st) {
  k_mask_flags<<<256, 256, 0, st>>>(pv, mask);
  count_launch();
}
void launch_miss_check(const PoolView& pv, const int8_t* skip, const int32_t* skip_key, int32_t* counts,
                  cudaStream_t st) {
  k_miss_check<<<256, 256, 0, st>>>(pv, skip, skip_key, counts);
  count_launch();
}
void launch_skip_key(const PoolView& pv, const int8_t* skip, int32_t* skip_key, cudaStream_t st) {
  k_skip_key<<<256, 256, 0, st>>>(pv, skip, skip_key);
  count_launch();
}
void launch_sample_keys(const PoolView& pv, int32_t* key, int64_t base, cudaStream_t st) {
  k_sample_keys<<<256, 256, 0, st>>>(pv, key, base);
  count_launch();
}
void launch_label(const PoolView& pv, const int32_t* key, const float* mpre, int64_t n, float* label,
                  cudaStream_t st) {
  k_label<<<256, 256, 0, st>>>(pv, key, mpre, n, label);
  count_launch();
}

}  // namespace mr
