// Navier-Stokes kernels (Sec. 4): the RK stages in the flux form and in the
// skew-symmetric form, and the shock-capturing filter applied after each step.
// Instantiated in mr_ns.cu.
//
// Tiles hold the four variables of a node side by side: a neighbour of a node is one
// 16-byte load instead of four, and 8 lanes of such a load read 128 consecutive
// bytes, also where a warp passes from one row of the block to the next (the rows of
// the tile, B + 8 nodes, are 8 nodes = 128 bytes longer than the block's), so the
// stencils read shared memory without bank conflicts.  With one array per variable
// every such load took two wavefronts, 73 % of what the shared-memory pipe carries.
#pragma once
#include "mr_kernels.cuh"

namespace mr {

template <typename T>
struct Vec4 {
  T a, b, c, d;
};
template <typename T>
struct Vec2 {
  T a, b;
};
__device__ __forceinline__ Vec4<float> ld4(const float* p) {
  const float4 v = *reinterpret_cast<const float4*>(p);
  return {v.x, v.y, v.z, v.w};
}
__device__ __forceinline__ Vec4<double> ld4(const double* p) {
  const double2 v = *reinterpret_cast<const double2*>(p), w = *reinterpret_cast<const double2*>(p + 2);
  return {v.x, v.y, w.x, w.y};
}
__device__ __forceinline__ void st4(float* p, float a, float b, float c, float d) {
  *reinterpret_cast<float4*>(p) = make_float4(a, b, c, d);
}
__device__ __forceinline__ void st4(double* p, double a, double b, double c, double d) {
  *reinterpret_cast<double2*>(p) = make_double2(a, b);
  *reinterpret_cast<double2*>(p + 2) = make_double2(c, d);
}
__device__ __forceinline__ Vec2<float> ld2(const float* p) {
  const float2 v = *reinterpret_cast<const float2*>(p);
  return {v.x, v.y};
}
__device__ __forceinline__ Vec2<double> ld2(const double* p) {
  const double2 v = *reinterpret_cast<const double2*>(p);
  return {v.x, v.y};
}
__device__ __forceinline__ void st2(float* p, float a, float b) { *reinterpret_cast<float2*>(p) = make_float2(a, b); }
__device__ __forceinline__ void st2(double* p, double a, double b) {
  *reinterpret_cast<double2*>(p) = make_double2(a, b);
}

// Ghost gather of the full tile (width 4, four variables) for a block with a
// uniform neighbourhood; nbo: pool offsets of the 3 x 3 blocks.  With commit,
// block-edge nodes held by a neighbour are stored where the block's copy differs.
template <int B, int NT, typename TF, typename TC>
__device__ __forceinline__ void gather4(const PoolView& pv, const int64_t* nbo, const TF* F, TF* Fw, TC* tile,
                                        bool commit) {
  // U nodes per thread and pass, 4 U loads in flight
  constexpr int G = kG, T = B + 2 * G, NP = T * T, UM = sizeof(TF) == 4 ? 3 : 2;
  constexpr int R = (NP + NT - 1) / NT, PASSES = (R + UM - 1) / UM, U = (R + PASSES - 1) / PASSES;
  const int64_t vs = pv.vs;
#pragma unroll 1
  for (int q0 = threadIdx.x; q0 < NP; q0 += U * NT) {
    TF v[U][4];
    int ed[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int q = q0 + u * NT;
      ed[u] = -1;
      if (q >= NP) continue;
      const int i = q % T - G, j = q / T - G;
      const int sx = (i >= 0) + (i >= B - 1), sy = (j >= 0) + (j >= B - 1);
      const TF* p = F + nbo[sx + 3 * sy] + (i - (sx - 1) * (B - 1)) + B * (j - (sy - 1) * (B - 1));
#pragma unroll
      for (int w = 0; w < 4; ++w) v[u][w] = p[w * vs];
      if (commit && i >= 0 && i <= B - 1 && j >= 0 && j <= B - 1 && (sx == 2 || sy == 2)) ed[u] = j * B + i;
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int q = q0 + u * NT;
      if (q >= NP) continue;
      st4(tile + 4 * q, to_tile<TC>(v[u][0]), to_tile<TC>(v[u][1]), to_tile<TC>(v[u][2]), to_tile<TC>(v[u][3]));
      if (ed[u] >= 0) {
        const int64_t me = nbo[4] + ed[u];
#pragma unroll
        for (int w = 0; w < 4; ++w)
          if (differs(F[me + w * vs], v[u][w])) Fw[me + w * vs] = v[u][w];
      }
    }
  }
}

// RK update of one variable of one node (the 3-register form of the advection
// stage).  With an FP64 state and FP32 stages the increments dt k are formed in
// FP32 and only accumulated in FP64 (FP64 arithmetic is a small fraction of the
// FP32 rate here), and the next stage field needs y_n only in FP32: stage 0 takes
// it from the tile (the committed state, rounded) and keeps it in yn for stages 1
// and 2, which then read no FP64 state.  With copy_state the last stage also stores
// the new state in the stage type into ynext, the shock filter's source.
// INT: widen the increments on the integer pipes (flux form, 2944 blocks of 33^2: 735 ->
// 717 us per step; the skew form, 16384 of 17^2, has no issue slots left: 845 -> 856).
template <typename TS, typename TC, bool INT>
struct NsUpdate {
  static constexpr bool MIX = sizeof(TS) == 8 && sizeof(TC) == 4;
  TS yv, av;
  TC yf;
  __device__ __forceinline__ static TS wide(TC v) {
    if constexpr (INT) return to_state<TS>(v);
    else return (TS)v;
  }
  __device__ __forceinline__ void load(const TS* y, const TS* acc, const TC* yn, int64_t at, int stage) {
    // stage 0 of one type takes the committed state from the tile
    yv = (MIX ? stage == 0 : stage == 1 || stage == 2) ? y[at] : TS(0);
    av = stage >= 1 ? acc[at] : TS(0);
    yf = TC(0);
    if (MIX && (stage == 1 || stage == 2)) yf = yn[at];
  }
  __device__ __forceinline__ void store(TS* y, TS* acc, TC* ynext, TC* yn, int64_t at, int stage, TC k, TC tile0,
                                        const StageCoef<TS>& cs, const StageCoef<TC>& cf, int copy_state) {
    if constexpr (MIX) {
      if (stage == 0) {
        yn[at] = tile0;
        acc[at] = yv + wide(cf.ca * k);
        ynext[at] = tile0 + cf.cy * k;
      } else if (stage == 1 || stage == 2) {
        acc[at] = av + wide(cf.ca * k);
        ynext[at] = yf + cf.cy * k;
      } else {
        const TS n = av + wide(cf.ca * k);
        y[at] = n;
        if (copy_state) ynext[at] = to_tile<TC>(n);
      }
    } else {
      const TS kk = (TS)k;
      if (stage == 0) {
        acc[at] = (TS)tile0 + cs.ca * kk;
        ynext[at] = (TC)((TS)tile0 + cs.cy * kk);
      } else if (stage == 1 || stage == 2) {
        acc[at] = av + cs.ca * kk;
        ynext[at] = (TC)(yv + cs.cy * kk);
      } else {
        const TS n = av + cs.ca * kk;
        y[at] = n;
        if (copy_state) ynext[at] = (TC)n;
      }
    }
  }
};

// Plans of a CTA's blocks: the next block's plan is fetched while one is processed.
struct NsPlan {
  int32_t pl[2][Plan<2>::INTS];
  int64_t nbo[2][Plan<2>::NB];
  __device__ __forceinline__ void put(const PoolView& pv, int buf, int32_t v) {
    using PL = Plan<2>;
    if (threadIdx.x >= PL::INTS) return;
    pl[buf][threadIdx.x] = v;
    if (threadIdx.x >= PL::NBO && threadIdx.x < PL::NBO + PL::NB)
      nbo[buf][threadIdx.x - PL::NBO] = (int64_t)v * 4 * pv.vs;
  }
  __device__ __forceinline__ static int32_t fetch(const PoolView& pv, int p, int nact) {
    return p < nact && threadIdx.x < Plan<2>::INTS ? pv.plan[(int64_t)p * Plan<2>::INTS + threadIdx.x] : 0;
  }
};

// ---------------------------------------------------- NS stage, flux form ----
// One RK4 stage of the 2D compressible Navier-Stokes equations (Sec. 4), ideal
// gas with constant c_p, in conservative flux form, q = (rho, rho u, rho v, E):
//   N(q) = -(dF/dx + dG/dy),
//   F = (rho u, rho u u + p - txx, rho u v - txy, (E + p) u - (u txx + v txy) - kap dth/dx),
//   G = (rho v, rho v u - txy, rho v v + p - tyy, (E + p) v - (u txy + v tyy) - kap dth/dy),
//   txx = mu (2 ux - 2/3 div), tyy = mu (2 vy - 2/3 div), txy = mu (uy + vx),
//   p = (gamma - 1)(E - (rho u u + rho v v)/2), th = p / rho,
//   kap = mu gamma / ((gamma - 1) Pr)  (R_s cancels in the heat flux),
// every derivative the 4th-order central D1.  Primitives on the whole tile,
// gradients and fluxes on nodes -2..B+1, flux divergence on the interior.
// Bound by issue slots and shared wavefronts: node-major tiles read the four
// variables of a neighbour in one 16-byte load.  Measured per launch (2944 blocks
// of 33^2, FP32 stages, FP64 state, 2 CTAs per SM): 183 us with 384 threads, 188
// with 512, 212 with 256; one CTA of 576 threads per SM 250; variable-major
// tiles 230.
template <int B, typename TY>
struct NsSmem {
  static constexpr int T = B + 2 * kG, TILE = T * T;
  static constexpr int FP = B + 8;            // pitch of F rows: i in [-2, B+1], j in [0, B-1]
  static constexpr int NF = B * FP;
  static constexpr int NG = (B + 4) * B;      // G: i in [0, B-1], j in [-2, B+1]
  using Bx = Box<2, B, kG>;
  static_assert(4 * Bx::SCR <= 4 * TILE, "prediction scratch fits in the primitives");
  static_assert(4 * Bx::CBOX <= 4 * (NF + NG), "coarse box fits in the fluxes");
  static constexpr size_t RING = ((size_t)kRingBytesD<2> + 15) / 16 * 16;
  static constexpr size_t BYTES = RING + sizeof(TY) * 4 * (2 * TILE + NF + NG);
};

// FP64 stages: the tiles of 33^2 leave room for one CTA per SM
template <int B, typename TY>
struct NsCfg {
  static constexpr int NT = B == 17 ? 256 : 384;
  static constexpr int MINB = B == 17 ? 3 : (sizeof(TY) == 8 ? 1 : 2);
};

template <int B, typename TS, typename TY, typename TSRC>
__global__ void __launch_bounds__(NsCfg<B, TY>::NT, NsCfg<B, TY>::MINB) k_stage_ns(PoolView pv, const TSRC* __restrict__ src,
                                                  TS* __restrict__ y, TS* __restrict__ acc, TY* __restrict__ ynext,
                                                  TY* __restrict__ yn, int stage, StageArgs sa) {
  pdl_enter();
  using TC = TY;
  using SM = NsSmem<B, TY>;
  constexpr int T = SM::T, G = kG, FP = SM::FP, NI = B * B, NT = NsCfg<B, TY>::NT;
  RingD<2>& R = *smem_as<RingD<2>>(0);
  TC* tile = smem_as<TC>(SM::RING);  // rho, rho u, rho v, E
  TC* pr = tile + 4 * SM::TILE;      // u, v, p, th
  TC* F = pr + 4 * SM::TILE;
  TC* Gf = F + 4 * SM::NF;
  __shared__ NsPlan sp;
  const int nact = pv.cnt->n_act;
  if ((int)blockIdx.x >= nact) return;  // no block for this CTA
  if (blockIdx.x == 0 && threadIdx.x == 0) atomicAdd(&pv.cnt->stage_blocks, (unsigned long long)nact);
  auto I = [&](int i, int j) { return 4 * ((j + G) * T + (i + G)); };
  auto fI = [&](int i, int j) { return 4 * (j * FP + (i + 2)); };
  auto gI = [&](int i, int j) { return 4 * ((j + 2) * B + i); };
  sp.put(pv, 0, NsPlan::fetch(pv, blockIdx.x, nact));
  __syncthreads();
  int buf = 0;
  for (int p = blockIdx.x; p < nact; p += gridDim.x, buf ^= 1) {
    const int32_t pre = NsPlan::fetch(pv, p + gridDim.x, nact);
    const int32_t* pl = sp.pl[buf];
    const BlockInfo b = plan_block<2>(pl);
    const TreeDev& td = pv.trees[b.tree];
    if ((pl[1] >> 30) & 1) {
      gather4<B, NT, TSRC, TC>(pv, sp.nbo[buf], src, (TSRC*)src, tile, stage == 0);
    } else {
      load_regions<2, CtaGroup>(pv, p, R);
      __syncthreads();
      fill_tile<2, B, TSRC, TC, kG, CtaGroup, 4>(pv, b, src, (TSRC*)src, tile, stage == 0, R, F, pr, true);
    }
    __syncthreads();
    // gamma - 1, mu and kappa = mu gamma / ((gamma - 1) Pr), formed once per tree
    TC gm1, mu, kap;
    if constexpr (sizeof(TC) == 4) { gm1 = td.nsf[0]; mu = td.nsf[1]; kap = td.nsf[2]; }
    else { gm1 = td.nsd[0]; mu = td.nsd[1]; kap = td.nsd[2]; }
    const TC c23 = (TC)(2.0 / 3.0);
    const TC c = tree_cD<TC>(td, b.lvl);
    for (int idx = threadIdx.x; idx < SM::TILE; idx += blockDim.x) {
      const Vec4<TC> q = ld4(tile + 4 * idx);
      const TC uu = q.b / q.a, vv = q.c / q.a;
      const TC prs = gm1 * (q.d - TC(0.5) * (q.b * uu + q.c * vv));
      st4(pr + 4 * idx, uu, vv, prs, prs / q.a);
    }
    __syncthreads();
    constexpr int W = B + 4;
    for (int idx = threadIdx.x; idx < W * W; idx += blockDim.x) {
      const int i = idx % W - 2, j = idx / W - 2;
      const bool needF = j >= 0 && j < B, needG = i >= 0 && i < B;
      if (!needF && !needG) continue;
      const TC* p0 = pr + I(i, j);
      const Vec4<TC> xa = ld4(p0 - 8), xb = ld4(p0 - 4), xc = ld4(p0 + 4), xd = ld4(p0 + 8);
      const Vec4<TC> ya = ld4(p0 - 8 * T), yb = ld4(p0 - 4 * T), yc = ld4(p0 + 4 * T), yd = ld4(p0 + 8 * T);
      const TC ux = d1_sum(xa.a, xb.a, xc.a, xd.a) * c, vx = d1_sum(xa.b, xb.b, xc.b, xd.b) * c;
      const TC uy = d1_sum(ya.a, yb.a, yc.a, yd.a) * c, vy = d1_sum(ya.b, yb.b, yc.b, yd.b) * c;
      const TC div = ux + vy;
      const TC txy = mu * (uy + vx);
      const Vec4<TC> q = ld4(tile + I(i, j)), w = ld4(p0);
      const TC m1 = q.b, m2 = q.c, E = q.d, uu = w.a, vv = w.b, prs = w.c;
      if (needF) {
        const TC txx = mu * (TC(2) * ux - c23 * div);
        const TC thx = d1_sum(xa.d, xb.d, xc.d, xd.d) * c;
        st4(F + fI(i, j), m1, m1 * uu + prs - txx, m1 * vv - txy,
            (E + prs) * uu - (uu * txx + vv * txy) - kap * thx);
      }
      if (needG) {
        const TC tyy = mu * (TC(2) * vy - c23 * div);
        const TC thy = d1_sum(ya.d, yb.d, yc.d, yd.d) * c;
        st4(Gf + gI(i, j), m2, m2 * uu - txy, m2 * vv + prs - tyy,
            (E + prs) * vv - (uu * txy + vv * tyy) - kap * thy);
      }
    }
    __syncthreads();
    const StageCoef<TS> cs(pv, sa, b.tree, stage);  // RK weights in the state type
    const StageCoef<TC> cf(pv, sa, b.tree, stage);  // and in the stage type
    const int64_t base = (int64_t)b.slot * 4 * pv.vs;
    const TS* yc = y;
    if constexpr (sizeof(TS) != sizeof(TC)) yc = committed(y, src);
    for (int q = threadIdx.x; q < NI; q += blockDim.x) {
      const int i = q % B, j = q / B;
      NsUpdate<TS, TC, true> up[4];
#pragma unroll
      for (int v = 0; v < 4; ++v) up[v].load(yc, acc, yn, base + v * pv.vs + q, stage);
      const TC* f0 = F + fI(i, j);
      const TC* g0 = Gf + gI(i, j);
      const Vec4<TC> fa = ld4(f0 - 8), fb = ld4(f0 - 4), fc = ld4(f0 + 4), fd = ld4(f0 + 8);
      const Vec4<TC> ga = ld4(g0 - 8 * B), gb = ld4(g0 - 4 * B), gc = ld4(g0 + 4 * B), gd = ld4(g0 + 8 * B);
      const Vec4<TC> t0 = ld4(tile + I(i, j));
      const TC k[4] = {-(d1_sum(fa.a, fb.a, fc.a, fd.a) * c + d1_sum(ga.a, gb.a, gc.a, gd.a) * c),
                       -(d1_sum(fa.b, fb.b, fc.b, fd.b) * c + d1_sum(ga.b, gb.b, gc.b, gd.b) * c),
                       -(d1_sum(fa.c, fb.c, fc.c, fd.c) * c + d1_sum(ga.c, gb.c, gc.c, gd.c) * c),
                       -(d1_sum(fa.d, fb.d, fc.d, fd.d) * c + d1_sum(ga.d, gb.d, gc.d, gd.d) * c)};
      const TC tv[4] = {t0.a, t0.b, t0.c, t0.d};
#pragma unroll
      for (int v = 0; v < 4; ++v)
        up[v].store(y, acc, ynext, yn, base + v * pv.vs + q, stage, k[v], tv[v], cs, cf, sa.copy_state);
    }
    sp.put(pv, buf ^ 1, pre);
    __syncthreads();
  }
}

// ------------------------------------------------ NS stage, skew form -------
// One RK4 stage of the 2D compressible Navier-Stokes equations in the
// skew-symmetric form of Reiss & Sesterhenn (2014), named in Sec. 4, on the
// square-root variables q = (phi, psi_x, psi_y, p), phi = sqrt(rho),
// psi = phi u (u = psi / phi, th = p / phi^2):
//   d phi/dt   = -1/2 sum_j (D_j psi_j + u_j D_j phi)
//   d psi_i/dt = -1/2 sum_j (D_j(psi_i u_j) + u_j D_j psi_i) - (D_i p - sum_j D_j tau_ij) / phi
//   d p/dt     = -gamma sum_j D_j(p u_j) + (gamma - 1) sum_j u_j D_j p
//                + (gamma - 1) (sum_ij tau_ij D_j u_i + sum_j D_j(kap D_j th)),
// tau_xx = mu (2 u_x - 2/3 div), tau_yy = mu (2 v_y - 2/3 div), tau_xy = mu (u_y + v_x),
// kap = mu gamma / ((gamma - 1) Pr); D is the 4th-order central D1 everywhere.
// The stresses and kap D th are formed on the arms of the interior that their
// second derivative reads (x-arm: i in [-2, B+1] on rows 0..B-1; y-arm: the
// transpose), then every interior node evaluates its four rates at once and
// applies the 3-register RK update of the advection stage.
// Bound by issue slots and shared wavefronts, then by the latency of the gather.
// Measured per launch (FP32 stages, FP64 state, 17^2) on 16384 blocks and on the
// 2944 of an adapted grid: 160 threads, 5 CTAs per SM 228 and 62 us; 128 x 6 220
// and 68; 192 x 4 238 and 74; 224 x 4 248 and 75; variable-major tiles 240 and
// 67.  The adapted grid, the ordinary case, decides.
template <int B, typename TY>
struct NssSmem {
  static constexpr int T = B + 2 * kG, TILE = T * T;
  static constexpr int XP = B + 8;            // pitch of x-arm rows
  static constexpr int NX = B * XP;           // x-arm: tau_xx, tau_xy, kap th_x, -
  static constexpr int NY = (B + 4) * B;      // y-arm: tau_xy, tau_yy, kap th_y, -
  using Bx = Box<2, B, kG>;
  static_assert(4 * Bx::SCR <= 3 * TILE, "prediction scratch fits in the primitives");
  static_assert(4 * Bx::CBOX <= 4 * (NX + NY), "coarse box fits in the arms");
  static constexpr int UV = (2 * TILE + 3) / 4 * 4, TH = (TILE + 3) / 4 * 4;
  static constexpr size_t RING = ((size_t)kRingBytesD<2> + 15) / 16 * 16;
  static constexpr size_t BYTES = RING + sizeof(TY) * (4 * TILE + UV + TH + 4 * (NX + NY));
};

// FP64 stages: shared memory holds three CTAs of 17^2 per SM, or one of 33^2
template <int B, typename TY>
struct NssCfg {
  static constexpr bool F64 = sizeof(TY) == 8;
  static constexpr int NT = B == 17 ? (F64 ? 192 : 160) : 384;
  static constexpr int MINB = B == 17 ? (F64 ? 3 : 5) : (F64 ? 1 : 2);
};

template <int B, typename TS, typename TY, typename TSRC>
__global__ void __launch_bounds__(NssCfg<B, TY>::NT, NssCfg<B, TY>::MINB) k_stage_nss(PoolView pv, const TSRC* __restrict__ src,
                                                   TS* __restrict__ y, TS* __restrict__ acc,
                                                   TY* __restrict__ ynext, TY* __restrict__ yn, int stage,
                                                   StageArgs sa) {
  pdl_enter();
  using TC = TY;
  using SM = NssSmem<B, TY>;
  constexpr int T = SM::T, G = kG, XP = SM::XP, NI = B * B, NT = NssCfg<B, TY>::NT;
  RingD<2>& R = *smem_as<RingD<2>>(0);
  TC* tile = smem_as<TC>(SM::RING);  // phi, psi_x, psi_y, p
  TC* uv = tile + 4 * SM::TILE;      // u, v
  TC* th = uv + SM::UV;
  TC* ax = th + SM::TH;
  TC* ay = ax + 4 * SM::NX;
  __shared__ NsPlan sp;
  const int nact = pv.cnt->n_act;
  if ((int)blockIdx.x >= nact) return;  // no block for this CTA
  if (blockIdx.x == 0 && threadIdx.x == 0) atomicAdd(&pv.cnt->stage_blocks, (unsigned long long)nact);
  auto I = [&](int i, int j) { return (j + G) * T + (i + G); };
  auto xI = [&](int i, int j) { return 4 * (j * XP + (i + 2)); };
  auto yI = [&](int i, int j) { return 4 * ((j + 2) * B + i); };
  sp.put(pv, 0, NsPlan::fetch(pv, blockIdx.x, nact));
  __syncthreads();
  int buf = 0;
  for (int p = blockIdx.x; p < nact; p += gridDim.x, buf ^= 1) {
    const int32_t pre = NsPlan::fetch(pv, p + gridDim.x, nact);
    const int32_t* pl = sp.pl[buf];
    const BlockInfo b = plan_block<2>(pl);
    const TreeDev& td = pv.trees[b.tree];
    if ((pl[1] >> 30) & 1) {
      gather4<B, NT, TSRC, TC>(pv, sp.nbo[buf], src, (TSRC*)src, tile, stage == 0);
    } else {
      load_regions<2, CtaGroup>(pv, p, R);
      __syncthreads();
      fill_tile<2, B, TSRC, TC, kG, CtaGroup, 4>(pv, b, src, (TSRC*)src, tile, stage == 0, R, ax, uv, true);
    }
    __syncthreads();
    TC gm1, mu, kap, gam;
    if constexpr (sizeof(TC) == 4) { gm1 = td.nsf[0]; mu = td.nsf[1]; kap = td.nsf[2]; gam = td.nsf[3]; }
    else { gm1 = td.nsd[0]; mu = td.nsd[1]; kap = td.nsd[2]; gam = td.nsd[3]; }
    const TC c23 = (TC)(2.0 / 3.0);
    const TC c = tree_cD<TC>(td, b.lvl);
    for (int idx = threadIdx.x; idx < SM::TILE; idx += blockDim.x) {
      const Vec4<TC> q = ld4(tile + 4 * idx);
      const TC f = q.a;
      if constexpr (sizeof(TC) == 4) {
        // FP32 stages: one reciprocal instead of three divisions
        const TC rf = TC(1) / f;
        st2(uv + 2 * idx, q.b * rf, q.c * rf);
        th[idx] = (q.d * rf) * rf;
      } else {
        st2(uv + 2 * idx, q.b / f, q.c / f);
        th[idx] = q.d / (f * f);
      }
    }
    __syncthreads();
    constexpr int W = B + 4;
    for (int idx = threadIdx.x; idx < W * W; idx += blockDim.x) {
      const int i = idx % W - 2, j = idx / W - 2;
      const bool needX = j >= 0 && j < B, needY = i >= 0 && i < B;
      if (!needX && !needY) continue;
      const int o = I(i, j);
      const TC* w = uv + 2 * o;
      const Vec2<TC> xa = ld2(w - 4), xb = ld2(w - 2), xc = ld2(w + 2), xd = ld2(w + 4);
      const Vec2<TC> ya = ld2(w - 4 * T), yb = ld2(w - 2 * T), yc = ld2(w + 2 * T), yd = ld2(w + 4 * T);
      const TC ux = d1_sum(xa.a, xb.a, xc.a, xd.a) * c, vx = d1_sum(xa.b, xb.b, xc.b, xd.b) * c;
      const TC uy = d1_sum(ya.a, yb.a, yc.a, yd.a) * c, vy = d1_sum(ya.b, yb.b, yc.b, yd.b) * c;
      const TC div = ux + vy;
      const TC txy = mu * (uy + vx);
      const TC* t0 = th + o;
      if (needX)
        st4(ax + xI(i, j), mu * (TC(2) * ux - c23 * div), txy, kap * (d1_sum(t0[-2], t0[-1], t0[1], t0[2]) * c), TC(0));
      if (needY)
        st4(ay + yI(i, j), txy, mu * (TC(2) * vy - c23 * div),
            kap * (d1_sum(t0[-2 * T], t0[-T], t0[T], t0[2 * T]) * c), TC(0));
    }
    __syncthreads();
    const StageCoef<TS> cs(pv, sa, b.tree, stage);
    const StageCoef<TC> cf(pv, sa, b.tree, stage);
    const int64_t base = (int64_t)b.slot * 4 * pv.vs;
    const TS* yc = y;
    if constexpr (sizeof(TS) != sizeof(TC)) yc = committed(y, src);
    for (int q = threadIdx.x; q < NI; q += blockDim.x) {
      const int i = q % B, j = q / B;
      const int o = I(i, j);
      NsUpdate<TS, TC, false> up[4];
#pragma unroll
      for (int v = 0; v < 4; ++v) up[v].load(yc, acc, yn, base + v * pv.vs + q, stage);
      const Vec2<TC> w0 = ld2(uv + 2 * o);
      const Vec4<TC> s0 = ld4(tile + 4 * o);
      const TC uu = w0.a, vv = w0.b, f = s0.a;
      // derivatives along one axis (neighbours d nodes apart) of the variables, the
      // velocity, and the variables' products with the velocity component `comp`
      struct Der { TC ph, sx, sy, p, u, v, msx, msy, mp; };
      auto along = [&](int d, auto comp) -> Der {
        const Vec4<TC> a = ld4(tile + 4 * (o - 2 * d)), bq = ld4(tile + 4 * (o - d)), cq = ld4(tile + 4 * (o + d)),
                       e = ld4(tile + 4 * (o + 2 * d));
        const Vec2<TC> wa = ld2(uv + 2 * (o - 2 * d)), wb = ld2(uv + 2 * (o - d)), wc = ld2(uv + 2 * (o + d)),
                       we = ld2(uv + 2 * (o + 2 * d));
        const TC ga = comp(wa), gb = comp(wb), gc = comp(wc), ge = comp(we);
        Der r;
        r.ph = d1_sum(a.a, bq.a, cq.a, e.a) * c;
        r.sx = d1_sum(a.b, bq.b, cq.b, e.b) * c;
        r.sy = d1_sum(a.c, bq.c, cq.c, e.c) * c;
        r.p = d1_sum(a.d, bq.d, cq.d, e.d) * c;
        r.u = d1_sum(wa.a, wb.a, wc.a, we.a) * c;
        r.v = d1_sum(wa.b, wb.b, wc.b, we.b) * c;
        r.msx = d1_sum(a.b * ga, bq.b * gb, cq.b * gc, e.b * ge) * c;
        r.msy = d1_sum(a.c * ga, bq.c * gb, cq.c * gc, e.c * ge) * c;
        r.mp = d1_sum(a.d * ga, bq.d * gb, cq.d * gc, e.d * ge) * c;
        return r;
      };
      const Der X = along(1, [](const Vec2<TC>& w) { return w.a; });
      const Der Y = along(T, [](const Vec2<TC>& w) { return w.b; });
      TC k[4];
      // mass
      k[0] = TC(-0.5) * ((X.sx + uu * X.ph) + (Y.sy + vv * Y.ph));
      // momentum
      const TC cx = (X.msx + uu * X.sx) + (Y.msx + vv * Y.sx);
      const TC cy = (X.msy + uu * X.sy) + (Y.msy + vv * Y.sy);
      const TC* a0 = ax + xI(i, j);
      const TC* b0 = ay + yI(i, j);
      const Vec4<TC> aa = ld4(a0 - 8), ab = ld4(a0 - 4), ac = ld4(a0 + 4), ad = ld4(a0 + 8);
      const Vec4<TC> ba = ld4(b0 - 8 * B), bb = ld4(b0 - 4 * B), bc = ld4(b0 + 4 * B), bd = ld4(b0 + 8 * B);
      const TC fx = X.p - (d1_sum(aa.a, ab.a, ac.a, ad.a) * c + d1_sum(ba.a, bb.a, bc.a, bd.a) * c);
      const TC fy = Y.p - (d1_sum(aa.b, ab.b, ac.b, ad.b) * c + d1_sum(ba.b, bb.b, bc.b, bd.b) * c);
      if constexpr (sizeof(TC) == 4) {
        const TC rf = TC(1) / f;
        k[1] = TC(-0.5) * cx - fx * rf;
        k[2] = TC(-0.5) * cy - fy * rf;
      } else {
        k[1] = TC(-0.5) * cx - fx / f;
        k[2] = TC(-0.5) * cy - fy / f;
      }
      // pressure
      const Vec2<TC> ta = ld2(a0);
      const TC tyy = b0[1];
      const TC phiv = (ta.a * X.u + ta.b * (Y.u + X.v)) + tyy * Y.v;
      const TC heat = d1_sum(aa.c, ab.c, ac.c, ad.c) * c + d1_sum(ba.c, bb.c, bc.c, bd.c) * c;
      k[3] = (-gam * (X.mp + Y.mp) + gm1 * (uu * X.p + vv * Y.p)) + gm1 * (phiv + heat);
      const TC tv[4] = {s0.a, s0.b, s0.c, s0.d};
#pragma unroll
      for (int v = 0; v < 4; ++v)
        up[v].store(y, acc, ynext, yn, base + v * pv.vs + q, stage, k[v], tv[v], cs, cf, sa.copy_state);
    }
    sp.put(pv, buf ^ 1, pre);
    __syncthreads();
  }
}

// ------------------------------------------------------- shock filter -------
// Shock-capturing filter of Bogey, de Cacqueray & Bailly (2009), applied after
// every time step in Sec. 4 (threshold r_th of the block's tree), in place on
// the state y.  The synchronised tiles are gathered from `ys`, a copy of the
// state in the stage type that no CTA writes meanwhile (the last RK stage
// stores it), so every CTA updates its own block's interior in y while the
// others read their ghosts.  Per direction a, node n:
//   th_n = (u_{n+1} - u_{n-1}) / (2 dx) + (v_{n+1} - v_{n-1}) / (2 dx)  (each along its axis)
//   Dth_n = (-th_{n+1} + 2 th_n - th_{n-1}) / 4
//   M_n = ((Dth_n - Dth_{n+1})^2 + (Dth_n - Dth_{n-1})^2) / 2
//   r_n = M_n / (c_n^2 / dx^2) + 1e-16,  c^2 = gamma p / rho
//   s_n = (1 - r_th / r_n + |1 - r_th / r_n|) / 2
//   q_n <- q_n - sum_a (s_{n+1/2} F_{n+1/2} - s_{n-1/2} F_{n-1/2}),
//   F_{n+1/2} = -(q_{n+1} - q_n) / 4, s_{n+1/2} = (s_n + s_{n+1}) / 2,
// both directions from the unfiltered tile.  The stencil reaches four nodes
// along a and one across.  Everything is evaluated in TC.  With TS = TC every
// interior node becomes its synchronised value minus the increment (as in
// the oracle); with an FP64 state and FP32 arithmetic the FP32 increment is
// subtracted from the FP64 state where it is not zero (block-edge nodes owned
// by a finer neighbour keep their own value until the next synchronisation
// replaces it by the owner's, as after every RK stage).
// KIND: MR_RHS_NS (q = rho, rho u, rho v, E) or MR_RHS_NS_SKEW (phi, psi, p).
// Instruction-bound (the four variables of a node share the strengths).  Measured
// (16384 blocks of 17^2, FP32 arithmetic on an FP64 state): 149 us with three nodes
// of the gather in flight per thread, 156 with five; 182 with variable-major tiles.
template <int B, typename TC>
struct FilterSmem {
  static constexpr int T = B + 2 * kG, TILE = T * T;
  using Bx = Box<2, B, kG>;
  static constexpr int UV = (2 * TILE + 3) / 4 * 4, C2 = (TILE + 3) / 4 * 4;
  static constexpr int SG = ((B + 2) * B + 3) / 4 * 4;  // strengths of one axis
  static_assert(4 * Bx::SCR <= UV + C2, "prediction scratch fits in the primitives");
  static_assert(4 * Bx::CBOX <= C2 + 2 * SG, "coarse box fits in the dilatation and strengths");
  static constexpr size_t RING = ((size_t)kRingBytesD<2> + 15) / 16 * 16;
  static constexpr size_t BYTES = RING + sizeof(TC) * (4 * TILE + UV + 2 * C2 + 2 * SG);
};

// 160 threads, 5 CTAs per SM
constexpr int kFilterThreads = 160;

template <int B, typename TS, typename TC, int KIND>
__global__ void __launch_bounds__(kFilterThreads, 5) k_filter(PoolView pv, const TC* __restrict__ ys, TS* __restrict__ y) {
  pdl_enter();
  using SM = FilterSmem<B, TC>;
  constexpr int T = SM::T, G = kG, NI = B * B;
  constexpr bool MIX = sizeof(TS) != sizeof(TC);
  RingD<2>& R = *smem_as<RingD<2>>(0);
  TC* tile = smem_as<TC>(SM::RING);
  TC* uv = tile + 4 * SM::TILE;  // u, v
  TC* pc = uv + SM::UV;          // c^2
  TC* th = pc + SM::C2;          // dilatation
  TC* sgx = th + SM::C2;         // s at i in [-1, B], j in [0, B-1]
  TC* sgy = sgx + SM::SG;        // s at i in [0, B-1], j in [-1, B]
  __shared__ NsPlan sp;
  const int nact = pv.cnt->n_act;
  if ((int)blockIdx.x >= nact) return;  // no block for this CTA
  auto I = [&](int i, int j) { return (j + G) * T + (i + G); };
  sp.put(pv, 0, NsPlan::fetch(pv, blockIdx.x, nact));
  __syncthreads();
  int buf = 0;
  for (int p = blockIdx.x; p < nact; p += gridDim.x, buf ^= 1) {
    const int32_t pre = NsPlan::fetch(pv, p + gridDim.x, nact);
    const int32_t* pl = sp.pl[buf];
    const BlockInfo b = plan_block<2>(pl);
    const TreeDev& td = pv.trees[b.tree];
    const int64_t base = (int64_t)b.slot * 4 * pv.vs;
    if (!(td.rth > 0.0)) {  // no filter on this tree
      sp.put(pv, buf ^ 1, pre);
      __syncthreads();
      continue;
    }
    if ((pl[1] >> 30) & 1) {
      gather4<B, kFilterThreads, TC, TC>(pv, sp.nbo[buf], ys, (TC*)ys, tile, false);
    } else {
      load_regions<2, CtaGroup>(pv, p, R);
      __syncthreads();
      fill_tile<2, B, TC, TC, kG, CtaGroup, 4>(pv, b, ys, (TC*)ys, tile, false, R, th, uv, true);
    }
    __syncthreads();
    TC gm1, gam, rth, h2, dx2;
    if constexpr (sizeof(TC) == 4) {
      gm1 = td.nsf[0]; gam = td.nsf[3]; rth = td.rthf; h2 = td.fh2[b.lvl]; dx2 = td.fdx2[b.lvl];
    } else {
      const double dxl = td.dx[b.lvl];
      gm1 = td.nsd[0]; gam = td.nsd[3]; rth = td.rth; h2 = 0.5 / dxl; dx2 = dxl * dxl;
    }
    for (int idx = threadIdx.x; idx < SM::TILE; idx += blockDim.x) {
      const Vec4<TC> q = ld4(tile + 4 * idx);
      const TC u = q.b / q.a, v = q.c / q.a;
      TC rho, pp;
      if constexpr (KIND == MR_RHS_NS) {
        rho = q.a;
        pp = gm1 * (q.d - TC(0.5) * (q.b * u + q.c * v));
      } else {
        rho = q.a * q.a;
        pp = q.d;
      }
      st2(uv + 2 * idx, u, v);
      pc[idx] = gam * pp / rho;
    }
    __syncthreads();
    // dilatation on [-3, B+2]^2 (only the cross of the interior is read)
    constexpr int W3 = B + 6;
    for (int idx = threadIdx.x; idx < W3 * W3; idx += blockDim.x) {
      const int o = I(idx % W3 - 3, idx / W3 - 3);
      const TC* w = uv + 2 * o;
      th[o] = (w[2] - w[-2]) * h2 + (w[2 * T + 1] - w[-2 * T + 1]) * h2;
    }
    __syncthreads();
    // strengths: x-arm then y-arm, (B+2) B nodes each
    for (int idx = threadIdx.x; idx < 2 * (B + 2) * B; idx += blockDim.x) {
      const int axis = idx < (B + 2) * B ? 0 : 1;
      const int e = idx - axis * (B + 2) * B;
      const int i = axis == 0 ? e % (B + 2) - 1 : e % B;
      const int j = axis == 0 ? e / (B + 2) : e / B - 1;
      const int o = I(i, j), d = axis == 0 ? 1 : T;
      const TC t0 = th[o - 2 * d], t1 = th[o - d], t2 = th[o], t3 = th[o + d], t4 = th[o + 2 * d];
      const TC d0 = (-t3 + TC(2) * t2 - t1) / TC(4), dp = (-t4 + TC(2) * t3 - t2) / TC(4),
               dm = (-t2 + TC(2) * t1 - t0) / TC(4);
      const TC M = TC(0.5) * ((d0 - dp) * (d0 - dp) + (d0 - dm) * (d0 - dm));
      const TC r = M / (pc[o] / dx2) + TC(1e-16);
      const TC z = TC(1) - rth / r;
      (axis == 0 ? sgx : sgy)[e] = TC(0.5) * (z + (z < TC(0) ? -z : z));
    }
    __syncthreads();
    for (int q = threadIdx.x; q < NI; q += blockDim.x) {
      const int i = q % B, j = q / B;
      const TC* sx = sgx + j * (B + 2) + (i + 1);
      const TC* sy = sgy + (j + 1) * B + i;
      const TC sxp = TC(0.5) * (sx[0] + sx[1]), sxm = TC(0.5) * (sx[-1] + sx[0]);
      const TC syp = TC(0.5) * (sy[0] + sy[B]), sym = TC(0.5) * (sy[-B] + sy[0]);
      const TC* t0 = tile + 4 * I(i, j);
      const Vec4<TC> c = ld4(t0), xp = ld4(t0 + 4), xm = ld4(t0 - 4), yp = ld4(t0 + 4 * T), ym = ld4(t0 - 4 * T);
      auto increment = [&](TC q0, TC qxp, TC qxm, TC qyp, TC qym) -> TC {
        const TC fxp = TC(-0.25) * (qxp - q0), fxm = TC(-0.25) * (q0 - qxm);
        const TC fyp = TC(-0.25) * (qyp - q0), fym = TC(-0.25) * (q0 - qym);
        const TC ddx = sxp * fxp - sxm * fxm;
        const TC ddy = syp * fyp - sym * fym;
        return ddx + ddy;
      };
      const TC d[4] = {increment(c.a, xp.a, xm.a, yp.a, ym.a), increment(c.b, xp.b, xm.b, yp.b, ym.b),
                       increment(c.c, xp.c, xm.c, yp.c, ym.c), increment(c.d, xp.d, xm.d, yp.d, ym.d)};
      TS* at = y + base + q;
      if constexpr (MIX) {
        // most nodes of a flow are left alone: no FP64 work for them
        if (d[0] != TC(0) || d[1] != TC(0) || d[2] != TC(0) || d[3] != TC(0)) {
#pragma unroll 1
          for (int v = 0; v < 4; ++v) {
            const TC dv = v == 0 ? d[0] : v == 1 ? d[1] : v == 2 ? d[2] : d[3];
            if (dv != TC(0)) at[v * pv.vs] = at[v * pv.vs] - (TS)dv;
          }
        }
      } else {
        at[0] = c.a - d[0];
        at[pv.vs] = c.b - d[1];
        at[2 * pv.vs] = c.c - d[2];
        at[3 * pv.vs] = c.d - d[3];
      }
    }
    sp.put(pv, buf ^ 1, pre);
    __syncthreads();
  }
}

// Copies the interiors (nvar x vs values) of every active block from the state
// y to `to` in the stage type (the filter's source when it runs outside a step).
template <typename TS, typename TC>
__global__ void k_state_copy(PoolView pv, const TS* __restrict__ y, TC* __restrict__ to) {
  pdl_enter();
  const int nact = pv.cnt->n_act;
  const int64_t per = (int64_t)pv.nvar * pv.vs;
  const int64_t n = (int64_t)nact * per;
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x) {
    const int p = (int)(k / per);
    const int64_t at = (int64_t)pv.act[p] * per + (k - (int64_t)p * per);
    to[at] = (TC)y[at];
  }
}

}  // namespace mr
