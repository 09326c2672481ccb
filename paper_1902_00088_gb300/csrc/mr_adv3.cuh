// 3D advection kernels on 17^3 blocks: the RK stage and the wavelet details.
// One CTA per block, one thread per z-column (x, y) of the block: a thread keeps
// its column in registers, so z-neighbours never touch shared memory, and
// everything that depends on z alone folds into constants of the unrolled loop.
#pragma once
#include "mr_kernels.cuh"


namespace mr {

// Column geometry: 289 columns on 10 warps.
struct Col3 {
  static constexpr int B = 17, NQ = B * B, NT = 320;
  static constexpr int NREG = RingD<3>::NREG;
};

// Owner of the nodes of column (i, j) in one class box: node k is at
// at(k) in the field when node(k), else it lies between the owner's nodes.
struct ColOwn {
  int64_t base;
  int slot, m, sh, ow, frac;
  __device__ __forceinline__ ColOwn(const int4 e, int l1, int i, int j, int64_t vs) {
    slot = e.x;
    m = e.y;
    sh = l1 - m;
    const int ox = 2 * i - (int)(int16_t)(e.z & 0xffff), oy = 2 * j - (e.z >> 16);
    ow = e.w;
    frac = (ox | oy) & ((1 << sh) - 1);
    base = (int64_t)slot * vs + (ox >> sh) + Col3::B * (oy >> sh);
  }
  __device__ __forceinline__ int64_t at(int k) const { return base + Col3::NQ * ((2 * k - ow) >> sh); }
  __device__ __forceinline__ bool node(int k) const { return ((frac | (2 * k - ow)) & ((1 << sh) - 1)) == 0; }
};

// ------------------------------------------------------------------ stage ----
// RK4 stage of the 3D advection equation (k_stage2's formulas and order of
// operations).  The stencil is a cross, so only the six face layers of width 2
// are gathered: 3468 ghost nodes per block instead of the 4348 with edges and
// corners, and of a coarser neighbour only the layers of its face are
// predicted (at most one face per axis: the other side of a block is its
// mother's).  The z-columns are taken in halves (nodes 0..8 and 8..16) whose
// z-neighbours stay in registers, which leaves the x and y differences to shared
// memory: 8 shared loads per node instead of 13.  The state and accumulator rows of the
// update are brought to shared memory by the bulk-copy engine meanwhile (FP32
// state), so the registers allow two CTAs of 20 warps per SM.
//
// Shared memory: 17 planes of the tile; the staged rows, which share their
// memory with the owner table and the prediction scratch of a block whose
// neighbourhood is not uniform.  A plane holds the rows y = -2 .. 18 of 17 nodes
// one after the other, so the lanes of a warp (consecutive columns) read
// consecutive words at every y neighbour, and the four x ghosts of each row
// apart, each in the bank that the missing neighbour in the row would have had:
// no load of the differences has a bank conflict.
template <typename TC, typename TS>
struct Stage3Smem {
  // threads of a half; halves per thread: both at once on 20 warps (FP32), one
  // after the other on 10 (FP64 state: the registers of two CTAs per SM)
  static constexpr int HT = 320, HPT = sizeof(TS) == 4 ? 1 : 2, NT = HT * 2 / HPT;
  static constexpr int R0 = 2 * Col3::B;               // node (0, 0) of a plane
  static constexpr int XG = R0 + 352, P = XG + 4 * 32;  // x ghosts, plane pitch
  static_assert(352 % 32 == 0 && 352 >= 19 * Col3::B, "banks of the x ghosts; rows up to y = 18");
  // node (x, y) of a plane, -2 <= x, y <= 18 (x or y inside the block)
  __device__ static __forceinline__ int at(int x, int y) {
    const int n = Col3::B * y + x;
    return x < 0 ? XG + 32 * (x + 2) + (n & 31) : x >= Col3::B ? XG + 32 * (x - 15) + (n & 31) : R0 + n;
  }
  static constexpr int TILE = (Col3::B * P + 3) / 4 * 4;
  // face prediction, the three faces side by side: coarse patches 4 x 11 x 11
  // (then the y pass), and the x pass
  static constexpr int CN = 11;                        // coarse nodes -1 .. 9 along a face
  static constexpr int PATCH = 4 * CN * CN;
  static constexpr int X0 = 0, X1 = X0 + 2 * CN * CN, X2 = X1 + Col3::B * 4 * CN, XE = X2 + Col3::B * CN * 4;
  static constexpr int Y0 = 0, Y1 = Y0 + 2 * Col3::B * CN, Y2 = Y1 + Col3::B * 2 * CN, YE = Y2 + Col3::NQ * 4;
  static constexpr int SA = ((3 * PATCH > YE ? 3 * PATCH : YE) + 3) / 4 * 4, SB = (XE + 3) / 4 * 4;
  static constexpr size_t TAB = sizeof(int4) * (Col3::NREG + 1);
  static constexpr size_t RING = TAB + sizeof(TC) * (SA + SB);
  static constexpr int VS = (Col3::B * Col3::NQ + 3) / 4 * 4;  // padded block, the pool's stride
  static constexpr size_t ROWS = sizeof(TS) == 4 ? 2 * sizeof(TS) * VS : 0;
  static constexpr size_t UNION = ((RING > ROWS ? RING : ROWS) + 15) / 16 * 16;
  static constexpr size_t BYTES = UNION + sizeof(TC) * TILE;
};

// Faces (bit a = axis a) of a block whose ghost layer holds a class box owned by
// a coarser leaf.  Only the outer side of the block's position in its mother
// can: lower for even coordinates, upper for odd ones.
__device__ __forceinline__ int coarse_face(const int4* reg, int lvl, const int64_t c[3], int t) {
  // t in [0, 75): face axis t / 25, one class box of the face's layer each
  const int a = t / 25, r = t % 25;
  const int n = ((a == 0 ? c[0] : a == 1 ? c[1] : c[2]) & 1) ? 6 : 0;
  const int u = r % 5 + 1, v = r / 5 + 1;
  const int cx = a == 0 ? n : u, cy = a == 1 ? n : (a == 0 ? u : v), cz = a == 2 ? n : v;
  return reg[cx + 7 * cy + 49 * cz].y < lvl ? 1 << a : 0;
}

template <typename TS, typename TY, typename TSRC, int ST>
__global__ void __launch_bounds__(Stage3Smem<TY, TS>::NT, 2) k_stage3(PoolView pv, const TSRC* __restrict__ src,
                                                                      TS* __restrict__ y, TS* __restrict__ acc,
                                                                      TY* __restrict__ ynext, StageArgs sa) {
  pdl_enter();
  using TC = TY;
  using SM = Stage3Smem<TC, TS>;
  constexpr int B = Col3::B, NQ = Col3::NQ, NT = SM::NT, P = SM::P, CN = SM::CN;
  constexpr int NZ = 9;  // nodes of a half column: z = z0 .. z0 + 8
  constexpr int HPT = SM::HPT;
  using PL = Plan<3>;
  constexpr bool ROWS = sizeof(TS) == 4 && ST >= 1;  // rows staged (y: stages 1 and 2; acc: 1 to 3)
  constexpr bool NEEDY = ST == 1 || ST == 2;
  // the committed state of stage 0 from memory: where neither the thread's
  // registers nor the tile hold it in the state's type
  constexpr bool Y0MEM = ST == 0 && HPT == 2 && sizeof(TS) != sizeof(TC);
  int4* reg = smem_as<int4>(0);
  TC* sca = smem_as<TC>(SM::TAB);
  TC* scb = sca + SM::SA;
  TS* yrow = smem_as<TS>(0);
  TS* arow = yrow + SM::VS;
  TC* tile = smem_as<TC>(SM::UNION);
  __shared__ __align__(8) uint64_t bar;
  __shared__ int32_t splan[2][PL::INTS];
  __shared__ int64_t snb[2][PL::NB];
  __shared__ int sface;
  __shared__ TC zl[B + 4];  // nodes -2 .. 18 of the last column
  const int nact = pv.cnt->n_act;
  if (blockIdx.x == 0 && threadIdx.x == 0) atomicAdd(&pv.cnt->stage_blocks, (unsigned long long)nact);
  if (ROWS && threadIdx.x == 0) mbar_init(&bar, 1);
  if (blockIdx.x < nact && threadIdx.x < PL::INTS) {
    const int32_t v = pv.plan[(int64_t)blockIdx.x * PL::INTS + threadIdx.x];
    splan[0][threadIdx.x] = v;
    if (threadIdx.x >= PL::NBO && threadIdx.x < PL::NBO + PL::NB) snb[0][threadIdx.x - PL::NBO] = (int64_t)v * pv.vs;
  }
  __syncthreads();
  const int half0 = HPT == 1 && threadIdx.x >= SM::HT ? 1 : 0;  // (first) half of the thread's warp: 0 lower, 1 upper
  const int t = threadIdx.x - half0 * SM::HT;
  const bool col = t < NQ;  // this thread has a column of the block
  const int x = t % B, yy = (t / B) % B;
  // ghost column of the threads from 184 on: 2 layers on each side of x, then
  // of y, at 17 positions along the side
  const int gt = t - (SM::HT - 8 * B);
  int gx = 0, gy = 0;
  if (gt >= 0) {
    const int l = gt < 4 * B ? gt % 4 : (gt - 4 * B) / B, w = gt < 4 * B ? gt / 4 : (gt - 4 * B) % B;
    const int d = l < 2 ? l - 2 : B - 2 + l;  // -2, -1, 17, 18
    gx = gt < 4 * B ? d : w;
    gy = gt < 4 * B ? w : d;
  }
  TC* const gdc = tile + SM::at(gx, gy);
  TC* const tc = tile + SM::at(x, yy);
  unsigned phase = 0;
  int buf = 0;
  for (int p = blockIdx.x; p < nact; p += gridDim.x, buf ^= 1) {
    const int pn = p + gridDim.x;
    int32_t pre = 0;
    if (pn < nact && threadIdx.x < PL::INTS) pre = pv.plan[(int64_t)pn * PL::INTS + threadIdx.x];
    const int32_t* pl = splan[buf];
    const BlockInfo b = plan_block<3>(pl);
    const bool uni = (pl[1] >> 30) & 1;
    const int64_t own = (int64_t)b.slot * pv.vs;
    TSRC raw[NZ];          // nodes z0 .. z0 + 8 (z0 = 8 half)
    TSRC gz[HPT][2];       // ghosts -2, -1 (lower half) or 17, 18 (upper)
    unsigned gzp = 0;      // ghosts (bit 2 i + d for half half0 + i) predicted from the coarse lattice
    unsigned gpred[HPT];   // predicted nodes of the ghost column
    bool bad = false;
    auto stage_rows = [&]() {
      if (ROWS && threadIdx.x == 0) {
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        mbar_expect_tx(&bar, (NEEDY ? 2 : 1) * sizeof(TS) * SM::VS);
        if (NEEDY) bulk_g2s(yrow, y + own, sizeof(TS) * SM::VS, &bar);
        bulk_g2s(arow, acc + own, sizeof(TS) * SM::VS, &bar);
      }
    };
    // block-edge nodes held by another block: its copy is the value (stage 0
    // stores it, Sec. 2.5); after stage 0 all equal-level copies are identical.
    // Node 8 belongs to the lower half.
    auto commit = [&](int half, int j) {
      const int64_t at = own + t + NQ * (8 * half + j);
      if (ST == 0 && !(half && j == 0) && differs(src[at], raw[j])) const_cast<TSRC*>(src)[at] = raw[j];
    };
    auto put = [&](int half) {  // the half column to the tile
#pragma unroll
      for (int j = 0; j < NZ; ++j) tc[(8 * half + j) * P] = (TC)raw[j];
    };
    if (uni) {
      // the rows' memory is free: they travel with the gather
      stage_rows();
      const int64_t* nb = snb[buf];
#pragma unroll
      for (int i = 0; i < HPT; ++i) {
        const int half = half0 + i, z0 = 8 * half;
        if (col) {
          const int sx = ST == 0 && x == B - 1 ? 2 : 1, sy = ST == 0 && yy == B - 1 ? 2 : 1;
          const int lxy = (x - (sx - 1) * (B - 1)) + B * (yy - (sy - 1) * (B - 1));
          const int r = sx + 3 * sy;
          const TSRC* mid = src + nb[r + 9] + lxy + NQ * z0;
          // beyond the half: nodes 14, 15 of the lower or 0, 1, 2 of the upper neighbour
          const TSRC* out = src + nb[r + 18 * half] + lxy + (half ? 0 : NQ * (B - 3));
#pragma unroll
          for (int j = 0; j < NZ - 1; ++j) raw[j] = mid[NQ * j];
          raw[NZ - 1] = ST == 0 && half ? out[0] : mid[NQ * (NZ - 1)];
          gz[i][0] = out[half ? NQ : 0];
          gz[i][1] = out[half ? 2 * NQ : NQ];
        }
        if (gt >= 0) {
          const int sx = gx < 0 ? 0 : (gx >= B ? 2 : (ST == 0 && gx == B - 1 ? 2 : 1));
          const int sy = gy < 0 ? 0 : (gy >= B ? 2 : (ST == 0 && gy == B - 1 ? 2 : 1));
          const int r = sx + 3 * sy;
          const int lxy = (gx - (sx - 1) * (B - 1)) + B * (gy - (sy - 1) * (B - 1));
          const TSRC* mid = src + nb[r + 9] + lxy + NQ * z0;
          const TSRC* last = ST == 0 && half ? src + nb[r + 18] + lxy : mid + NQ * (NZ - 1);
          TC* gd = gdc + z0 * P;
#pragma unroll
          for (int j = 0; j < NZ; ++j) {
            const TSRC* a = j < NZ - 1 ? mid + NQ * j : last;
            if constexpr (std::is_same<TSRC, TC>::value) cp_async(gd + j * P, a);
            else gd[j * P] = (TC)*a;
          }
        }
        if (col) {
          if (ST == 0) {
#pragma unroll
            for (int j = 0; j < NZ; ++j)
              if (x == B - 1 || yy == B - 1 || (half && j == NZ - 1)) commit(half, j);
          }
          put(half);
        }
      }
    } else {
      const int4* rsrc = plan_regions<3>(pv, p);
      for (int r = threadIdx.x; r < Col3::NREG; r += NT) reg[r] = rsrc[r];
      if (threadIdx.x == 0) sface = 0;
      __syncthreads();
      const int l1 = b.lvl + 1;
      if (threadIdx.x < 75) {
        const int f = coarse_face(reg, b.lvl, b.c, threadIdx.x);
        if (f) atomicOr(&sface, f);
      }
#pragma unroll
      for (int i = 0; i < HPT; ++i) {
        const int half = half0 + i, z0 = 8 * half;
        // class boxes along z of the half: node z0, nodes z0 + 1 .. z0 + 7, node
        // z0 + 8, ghosts
        const int c0 = half ? 3 : 1;
        if (col) {
          const int rb = reg_class<B>(x) + 7 * reg_class<B>(yy);
          const bool core = x >= 1 && x <= B - 2 && yy >= 1 && yy <= B - 2;
          const TSRC* mine = src + own + t + NQ * z0;
          unsigned other = 0;  // nodes held by another block
          static_for<0, 3>([&](auto cc) {
            constexpr int C = decltype(cc)::value;
            constexpr int J0 = C == 0 ? 0 : C == 1 ? 1 : 8, J1 = C == 0 ? 0 : C == 1 ? 7 : 8;
            const int4 e = reg[rb + 49 * (c0 + C)];
            if ((C == 1 && core) || e.x == b.slot) {
#pragma unroll
              for (int j = J0; j <= J1; ++j) raw[j] = mine[NQ * j];
              return;
            }
            if (e.x < 0) {  // no owner: zero in the tile, the pool stays as it is
              bad = true;
#pragma unroll
              for (int j = J0; j <= J1; ++j) raw[j] = TSRC(0);
              return;
            }
            other |= C == 0 ? 1u : C == 1 ? 0xfeu : 0x100u;
            const ColOwn o(e, l1, x, yy, pv.vs);
#pragma unroll
            for (int j = J0; j <= J1; ++j) raw[j] = src[o.at(z0 + j)];
          });
          const int4 e = reg[rb + 49 * (half ? 6 : 0)];
          gz[i][0] = gz[i][1] = TSRC(0);
          if (e.x < 0) {
            bad = true;
          } else {
            const ColOwn o(e, l1, x, yy, pv.vs);
            const int k0 = half ? B : -2;
#pragma unroll
            for (int d = 0; d < 2; ++d) {
              if (o.m >= b.lvl || o.node(k0 + d)) {
                gz[i][d] = src[o.at(k0 + d)];
              } else {
                bad |= o.m != b.lvl - 1;
                gzp |= 1u << (2 * i + d);
              }
            }
          }
          if (ST == 0) {
#pragma unroll
            for (int j = 0; j < NZ; ++j)
              if ((other >> j) & 1) commit(half, j);
          }
          put(half);
        }
        gpred[i] = 0;
        if (gt >= 0) {
          TC* gd = gdc + z0 * P;
          const int rb = reg_class<B>(gx) + 7 * reg_class<B>(gy);
          static_for<0, 3>([&](auto cc) {
            constexpr int C = decltype(cc)::value;
            constexpr int J0 = C == 0 ? 0 : C == 1 ? 1 : 8, J1 = C == 0 ? 0 : C == 1 ? 7 : 8;
            const int4 e = reg[rb + 49 * (c0 + C)];
            if (e.x < 0) {
              bad = true;
#pragma unroll
              for (int j = J0; j <= J1; ++j) gd[j * P] = TC(0);
              return;
            }
            const ColOwn o(e, l1, gx, gy, pv.vs);
#pragma unroll
            for (int j = J0; j <= J1; ++j) {
              if (o.m >= b.lvl || o.node(z0 + j)) {
                if constexpr (std::is_same<TSRC, TC>::value) cp_async(gd + j * P, src + o.at(z0 + j));
                else gd[j * P] = (TC)src[o.at(z0 + j)];
              } else {
                bad |= o.m != b.lvl - 1;
                gpred[i] |= 1u << j;
              }
            }
          });
        }
      }
      __syncthreads();
      const int fm = sface;
      if (fm) {
        // Prediction of the face layers: x first, then y, then z (the order of
        // predict_box), each face from a patch of 4 coarse nodes across it
        // and 11 x 11 along it.  n0: first coarse node across the face.  The
        // passes take the odd nodes (4 products and sums) before the even ones
        // (copies), so that their warps hold one kind.
        const int n0[3] = {(b.c[0] & 1) ? 7 : -2, (b.c[1] & 1) ? 7 : -2, (b.c[2] & 1) ? 7 : -2};
        for (int q = threadIdx.x; q < 3 * SM::PATCH; q += NT) {
          const int a = q / SM::PATCH, r = q % SM::PATCH;
          if (!((fm >> a) & 1)) continue;
          // patch layout: x fastest, then y, then z, with 4 nodes along the face's axis
          const int wx = a == 0 ? 4 : CN, wy = a == 1 ? 4 : CN;
          const int ix = r % wx, iy = (r / wx) % wy, iz = r / (wx * wy);
          const int nx = ix + (a == 0 ? n0[0] : -1), ny = iy + (a == 1 ? n0[1] : -1), nz = iz + (a == 2 ? n0[2] : -1);
          const int4 e = reg[reg_class<B>(2 * nx) + 7 * reg_class<B>(2 * ny) + 49 * reg_class<B>(2 * nz)];
          TC v = TC(0);
          if (e.x < 0 || e.y < b.lvl - 1) {
            bad = true;
          } else {
            const ColOwn o(e, l1, 2 * nx, 2 * ny, pv.vs);
            v = (TC)src[o.at(2 * nz)];
          }
          sca[q] = v;
        }
        __syncthreads();
        // layer d = 0, 1 of a face: tile index -2, -1 (lower) or 17, 18 (upper);
        // the odd layer is d = 1 (lower) or 0 (upper), the other a coarse node.
        // x pass: 121 rows of 2 layers, then 44 rows of 17 nodes of each other face
        constexpr int XO = CN * CN, XR = 4 * CN;
        for (int q = threadIdx.x; q < 2 * XO + 2 * XR * B; q += NT) {
          // odd: [0, XO + 16 XR), even: the rest
          const bool odd = q < XO + 16 * XR;
          const int u = odd ? q : q - (XO + 16 * XR);
          if (u < XO) {  // face across x
            if (!(fm & 1)) continue;
            const TC* c4 = sca + 4 * u;
            const bool low = n0[0] < 0;
            scb[SM::X0 + 2 * u + (odd == low ? 1 : 0)] = odd ? dd4(c4[0], c4[1], c4[2], c4[3]) : c4[low ? 1 : 2];
          } else {
            const int per = odd ? 8 : 9;
            const int v = u - XO, row2 = v / per, m = v % per;
            const int a = row2 < XR ? 1 : 2, row = row2 - (a - 1) * XR;
            if (!((fm >> a) & 1)) continue;
            const TC* c = sca + a * SM::PATCH + CN * row + m;  // patch rows: 11 coarse x nodes, from -1
            scb[(a == 1 ? SM::X1 : SM::X2) + B * row + 2 * m + (odd ? 1 : 0)] = odd ? dd4(c[0], c[1], c[2], c[3]) : c[1];
          }
        }
        __syncthreads();
        // y pass (over the patches, no longer needed): the face across x [nz][y][2],
        // across y [nz][d][x], across z [nz][y][x]
        constexpr int YA = 2 * CN, YB = CN * B, YC = 4 * B;  // values per node along y (a 0 and 2); per layer (a 1)
        constexpr int YODD = 8 * (YA + YC) + YB, YALL = 17 * (YA + YC) + 2 * YB;
        for (int q = threadIdx.x; q < YALL; q += NT) {
          const bool odd = q < YODD;
          int u = odd ? q : q - YODD;
          if (u < YB) {  // face across y: one layer
            if (!(fm & 2)) continue;
            const int xx = u % B, iz = u / B;
            const bool low = n0[1] < 0;
            const TC* c = scb + SM::X1 + 4 * iz * B + xx;
            sca[SM::Y1 + (2 * iz + (odd == low ? 1 : 0)) * B + xx] =
                odd ? dd4(c[0], c[B], c[2 * B], c[3 * B]) : c[(low ? 1 : 2) * B];
            continue;
          }
          u -= YB;
          const int per = odd ? 8 : 9;
          const int a = u < per * YA ? 0 : 2;
          if (!((fm >> a) & 1)) continue;
          if (a == 2) u -= per * YA;
          const int w = a == 0 ? 2 : B;
          const int xx = u % w, m = (u / w) % per, iz = u / (w * per);
          const TC* c = scb + (a == 0 ? SM::X0 : SM::X2) + (iz * CN + m) * w + xx;
          sca[(a == 0 ? SM::Y0 : SM::Y2) + (iz * B + 2 * m + (odd ? 1 : 0)) * w + xx] =
              odd ? dd4(c[0], c[w], c[2 * w], c[3 * w]) : c[w];
        }
        __syncthreads();
        // z pass, at the predicted nodes
#pragma unroll
        for (int i = 0; i < HPT; ++i) {
          const int half = half0 + i;
          if (gpred[i]) {
            const bool fx = gx < 0 || gx >= B;  // layer across x, else across y
            const int d = fx ? (gx < 0 ? gx + 2 : gx - B) : (gy < 0 ? gy + 2 : gy - B);
            constexpr int st = 2 * B;  // both layouts hold 34 values per coarse z
            const TC* c = (fx ? sca + SM::Y0 + 2 * gy + d : sca + SM::Y1 + d * B + gx) + 4 * half * st;
            TC* gd = gdc + 8 * half * P;
#pragma unroll
            for (int j = 0; j < NZ; ++j) {
              if (!((gpred[i] >> j) & 1)) continue;
              const TC* ck = c + (j >> 1) * st;
              gd[j * P] = (j & 1) ? dd4(ck[0], ck[st], ck[2 * st], ck[3 * st]) : ck[st];
            }
          }
          if ((gzp >> (2 * i)) & 3) {
            // lower: the layers -2 (a coarse node) and -1; upper: 17 and 18 (a coarse node)
            const TC* c = sca + SM::Y2 + yy * B + x;
            const TC mid4 = dd4(c[0], c[NQ], c[2 * NQ], c[3 * NQ]), node = half ? c[2 * NQ] : c[NQ];
            if ((gzp >> (2 * i)) & 1) gz[i][0] = (TSRC)(half ? mid4 : node);
            if ((gzp >> (2 * i)) & 2) gz[i][1] = (TSRC)(half ? node : mid4);
          }
        }
      }
      if (bad) set_err(pv, kErrGraded);
    }
    if (t == NQ - 1) {  // the last column, for the lanes that compute it
#pragma unroll
      for (int i = 0; i < HPT; ++i) {
        const int half = half0 + i;
#pragma unroll
        for (int d = 0; d < 2; ++d) zl[half ? B + 2 + d : d] = (TC)gz[i][d];
#pragma unroll
        for (int j = 0; j < NZ; ++j) zl[8 * half + j + 2] = tc[(8 * half + j) * P];
      }
    }
    if constexpr (std::is_same<TSRC, TC>::value) cp_async_wait_all();
    __syncthreads();
    if (!uni) stage_rows();
    if (ROWS) {
      if (!bulk_landed(pv, &bar, phase)) return;
      phase ^= 1;
    }
    const TreeDev& td = pv.trees[b.tree];
    const TC cd = tree_cD<TC>(td, b.lvl);
    const StageCoef<TS> cs(pv, sa, b.tree, ST);
    const TS cas = cs.ca, cys = cs.cy;
    const TC u0 = tree_rhs<TC>(td, 0), u1 = tree_rhs<TC>(td, 1), u2 = tree_rhs<TC>(td, 2);
    // node q = column + 289 z: tk its place in the tile, xo the x neighbours'
    // places, z2 .. the column's values around it, yk / ak state and accumulator
    auto node = [&](int64_t at, const TC* tk, const TC* xa, const TC* xb, const TC* xc, const TC* xd, TC zm2, TC zm1,
                    TC zp1, TC zp2, TS yk, TS ak) {
      const TC dxv = d1_sum(*xa, *xb, *xc, *xd) * cd;
      const TC dyv = d1_sum(tk[-2 * B], tk[-B], tk[B], tk[2 * B]) * cd;
      const TC dzv = d1_sum(zm2, zm1, zp1, zp2) * cd;
      TC s = u0 * dxv + u1 * dyv;
      s = s + u2 * dzv;
      const TS kk = to_state<TS>(-s);
      if (ST == 0) {
        acc[at] = yk + cas * kk;
        ynext[at] = to_tile<TY>(yk + cys * kk);
      } else if (ST == 1 || ST == 2) {
        acc[at] = ak + cas * kk;
        ynext[at] = to_tile<TY>(yk + cys * kk);
      } else {
        y[at] = ak + cas * kk;
      }
    };
    if (t < NQ - 1) {
      const TC *xa = tile + SM::at(x - 2, yy), *xb = tile + SM::at(x - 1, yy), *xc = tile + SM::at(x + 1, yy),
               *xd = tile + SM::at(x + 2, yy);
#pragma unroll
      for (int i = 0; i < HPT; ++i) {
        const int half = half0 + i, z0 = 8 * half;
        const int64_t me = own + t + NQ * z0;
        // FP64 state: the half's values of the update, loaded together
        constexpr bool PRE = !ROWS && (ST >= 1 || Y0MEM);
        TS yv[PRE ? NZ : 1], av[PRE ? NZ : 1];
        if constexpr (PRE) {
#pragma unroll
          for (int j = 0; j < NZ; ++j) {
            if constexpr (NEEDY || Y0MEM) yv[j] = (Y0MEM ? committed(y, src) : y)[me + NQ * j];
            if constexpr (ST >= 1) av[j] = acc[me + NQ * j];
          }
        }
        // the column from two nodes below to two above: the other half's nodes from the tile
        TC c[NZ + 4];
#pragma unroll
        for (int j = 0; j < NZ; ++j) c[j + 2] = HPT == 1 ? (TC)raw[j] : tc[(z0 + j) * P];
        {
          const TC* in = tc + (half ? 6 * P : NZ * P);
          const TC l0 = in[0], l1v = in[P];
          c[0] = half ? l0 : (TC)gz[i][0];
          c[1] = half ? l1v : (TC)gz[i][1];
          c[NZ + 2] = half ? (TC)gz[i][0] : l0;
          c[NZ + 3] = half ? (TC)gz[i][1] : l1v;
        }
#pragma unroll
        for (int j = 0; j < NZ; ++j) {
          if (j == 0 && half) continue;  // node 8: the lower half's
          const int k = (z0 + j) * P;
          TS yk = TS(0), ak = TS(0);
          if constexpr (ROWS) {
            if (NEEDY) yk = yrow[t + NQ * (z0 + j)];
            ak = arow[t + NQ * (z0 + j)];
          } else if constexpr (PRE) {
            if constexpr (NEEDY || Y0MEM) yk = yv[j];
            if constexpr (ST >= 1) ak = av[j];
          }
          // stage 0: the committed (synchronised) state is the column itself
          if (ST == 0 && !Y0MEM) yk = HPT == 1 ? (TS)raw[j] : (TS)c[j + 2];
          node(me + NQ * j, tc + k, xa + k, xb + k, xc + k, xd + k, c[j], c[j + 1], c[j + 3], c[j + 4], yk, ak);
        }
      }
    } else if (half0 == 0 && t < NQ - 1 + B) {
      // the last column: one node per lane instead of 17 on one lane of a warp
      const int z = t - (NQ - 1), k = z * P, q = NQ - 1 + NQ * z;
      TS yk = TS(0), ak = TS(0);
      if (NEEDY) yk = ROWS ? yrow[q] : y[own + q];
      if (ST >= 1) ak = ROWS ? arow[q] : acc[own + q];
      if (ST == 0) yk = sizeof(TS) == sizeof(TC) ? (TS)zl[z + 2] : committed(y, src)[own + q];
      node(own + q, tile + SM::at(B - 1, B - 1) + k, tile + SM::at(B - 3, B - 1) + k, tile + SM::at(B - 2, B - 1) + k,
           tile + SM::at(B, B - 1) + k, tile + SM::at(B + 1, B - 1) + k, zl[z], zl[z + 1], zl[z + 3], zl[z + 4], yk, ak);
    }
    if (pn < nact && threadIdx.x < PL::INTS) {
      splan[buf ^ 1][threadIdx.x] = pre;
      if (threadIdx.x >= PL::NBO && threadIdx.x < PL::NBO + PL::NB)
        snb[buf ^ 1][threadIdx.x - PL::NBO] = (int64_t)pre * pv.vs;
    }
    __syncthreads();
  }
}

// ---------------------------------------------------------------- details ----
// Details of 17^3 blocks (Sec. 2.3: D = B - P(R(B)), x then y then z).  P(R(B)) reads the coarse
// lattice of the tile only, and every coarse-lattice node of the ghost layer is
// a node of its owner whatever the owner's level: 602 ghost nodes per block
// (11^3 coarse nodes less the block's own 9^3) are all that is gathered, and
// nothing is predicted.  The x pass goes to shared memory (11 x 11 rows), the y
// pass of a column is kept in its thread's registers and feeds the z pass, and
// the block's own values go from memory straight to registers.  Per-block latency
// bounds it (four barriers per block, 3 CTAs per SM; 4 CTAs spill: 487 us instead of
// 460, with three more barriers).  Measured, before with a gathered 21^3 tile and its
// predicted ghosts: 2078 -> 400 us on a uniform grid of 32768 blocks (FP32); the three
// rounds of an adaptive FP32 step with 1632 blocks 426 -> 120 us; of an FP64 step with
// 2584 blocks 1750 -> 470 us, where maxima, the non-finite test and the division by 16
// are kept off the FP64 pipe.
template <typename TT, typename TD>
struct Det3Smem {
  static constexpr int CN = 11;
  static constexpr int E = (CN * CN * CN + 3) / 4 * 4;        // coarse lattice, type TT
  static constexpr int X = CN * CN * Col3::B;                 // x pass, type TT or TD
  static constexpr int NG = CN * CN * CN - 9 * 9 * 9;         // ghost nodes of the lattice
  static constexpr size_t XB = (X * (sizeof(TD) > sizeof(TT) ? sizeof(TD) : sizeof(TT)) + 15) / 16 * 16;
  static constexpr size_t TAB = ((size_t)kRingBytesD<3> + 15) / 16 * 16;
  static constexpr size_t GT = (4 * NG + 15) / 16 * 16;
  static constexpr size_t BYTES = TAB + GT + XB + sizeof(TT) * E;
};

template <typename TS, typename TD, typename TT>
__global__ void __launch_bounds__(Col3::NT, sizeof(TS) == 8 ? 2 : 3) k_details3(PoolView pv, TS* __restrict__ y) {
  pdl_enter();
  using SM = Det3Smem<TT, TD>;
  constexpr int B = Col3::B, NQ = Col3::NQ, NT = Col3::NT, CN = SM::CN, CP = CN * CN;
  using PL = Plan<3>;
  RingD<3>& R = *smem_as<RingD<3>>(0);
  int32_t* gtab = smem_as<int32_t>(SM::TAB);
  TD* X64 = smem_as<TD>(SM::TAB + SM::GT);
  TT* E = smem_as<TT>(SM::TAB + SM::GT + SM::XB);
  __shared__ double red[2][32];
  __shared__ int32_t splan[2][PL::INTS];
  __shared__ int32_t snb[PL::NB];
  __shared__ int nonfinite;
  __shared__ double csv;
  __shared__ int csv_tree;
  const int t = threadIdx.x;
  const int nact = pv.cnt->n_round;
  if ((int)blockIdx.x >= nact) return;  // no block for this CTA (small grids)
  const bool all_blocks = pv.cnt->first_round != 0;
  const int prev = pv.cnt->round_id - 1;
  const bool plan_ok = pv.cnt->plan_topo == pv.cnt->topo;
  // ghost nodes of the coarse lattice: lattice index | neighbour << 11 | offset
  // in that neighbour (of a uniform neighbourhood) << 16
  for (int g = t; g < SM::NG; g += NT) {
    int n[3];  // lattice position 0 .. 10, at node 2 (n - 1)
    if (g < 2 * CP) {
      n[0] = g % CN;
      n[1] = (g / CN) % CN;
      n[2] = g < CP ? 0 : CN - 1;
    } else if (g < 2 * CP + 2 * 9 * CN) {
      const int r = g - 2 * CP;
      n[0] = r % CN;
      n[1] = (r / CN) % 2 ? CN - 1 : 0;
      n[2] = r / (2 * CN) + 1;
    } else {
      const int r = g - 2 * CP - 2 * 9 * CN;
      n[0] = r % 2 ? CN - 1 : 0;
      n[1] = (r / 2) % 9 + 1;
      n[2] = r / 18 + 1;
    }
    int nb = 0, off = 0, mul = 1, lm = 1;
    for (int a = 0; a < 3; ++a) {
      const int k = 2 * (n[a] - 1);
      const int s = k < 0 ? 0 : (k <= B - 2 ? 1 : 2);
      nb += s * mul;
      off += (k - (s - 1) * (B - 1)) * lm;
      mul *= 3;
      lm *= B;
    }
    gtab[g] = (n[2] * CP + n[1] * CN + n[0]) | (nb << 11) | (off << 16);
  }
  unsigned long long ndet = 0;
  if (t == 0) {
    csv = 0.0;
    csv_tree = -1;
    nonfinite = 0;
  }
  auto flush_csv = [&]() {
    if (csv_tree >= 0 && t == 0 && csv > 0.0) atomic_max_pos(&pv.svar[csv_tree], csv);
  };
  if (plan_ok && blockIdx.x < nact && t < PL::INTS) splan[0][t] = pv.plan[(int64_t)blockIdx.x * PL::INTS + t];
  __syncthreads();
  // column of the thread: rows with even y first, so that the warps of a y pass
  // take one branch
  const bool col = t < NQ;
  const int x = t % B, ry = (t / B) % B, yy = ry < 9 ? 2 * ry : 2 * (ry - 9) + 1;
  const int cq = yy * B + x;
  int buf = 0;
  for (int p = blockIdx.x; p < nact; p += gridDim.x, buf ^= 1) {
    const int pn = p + gridDim.x;
    int32_t pre = 0;
    if (plan_ok && pn < nact && t < PL::INTS) pre = pv.plan[(int64_t)pn * PL::INTS + t];
    BlockInfo b;
    int q = 0;
    if (plan_ok) {
      b = plan_block<3>(splan[buf]);
      q = t < PL::NB ? splan[buf][PL::NBO + t] : b.slot;
    } else {
      b = load_block(pv, pv.act[p]);
      q = b.slot;
      if (t < PL::NB && t != 13) {
        const int64_t cn[3] = {b.c[0] + t % 3 - 1, b.c[1] + (t / 3) % 3 - 1, b.c[2] + t / 9 - 1};
        q = tab_get<3>(pv, pv.trees[b.tree], b.lvl, cn);
      }
    }
    const TreeDev& td = pv.trees[b.tree];
    if (pv.norm_kind == 1 && b.tree != csv_tree) {  // block of another tree: flush the scale
      flush_csv();
      __syncthreads();
      if (t == 0) {
        csv = 0.0;
        csv_tree = b.tree;
      }
    }
    // With a plan and every block due (the first round of a step) a block with a
    // uniform neighbourhood gathers without a barrier.
    bool uni;
    if (plan_ok) {
      uni = (splan[buf][1] >> 30) & 1;
    } else {
      if (t < PL::NB) snb[t] = q;
      uni = __syncthreads_and(q >= 0);
    }
    const int32_t* nbs = plan_ok ? splan[buf] + PL::NBO : snb;  // slots of the 3^3 blocks
    if (!uni) {
      if (plan_ok && all_blocks) {
        const int4* rsrc = plan_regions<3>(pv, p);
        for (int r = t; r < Col3::NREG; r += NT) R.reg[r] = rsrc[r];
      } else {
        build_ring<3, B>(pv, td, b, R);
      }
      __syncthreads();
    }
    bool dirty = all_blocks;
    if (!all_blocks)
      dirty = __syncthreads_or(uni ? t < PL::NB && pv.stamp[q] == prev
                                   : t < Geo<3, B>::NR && R.slot[t] >= 0 && pv.stamp[R.slot[t]] == prev);
    if (!dirty) {
      // no leaf of the ring changed in the previous round: the stored details
      // and norms are those of the unchanged tile
      if (pv.norm_kind == 1 && t == 0) csv = fmax(csv, pv.bmax[b.slot]);
      if (plan_ok && pn < nact && t < PL::INTS) splan[buf ^ 1][t] = pre;
      __syncthreads();
      continue;
    }
    ndet += 1;
    const int64_t own = (int64_t)b.slot * pv.vs;
    const int64_t me = own + cq;
    TT v[B];
    // block-edge nodes held by another block take (and store) its value
    if (uni) {
      if (col) {
        const int sx = x == B - 1 ? 2 : 1, sy = yy == B - 1 ? 2 : 1;
        const int lxy = (x - (sx - 1) * (B - 1)) + B * (yy - (sy - 1) * (B - 1));
        const TS* mid = y + (int64_t)nbs[sx + 3 * sy + 9] * pv.vs + lxy;
        const TS* top = y + (int64_t)nbs[sx + 3 * sy + 18] * pv.vs + lxy;
        TS raw[B];
#pragma unroll
        for (int k = 0; k < B; ++k) raw[k] = k < B - 1 ? mid[NQ * k] : *top;
#pragma unroll
        for (int k = 0; k < B; ++k) {
          if ((x == B - 1 || yy == B - 1 || k == B - 1) && differs(y[me + NQ * k], raw[k])) y[me + NQ * k] = raw[k];
          v[k] = to_tile<TT>(raw[k]);
        }
      }
      for (int g = t; g < SM::NG; g += NT) {
        const int e = gtab[g];
        E[e & 2047] = (TT)y[(int64_t)nbs[(e >> 11) & 31] * pv.vs + (e >> 16)];
      }
    } else {
      if (!(plan_ok && all_blocks)) {
        build_regions<3, B, CtaGroup>(b, R);
        __syncthreads();
      }
      const int l1 = b.lvl + 1;
      bool lost = false;
      if (col) {
        const int rb = reg_class<B>(x) + 7 * reg_class<B>(yy);
        const bool core = x >= 1 && x <= B - 2 && yy >= 1 && yy <= B - 2;
        TS raw[B];
        unsigned other = 0;  // nodes held by another block
        static_for<1, 6>([&](auto cc) {
          constexpr int C = decltype(cc)::value;
          constexpr int K0 = C == 1 ? 0 : C == 2 ? 1 : C == 3 ? 8 : C == 4 ? 9 : 16;
          constexpr int K1 = C == 1 ? 0 : C == 2 ? 7 : C == 3 ? 8 : C == 4 ? 15 : 16;
          if (C >= 2 && C <= 4 && core) {
#pragma unroll
            for (int k = K0; k <= K1; ++k) raw[k] = y[me + NQ * k];
            return;
          }
          const int4 e = R.reg[rb + 49 * C];
          if (e.x < 0) {
            lost = true;
#pragma unroll
            for (int k = K0; k <= K1; ++k) raw[k] = TS(0);
            return;
          }
          const ColOwn o(e, l1, x, yy, pv.vs);
          const bool self = o.slot == b.slot;
#pragma unroll
          for (int k = K0; k <= K1; ++k) {
            raw[k] = self ? y[me + NQ * k] : y[o.at(k)];
            if (!self) other |= 1u << k;
          }
        });
#pragma unroll
        for (int k = 0; k < B; ++k) {
          if (((other >> k) & 1) && differs(y[me + NQ * k], raw[k])) y[me + NQ * k] = raw[k];
          v[k] = to_tile<TT>(raw[k]);
        }
      }
      for (int g = t; g < SM::NG; g += NT) {
        const int at = gtab[g] & 2047;
        const int n0 = 2 * (at % CN - 1), n1 = 2 * ((at / CN) % CN - 1), n2 = 2 * (at / CP - 1);
        const int4 e = R.reg[reg_class<B>(n0) + 7 * reg_class<B>(n1) + 49 * reg_class<B>(n2)];
        TT val = TT(0);
        if (e.x < 0 || e.y < b.lvl - 1) {
          lost = true;
        } else {
          const ColOwn o(e, l1, n0, n1, pv.vs);
          val = (TT)y[o.at(n2)];
        }
        E[at] = val;
      }
      if (lost) set_err(pv, kErrGraded);
    }
    // largest |value| of the interior and the non-finite test
    AbsMax<TT> mqa;
    bool bad = false;
    if (col) {
#pragma unroll
      for (int k = 0; k < B; ++k) {
        mqa.add(v[k]);
        bad |= !finite(v[k]);
      }
      if (((x | yy) & 1) == 0) {
        TT* e0 = E + CP + (yy / 2 + 1) * CN + x / 2 + 1;
#pragma unroll
        for (int k = 0; k < B; k += 2) e0[CP * (k / 2)] = v[k];
      }
    }
    if (bad) nonfinite = 1;
    __syncthreads();
    // x pass on the coarse rows into X, y pass of the column, z pass and the
    // detail at every odd node; with EX also the coarse lattice's largest |value|
    float mt = 0.f;
    auto pass = [&](auto tag, auto exc) -> decltype(tag) {
      using A = decltype(tag);
      constexpr bool EX = decltype(exc)::value;
      A* XA = reinterpret_cast<A*>(X64);
      for (int idx = t; idx < CP * 8; idx += NT) {
        const int row = idx >> 3, m = idx & 7;
        const TT* e = E + row * CN + m;
        const TT e0 = e[0], e1 = e[1], e2 = e[2], e3 = e[3];
        if constexpr (EX)
          mt = fmaxf(fmaxf(mt, fmaxf(fabsf((float)e0), fabsf((float)e1))), fmaxf(fabsf((float)e2), fabsf((float)e3)));
        XA[row * B + 2 * m + 1] = dd4((A)e0, (A)e1, (A)e2, (A)e3);
      }
      for (int idx = t; idx < CP * 9; idx += NT) {
        const int row = idx / 9, m = idx % 9;
        XA[row * B + 2 * m] = (A)E[row * CN + m + 1];
      }
      __syncthreads();
      AbsMax<A> md;
      if (col) {
        A yv[CN];  // y pass on the coarse z planes
        const A* x0 = XA + (yy >> 1) * B + x;
        if (yy & 1) {
#pragma unroll
          for (int z = 0; z < CN; ++z) {
            const A* r = x0 + z * CN * B;
            yv[z] = dd4(r[0], r[B], r[2 * B], r[3 * B]);
          }
        } else {
#pragma unroll
          for (int z = 0; z < CN; ++z) yv[z] = x0[z * CN * B + B];
        }
        const bool odd = (x | yy) & 1;
#pragma unroll
        for (int k = 0; k < B; ++k) {
          if (k & 1) {
            const int m = k / 2;
            md.add((A)v[k] - dd4(yv[m], yv[m + 1], yv[m + 2], yv[m + 3]));
          } else if (odd) {
            md.add((A)v[k] - yv[k / 2 + 1]);
          }
        }
      }
      return md.get();
    };
    constexpr bool cert = sizeof(TT) == 4 && sizeof(TD) == 8;
    using A0 = std::conditional_t<cert, float, TD>;
    A0 m0 = pass(A0(0), std::true_type{});
    TT mq = mqa.get();
    float mtr = mt;
    block_max3<A0, TT, float>(m0, mq, mtr, reinterpret_cast<A0*>(red[0]), reinterpret_cast<TT*>(red[1]),
                              reinterpret_cast<float*>(red[1]) + 32);
    double md = 0.0;  // thread 0's value is stored
    if constexpr (cert) {
      // FP32 values, FP64 decision: the FP32 evaluation differs from the FP64 one
      // by at most ~20 u max|tile| (u = 2^-24, x/y/z passes of the 4-point rule and
      // the subtraction); where its maximum is farther than 32 u max|tile| from eps
      // the threshold decision (Sec. 2.3) is the FP64 one, otherwise the block is
      // evaluated again in FP64
      const float err = 0x1p-19f * fmaxf(mtr, (float)mq) + 1e-37f;
      if (pv.norm_kind == 0 && certain_vs_eps(m0, err, td)) {
        md = (double)m0;
      } else {
        const double m64 = pass(double(0), std::false_type{});
        md = block_max<double>(m64, red[0]);
      }
    } else {
      md = (double)m0;
    }
    if (t == 0) {
      if (nonfinite) md = __longlong_as_double(0x7ff8000000000000LL);
      nonfinite = 0;
      pv.md[b.slot] = md;
      pv.bmax[b.slot] = (double)mq;
      if (pv.norm_kind == 1) csv = fmax(csv, (double)mq);
    }
    if (plan_ok && pn < nact && t < PL::INTS) splan[buf ^ 1][t] = pre;
    __syncthreads();
  }
  __syncthreads();
  if (pv.norm_kind == 1) flush_csv();
  if (t == 0 && ndet) atomicAdd(&pv.cnt->det_blocks, ndet);
}

// ----------------------------------------------------------------- refine ----
// Refinement of 17^3 blocks (k_refine's values).  A mother is split among four
// CTAs by the quadrant of its children in x and y: each gathers the 11 x 11 x 19
// mother nodes that its 17 x 17 fine columns read, upsamples along x in shared
// memory and keeps the y pass of a column in registers, once per coarse z plane,
// for the 33 fine nodes along z (both children of the column).  One CTA per mother
// left most SMs waiting (204 mothers on 304 CTAs) and evaluated the y pass again
// for each of the four z taps: 107 -> 60 us for 204 mothers (FP32), 694 -> 229 us
// for 295 (FP64, whose pipe is then 73 % busy).
template <typename TS>
struct Refine3Smem {
  static constexpr int CN = 11, CZ = 19;
  static constexpr int TILE = CN * CN * CZ;          // mother nodes of the quadrant
  static constexpr int KN = 9, KZ = 13;              // coarser nodes their prediction reads
  static constexpr int KB = KN * KN * KZ;            // coarse box, then
  static constexpr int KX = CN * KN * KZ;            // ... its x pass
  static constexpr int KY = CN * CN * KZ;            // ... and y pass
  static constexpr int X = CZ * CN * Col3::B;        // x pass of the upsampling (over box and x pass)
  static_assert(KB + KX <= X, "the gather's scratch fits under the x pass");
  static constexpr size_t RING = ((size_t)kRingBytesD<3> + 15) / 16 * 16;
  static constexpr size_t BYTES = RING + sizeof(TS) * (TILE + X + KY);
};

template <typename TS>
__global__ void __launch_bounds__(Col3::NT, sizeof(TS) == 8 ? 2 : 3) k_refine3(PoolView pv, TS* __restrict__ y) {
  pdl_enter();
  using SM = Refine3Smem<TS>;
  constexpr int B = Col3::B, NQ = Col3::NQ, NT = Col3::NT, CN = SM::CN, CZ = SM::CZ, KN = SM::KN, KZ = SM::KZ;
  RingD<3>& R = *smem_as<RingD<3>>(0);
  TS* T = smem_as<TS>(SM::RING);
  TS* X = T + SM::TILE;
  TS* kb = X;               // coarse box and its x pass, before the upsampling
  TS* kx = X + SM::KB;
  TS* ky = X + SM::X;
  const int t = threadIdx.x;
  const int nact = pv.cnt->n_act;
  const int n_alloc = pv.cnt->n_alloc, n_free = pv.cnt->n_free;
  if (n_alloc > n_free) {
    if (blockIdx.x == 0 && t == 0) set_err(pv, kErrCapacity);
    return;
  }
  if (n_alloc == 0) return;  // no block refines: the list stays as it is
  // fine column of the thread (even rows first: the warps of the y pass take one branch)
  const bool col = t < NQ;
  const int fx = t % B, ry = (t / B) % B, fy = ry < 9 ? 2 * ry : 2 * (ry - 9) + 1;
  // half of a gathered column: z = -1 .. 8 or 9 .. 17
  const int gh = t >= CN * CN ? 1 : 0, gc = t - gh * CN * CN;
  const bool gat = gc < CN * CN;
  for (int it = blockIdx.x; it < 4 * nact; it += gridDim.x) {
    const int p = it >> 2, quad = it & 3, qx = quad & 1, qy = quad >> 1;
    const int slot = pv.act[p];
    const int2 off = new_offset(pv, p);
    const int e0 = off.x, a0 = off.y;
    if (pv.flag[slot] != 1) {
      if (quad == 0 && t == 0) pv.act_next[e0] = slot;
      continue;
    }
    const BlockInfo b = load_block(pv, slot);
    const TreeDev& td = pv.trees[b.tree];
    build_ring<3, B>(pv, td, b, R);
    __syncthreads();
    const bool mixed = R.mixed != 0;
    build_regions<3, B, CtaGroup>(b, R);
    __syncthreads();
    const int l1 = b.lvl + 1;
    const int bx = qx ? 7 : -1, by = qy ? 7 : -1;  // first mother node of the quadrant
    bool bad = false;
    unsigned pred = 0;  // nodes of the half column predicted from the coarse lattice
    const int gi = gc % CN + bx, gj = (gc / CN) % CN + by;
    TS* gd = T + (gc % CN) + CN * ((gc / CN) % CN) + (gh ? 10 * CN * CN : 0);  // the half's first node
    if (gat) {
      const int rb = reg_class<B>(gi) + 7 * reg_class<B>(gj);
      static_for<0, 4>([&](auto cc) {
        constexpr int C = decltype(cc)::value;
        // lower half: classes 0 .. 3 at nodes -1, 0, 1..7, 8; upper: 4 .. 6 at 9..15, 16, 17
        if (C == 3 && gh) return;
        const int cls = gh ? C + 4 : C;
        const int k0 = gh ? (C == 0 ? 9 : 15 + C) : (C == 0 ? -1 : C == 1 ? 0 : C == 2 ? 1 : 8);
        const int k1 = gh ? (C == 0 ? 15 : 15 + C) : (C == 0 ? -1 : C == 1 ? 0 : C == 2 ? 7 : 8);
        const int f0 = gh ? 9 : -1;
        const int4 e = R.reg[rb + 49 * cls];
        if (e.x < 0) {
          bad = true;
          for (int k = k0; k <= k1; ++k) gd[(k - f0) * CN * CN] = TS(0);
          return;
        }
        const ColOwn o(e, l1, gi, gj, pv.vs);
        const bool all = o.m >= b.lvl;
        for (int k = k0; k <= k1; ++k) {
          if (all || o.node(k)) {
            cp_async(gd + (k - f0) * CN * CN, (const TS*)y + o.at(k));
          } else {
            bad |= o.m != b.lvl - 1;
            pred |= 1u << (k - f0);
          }
        }
      });
    }
    if (mixed && R.coarser && R.cmask) {
      // predicted nodes: the span, per axis, of the classes owned by a coarser
      // leaf, within the quadrant; nlo / nhi: the coarse nodes they read
      int lo[3], hi[3], nlo[3], nhi[3];
      bool any = true;
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        const int m = (R.cmask >> (7 * a)) & 127;
        const int o0 = a == 0 ? bx : a == 1 ? by : -1, o1 = o0 + (a == 2 ? CZ : CN) - 1;
        const int cl = m ? __ffs(m) - 1 : 0, ch = m ? 31 - __clz(m) : 0;
        const int l = cl == 0 ? -1 : cl == 1 ? 0 : cl == 2 ? 1 : cl == 3 ? 8 : cl == 4 ? 9 : cl == 5 ? 16 : 17;
        const int h = ch == 0 ? -1 : ch == 1 ? 0 : ch == 2 ? 7 : ch == 3 ? 8 : ch == 4 ? 15 : ch == 5 ? 16 : 17;
        lo[a] = max(l, o0);
        hi[a] = min(h, o1);
        any &= lo[a] <= hi[a];
        nlo[a] = (lo[a] >> 1) - 1;
        nhi[a] = (hi[a] >> 1) + 2;
      }
      if (any) {
        // box origins: coarse node kx0 .. kx0 + 8 (x, y), -2 .. 10 (z)
        const int kx0 = qx ? 2 : -2, ky0 = qy ? 2 : -2;
        for (int q = t; q < SM::KB; q += NT) {
          const int nx = q % KN + kx0, ny = (q / KN) % KN + ky0, nz = q / (KN * KN) - 2;
          if (nx < nlo[0] || nx > nhi[0] || ny < nlo[1] || ny > nhi[1] || nz < nlo[2] || nz > nhi[2]) continue;
          const int4 e = R.reg[reg_class<B>(2 * nx) + 7 * reg_class<B>(2 * ny) + 49 * reg_class<B>(2 * nz)];
          if (e.x < 0 || e.y < b.lvl - 1) {
            bad = true;
            kb[q] = TS(0);
          } else {
            const ColOwn o(e, l1, 2 * nx, 2 * ny, pv.vs);
            cp_async(kb + q, (const TS*)y + o.at(2 * nz));
          }
        }
        cp_async_wait_all();
        __syncthreads();
        // x, then y (then z at the node): the order of predict_box
        const int ex = hi[0] - lo[0] + 1, ey = nhi[1] - nlo[1] + 1, ez = nhi[2] - nlo[2] + 1, fyn = hi[1] - lo[1] + 1;
        for (int q = t; q < ex * ey * ez; q += NT) {
          const int xx = q % ex + lo[0], ny = (q / ex) % ey + nlo[1] - ky0, nz = q / (ex * ey) + nlo[2] + 2;
          const TS* c = kb + (nz * KN + ny) * KN + (xx >> 1) - kx0;
          kx[(nz * KN + ny) * CN + xx - bx] = (xx & 1) ? dd4(c[-1], c[0], c[1], c[2]) : c[0];
        }
        __syncthreads();
        for (int q = t; q < ex * fyn * ez; q += NT) {
          const int xx = q % ex + lo[0] - bx, yy = (q / ex) % fyn + lo[1], nz = q / (ex * fyn) + nlo[2] + 2;
          const TS* c = kx + (nz * KN + (yy >> 1) - ky0) * CN + xx;
          ky[(nz * CN + yy - by) * CN + xx] = (yy & 1) ? dd4(c[-CN], c[0], c[CN], c[2 * CN]) : c[0];
        }
        __syncthreads();
      }
    }
    if (pred) {
      const int f0 = gh ? 9 : -1;
      const TS* c = ky + (gj - by) * CN + gi - bx;
      constexpr int st = CN * CN;
#pragma unroll
      for (int d = 0; d < 10; ++d) {
        if (!((pred >> d) & 1)) continue;
        const int k = f0 + d;
        const TS* ck = c + ((k >> 1) + 2) * st;
        gd[d * CN * CN] = (k & 1) ? dd4(ck[-st], ck[0], ck[st], ck[2 * st]) : ck[0];
      }
    }
    if (bad) set_err(pv, kErrGraded);
    if (quad == 0 && t < 8) {
      // light data of the children, in the order of their Hilbert keys
      int32_t c[3] = {(int32_t)(2 * b.c[0] + (t & 1)), (int32_t)(2 * b.c[1] + ((t >> 1) & 1)), (int32_t)(2 * b.c[2] + (t >> 2))};
      const int cs = pv.freelist[n_free - n_alloc + a0 + t];
      const uint64_t key = block_key<3>(c, l1, td.Jmax);
      int rank = 0;
      for (int o = 0; o < 8; ++o) rank += __shfl_sync(0xffu, key, o) < key;
      pv.act_next[e0 + rank] = cs;
      pv.lvl[cs] = (int8_t)l1;
      pv.tree[cs] = (int16_t)b.tree;
      for (int a = 0; a < 3; ++a) pv.crd[3 * cs + a] = c[a];
      pv.hkey[cs] = key;
      pv.flag[cs] = 0;
    }
    const int c0 = pv.freelist[n_free - n_alloc + a0 + quad], c1 = pv.freelist[n_free - n_alloc + a0 + quad + 4];
    cp_async_wait_all();
    __syncthreads();
    // x pass of the upsampling on the rows (y, z) of the quadrant: odd, then even fine nodes
    for (int q = t; q < CN * CZ * 8; q += NT) {
      const int row = q >> 3, m = q & 7;
      const TS* c = T + row * CN + m;
      X[row * B + 2 * m + 1] = dd4(c[0], c[1], c[2], c[3]);
    }
    for (int q = t; q < CN * CZ * 9; q += NT) {
      const int row = q / 9, m = q % 9;
      X[row * B + 2 * m] = T[row * CN + m + 1];
    }
    __syncthreads();
    if (col) {
      TS yv[CZ];  // y pass on the mother's z planes -1 .. 17
      const TS* x0 = X + (fy >> 1) * B + fx;
      if (fy & 1) {
#pragma unroll
        for (int z = 0; z < CZ; ++z) {
          const TS* r = x0 + z * CN * B;
          yv[z] = dd4(r[0], r[B], r[2 * B], r[3 * B]);
        }
      } else {
#pragma unroll
        for (int z = 0; z < CZ; ++z) yv[z] = x0[z * CN * B + B];
      }
      TS* lo = y + (int64_t)c0 * pv.vs + fy * B + fx;
      TS* up = y + (int64_t)c1 * pv.vs + fy * B + fx;
#pragma unroll
      for (int z = 0; z < 33; ++z) {
        const TS v = (z & 1) ? dd4(yv[z / 2], yv[z / 2 + 1], yv[z / 2 + 2], yv[z / 2 + 3]) : yv[z / 2 + 1];
        if (z <= 16) lo[NQ * z] = v;
        if (z >= 16) up[NQ * (z - 16)] = v;
      }
    }
    __syncthreads();
  }
}

}  // namespace mr
