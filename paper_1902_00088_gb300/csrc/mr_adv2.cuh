// 2D advection stage on blocks of 17^2 or 33^2 nodes: a group of threads (a warp
// or a CTA) per block.
#pragma once
#include "mr_kernels.cuh"

namespace mr {

// Geometry of the stage kernel.  GT: threads per block (32 or a CTA); NW: blocks
// per CTA (1 unless GT is 32).
//
// Tile: the block's own nodes row after row without padding, as they lie in the
// pool, so that the bulk-copy engine brings them; the ghost rows below and above
// follow at the same pitch.  The x ghosts of row y lie GO words behind the place
// that node (x, y) of that pitch would have: consecutive lanes (consecutive nodes)
// read consecutive banks at every neighbour, also where a row ends.  No corners:
// the stencil is a cross.
template <int B, typename TS, typename TY, int GT, int NW, int ST>
struct Stage2 {
  static constexpr int NI = B * B;
  static constexpr int R0 = (2 * B + 2 + 3) / 4 * 4;                  // node (0, 0), 16-byte aligned
  static constexpr int GO = (NI + 2 * B + 2 + 31) / 32 * 32;          // x ghosts
  static constexpr int TILE = (R0 + GO + NI + 2 + 3) / 4 * 4;
  static constexpr int VS = (NI + 3) / 4 * 4;                         // padded block, the pool's stride
  static constexpr int CN = (B - 1) / 2 + 3;                          // coarse nodes -1 .. (B + 1) / 2 along a face
  static constexpr int PATCH = 4 * CN;                                // 4 coarse nodes across a face
  static constexpr int X0 = 0, X1 = 2 * CN, XE = X1 + 4 * B;          // x pass: face across x [ny][2], across y [ny][x]
  static constexpr int NREG = RingD<2>::NREG;
  static constexpr bool ROWS = sizeof(TS) == 4 && ST >= 1;            // state / accumulator rows by bulk copies
  static constexpr bool Y0 = ST == 0 && sizeof(TS) != sizeof(TY);     // the state beside a tile of another type
  static constexpr size_t up(size_t x) { return (x + 15) / 16 * 16; }
  static constexpr size_t TAB = 16;                                   // after the mbarrier
  static constexpr size_t SCR = TAB + up(sizeof(int4) * (NREG + 1));
  static constexpr size_t FAC = SCR + up(sizeof(TY) * (2 * PATCH + XE));
  static constexpr size_t TIL = FAC + up(sizeof(TY) * 4 * B);
  static constexpr size_t ROW = TIL + sizeof(TY) * TILE;
  static constexpr size_t AREA = up(ROW + (ROWS ? 2 : Y0 ? 1 : 0) * sizeof(TS) * VS);
  static constexpr size_t BYTES = NW * AREA;
  static_assert(GT == 32 || NW == 1, "a CTA or its warps");
  static_assert(sizeof(TY) * TILE % 16 == 0, "aligned rows");
};

// One RK4 stage on every block (Sec. 3: 4th-order central FD + classic RK4):
//   k = N(Y_s) on the synchronised tile, then the 3-register update
//   s0: acc = y + dt/6 k, Y1 = y + dt/2 k      s1: acc += dt/3 k, Y2 = y + dt/2 k
//   s2: acc += dt/3 k,    Y3 = y + dt k        s3: y = acc + dt/6 k
// Advection RHS: -(u Dx phi + v Dy phi),
//   D1 f = ((f[-2] - f[2]) + 8 (f[1] - f[-1])) / (12 dx).
//
// The block's own nodes come by one bulk copy; only the four ghost strips of width
// 2 are gathered, in stage 0 also the edge nodes that another block holds (its copy
// is the value, stored back, Sec. 2.5; after stage 0 equal-level copies are
// identical).  Next to coarser leaves only the strips of those faces are predicted:
// at most one face per axis, the outer one of the block's place in its mother.
//
// Bound by the shared and global wavefronts of the load/store unit, then by HBM:
// 62 us per launch on 65536 blocks of 17^2 (FP32, one warp per block), where the
// five arrays of stages 1 and 2 alone take 58; 89 with the whole tile of width 2
// gathered node by node.  7472 blocks of an adapted forest: 19 us, 36 before.
// Warps per SM for one warp per block, FP32 advection: 20 (96 registers, nothing
// spilled) 62 us, 16 65, 24 64, 28 70, 32 (64 registers, 150 bytes spilled) 73.  At 20
// the FP32 swirl spills 8 to 16 bytes and the FP64 states, bound by the FP64 pipe, up
// to 100.
template <int B, int RHS, typename TS, typename TY, typename TSRC, int GT, int NW, int ST>
__global__ void __launch_bounds__(GT * NW, GT == 32 ? 20 / NW : 1024 / GT) k_stage2(PoolView pv, const TSRC* __restrict__ src,
                                                                     TS* __restrict__ y, TS* __restrict__ acc,
                                                                     TY* __restrict__ ynext, int staging,
                                                                     StageArgs sa) {
  pdl_enter();
  using SM = Stage2<B, TS, TY, GT, NW, ST>;
  using PL = Plan<2>;
  using TC = TY;
  using Grp = std::conditional_t<GT == 32, WarpGroup, CtaGroup>;
  const Grp g{};
  constexpr int NI = SM::NI, GO = SM::GO, CN = SM::CN, PATCH = SM::PATCH;
  constexpr bool BULK = std::is_same<TSRC, TC>::value;  // own nodes by a bulk copy
  constexpr bool ROWS = SM::ROWS, NEEDY = ST == 1 || ST == 2;
  constexpr bool Y0 = SM::Y0;  // stage 0: the committed state is kept in ys; else the tile holds it
  static_assert(Y0 == (ST == 0 && !BULK), "stage 0 reads the state");
  const int r = g.rank(), grp = GT == 32 ? threadIdx.x >> 5 : 0;
  unsigned char* area = smem_as<unsigned char>(0) + grp * SM::AREA;
  uint64_t* bar = reinterpret_cast<uint64_t*>(area);
  int4* reg = reinterpret_cast<int4*>(area + SM::TAB);
  TC* patch = reinterpret_cast<TC*>(area + SM::SCR);
  TC* xp = patch + 2 * PATCH;
  TC* fac = reinterpret_cast<TC*>(area + SM::FAC);
  TC* tile = reinterpret_cast<TC*>(area + SM::TIL) + SM::R0;  // node (0, 0)
  TS* ys = reinterpret_cast<TS*>(area + SM::ROW);
  TS* as = ys + SM::VS;
  __shared__ int32_t splan[NW][PL::INTS];
  __shared__ int64_t snb[NW][PL::NB];  // pool offsets of the plan's neighbours
  const int nact = pv.cnt->n_act;
  const int p0 = blockIdx.x * NW + grp, np = gridDim.x * NW;
  if (blockIdx.x * NW >= nact) return;  // no block for this CTA (small grids)
  if (blockIdx.x == 0 && threadIdx.x == 0) atomicAdd(&pv.cnt->stage_blocks, (unsigned long long)nact);
  if ((BULK || ROWS) && r == 0) mbar_init(bar, 1);
  int32_t cur = p0 < nact && r < PL::INTS ? pv.plan[(int64_t)p0 * PL::INTS + r] : 0;
  unsigned phase = 0;
  // place of node (i, j) in the tile
  auto at_tile = [](int i, int j) { return B * j + i + (i < 0 || i >= B ? GO : 0); };
  for (int p = p0; p < nact; p += np) {
    if (r < PL::INTS) splan[grp][r] = cur;
    if (r >= PL::NBO && r < PL::NBO + PL::NB) snb[grp][r - PL::NBO] = (int64_t)cur * pv.vs;
    g.sync();  // also: the previous block's tile and rows have been read
    const int pn = p + np;
    cur = pn < nact && r < PL::INTS ? pv.plan[(int64_t)pn * PL::INTS + r] : 0;
    const int32_t* pl = splan[grp];
    const BlockInfo b = plan_block<2>(pl);
    const bool uni = (pl[1] >> 30) & 1;
    const int64_t own = (int64_t)b.slot * pv.vs;
    const bool staged = ROWS && staging != 0;
    if ((BULK || staged) && r == 0) {
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      mbar_expect_tx(bar, (BULK ? sizeof(TC) * SM::VS : 0) + (staged ? (NEEDY ? 2 : 1) * sizeof(TS) * SM::VS : 0));
      if (BULK) bulk_g2s(tile, src + own, sizeof(TC) * SM::VS, bar);
      if (staged) {
        if (NEEDY) bulk_g2s(ys, y + own, sizeof(TS) * SM::VS, bar);
        bulk_g2s(as, acc + own, sizeof(TS) * SM::VS, bar);
      }
    }
    const TreeDev& td = pv.trees[b.tree];
    if (RHS == MR_RHS_SWIRL) {
      // factors of the velocity along x, then along y
      const TC* A = lattice<TC>(pv) + td.lat_off + (int64_t)kLatSwA * td.N;
      const TC* Bt = lattice<TC>(pv) + td.lat_off + (int64_t)kLatSwB * td.N;
      for (int q = r; q < 2 * B; q += GT) {
        const int64_t U = pmod64(((q < B ? b.c[0] : b.c[1]) * (B - 1) + q % B) << (td.Jmax - b.lvl), td.N);
        fac[2 * q] = A[U];
        fac[2 * q + 1] = Bt[U];
      }
    }
    if (!BULK) {
#pragma unroll 5
      for (int q = r; q < NI; q += GT) {
        const TSRC v = src[own + q];
        tile[q] = to_tile<TC>(v);
        if constexpr (Y0) ys[q] = v;
      }
    }
    // edge node q of another block: its copy, stored where it differs
    auto commit = [&](int i, int j, TSRC v) {
      const int q = B * j + i;
      if (ST == 0) {
        TSRC mine;
        if constexpr (BULK) mine = tile[q];
        else mine = ys[q];
        if (differs(mine, v)) const_cast<TSRC*>(src)[own + q] = v;
        if constexpr (Y0) ys[q] = v;
      }
      tile[q] = to_tile<TC>(v);
    };
    auto landed = [&]() -> bool {
      if (!BULK) g.sync();
      if (!BULK && !staged) return true;
      phase ^= 1;
      return bulk_landed(pv, bar, phase ^ 1);
    };
    // ghost h: rows -2, -1, B, B + 1, then the pairs left and right of each row
    auto ghost = [](int h, int& i, int& j) {
      if (h < 4 * B) {
        const int l = h / B;
        i = h - l * B;
        j = l < 2 ? l - 2 : B - 2 + l;
      } else {
        const int e = h - 4 * B, s = e >= 2 * B, w = e - s * 2 * B;
        j = w >> 1;
        i = s ? B + (w & 1) : (w & 1) - 2;
      }
    };
    if (uni) {
      constexpr int NG = 8 * B, NE = ST == 0 ? 2 * B - 1 : 0, RN = (NG + NE + GT - 1) / GT;
      const int64_t* nb = snb[grp];
      TSRC val[RN];
#pragma unroll
      for (int u = 0; u < RN; ++u) {
        const int h = r + u * GT;
        if (h >= NG + NE) continue;
        int i, j;
        ghost(h, i, j);
        if (NE && h >= NG) {  // edge nodes held by the upper neighbours: column B - 1, row B - 1
          const int e = h - NG;
          i = e < B ? B - 1 : e - B;
          j = e < B ? e : B - 1;
        }
        const int sx = i < 0 ? 0 : i >= B || (NE && i == B - 1 && h >= NG) ? 2 : 1;
        const int sy = j < 0 ? 0 : j >= B || (NE && j == B - 1 && h >= NG) ? 2 : 1;
        // a ghost in row or column B - 1 (stage 0): its holder is the next block
        const int ex = NE && h < NG && i == B - 1 ? 2 : sx, ey = NE && h < NG && j == B - 1 ? 2 : sy;
        val[u] = src[nb[ex + 3 * ey] + (i - (ex - 1) * (B - 1)) + B * (j - (ey - 1) * (B - 1))];
      }
      if (!landed()) return;
#pragma unroll
      for (int u = 0; u < RN; ++u) {
        const int h = r + u * GT;
        if (h >= NG + NE) continue;
        if (NE && h >= NG) {
          const int e = h - NG;
          commit(e < B ? B - 1 : e - B, e < B ? e : B - 1, val[u]);
        } else {
          int i, j;
          ghost(h, i, j);
          tile[at_tile(i, j)] = to_tile<TC>(val[u]);
        }
      }
    } else {
      const int4* rsrc = plan_regions<2>(pv, p);
      for (int q = r; q < SM::NREG; q += GT) reg[q] = rsrc[q];
      g.sync();
      const int l1 = b.lvl + 1;
      bool bad = false;
      // n: first coarse node across the axis' face; faces with a coarser leaf
      const int n0[2] = {(b.c[0] & 1) ? (B - 1) / 2 - 1 : -2, (b.c[1] & 1) ? (B - 1) / 2 - 1 : -2};
      auto coarse = [&](int t) {  // t in [0, 10): axis t / 5, one class box of the face each
        const int w = t % 5 + 1, n = n0[t / 5] < 0 ? 0 : 6;
        return reg[t < 5 ? n + 7 * w : w + 7 * n].y < b.lvl;
      };
      bool fx = false, fy = false;
      if constexpr (GT == 32) {
        const unsigned m = __ballot_sync(0xffffffffu, r < 10 && coarse(r));
        fx = m & 31;
        fy = m & 992;
      } else {
#pragma unroll
        for (int t = 0; t < 5; ++t) {
          fx |= coarse(t);
          fy |= coarse(t + 5);
        }
      }
      // ghosts, the edge nodes, then the patches of coarse nodes at the two faces
      constexpr int NG = 8 * B, NE = 4 * (B - 1), RN = (NG + NE + GT - 1) / GT;
      TSRC val[RN];
      unsigned have = 0, pred = 0;
#pragma unroll
      for (int u = 0; u < RN; ++u) {
        const int h = r + u * GT;
        val[u] = TSRC(0);
        if (h >= NG + NE) continue;
        int i, j;
        ghost(h, i, j);
        if (h >= NG) {
          const int e = h - NG, s = e / (B - 1), w = e - s * (B - 1);
          i = s == 0 ? w : s == 1 ? B - 1 : s == 2 ? w + 1 : 0;
          j = s == 0 ? 0 : s == 1 ? w : s == 2 ? B - 1 : w + 1;
        }
        const int4 e = reg[reg_class<B>(i) + 7 * reg_class<B>(j)];
        if (h >= NG && e.x == b.slot) continue;
        if (e.x < 0) {
          bad = true;  // zero; of an edge node in the tile only: the pool stays as it is
          (h >= NG ? pred : have) |= 1u << u;
          continue;
        }
        const int sh = l1 - e.y, ox = 2 * i - (int)(int16_t)(e.z & 0xffff), oy = 2 * j - (e.z >> 16);
        if (h >= NG || e.y >= b.lvl || ((ox | oy) & ((1 << sh) - 1)) == 0) {
          val[u] = src[(int64_t)e.x * pv.vs + (ox >> sh) + B * (oy >> sh)];
          have |= 1u << u;
        } else {
          bad |= e.y != b.lvl - 1;
          pred |= 1u << u;
        }
      }
      if (fx || fy) {
        // patch of the face across x: [ny][4], across y: [4][nx]
        constexpr int RP = (2 * PATCH + GT - 1) / GT;
#pragma unroll
        for (int u = 0; u < RP; ++u) {
          const int q = r + u * GT;
          if (q >= 2 * PATCH || !(q < PATCH ? fx : fy)) continue;
          const int w = q < PATCH ? q : q - PATCH;
          const int nx = q < PATCH ? n0[0] + (w & 3) : w % CN - 1, ny = q < PATCH ? (w >> 2) - 1 : n0[1] + w / CN;
          const int4 e = reg[reg_class<B>(2 * nx) + 7 * reg_class<B>(2 * ny)];
          TC v = TC(0);
          if (e.x < 0 || e.y < b.lvl - 1) {
            bad = true;
          } else {
            const int sh = l1 - e.y;
            v = to_tile<TC>(src[(int64_t)e.x * pv.vs + ((4 * nx - (int)(int16_t)(e.z & 0xffff)) >> sh) +
                                B * ((4 * ny - (e.z >> 16)) >> sh)]);
          }
          patch[q] = v;
        }
        g.sync();
        // x pass; the odd layer of a face is predicted, the even one a coarse node
        for (int q = r; q < SM::XE; q += GT) {
          if (!(q < SM::X1 ? fx : fy)) continue;
          if (q < SM::X1) {
            const TC* c = patch + 4 * (q >> 1);
            const bool low = n0[0] < 0;
            xp[q] = ((q & 1) != 0) == low ? dd4(c[0], c[1], c[2], c[3]) : c[low ? 1 : 2];
          } else {
            const int w = q - SM::X1, row = w / B, x = w - row * B;
            const TC* c = patch + PATCH + CN * row + (x >> 1);
            xp[q] = (x & 1) ? dd4(c[0], c[1], c[2], c[3]) : c[1];
          }
        }
        g.sync();
      }
      if (!landed()) return;
#pragma unroll
      for (int u = 0; u < RN; ++u) {
        const int h = r + u * GT;
        if (h >= NG + NE) continue;
        int i, j;
        ghost(h, i, j);
        if (h >= NG) {
          const int e = h - NG, s = e / (B - 1), w = e - s * (B - 1);
          i = s == 0 ? w : s == 1 ? B - 1 : s == 2 ? w + 1 : 0;
          j = s == 0 ? 0 : s == 1 ? w : s == 2 ? B - 1 : w + 1;
          if ((have >> u) & 1) commit(i, j, val[u]);
          if ((pred >> u) & 1) tile[B * j + i] = TC(0);
          continue;
        }
        TC v = to_tile<TC>(val[u]);
        if ((pred >> u) & 1) {  // y pass at the node
          const bool ax = i < 0 || i >= B;
          const TC* c = ax ? xp + (j >> 1) * 2 + (i < 0 ? i + 2 : i - B) : xp + SM::X1 + i;
          const int st = ax ? 2 : B;
          const bool odd = j & 1;
          if (odd) v = dd4(c[0], c[st], c[2 * st], c[3 * st]);
          else v = c[ax ? st : (j < 0 ? 1 : 2) * st];
        }
        tile[at_tile(i, j)] = v;
      }
      if (bad) set_err(pv, kErrGraded);
    }
    const TC c = tree_cD<TC>(td, b.lvl);
    const StageCoef<TS> cs(pv, sa, b.tree, ST);
    const TC ct = StageCoef<TC>(pv, sa, b.tree, ST).ct;
    const TS cas = cs.ca, cys = cs.cy;
    const TC uc0 = tree_rhs<TC>(td, 0), uc1 = tree_rhs<TC>(td, 1);
    // nodes q = r + GT u, U at a time: the loads of the state first
    constexpr int RQ = (NI + GT - 1) / GT, U = RQ < 5 ? RQ : 5;
    constexpr bool EARLY = !ROWS && RQ <= 5 && ST >= 1;  // loads that need not wait for the tile
    TS yv[U], av[U];
    auto load = [&](int u, int q) {
      if (NEEDY) yv[u] = staged ? ys[q] : y[own + q];
      if (ST >= 1) av[u] = staged ? as[q] : acc[own + q];
    };
    if (EARLY) {
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (r + u * GT < NI) load(u, r + u * GT);
    }
    g.sync();
#pragma unroll
    for (int q0 = 0; q0 < RQ * GT; q0 += U * GT) {
      if (!EARLY) {
#pragma unroll
        for (int u = 0; u < U; ++u)
          if (q0 + u * GT + r < NI) load(u, q0 + u * GT + r);
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int q = q0 + u * GT + r;
        if (q >= NI) continue;
        const int i = q % B;
        const TC* t0 = tile + q;
        const TC dxv = d1_sum(t0[i < 2 ? GO - 2 : -2], t0[i < 1 ? GO - 1 : -1], t0[i > B - 2 ? GO + 1 : 1],
                              t0[i > B - 3 ? GO + 2 : 2]) * c;
        const TC dyv = d1_sum(t0[-2 * B], t0[-B], t0[B], t0[2 * B]) * c;
        TC u0 = uc0, u1 = uc1;
        if (RHS == MR_RHS_SWIRL) {
          const int j = q / B;
          u0 = ct * (fac[2 * i] * fac[2 * (B + j) + 1]);
          u1 = -(ct * (fac[2 * (B + j)] * fac[2 * i + 1]));
        }
        const TC s = u0 * dxv + u1 * dyv;
        const TS kk = to_state<TS>(-s);
        const int64_t at = own + q;
        if (ST == 0) {
          TS y0;
          if constexpr (Y0) y0 = ys[q];
          else y0 = t0[0];
          acc[at] = y0 + cas * kk;
          ynext[at] = to_tile<TY>(y0 + cys * kk);
        } else if (NEEDY) {
          acc[at] = av[u] + cas * kk;
          ynext[at] = to_tile<TY>(yv[u] + cys * kk);
        } else {
          y[at] = av[u] + cas * kk;
        }
      }
    }
  }
}
}  // namespace mr
