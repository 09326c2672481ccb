// Wavelet details of 2D blocks (Sec. 2.3), one variable of one block per thread
// group: a warp for 17^2 blocks, a CTA of 128 threads for 33^2 ones.
#pragma once
#include "mr_kernels.cuh"

namespace mr {

// D = B - P(R(B)) reads, of the tile, the block's own nodes and the coarse
// lattice (every second node, one beyond each side).  A coarse-lattice node of
// the ghost layer is a node of its owner whatever the owner's level, so 40 (17^2)
// or 72 (33^2) ghost nodes are gathered and none is predicted.
//
// Rows of the work array, one per coarse y (-1 .. NC - 2): the NC coarse nodes,
// then the x pass at the odd nodes between them.
template <int B>
struct Det2 {
  static constexpr int NC = (B + 1) / 2 + 2, NO = (B - 1) / 2;
  static constexpr int RP = NC + NO, SZ = NC * RP;
  static constexpr int NI = B * B;
  static constexpr int NG = NC * NC - ((B + 1) / 2) * ((B + 1) / 2);
  static constexpr int GS = B == 17 ? 32 : 128;        // threads per item
  static constexpr int NT = 128, ITEMS = NT / GS;      // threads and items per CTA
  static constexpr int K = (NI + GS - 1) / GS;         // nodes per thread
  static constexpr int NE = 4 * (B - 1);               // edge nodes
  // edge node e: lower edge from x = 0, right edge upward, upper edge back, left edge down
  __device__ static __forceinline__ void edge(int e, int& i, int& j) {
    const int s = e / (B - 1), r = e % (B - 1);
    i = s == 0 ? r : s == 1 ? B - 1 : s == 2 ? B - 1 - r : 0;
    j = s == 0 ? 0 : s == 1 ? r : s == 2 ? B - 1 : B - 1 - r;
  }
  __device__ static __forceinline__ int edge_of(int i, int j) {  // -1: not an edge node
    return j == 0 && i < B - 1 ? i : i == B - 1 && j < B - 1 ? B - 1 + j : j == B - 1 && i > 0 ? 3 * (B - 1) - i
           : i == 0 ? 4 * (B - 1) - j : -1;
  }
  // place of node x in a row: coarse nodes (even x) from 1, odd ones after them
  __host__ __device__ static constexpr int place(int x) { return (x & 1) ? NC + x / 2 : 1 + x / 2; }
};

template <int B, typename TS, typename TT, typename TD>
struct Det2Smem {
  using D2 = Det2<B>;
  static constexpr size_t TABS = (4 * (D2::NI + D2::NG) + 15) / 16 * 16;  // per CTA
  static constexpr size_t RING = ((size_t)kRingBytesD<2> + 15) / 16 * 16;
  static constexpr size_t W = (sizeof(TT) * D2::SZ + 15) / 16 * 16;
  // x pass of the FP64 evaluation of FP32 values
  static constexpr size_t XD = sizeof(TD) > sizeof(TT) ? sizeof(TD) * D2::NC * D2::NO : 0;
  static constexpr size_t NB = 80;                                          // neighbours' pool offsets
  static constexpr size_t EV = sizeof(TS) * D2::NE;  // edge values (a multiple of 16 bytes)
  static constexpr size_t ITEM = RING + W + (XD + 15) / 16 * 16 + EV + NB;
  static constexpr size_t BYTES = TABS + D2::ITEMS * ITEM;
};

// Bound by instruction issue and latency (48 % of the issue slots used); 12 CTAs per SM
// spill, 6 hide less latency: 8 CTAs of 4 warps.  Measured, before with one CTA (or warp) per block over the gathered and
// predicted 21^2 tile, variable after variable: 65536 FP32 blocks of 17^2 104 -> 78 us;
// 16384 blocks of 4 FP64 variables 165 -> 101 us; the rounds of an adaptive step with 64
// trees 168 -> 94 us, with 33^2 blocks of 4 variables 443 -> 238 us (a third of it by
// looking the owners of a block's edge nodes up apart from its own nodes).
template <int B, typename TS, typename TD, typename TT>
__global__ void __launch_bounds__(128, 8) k_details2(PoolView pv, TS* __restrict__ y) {
  pdl_enter();
  using D2 = Det2<B>;
  using SM = Det2Smem<B, TS, TT, TD>;
  using PL = Plan<2>;
  using G = std::conditional_t<D2::GS == 32, WarpGroup, CtaGroup>;
  constexpr int NC = D2::NC, NO = D2::NO, RP = D2::RP, NI = D2::NI, GS = D2::GS, K = D2::K;
  const G g{};
  const int rank = threadIdx.x % GS, item = threadIdx.x / GS;
  unsigned char* sm = smem_as<unsigned char>(0);
  int32_t* ntab = reinterpret_cast<int32_t*>(sm);
  int32_t* gtab = ntab + NI;
  unsigned char* mem = sm + SM::TABS + item * SM::ITEM;
  RingD<2>& R = *reinterpret_cast<RingD<2>*>(mem);
  TT* E = reinterpret_cast<TT*>(mem + SM::RING);
  TD* XD = reinterpret_cast<TD*>(mem + SM::RING + SM::W);
  int64_t* nbo = reinterpret_cast<int64_t*>(mem + SM::ITEM - SM::NB);
  TS* ev = reinterpret_cast<TS*>(mem + SM::ITEM - SM::NB - SM::EV);
  __shared__ double red[4];
  const int nact = pv.cnt->n_round, nv = pv.nvar;
  if ((int64_t)blockIdx.x * D2::ITEMS >= (int64_t)nact * nv) return;  // no item for this CTA (small grids)
  // nodes: place in the work array | kind << 12 (0 coarse, 1 odd x on a coarse row, 2
  // odd y) | upper edge in x << 14, in y << 15 | edge node << 16 (0: none, else + 1)
  for (int q = threadIdx.x; q < NI; q += blockDim.x) {
    const int i = q % B, j = q / B;
    const int row = (j & 1) ? j / 2 : j / 2 + 1;  // first row of the y pass, or the node's own
    const int kind = (j & 1) ? 2 : (i & 1);
    ntab[q] = (row * RP + D2::place(i)) | (kind << 12) | (i == B - 1 ? 1 << 14 : 0) | (j == B - 1 ? 1 << 15 : 0) |
              ((D2::edge_of(i, j) + 1) << 16);
  }
  // ghost nodes: place | neighbour << 12 | offset in that neighbour (of a uniform
  // neighbourhood) << 16
  for (int q = threadIdx.x; q < D2::NG; q += blockDim.x) {
    int n[2];  // coarse lattice position, at node 2 (n - 1)
    if (q < 2 * NC) {
      n[0] = q % NC;
      n[1] = q < NC ? 0 : NC - 1;
    } else {
      const int r = q - 2 * NC;
      n[0] = r % 2 ? NC - 1 : 0;
      n[1] = r / 2 + 1;
    }
    int nb = 0, off = 0, mul = 1, lm = 1;
    for (int a = 0; a < 2; ++a) {
      const int k = 2 * (n[a] - 1);
      const int s = k < 0 ? 0 : (k <= B - 2 ? 1 : 2);
      nb += s * mul;
      off += (k - (s - 1) * (B - 1)) * lm;
      mul *= 3;
      lm *= B;
    }
    gtab[q] = (n[1] * RP + n[0]) | (nb << 12) | (off << 16);
  }
  __syncthreads();
  auto group_and = [&](bool p) -> bool {
    if constexpr (GS == 32) return __all_sync(0xffffffffu, p);
    else return __syncthreads_and(p);
  };
  auto group_or = [&](bool p) -> bool {
    if constexpr (GS == 32) return __any_sync(0xffffffffu, p);
    else return __syncthreads_or(p);
  };
  const bool all_blocks = pv.cnt->first_round != 0;
  const int prev = pv.cnt->round_id - 1;
  const bool plan_ok = pv.cnt->plan_topo == pv.cnt->topo;
  // items: (block, variable); the stride is a multiple of nv, so a group keeps its
  // variable
  const int64_t first = (int64_t)blockIdx.x * D2::ITEMS + item, stride = (int64_t)gridDim.x * D2::ITEMS;
  const int v = (int)(first % nv);
  unsigned ndet = 0;
  double scale = 0.0;  // largest |value| of the tree's blocks seen by this group
  int scale_tree = -1;
  auto flush = [&]() {
    if (rank == 0 && scale_tree >= 0 && scale > 0.0) atomic_max_pos(&pv.svar[scale_tree * nv + v], scale);
  };
  for (int64_t it = first; it < (int64_t)nact * nv; it += stride) {
    const int p = (int)(it / nv);
    BlockInfo b;
    int q = 0;
    if (plan_ok) {
      const int32_t* pl = pv.plan + (int64_t)p * PL::INTS;
      b = plan_block<2>(pl);
      q = rank < PL::NB ? pl[PL::NBO + rank] : b.slot;
    } else {
      b = load_block(pv, pv.act[p]);
      q = b.slot;
      if (rank < PL::NB && rank != 4) {
        const int64_t cn[3] = {b.c[0] + rank % 3 - 1, b.c[1] + rank / 3 - 1, 0};
        q = tab_get<2>(pv, pv.trees[b.tree], b.lvl, cn);
      }
    }
    const TreeDev& td = pv.trees[b.tree];
    if (pv.norm_kind == 1 && b.tree != scale_tree) {
      flush();
      scale = 0.0;
      scale_tree = b.tree;
    }
    const bool uni = group_and(q >= 0);
    bool ring = false, dirty = all_blocks;
    if (!all_blocks) {
      if (uni) {
        dirty = group_or(rank < PL::NB && pv.stamp[q] == prev);
      } else {
        build_ring<2, B, G>(pv, td, b, R);
        g.sync();
        ring = true;
        dirty = group_or(rank < Geo<2, B>::NR && R.slot[rank] >= 0 && pv.stamp[R.slot[rank]] == prev);
      }
    }
    if (!dirty) {
      // no leaf of the ring changed in the previous round: the stored details
      // and norms are those of the unchanged tile
      if (pv.norm_kind == 1) scale = fmax(scale, pv.bmax[(int64_t)b.slot * nv + v]);
      continue;
    }
    ndet += v == 0;
    const int64_t vo = (int64_t)v * pv.vs, bs = (int64_t)nv * pv.vs;  // variable offset, block stride
    TS* const me = y + (int64_t)b.slot * bs + vo;
    // the thread's nodes; block-edge nodes held by another block take (and
    // store) its value
    TS raw[K];
    if (uni) {
      if (rank < PL::NB) nbo[rank] = (int64_t)q * bs + vo;
      g.sync();
#pragma unroll
      for (int k = 0; k < K; ++k) {
        const int n = rank + k * GS;
        if (n >= NI) continue;
        const int e = ntab[n];
        const int ux = (e >> 14) & 1, uy = (e >> 15) & 1;
        raw[k] = y[nbo[4 + ux + 3 * uy] + n - ux * (B - 1) - uy * (B * (B - 1))];
      }
      for (int k = rank; k < D2::NG; k += GS) {
        const int e = gtab[k];
        E[e & 0xfff] = to_tile<TT>(y[nbo[(e >> 12) & 15] + (e >> 16)]);
      }
#pragma unroll
      for (int k = 0; k < K; ++k) {
        const int n = rank + k * GS;
        if (n < NI && (ntab[n] & (3 << 14)) && differs(me[n], raw[k])) me[n] = raw[k];
      }
    } else {
      if (!ring && plan_ok) {  // the stage plan's owner table
        const int4* src = plan_regions<2>(pv, p);
        for (int r = rank; r < RingD<2>::NREG; r += GS) R.reg[r] = src[r];
      } else {
        if (!ring) {
          build_ring<2, B, G>(pv, td, b, R);
          g.sync();
        }
        build_regions<2, B, G>(b, R);
      }
      g.sync();
      const int l1 = b.lvl + 1;
      bool lost = false;
      auto owned = [&](const int4 e, int i, int j) -> int64_t {
        const int sh = l1 - e.y;
        const int ox = 2 * i - (int)(int16_t)(e.z & 0xffff), oy = 2 * j - (e.z >> 16);
        return (int64_t)e.x * bs + vo + (ox >> sh) + B * (oy >> sh);
      };
#pragma unroll
      for (int k = 0; k < K; ++k) {
        const int n = rank + k * GS;
        if (n < NI) raw[k] = me[n];
      }
      for (int k = rank; k < D2::NE; k += GS) {
        int i, j;
        D2::edge(k, i, j);
        const int4 e = R.reg[reg_class<B>(i) + 7 * reg_class<B>(j)];
        const int n = j * B + i;
        TS val = me[n];
        if (e.x < 0) {
          lost = true;
          val = TS(0);
        } else if (e.x != b.slot) {
          const TS mine = val;
          val = y[owned(e, i, j)];
          if (differs(mine, val)) me[n] = val;
        }
        ev[k] = val;
      }
      for (int k = rank; k < D2::NG; k += GS) {
        const int at = gtab[k] & 0xfff;
        const int i = 2 * (at % RP - 1), j = 2 * (at / RP - 1);
        const int4 e = R.reg[reg_class<B>(i) + 7 * reg_class<B>(j)];
        const bool ok = e.x >= 0 && e.y >= b.lvl - 1;
        lost |= !ok;
        E[at] = ok ? to_tile<TT>(y[owned(e, i, j)]) : TT(0);
      }
      g.sync();
#pragma unroll
      for (int k = 0; k < K; ++k) {
        const int n = rank + k * GS;
        if (n < NI && (ntab[n] >> 16)) raw[k] = ev[(ntab[n] >> 16) - 1];
      }
      if (lost) set_err(pv, kErrGraded);
    }
    // largest |value| of the interior, non-finite test, coarse nodes to the work array
    AbsMax<TT> mqa;
    bool bad = false;
    TT val[K];
#pragma unroll
    for (int k = 0; k < K; ++k) {
      const int n = rank + k * GS;
      if (n >= NI) continue;
      const TT t = val[k] = to_tile<TT>(raw[k]);
      mqa.add(t);
      bad |= !finite(t);
      const int e = ntab[n];
      if (((e >> 12) & 3) == 0) E[e & 0xfff] = t;
    }
    g.sync();
    // x pass, then the y pass and the detail at the thread's odd nodes
    float mt = 0.f;  // largest |value| of the coarse lattice
    AbsMax<TT> md;
    for (int k = rank; k < NC * NO; k += GS) {
      TT* r = E + (k / NO) * RP;
      const int m = k % NO;
      const TT a = r[m], c = r[m + 1], d = r[m + 2], f = r[m + 3];
      mt = fmaxf(fmaxf(mt, fmaxf(fabsf((float)a), fabsf((float)c))), fmaxf(fabsf((float)d), fabsf((float)f)));
      r[NC + m] = dd4(a, c, d, f);
    }
    g.sync();
#pragma unroll
    for (int k = 0; k < K; ++k) {
      const int n = rank + k * GS;
      if (n >= NI) continue;
      const int e = ntab[n], kind = (e >> 12) & 3;
      if (kind == 0) continue;
      const TT* r = E + (e & 0xfff);
      const TT pr = kind == 2 ? dd4(r[0], r[RP], r[2 * RP], r[3 * RP]) : r[0];
      md.add(val[k] - pr);
    }
    constexpr bool cert = sizeof(TT) == 4 && sizeof(TD) == 8;
    auto group_max = [&](auto m) {
      using A = decltype(m);
      m = warp_max_pos(m);
      if constexpr (GS > 32) {
        A* r = reinterpret_cast<A*>(red);
        __syncthreads();
        if ((threadIdx.x & 31) == 0) r[threadIdx.x >> 5] = m;
        __syncthreads();
        const int w = threadIdx.x & 31;
        m = warp_max_pos(w < 4 ? r[w] : A(0));
      }
      return m;
    };
    const TT m0 = group_max(md.get());
    const TT mq = group_max(mqa.get());
    double m = (double)m0;
    if constexpr (cert) {
      // certified as in k_details3: err bounds the FP32 evaluation's error
      const float err = 0x1p-19f * fmaxf(group_max(mt), (float)mq) + 1e-37f;
      if (!(pv.norm_kind == 0 && certain_vs_eps(m0, err, td))) {
        for (int k = rank; k < NC * NO; k += GS) {
          const TT* r = E + (k / NO) * RP + k % NO;
          XD[k] = dd4((TD)r[0], (TD)r[1], (TD)r[2], (TD)r[3]);
        }
        g.sync();
        AbsMax<TD> md64;
#pragma unroll
        for (int k = 0; k < K; ++k) {
          const int n = rank + k * GS;
          if (n >= NI) continue;
          const int e = ntab[n], kind = (e >> 12) & 3;
          if (kind == 0) continue;
          const int row = (e & 0xfff) / RP, c = (e & 0xfff) % RP;
          auto at = [&](int r) -> TD { return c < NC ? (TD)E[r * RP + c] : XD[r * NO + c - NC]; };
          const TD pr = kind == 2 ? dd4(at(row), at(row + 1), at(row + 2), at(row + 3)) : at(row);
          md64.add((TD)val[k] - pr);
        }
        m = (double)group_max(md64.get());
      }
    }
    if (group_or(bad)) m = __longlong_as_double(0x7ff8000000000000LL);
    if (rank == 0) {
      pv.md[(int64_t)b.slot * nv + v] = m;
      pv.bmax[(int64_t)b.slot * nv + v] = (double)mq;
    }
    if (pv.norm_kind == 1) scale = fmax(scale, (double)mq);
    g.sync();
  }
  if (pv.norm_kind == 1) flush();
  if (rank == 0 && ndet) atomicAdd(&pv.cnt->det_blocks, (unsigned long long)ndet);
}

}  // namespace mr
