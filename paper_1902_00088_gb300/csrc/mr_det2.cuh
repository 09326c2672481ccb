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
// Work array S: the block's own nodes row after row without padding, as they lie in
// the pool (one bulk copy), the ghost rows y = -2 and B + 1 where that pitch puts
// them, and the coarse ghosts x = -2 and B + 1 of every coarse row apart.  The x pass
// takes the detail of an odd node of an even row and leaves its prediction in the
// node's place; the y pass then reads rows y -+ 1 and y -+ 3 at every x alike.
template <int B>
struct Det2 {
  static constexpr int NC = (B + 1) / 2 + 2, NO = (B - 1) / 2;
  static constexpr int NI = B * B, VS = (NI + 3) / 4 * 4;
  static constexpr int NG = NC * NC - ((B + 1) / 2) * ((B + 1) / 2);
  static constexpr int GS = B == 17 ? 32 : 128;        // threads per item
  static constexpr int NT = 128, ITEMS = NT / GS;      // threads and items per CTA
  static constexpr int NE = 4 * (B - 1);               // edge nodes
  static constexpr int NU = 2 * B - 1;                 // ... held by the upper neighbours
  static constexpr int R0 = (2 * B + 3) / 4 * 4;       // node (0, 0), 16-byte aligned
  static constexpr int GL = R0 + B * (B + 2), GR = GL + NC, SZ = GR + NC;
  // edge node e: lower edge from x = 0, right edge upward, upper edge back, left edge down
  __device__ static __forceinline__ void edge(int e, int& i, int& j) {
    const int s = e / (B - 1), r = e % (B - 1);
    i = s == 0 ? r : s == 1 ? B - 1 : s == 2 ? B - 1 - r : 0;
    j = s == 0 ? 0 : s == 1 ? r : s == 2 ? B - 1 : B - 1 - r;
  }
  // coarse lattice position (0 .. NC - 1, at node 2 (n - 1)) of ghost node k: lower and
  // upper row, then the pairs left and right of the rows between
  __device__ static __forceinline__ void ghost(int k, int& nx, int& ny) {
    if (k < 2 * NC) {
      nx = k < NC ? k : k - NC;
      ny = k < NC ? 0 : NC - 1;
    } else {
      nx = (k & 1) ? NC - 1 : 0;
      ny = (k - 2 * NC) / 2 + 1;
    }
  }
  __device__ static __forceinline__ int at_ghost(int nx, int ny) {
    return nx == 0 ? GL + ny : nx == NC - 1 ? GR + ny : R0 + 2 * B * (ny - 1) + 2 * (nx - 1);
  }
};

template <int B, typename TS, typename TT, typename TD>
struct Det2Smem {
  using D2 = Det2<B>;
  static constexpr size_t up(size_t x) { return (x + 15) / 16 * 16; }
  static constexpr size_t TABS = up(4 * D2::NG);  // per CTA
  static constexpr size_t RING = up(kRingBytesD<2>);
  static constexpr size_t W = up(sizeof(TT) * D2::SZ);
  // x pass of the FP64 evaluation of FP32 values
  static constexpr size_t XD = sizeof(TD) > sizeof(TT) ? up(sizeof(TD) * D2::NC * D2::NO) : 0;
  static constexpr size_t NB = 96;  // mbarrier, the neighbours' pool offsets
  static constexpr size_t ITEM = NB + RING + W + XD;
  static constexpr size_t BYTES = TABS + D2::ITEMS * ITEM;
};

// Bound by instruction issue (66 % of the slots before the in-place x pass) and by
// shared wavefronts.  Measured, first with one CTA (or warp) per block over the
// gathered and predicted 21^2 tile, then with a table entry per node and a separate
// work array, now: 65536 FP32 blocks of 17^2 104, 75, 61 us; the rounds of an adaptive
// step with 64 trees 168, 92, 77; with 33^2 blocks of 4 variables 443, 238, 196; with 46
// FP64 blocks of 17^2 66, 49, 41.  CTAs per SM: 17^2 8 (10: 68 us, 12: 70, 6: 74 on 65536
// blocks), 33^2 12 (8: 241 us, 10: 206, 14: 204 on four variables).
template <int B, typename TS, typename TD, typename TT>
__global__ void __launch_bounds__(128, B == 17 ? 8 : 12) k_details2(PoolView pv, TS* __restrict__ y) {
  pdl_enter();
  using D2 = Det2<B>;
  using SM = Det2Smem<B, TS, TT, TD>;
  using PL = Plan<2>;
  using G = std::conditional_t<D2::GS == 32, WarpGroup, CtaGroup>;
  constexpr int NC = D2::NC, NO = D2::NO, NI = D2::NI, GS = D2::GS;
  constexpr bool BULK = std::is_same<TS, TT>::value;  // own nodes by a bulk copy
  const G g{};
  const int rank = threadIdx.x % GS, item = threadIdx.x / GS;
  unsigned char* sm = smem_as<unsigned char>(0);
  int32_t* gtab = reinterpret_cast<int32_t*>(sm);
  unsigned char* mem = sm + SM::TABS + item * SM::ITEM;
  uint64_t* bar = reinterpret_cast<uint64_t*>(mem);
  int64_t* nbo = reinterpret_cast<int64_t*>(mem + 16);
  RingD<2>& R = *reinterpret_cast<RingD<2>*>(mem + SM::NB);
  TT* E = reinterpret_cast<TT*>(mem + SM::NB + SM::RING);
  TT* S = E + D2::R0;  // node (0, 0)
  TD* XD = reinterpret_cast<TD*>(mem + SM::NB + SM::RING + SM::W);
  __shared__ double red[4];
  const int nact = pv.cnt->n_round, nv = pv.nvar;
  if ((int64_t)blockIdx.x * D2::ITEMS >= (int64_t)nact * nv) return;  // no item for this CTA (small grids)
  if (BULK && rank == 0) mbar_init(bar, 1);
  unsigned phase = 0;
  // ghost nodes: place | neighbour << 12 | offset in that neighbour (of a uniform
  // neighbourhood) << 16
  for (int k = threadIdx.x; k < D2::NG; k += blockDim.x) {
    int n[2];
    D2::ghost(k, n[0], n[1]);
    int nb = 0, off = 0, mul = 1, lm = 1;
    for (int a = 0; a < 2; ++a) {
      const int x = 2 * (n[a] - 1);
      const int s = x < 0 ? 0 : (x <= B - 2 ? 1 : 2);
      nb += s * mul;
      off += (x - (s - 1) * (B - 1)) * lm;
      mul *= 3;
      lm *= B;
    }
    gtab[k] = D2::at_ghost(n[0], n[1]) | (nb << 12) | (off << 16);
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
    // own nodes; block-edge nodes held by another block take (and store) its value
    if constexpr (BULK) {
      if (rank == 0) {
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        mbar_expect_tx(bar, sizeof(TT) * D2::VS);
        bulk_g2s(S, me, sizeof(TT) * D2::VS, bar);
      }
    } else {
#pragma unroll 5
      // conversion instructions: the FP64 pipe has time for them, the issue slots have
      // none for integer roundings (16384 blocks of 4 variables 89 us instead of 113)
      for (int n = rank; n < NI; n += GS) S[n] = (TT)(me[n]);
    }
    auto landed = [&]() -> bool {
      if constexpr (BULK) {
        phase ^= 1;
        return bulk_landed(pv, bar, phase ^ 1);
      } else {
        g.sync();
        return true;
      }
    };
    auto commit = [&](int n, TS v) {
      TS mine;
      if constexpr (BULK) mine = S[n];
      else mine = me[n];
      if (differs(mine, v)) me[n] = v;
      S[n] = (TT)(v);
    };
    if (uni) {
      if (rank < PL::NB) nbo[rank] = (int64_t)q * bs + vo;
      g.sync();
      constexpr int RE = (D2::NU + GS - 1) / GS, RG = (D2::NG + GS - 1) / GS;
      TS ve[RE], vg[RG];
#pragma unroll
      for (int u = 0; u < RE; ++u) {  // column B - 1, then row B - 1
        const int e = rank + u * GS;
        if (e >= D2::NU) continue;
        const int ux = e < B, uy = e >= B - 1;
        ve[u] = y[nbo[4 + ux + 3 * uy] + (e < B ? 0 : e - B) + (uy ? 0 : B * e)];
      }
#pragma unroll
      for (int u = 0; u < RG; ++u) {
        const int k = rank + u * GS;
        if (k >= D2::NG) continue;
        const int e = gtab[k];
        vg[u] = y[nbo[(e >> 12) & 15] + (e >> 16)];
      }
      if (!landed()) return;
#pragma unroll
      for (int u = 0; u < RE; ++u) {
        const int e = rank + u * GS;
        if (e < D2::NU) commit(e < B ? B * e + B - 1 : B * (B - 1) + e - B, ve[u]);
      }
#pragma unroll
      for (int u = 0; u < RG; ++u) {
        const int k = rank + u * GS;
        if (k < D2::NG) E[gtab[k] & 0xfff] = (TT)(vg[u]);
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
      constexpr int RE = (D2::NE + GS - 1) / GS, RG = (D2::NG + GS - 1) / GS;
      TS ve[RE], vg[RG];
      unsigned other = 0;  // edge nodes of other blocks
#pragma unroll
      for (int u = 0; u < RE; ++u) {
        const int k = rank + u * GS;
        if (k >= D2::NE) continue;
        int i, j;
        D2::edge(k, i, j);
        const int4 e = R.reg[reg_class<B>(i) + 7 * reg_class<B>(j)];
        ve[u] = TS(0);
        if (e.x < 0) lost = true;
        else if (e.x != b.slot) ve[u] = y[owned(e, i, j)];
        if (e.x != b.slot) other |= 1u << u;
      }
#pragma unroll
      for (int u = 0; u < RG; ++u) {
        const int k = rank + u * GS;
        if (k >= D2::NG) continue;
        int nx, ny;
        D2::ghost(k, nx, ny);
        const int i = 2 * (nx - 1), j = 2 * (ny - 1);
        const int4 e = R.reg[reg_class<B>(i) + 7 * reg_class<B>(j)];
        const bool ok = e.x >= 0 && e.y >= b.lvl - 1;
        lost |= !ok;
        vg[u] = ok ? y[owned(e, i, j)] : TS(0);
      }
      if (!landed()) return;
#pragma unroll
      for (int u = 0; u < RE; ++u) {
        if (!((other >> u) & 1)) continue;
        int i, j;
        D2::edge(rank + u * GS, i, j);
        if (lost) S[j * B + i] = TT(0);  // an error: the pool stays as it is
        else commit(j * B + i, ve[u]);
      }
#pragma unroll
      for (int u = 0; u < RG; ++u) {
        const int k = rank + u * GS;
        if (k < D2::NG) E[gtab[k] & 0xfff] = (TT)(vg[u]);
      }
      if (lost) set_err(pv, kErrGraded);
    }
    g.sync();
    // x pass with the details of the even rows, then the y pass with those of the odd
    // ones; every own node is read once: largest |value|, non-finite test
    AbsMax<TT> mqa, md;
    bool bad = false;
    auto seen = [&](TT t) {
      mqa.add(t);
      bad |= !finite(t);
    };
    float mt = 0.f;  // largest |value| of the coarse lattice
    for (int k = rank; k < NC * NO; k += GS) {
      const int r = k / NO, m = k % NO;
      TT* w = S + 2 * B * (r - 1) + 2 * m;
      const TT a = m == 0 ? E[D2::GL + r] : w[-2], c = w[0], d = w[2], f = m == NO - 1 ? E[D2::GR + r] : w[4];
      mt = fmaxf(fmaxf(mt, fmaxf(fabsf((float)a), fabsf((float)c))), fmaxf(fabsf((float)d), fabsf((float)f)));
      const TT pr = dd4(a, c, d, f);
      if (r >= 1 && r <= NC - 2) {
        seen(c);
        if (m == NO - 1) seen(d);
        const TT v = w[1];
        seen(v);
        md.add(v - pr);
      }
      w[1] = pr;
    }
    g.sync();
    for (int k = rank; k < NO * B; k += GS) {
      const int m = k / B;
      const TT* w = S + k + B * (m + 1);  // row 2 m + 1
      const TT v = w[0];
      seen(v);
      md.add(v - dd4(w[-3 * B], w[-B], w[B], w[3 * B]));
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
        // again in FP64; the odd nodes of the even rows are read back from the pool
        AbsMax<TD> md64;
        for (int k = rank; k < NC * NO; k += GS) {
          const int r = k / NO, m2 = k % NO;
          const TT* w = S + 2 * B * (r - 1) + 2 * m2;
          const TD pr = dd4((TD)(m2 == 0 ? E[D2::GL + r] : w[-2]), (TD)w[0], (TD)w[2],
                            (TD)(m2 == NO - 1 ? E[D2::GR + r] : w[4]));
          XD[r * NO + m2] = pr;
          if (r >= 1 && r <= NC - 2) md64.add((TD)me[2 * B * (r - 1) + 2 * m2 + 1] - pr);
        }
        g.sync();
        for (int k = rank; k < NO * B; k += GS) {
          const int m2 = k / B, x = k - m2 * B;
          const TT* w = S + k + B * (m2 + 1);
          const TD* xd = XD + m2 * NO + x / 2;
          const TD pr = (x & 1) ? dd4(xd[0], xd[NO], xd[2 * NO], xd[3 * NO])
                                : dd4((TD)w[-3 * B], (TD)w[-B], (TD)w[B], (TD)w[3 * B]);
          md64.add((TD)w[0] - pr);
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
