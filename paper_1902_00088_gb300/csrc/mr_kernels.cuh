// Kernel templates of the multiresolution step.  Instantiated per dimension in
// mr_k2*.cu / mr_k3*.cu.  Every persistent kernel loops over the active list with
// a grid-stride loop bounded by the device-side block count, so no launch
// needs a host round trip.
#pragma once
#include "mr_device.cuh"

namespace mr {

// Per-tree stage constants in the arithmetic type T.  The FP32 copies hold the
// FP64 values rounded once (on creation, or when the step's time is set), so
// an FP32 kernel reads them without an FP64 conversion per block.
template <typename T> struct StageCoef {
  T ca, cy, ct;
  __device__ __forceinline__ StageCoef(const PoolView& pv, const StageArgs& sa, int t, int s) {
    if constexpr (sizeof(T) == 4) {
      if (pv.tt) { ca = pv.tt[t].caf[s]; cy = pv.tt[t].cyf[s]; ct = pv.tt[t].ctf[s]; }
      else { ca = sa.caf[t]; cy = sa.cyf[t]; ct = sa.ctf[t]; }
    } else {
      if (pv.tt) { ca = pv.tt[t].ca[s]; cy = pv.tt[t].cy[s]; ct = pv.tt[t].ct[s]; }
      else { ca = sa.ca[t]; cy = sa.cy[t]; ct = sa.ct[t]; }
    }
  }
};
template <typename T> __device__ __forceinline__ T tree_cD(const TreeDev& td, int l) {
  if constexpr (sizeof(T) == 4) return td.cDf[l]; else return td.cD[l];
}
template <typename T> __device__ __forceinline__ T tree_rhs(const TreeDev& td, int a) {
  if constexpr (sizeof(T) == 4) return td.rhsf[a]; else return td.rhs[a];
}
template <typename T> __device__ __forceinline__ const T* lattice(const PoolView& pv) {
  if constexpr (sizeof(T) == 4) return pv.latf; else return pv.lat;
}


// (f[-2] - f[2]) + 8 (f[1] - f[-1]): the product with 8 is exact, so the fused
// form rounds the same value once (one instruction less per derivative).
__device__ __forceinline__ float d1_sum(float fm2, float fm1, float f1, float f2) {
  return __fmaf_rn(8.f, f1 - fm1, fm2 - f2);
}
__device__ __forceinline__ double d1_sum(double fm2, double fm1, double f1, double f2) {
  return __fma_rn(8.0, f1 - fm1, fm2 - f2);
}

// ------------------------------------------------------------- stage plans ----
// Stage plans of all active blocks, one warp per block (layout in Plan<D>):
// the 3^d - 1 equal-level neighbours, one lookup per lane in the dense leaf
// tables; for a block whose neighbourhood is not uniform, also its ring and
// class-box owner table (RingD), so that the four RK stages of the step and
// the first coarsening round gather without searching.  Both stay valid while
// the tree generation is unchanged.
template <int D, int B>
__global__ void __launch_bounds__(128) k_plan(PoolView pv) {
  pdl_enter();
  using PL = Plan<D>;
  static_assert(PL::NB <= 32 && PL::INTS <= 32, "one lane per neighbour");
  constexpr int NW = 4;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  RingD<D>& R = *smem_as<RingD<D>>((size_t)warp * kRingBytesD<D>);
  // The plans of this tree stand (a step on a grid that did not change): nothing to do.
  // plan_topo changes only after the last CTA has read it.  65536 blocks: 22 -> 4 us.
  if (pv.cnt->plan_topo == pv.cnt->topo) return;
  const int nact = pv.cnt->n_act;
  for (int p = blockIdx.x * NW + warp; p < nact; p += gridDim.x * NW) {
    const int s = pv.act[p];
    BlockInfo b;
    b.slot = s;
    b.lvl = pv.lvl[s];
    b.tree = pv.tree[s];
    for (int a = 0; a < 3; ++a) b.c[a] = a < D ? pv.crd[3 * s + a] : 0;
    const TreeDev& td = pv.trees[b.tree];
    int q = s;
    if (lane < PL::NB) {
      const int o[3] = {lane % 3 - 1, (lane / 3) % 3 - 1, D == 3 ? lane / 9 - 1 : 0};
      if (o[0] != 0 || o[1] != 0 || o[2] != 0) {
        const int64_t cn[3] = {b.c[0] + o[0], b.c[1] + o[1], b.c[2] + o[2]};
        q = tab_get<D>(pv, td, b.lvl, cn);
      }
    }
    const bool uni = __all_sync(0xffffffffu, q >= 0);
    int32_t* out = pv.plan + (int64_t)p * PL::INTS;
    if (lane == 0) out[0] = s;
    if (lane == 1) out[1] = b.lvl | (b.tree << 8) | (uni ? 1 << 30 : 0);
    if (lane >= 2 && lane < 2 + D) out[lane] = (int32_t)b.c[lane - 2];
    const int qs = __shfl_sync(0xffffffffu, q, (lane - PL::NBO) & 31);
    if (lane >= PL::NBO && lane < PL::NBO + PL::NB) out[lane] = qs;
    if (!uni) {
      build_ring<D, B, WarpGroup>(pv, td, b, R);
      __syncwarp();
      build_regions<D, B, WarpGroup>(b, R);
      __syncwarp();
      store_regions<D, WarpGroup>(pv, p, R);
      __syncwarp();
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    if (atomicAdd(&pv.cnt->ctas_done, 1u) == gridDim.x - 1) {
      pv.cnt->ctas_done = 0;
      pv.cnt->plan_topo = pv.cnt->topo;
    }
  }
}

// Start of a coarsening round: the blocks it works on (none once a round
// merged nothing), its id, and the per-tree threshold scales reset to v.
template <int D>
__global__ void k_round_begin(PoolView pv, double v) {
  pdl_enter();
  Counters* c = pv.cnt;
  if (threadIdx.x == 0) {
    c->n_round = c->done ? 0 : c->n_act;
    c->round_id += 1;
  }
  for (int i = threadIdx.x; i < pv.ntrees * pv.nvar; i += blockDim.x) pv.svar[i] = v;
}

// ------------------------------------------------------- new-list offsets ----
// New-list counts of 8 consecutive positions (one per warp of the CTA, in warp
// order): each position's exclusive prefix within them, and their total.  The
// totals are scanned later, so a scan works on an eighth of the list (7500 blocks
// of 64 trees: 18 -> 4 us in the last CTA of k_flags).
__device__ __forceinline__ void emit_group(const PoolView& pv, int g, int n, int2 (*sh)[8], int par, int2 e) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (lane == 0) sh[par][w] = e;
  __syncthreads();
  if (w == 0 && lane < 8) {
    const int2 own = sh[par][lane];
    int2 v = own;
    for (int o = 1; o < 8; o <<= 1) {
      const int x = __shfl_up_sync(0xffu, v.x, o), z = __shfl_up_sync(0xffu, v.y, o);
      if (lane >= o) { v.x += x; v.y += z; }
    }
    if (8 * g + lane < n) reinterpret_cast<int2*>(pv.eoff)[8 * g + lane] = make_int2(v.x - own.x, v.y - own.y);
    if (lane == 7) reinterpret_cast<int2*>(pv.grp)[g] = v;
  }
}
// Scan of the group totals by the calling (last) CTA of 256 threads.
__device__ __forceinline__ void scan_groups(const PoolView& pv, int n) {
  const int ng = (n + 7) >> 3;
  if (ng <= 1024) cta_scan2<256, 4>(pv.grp, pv.gof, ng, &pv.cnt->n_new);
  else cta_scan2<256, 16>(pv.grp, pv.gof, ng, &pv.cnt->n_new);
}
// Position of the first entry of list position p in the new list, and of its first
// slot among those requested (refinement) or freed (merge).
__device__ __forceinline__ int2 new_offset(const PoolView& pv, int p) {
  const int2 g = reinterpret_cast<const int2*>(pv.gof)[p >> 3], l = reinterpret_cast<const int2*>(pv.eoff)[p];
  return make_int2(g.x + l.x, g.y + l.y);
}

// ----------------------------------------------------------------- refine ----
// x pass of the upsampling: fine x in [0, 2(B-1)] on mother rows y in [-1, B]
template <int B>
struct RefGeo {
  static constexpr int NF = 2 * B - 1;
  static constexpr int NR = B + 2;
  static constexpr int NX = NF * NR;
};

// Sec. 2.3: the synchronised mother tile is upsampled by the 4th-order
// interpolating prediction and split into 2^d children (one treecode digit
// appended); children are placed in the new active list in Hilbert order.
// 2D blocks; 3D ones are refined by k_refine3 (mr_adv3.cuh).  One CTA per mother
// and variable: with the four variables of a mother in one CTA, 376 mothers of 33^2
// nodes were 1.2 waves of 304 CTAs (335 us); 216 us with 1504 items of a quarter of
// the shared memory, 138 us with odd and even nodes apart (see below).
//
// Launch shape of its own (not the stage's): a mother and variable keeps its CTA
// waiting on the ring, the owners and the nodes in turn, so CTAs in flight count.
// Refinement of a step, 17^2 blocks, 8 CTAs of 128 threads (64 registers) per SM against
// 4 of 160: 64 trees 43 and 53 us, double shear layer 61 and 70, 736 blocks of 4
// variables 41 and 48 (FP32), 49 and 56 (FP64); 5 of 192: 47, 63, 42, 47; 45 FP64
// blocks, where a launch is one wave, 28 with any of them.  33^2 blocks: mixing layer
// (FP64 state) 4 of 256 131, 3 of 288 135; 352 FP32 blocks 43 and 42.
template <int B, typename TS>
struct RefineCfg {
  using Bx = Box<2, B, 1>;
  static constexpr int NT = B == 17 ? 128 : 256, MINB = B == 17 ? 8 : 4;
  static constexpr int SCR = Bx::SCR > RefGeo<B>::NX ? Bx::SCR : RefGeo<B>::NX;
  static constexpr size_t BYTES = kRingBytesD<2> + sizeof(TS) * (Bx::TILE + Bx::CBOX + SCR);
};
template <int B, typename TS>
__global__ void __launch_bounds__(RefineCfg<B, TS>::NT, RefineCfg<B, TS>::MINB) k_refine(PoolView pv, TS* __restrict__ y) {
  pdl_enter();
  constexpr int D = 2;
  using Gm = Geo<D, B>;
  using Bx = Box<D, B, 1>;  // prediction of the children reaches one node
  using RG = RefGeo<B>;
  RingD<D>& R = *smem_as<RingD<D>>(0);
  __shared__ int cslot[8];
  TS* tile = smem_as<TS>(kRingBytesD<D>);
  TS* cbox = tile + Bx::TILE;
  TS* scr = cbox + Bx::CBOX;  // gather scratch, then the x pass of the upsampling
  TS* X = scr;
  const int nact = pv.cnt->n_act;
  const int n_alloc = pv.cnt->n_alloc, n_free = pv.cnt->n_free;
  if (n_alloc > n_free) {
    if (blockIdx.x == 0 && threadIdx.x == 0) set_err(pv, kErrCapacity);
    return;
  }
  if (n_alloc == 0) return;  // no block refines: the list stays as it is
  const int nv = pv.nvar;
  for (int64_t it = blockIdx.x; it < (int64_t)nact * nv; it += gridDim.x) {
    const int p = (int)(it / nv), v = (int)(it % nv);
    const int slot = pv.act[p];
    const int2 off = new_offset(pv, p);
    const int e = off.x, a = off.y;
    if (pv.flag[slot] != 1) {
      if (v == 0 && threadIdx.x == 0) pv.act_next[e] = slot;
      continue;
    }
    // variable v as the only variable of blocks nvar * vs apart
    PoolView pv1 = pv;
    pv1.nvar = 1;
    pv1.vs = pv.vs * nv;
    const TS* yv = y + v * pv.vs;
    const BlockInfo b = load_block(pv, slot);
    const TreeDev& td = pv.trees[b.tree];
    build_ring<D, B>(pv, td, b, R);
    __syncthreads();
    fill_tile<D, B, TS, TS, 1>(pv1, b, yv, (TS*)yv, tile, false, R, cbox, scr);
    if (threadIdx.x < Gm::NCH) {
      const int ch = threadIdx.x;
      const int cs = pv.freelist[n_free - n_alloc + a + ch];
      cslot[ch] = cs;
      if (v == 0) {
        // light data of the children, in the order of their Hilbert keys
        const int32_t cc[3] = {(int32_t)(2 * b.c[0] + (ch & 1)), (int32_t)(2 * b.c[1] + (ch >> 1)), 0};
        const uint64_t key = block_key<D>(cc, b.lvl + 1, td.Jmax);
        int rank = 0;
        for (int o = 0; o < Gm::NCH; ++o) rank += __shfl_sync((1u << Gm::NCH) - 1u, key, o) < key;
        pv.act_next[e + rank] = cs;
        pv.lvl[cs] = (int8_t)(b.lvl + 1);
        pv.tree[cs] = (int16_t)b.tree;
        for (int ax = 0; ax < 3; ++ax) pv.crd[3 * cs + ax] = cc[ax];
        pv.hkey[cs] = key;
        pv.flag[cs] = 0;
      }
    }
    __syncthreads();
    // Separable upsampling: X = prediction along x on the mother's rows (y in
    // [-1, B]), then y per child node -- the operations of the tensor product in
    // the same order; odd nodes (4-point rule) before even ones (copies), so that
    // their warps hold one kind (the rule on the FP64 pipe bounds the FP64 form).
    constexpr int H = B - 1, NR = RG::NR, NF = RG::NF;
    for (int idx = threadIdx.x; idx < NR * H; idx += blockDim.x) {
      const int row = idx / H, m = idx % H;
      const TS* t = tile + Bx::tix(m - 1, row - 1, 0);
      X[row * NF + 2 * m + 1] = dd4(t[0], t[1], t[2], t[3]);
    }
    for (int idx = threadIdx.x; idx < NR * B; idx += blockDim.x) {
      const int row = idx / B, m = idx % B;
      X[row * NF + 2 * m] = tile[Bx::tix(m, row - 1, 0)];
    }
    __syncthreads();
    // child ch, odd rows j = 2m + 1, then even ones j = 2m (fine row (ch >> 1)(B - 1) + j)
    constexpr int NO = H / 2, NE = NO + 1;
    for (int idx = threadIdx.x; idx < 4 * NO * B; idx += blockDim.x) {
      const int i = idx % B, m = (idx / B) % NO, ch = idx / (B * NO);
      const TS* t = X + ((ch >> 1) * NO + m) * NF + (ch & 1) * H + i;  // mother rows fl - 1 .. fl + 2, from -1
      y[((int64_t)cslot[ch] * nv + v) * pv.vs + (2 * m + 1) * B + i] = dd4(t[0], t[NF], t[2 * NF], t[3 * NF]);
    }
    for (int idx = threadIdx.x; idx < 4 * NE * B; idx += blockDim.x) {
      const int i = idx % B, m = (idx / B) % NE, ch = idx / (B * NE);
      y[((int64_t)cslot[ch] * nv + v) * pv.vs + 2 * m * B + i] = X[((ch >> 1) * NO + m + 1) * NF + (ch & 1) * H + i];
    }
    __syncthreads();
  }
}

// ---------------------------------------------------------------- details ----
// Common parts of the details kernels (k_details2 in mr_det2.cuh, k_details3 in
// mr_adv3.cuh).
// The FP32 maximum m32 is within E of the FP64 one, and m32 + E < eps or
// m32 - E >= eps holds in exact arithmetic: the sum is rounded up and compared
// with eps rounded down, the difference rounded down and compared with eps
// rounded up, so the threshold decision needs no FP64 evaluation.
__device__ __forceinline__ bool certain_vs_eps(float m32, float E, const TreeDev& td) {
  return __fadd_ru(m32, E) < td.epsf[0] || __fsub_rd(m32, E) >= td.epsf[1];
}

// Largest |value| added, NaN ignored (as fmax does).  FP64 values are compared
// on their bit patterns, which order as the magnitudes do: a comparison of
// doubles would take the FP64 pipe, the bound of the FP64 details.
template <typename T>
struct AbsMax {
  T m = T(0);
  __device__ __forceinline__ void add(T v) { m = fmax(m, (T)fabs(v)); }
  __device__ __forceinline__ T get() const { return m; }
};
template <>
struct AbsMax<double> {
  long long m = 0;
  __device__ __forceinline__ void add(double v) {
    const long long b = __double_as_longlong(v) & 0x7fffffffffffffffLL;
    if (b > m && b <= 0x7ff0000000000000LL) m = b;
  }
  __device__ __forceinline__ double get() const { return __longlong_as_double(m); }
};

// Maximum over the warp of non-negative values (not NaN), on their bit patterns.
__device__ __forceinline__ float warp_max_pos(float v) {
  return __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(v)));
}
__device__ __forceinline__ double warp_max_pos(double v) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(v);
  const unsigned hi = (unsigned)(b >> 32), top = __reduce_max_sync(0xffffffffu, hi);
  const unsigned lo = __reduce_max_sync(0xffffffffu, hi == top ? (unsigned)b : 0u);
  return __longlong_as_double((long long)(((unsigned long long)top << 32) | lo));
}

// Maximum over the CTA of non-negative values (not NaN), one per warp in red; every
// thread gets the result.  On bit patterns: FP64 maxima take the FP64 pipe, which
// yields two results per clock and SM (3D details, 2584 FP64 blocks: 593 -> 514 us).
template <typename T>
__device__ __forceinline__ T block_max(T v, T* red) {
  v = warp_max_pos(v);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  const int w = threadIdx.x & 31;
  return warp_max_pos(w < (int)(blockDim.x >> 5) ? red[w] : T(0));
}

// The same of a, b and c in one reduction (one value per warp in ra / rb / rc, which
// the CTA has read before its last barrier).
template <typename A, typename Bt, typename Ct>
__device__ __forceinline__ void block_max3(A& a, Bt& b, Ct& c, A* ra, Bt* rb, Ct* rc) {
  a = warp_max_pos(a);
  b = warp_max_pos(b);
  c = warp_max_pos(c);
  if ((threadIdx.x & 31) == 0) {
    ra[threadIdx.x >> 5] = a;
    rb[threadIdx.x >> 5] = b;
    rc[threadIdx.x >> 5] = c;
  }
  __syncthreads();
  const int w = threadIdx.x & 31;
  const bool in = w < (int)(blockDim.x >> 5);
  a = warp_max_pos(in ? ra[w] : A(0));
  b = warp_max_pos(in ? rb[w] : Bt(0));
  c = warp_max_pos(in ? rc[w] : Ct(0));
}

// ---------------------------------------------------------------- coarsen ----
// Sec. 2.3: 2^d sisters with status -2 merge into their mother by restriction
// (every second node); a mother node on a line shared by two children is read
// from the child in which it has local index 0.  The mother takes the slot of
// the family member that comes first in Hilbert order.
// One kernel per round: families are merged (the mother's data, then the
// family's table entries, light data and freed slots -- the family's 2^d
// members sit at consecutive list positions, a Hilbert-curve property), and
// the CTA that finishes last copies the new active list in place, updates the
// counters and prepares the next round (RoundCtl).

// Counters a round works with, read at its start (they change at its end).
struct RoundState {
  int nround, n_free, n_new, n_alloc, rid, rounds, topo;
  bool done, none;
  __device__ __forceinline__ explicit RoundState(const Counters* c) {
    nround = c->n_round;
    n_free = c->n_free;
    n_new = c->n_new;
    n_alloc = c->n_alloc;
    rid = c->round_id;
    rounds = c->rounds;
    topo = c->topo;
    done = c->done != 0;
    none = n_new == nround;  // no family merges: the tree and the list are unchanged
  }
};

// Table entry, light data and slot of member s (list position q, block m) of a
// merged family whose mother takes `slot`.
template <int D>
__device__ __forceinline__ void merge_member(const PoolView& pv, const TreeDev& td, const RoundState& rs, int q, int s,
                                             const BlockInfo& m, int slot) {
  pv.tab[td.tab_off[m.lvl] + (int64_t)morton<D>(m.c, m.lvl)] = -1;
  if (s == slot) {
    const int64_t pc[3] = {m.c[0] >> 1, m.c[1] >> 1, m.c[2] >> 1};
    pv.tab[td.tab_off[m.lvl - 1] + (int64_t)morton<D>(pc, m.lvl - 1)] = s;
    pv.stamp[s] = rs.rid;
    pv.lvl[s] = (int8_t)(m.lvl - 1);
    const int32_t c32[3] = {(int32_t)pc[0], (int32_t)pc[1], (int32_t)pc[2]};
    for (int a = 0; a < 3; ++a) pv.crd[3 * s + a] = c32[a];
    pv.hkey[s] = block_key<D>(c32, m.lvl - 1, td.Jmax);
  } else {
    pv.lvl[s] = -1;
    pv.freelist[rs.n_free + new_offset(pv, q).y] = s;
  }
}

// List position of work item it, nq = ceil(n / 2^d): the first members of the families
// sit 2^d positions apart, so consecutive items take positions 2^d apart (in list
// order with a grid of a multiple of 2^d CTAs, only every 2^d-th CTA had families).
template <int D>
__device__ __forceinline__ int merge_position(int it, int nq) {
  return (it % nq) * (1 << D) + it / nq;
}

// End of a round, by the CTA of the grid that finishes last: the new list in place
// (every entry of act_next is written by now), the counters, and the next round, if
// one runs (a family merged and fewer than max_rounds ran): the blocks it evaluates,
// its id, its threshold scales (the last round's stay for the next step's proposal
// features); in a captured step the while node's condition.
template <int D>
__device__ __forceinline__ void finish_round(const PoolView& pv, const RoundState& rs, const RoundCtl& rc) {
  const int ncopy = rs.done || rs.none ? 0 : rs.n_new;
  const int n4 = ncopy >> 2;
  const int4* from = reinterpret_cast<const int4*>(pv.act_next);
  int4* to = reinterpret_cast<int4*>(pv.act);
  for (int p = threadIdx.x; p < n4; p += 4 * blockDim.x) {
    int4 t[4];
#pragma unroll
    for (int r = 0; r < 4; ++r)
      if (p + r * (int)blockDim.x < n4) t[r] = __ldcg(from + p + r * blockDim.x);
#pragma unroll
    for (int r = 0; r < 4; ++r)
      if (p + r * (int)blockDim.x < n4) to[p + r * blockDim.x] = t[r];
  }
  if ((int)threadIdx.x < (ncopy & 3)) pv.act[4 * n4 + threadIdx.x] = __ldcg(pv.act_next + 4 * n4 + threadIdx.x);
  // a round that is not skipped works on the whole list
  const int merged = rs.done ? 0 : (rs.nround - rs.n_new) / ((1 << D) - 1);
  const bool done = rs.done || merged == 0;
  const bool next = !done && rs.rounds + 1 < rc.max_rounds;
  if (next)
    for (int i = threadIdx.x; i < pv.ntrees * pv.nvar; i += blockDim.x) pv.svar[i] = rc.svar_v;
  if (threadIdx.x == 0) {
    Counters* c = pv.cnt;
    c->first_round = 0;
    if (!rs.done) {
      c->merged = merged;
      c->n_free = rs.n_free + rs.n_alloc;
      c->n_act = rs.n_new;
      if (done) c->done = 1;
      else c->topo = rs.topo + 1;
    }
    c->rounds = rs.rounds + 1;
    c->n_round = done ? 0 : rs.n_new;
    if (next) c->round_id = rs.rid + 1;
    if (rc.has_h) {
      c->graph_rounds += 1;
      cudaGraphSetConditional(rc.h, next ? 1u : 0u);
    }
    c->ctas_done = 0;
  }
}

// 2D: one warp per family of 17^2 blocks with one variable, else one CTA (9 or 10
// values per thread, read before the first is written: the mother takes a child's
// slot).  Blocks that do not merge only enter the new list.  Latency-bound: a chain of
// list entry, block data, children's nodes and tables.  With a CTA of 256 threads per
// block, through shared memory, in list order: 47 -> 12 us for the first round of 64
// trees (7472 blocks), 64 -> 35 us for 2944 blocks of 33^2 x 4 FP64 values.
template <int B, int NV>
struct Coarsen2 {
  static constexpr int N = NV * B * B;
  static constexpr int GS = N <= 320 ? 32 : (N <= 1280 ? 128 : 512);  // threads per family
  static constexpr int NT = GS == 32 ? 128 : GS;
  static constexpr int K = (N + GS - 1) / GS;
};
template <int B, int NV, typename TS>
__global__ void __launch_bounds__(Coarsen2<B, NV>::NT) k_coarsen2(PoolView pv, TS* __restrict__ y, RoundCtl rc) {
  pdl_enter();
  using CO = Coarsen2<B, NV>;
  using G = std::conditional_t<CO::GS == 32, WarpGroup, CtaGroup>;
  constexpr int GS = CO::GS, K = CO::K, NI = B * B, ITEMS = CO::NT / GS;
  const G g{};
  const int rank = threadIdx.x % GS, item = threadIdx.x / GS;
  __shared__ int scs[ITEMS][4];
  int* cs = scs[item];
  const RoundState rs(pv.cnt);
  const int64_t bs = (int64_t)NV * pv.vs;
  const int nq = (rs.nround + 3) / 4;
  for (int it = blockIdx.x * ITEMS + item; !rs.none && it < 4 * nq; it += gridDim.x * ITEMS) {
    const int p = merge_position<2>(it, nq);
    if (p >= rs.nround || !pv.emit[2 * p]) continue;  // a member of a family merged at its first member
    const int slot = pv.act[p];
    if (rank == 0) pv.act_next[new_offset(pv, p).x] = slot;
    if (pv.flag[slot] != -2) continue;
    const BlockInfo b = load_block(pv, slot);
    const TreeDev& td = pv.trees[b.tree];
    // the family: positions p .. p + 3
    BlockInfo m = b;
    if (rank < 4) {
      cs[rank] = -1;
      if (p + rank < rs.nround) m = load_block(pv, pv.act[p + rank]);
      else m.tree = -1;
    }
    g.sync();
    if (rank < 4 && m.tree == b.tree && m.lvl == b.lvl && (m.c[0] >> 1) == (b.c[0] >> 1) &&
        (m.c[1] >> 1) == (b.c[1] >> 1))
      cs[(m.c[0] & 1) + 2 * (m.c[1] & 1)] = m.slot;
    g.sync();
    if (cs[0] < 0 || cs[1] < 0 || cs[2] < 0 || cs[3] < 0) {  // cannot happen for a complete family
      if (rank == 0) set_err(pv, kErrGraded);
      g.sync();
      continue;
    }
    TS val[K];
#pragma unroll
    for (int k = 0; k < K; ++k) {
      const int idx = rank + k * GS;
      if (idx >= CO::N) continue;
      const int v = idx / NI, q = idx % NI, i = q % B, j = q / B;
      const int bx = 2 * i >= B - 1, by = 2 * j >= B - 1;
      val[k] = y[(int64_t)cs[bx + 2 * by] * bs + v * pv.vs + (2 * i - bx * (B - 1)) + B * (2 * j - by * (B - 1))];
    }
    g.sync();
#pragma unroll
    for (int k = 0; k < K; ++k) {
      const int idx = rank + k * GS;
      if (idx >= CO::N) continue;
      const int v = idx / NI, q = idx % NI;
      y[(int64_t)slot * bs + v * pv.vs + q] = val[k];
    }
    if (rank < 4) merge_member<2>(pv, td, rs, p + rank, m.slot, m, slot);
    g.sync();
  }
  if (last_cta_all(pv.cnt)) finish_round<2>(pv, rs, rc);
}

// 3D: one CTA per family, the mother's nodes through shared memory.
template <int B, typename TS>
__global__ void __launch_bounds__(256) k_coarsen3(PoolView pv, TS* __restrict__ y, RoundCtl rc) {
  pdl_enter();
  using Gm = Geo<3, B>;
  TS* buf = smem_as<TS>(0);
  __shared__ int cs[8];
  const RoundState rs(pv.cnt);
  const int nq = (rs.nround + 7) / 8;
  for (int it = blockIdx.x; !rs.none && it < 8 * nq; it += gridDim.x) {
    const int p = merge_position<3>(it, nq);
    if (p >= rs.nround || !pv.emit[2 * p]) continue;  // a member of a family merged by the CTA of its first member
    const int slot = pv.act[p];
    if (threadIdx.x == 0) pv.act_next[new_offset(pv, p).x] = slot;
    if (pv.flag[slot] != -2) continue;
    const BlockInfo b = load_block(pv, slot);
    const TreeDev& td = pv.trees[b.tree];
    if (threadIdx.x < 8) {
      int64_t cc[3];
      for (int a = 0; a < 3; ++a) cc[a] = (b.c[a] & ~(int64_t)1) | ((threadIdx.x >> a) & 1);
      cs[threadIdx.x] = tab_get<3>(pv, td, b.lvl, cc);
    }
    __syncthreads();
    bool missing = false;
    for (int ch = 0; ch < 8; ++ch) missing |= cs[ch] < 0;
    if (missing) {  // cannot happen for a complete family; never read slot -1
      if (threadIdx.x == 0) set_err(pv, kErrGraded);
      __syncthreads();
      continue;
    }
#pragma unroll 4
    for (int q = threadIdx.x; q < Gm::NI; q += 256) {
      const int I[3] = {q % B, (q / B) % B, q / (B * B)};
      int cb = 0, li[3];
      for (int a = 0; a < 3; ++a) {
        const int bit = (2 * I[a] >= B - 1) ? 1 : 0;
        cb |= bit << a;
        li[a] = 2 * I[a] - bit * (B - 1);
      }
      buf[q] = y[(int64_t)cs[cb] * pv.vs + Gm::lin(li[0], li[1], li[2])];
    }
    __syncthreads();
    for (int q = threadIdx.x; q < Gm::NI; q += 256) y[(int64_t)slot * pv.vs + q] = buf[q];
    // the family's tables and light data (positions p .. p + 7)
    if (threadIdx.x < 8) {
      const int s = pv.act[p + threadIdx.x];
      merge_member<3>(pv, td, rs, p + threadIdx.x, s, load_block(pv, s), slot);
    }
    __syncthreads();
  }
  if (last_cta_all(pv.cnt)) finish_round<3>(pv, rs, rc);
}

// --------------------------------------------------------------------- IC ----
// Analytic fields from per-lattice factor tables: Gaussian as the product of
// its 1D factors (x, then y, then z); mixing layer q = (1, u(y), v, E) with
// v = amp (s(x) e(y)), E = p0/(gamma-1) + (u u + v v)/2; double shear layer
// (Sec. 4) from its layer profile s(x) and u(y), in the RHS kind's variables.
template <int D, int B, typename TS>
__global__ void k_ic(PoolView pv, TS* __restrict__ y) {
  pdl_enter();
  using Gm = Geo<D, B>;
  const int nact = pv.cnt->n_act;
  const int nv = pv.nvar;
  for (int p = blockIdx.x; p < nact; p += gridDim.x) {
    const BlockInfo b = load_block(pv, pv.act[p]);
    const TreeDev& td = pv.trees[b.tree];
    const int sh = td.Jmax - b.lvl;
    const double* lat = pv.lat + td.lat_off;
    for (int q = threadIdx.x; q < Gm::NI; q += blockDim.x) {
      const int ijk[3] = {q % B, (q / B) % B, D == 3 ? q / (B * B) : 0};
      int64_t U[3] = {0, 0, 0};
      for (int a = 0; a < D; ++a) U[a] = pmod64((b.c[a] * (B - 1) + ijk[a]) << sh, td.N);
      const int64_t at = (int64_t)b.slot * nv * pv.vs + q;
      if (td.ic_kind == MR_IC_GAUSS) {
        double f = lat[kLatGx * td.N + U[0]] * lat[kLatGy * td.N + U[1]];
        if (D == 3) f = f * lat[kLatGz * td.N + U[2]];
        y[at] = (TS)f;
      } else if (td.ic_kind == MR_IC_MIXING) {
        const double u = lat[kLatNsU * td.N + U[1]];
        const double v = td.ic_amp * (lat[kLatNsS * td.N + U[0]] * lat[kLatNsE * td.N + U[1]]);
        const double E = td.ic_e0 + 0.5 * (u * u + v * v);
        y[at] = (TS)1.0;
        y[at + pv.vs] = (TS)u;
        y[at + 2 * pv.vs] = (TS)v;
        y[at + 3 * pv.vs] = (TS)E;
      } else if (td.ic_kind == MR_IC_SHEAR_LAYER) {
        const double s = lat[kLatSlS * td.N + U[0]];
        const double rho = td.ic_sl[1] + (td.ic_sl[0] - td.ic_sl[1]) * s;
        const double v = td.ic_sl[3] + (td.ic_sl[2] - td.ic_sl[3]) * s;
        const double u = lat[kLatSlU * td.N + U[1]];
        double q[4];
        if (pv.rhs_kind == MR_RHS_NS_SKEW) {
          const double f = sqrt(rho);
          q[0] = f; q[1] = f * u; q[2] = f * v; q[3] = td.ic_sl[4];
        } else {
          const double m1 = rho * u, m2 = rho * v;
          q[0] = rho; q[1] = m1; q[2] = m2; q[3] = td.ic_sl[4] / td.nsd[0] + 0.5 * (m1 * u + m2 * v);
        }
        for (int w = 0; w < 4; ++w) y[at + w * pv.vs] = (TS)q[w];
      }
    }
  }
}

// ------------------------------------------------------------- sync export ---
// Ghost synchronisation of the current field: commits the block-edge nodes
// taken from finer blocks; optionally writes the full tile (double) to `tiles`
// at the block's list position.
template <int D, int B, typename TS>
__global__ void __launch_bounds__(256) k_sync(PoolView pv, TS* __restrict__ y, double* __restrict__ tiles) {
  pdl_enter();
  using Gm = Geo<D, B>;
  RingD<D>& R = *smem_as<RingD<D>>(0);
  double* tile = smem_as<double>(kRingBytesD<D>);
  double* cbox = tile + pv.nvar * Gm::TILE;
  const int nact = pv.cnt->n_act;
  const int nv = pv.nvar;
  for (int p = blockIdx.x; p < nact; p += gridDim.x) {
    const BlockInfo b = load_block(pv, pv.act[p]);
    const TreeDev& td = pv.trees[b.tree];
    build_ring<D, B>(pv, td, b, R);
    __syncthreads();
    fill_tile<D, B, TS, double>(pv, b, y, y, tile, true, R, cbox);
    __syncthreads();
    if (tiles)
      for (int idx = threadIdx.x; idx < nv * Gm::TILE; idx += blockDim.x)
        tiles[(int64_t)p * nv * Gm::TILE + idx] = tile[idx];
    __syncthreads();
  }
}

// ---------------------------------------------------------------- export -----
template <int D, int B, typename TS>
__global__ void k_export_fields(PoolView pv, const TS* __restrict__ y, double* __restrict__ out) {
  pdl_enter();
  using Gm = Geo<D, B>;
  const int nact = pv.cnt->n_act;
  const int nv = pv.nvar;
  for (int p = blockIdx.x; p < nact; p += gridDim.x) {
    const int slot = pv.act[p];
    for (int idx = threadIdx.x; idx < nv * Gm::NI; idx += blockDim.x) {
      const int v = idx / Gm::NI, q = idx % Gm::NI;
      out[(int64_t)p * nv * Gm::NI + idx] = (double)y[((int64_t)slot * nv + v) * pv.vs + q];
    }
  }
}

template <int D, int B, typename TS>
__global__ void k_import_fields(PoolView pv, TS* __restrict__ y, const double* __restrict__ in,
                                int64_t n) {
  pdl_enter();
  using Gm = Geo<D, B>;
  const int nv = pv.nvar;
  for (int64_t i = blockIdx.x; i < n; i += gridDim.x)
    for (int idx = threadIdx.x; idx < nv * Gm::NI; idx += blockDim.x) {
      const int v = idx / Gm::NI, q = idx % Gm::NI;
      y[(i * nv + v) * pv.vs + q] = (TS)in[i * nv * Gm::NI + idx];
    }
}

// ----------------------------------------------------------------- error -----
// Error against exact factor tables ex[3][N] of one tree over unique nodes
// (each block's last node per axis dropped), weights dx^d.
template <int D, int B, typename TS>
__global__ void k_error(PoolView pv, const TS* __restrict__ y, int tree, const double* ex,
                        double* out) {
  pdl_enter();
  const int nact = pv.cnt->n_act;
  const TreeDev& td = pv.trees[tree];
  constexpr int BZ = D == 3 ? B - 1 : 1;
  const int NU = (B - 1) * (B - 1) * BZ;
  double e2 = 0, x2 = 0, ei = 0, xi = 0;
  for (int p = blockIdx.x; p < nact; p += gridDim.x) {
    const BlockInfo b = load_block(pv, pv.act[p]);
    if (b.tree != tree) continue;
    const int sh = td.Jmax - b.lvl;
    const double dx = td.dx[b.lvl];
    const double w = D == 3 ? dx * dx * dx : dx * dx;
    for (int q = threadIdx.x; q < NU; q += blockDim.x) {
      const int ijk[3] = {q % (B - 1), (q / (B - 1)) % (B - 1), D == 3 ? q / ((B - 1) * (B - 1)) : 0};
      int64_t U[3] = {0, 0, 0};
      for (int a = 0; a < D; ++a) U[a] = pmod64((b.c[a] * (B - 1) + ijk[a]) << sh, td.N);
      double e = ex[U[0]] * ex[td.N + U[1]];
      if (D == 3) e = e * ex[2 * td.N + U[2]];
      const double a = (double)y[(int64_t)b.slot * pv.nvar * pv.vs + Geo<D, B>::lin(ijk[0], ijk[1], ijk[2])];
      e2 += w * (a - e) * (a - e);
      x2 += w * e * e;
      ei = fmax(ei, fabs(a - e));
      xi = fmax(xi, fabs(e));
    }
  }
  atomicAdd(&out[0], e2);
  atomicAdd(&out[1], x2);
  atomic_max_pos(&out[2], ei);
  atomic_max_pos(&out[3], xi);
}

// ------------------------------------------------------- tree maintenance ----
// One thread per block: its flag, and the new-list counts in groups of 8 positions
// (see emit_group).  SCAN: the CTA that finishes last also scans the group totals.
template <int D, bool SCAN>
__global__ void __launch_bounds__(256) k_refine_count(PoolView pv, int mode, const int8_t* mask) {
  pdl_enter();
  const int nact = pv.cnt->n_act;
  const int nch = 1 << D;
  for (int base = blockIdx.x * blockDim.x; base < nact; base += gridDim.x * blockDim.x) {
    const int p = base + threadIdx.x;
    int2 own = make_int2(0, 0);
    if (p < nact) {
      const int s = pv.act[p];
      const int l = pv.lvl[s];
      const TreeDev& td = pv.trees[pv.tree[s]];
      // mode 2: flags already set on the device (learned proposal + closure)
      const bool r = l < td.Jmax && (mode == MR_ADAPT_REFINE_ALL || (mode == 2 ? pv.flag[s] == 1 : (mask && mask[p] > 0)));
      pv.flag[s] = r ? 1 : 0;
      own = make_int2(r ? nch : 1, r ? nch : 0);
    }
    int2 v = own;
    for (int o = 1; o < 8; o <<= 1) {
      const int x = __shfl_up_sync(0xffffffffu, v.x, o, 8), z = __shfl_up_sync(0xffffffffu, v.y, o, 8);
      if ((threadIdx.x & 7) >= o) { v.x += x; v.y += z; }
    }
    if (p < nact) reinterpret_cast<int2*>(pv.eoff)[p] = make_int2(v.x - own.x, v.y - own.y);
    if ((threadIdx.x & 7) == 7 && (p & ~7) < nact) reinterpret_cast<int2*>(pv.grp)[p >> 3] = v;
  }
  if constexpr (SCAN) {
    if (last_cta_all(pv.cnt)) {
      scan_groups(pv, nact);
      if (threadIdx.x == 0) pv.cnt->ctas_done = 0;
    }
  }
}

// True in thread 0 of the CTA of the grid that finishes last; the writes of
// every other CTA of the grid are visible to it.
__device__ __forceinline__ bool last_cta(Counters* c) {
  __shared__ bool last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(&c->ctas_done, 1u) == gridDim.x - 1;
  __syncthreads();
  return last && threadIdx.x == 0;
}

// End of a refinement in one kernel: each refined mother's table entry is
// replaced by its children's and its slot freed, the new active list is copied
// in place (each index is read, then written, by one thread), and the counters
// are updated by the last CTA.
template <int D>
__global__ void k_refine_commit(PoolView pv) {
  pdl_enter();
  Counters* c = pv.cnt;
  const int nact = c->n_act, n_new = c->n_new, n_alloc = c->n_alloc, n_free = c->n_free;
  const bool ok = n_alloc <= n_free;
  const bool any = n_alloc > 0;  // some block refines (else the tree and the list are unchanged)
  const int nch = 1 << D;
  const int nmax = ok && any ? (nact > n_new ? nact : n_new) : 0;
  for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < nmax; p += gridDim.x * blockDim.x) {
    const int32_t nxt = p < n_new ? pv.act_next[p] : 0;
    if (p < nact) {
      const int s = pv.act[p];
      if (pv.flag[s] == 1) {
        const BlockInfo b = load_block(pv, s);
        const TreeDev& td = pv.trees[b.tree];
        pv.tab[td.tab_off[b.lvl] + (int64_t)morton<D>(b.c, b.lvl)] = -1;
        const int2 off = new_offset(pv, p);
        const int e = off.x;
        for (int r = 0; r < nch; ++r) {
          const int cs = pv.act_next[e + r];
          int64_t cc[3] = {pv.crd[3 * cs], pv.crd[3 * cs + 1], pv.crd[3 * cs + 2]};
          pv.tab[td.tab_off[b.lvl + 1] + (int64_t)morton<D>(cc, b.lvl + 1)] = cs;
        }
        pv.freelist[n_free - n_alloc + off.y / nch] = s;
        pv.lvl[s] = -1;
        pv.flag[s] = 0;
      }
    }
    if (p < n_new) pv.act[p] = nxt;
  }
  if (last_cta(c)) {
    if (ok && any) {
      c->n_free = n_free - n_alloc + n_alloc / nch;
      c->n_act = n_new;
      c->topo += 1;
    }
    c->ctas_done = 0;
  }
}

__device__ __forceinline__ bool same_family(const PoolView& pv, int s, int t) {
  if (pv.tree[s] != pv.tree[t] || pv.lvl[s] != pv.lvl[t]) return false;
  for (int a = 0; a < 3; ++a)
    if ((pv.crd[3 * s + a] >> 1) != (pv.crd[3 * t + a] >> 1)) return false;
  return true;
}

// Flags of one coarsening round (Sec. 2.3), one warp per block.  A block
// qualifies (-1) if its largest normalised detail is below eps (strict), it is
// above Jmin, all 2^d sisters are leaves, and no leaf one level finer touches
// it (gradedness after the merge).  A family coarsens (-2) only if all its
// sisters qualify (completeness); this is the fixpoint of the paper's -2
// assignment, reached here by evaluating the condition for the whole family.
// Also emits the new-list counts (first member of a merged family hosts the
// mother; other members free their slots).
template <int D, bool SCAN>
__global__ void __launch_bounds__(256) k_flags(PoolView pv) {
  pdl_enter();
  // A family (the 2^d sisters of a block) merges when every sister is a leaf
  // whose normalised detail is below eps, above Jmin, and no leaf one level
  // finer touches any sister: the cells of level l+1 around the family,
  // [-1, 4]^d relative to its lower corner minus the family itself (the
  // union of the sisters' rings).  One warp per block, a lane per sister and
  // variable: the FP64 division of the normalisation is one sequence per warp
  // (with a lane per sister it took 78 us for 16384 blocks of 4 variables, all
  // FP64 pipe); the ring lookups are spread over the lanes.
  constexpr int NS = 1 << D;
  constexpr int NBOX = D == 3 ? 6 * 6 * 6 : 6 * 6;  // [-1, 4]^d around a family
  static_assert(NS * kMaxVar <= 32 && kMaxVar == 4, "a lane per sister and variable");
  __shared__ int2 sh[2][8];
  const int nact = pv.cnt->n_round;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nv = pv.nvar;
  int par = 0;
  for (int g = blockIdx.x; 8 * g < nact; g += gridDim.x, par ^= 1) {
    const int p = 8 * g + warp;
    int2 e = make_int2(0, 0);
    if (p < nact) {
      const int s = pv.act[p];
      const BlockInfo b = load_block(pv, s);
      // lane 31: is the previous list entry a member of the same family
      const bool prev = lane == 31 && p > 0 && same_family(pv, s, pv.act[p - 1]);
      const TreeDev& td = pv.trees[b.tree];
      const int sis = lane >> 2, v = lane & 3;
      const int own = (int)((b.c[0] & 1) | ((b.c[1] & 1) << 1) | (D > 2 ? (b.c[2] & 1) << 2 : 0));
      int64_t fc[3] = {0, 0, 0};
      for (int a = 0; a < D; ++a) fc[a] = b.c[a] & ~(int64_t)1;
      // a family at Jmin never merges: only the block's own detail is recorded
      const bool above = b.lvl > td.Jmin;
      int t = -1;
      if (sis == own) {
        t = s;
      } else if (above && sis < NS) {
        int64_t c[3] = {0, 0, 0};
        for (int a = 0; a < D; ++a) c[a] = fc[a] | ((sis >> a) & 1);
        t = tab_get<D>(pv, td, b.lvl, c);
      }
      // normalised detail of the lane's sister: the maximum over the variables
      // of non-negative values (NaN if a variable's is), on their bit patterns,
      // which order as the values
      long long mb = 0;
      bool nan = false;
      if (t >= 0 && v < nv) {
        double mv = pv.md[(int64_t)t * nv + v];
        if (pv.norm_kind != 0) {
          double sv = pv.svar[b.tree * nv + v];
          if (sv == 0.0) sv = 1.0;
          mv = mv / sv;
        }
        mb = __double_as_longlong(mv);
        nan = (mb & 0x7fffffffffffffffLL) > 0x7ff0000000000000LL;
        if (nan) mb = 0;
      }
      for (int o = 1; o < 4; o <<= 1) {
        const long long x = __shfl_xor_sync(0xffffffffu, mb, o);
        mb = x > mb ? x : mb;
      }
      const unsigned nans = __ballot_sync(0xffffffffu, nan);
      nan = (nans >> (4 * sis)) & 15u;
      if (nan) mb = 0x7ff8000000000000LL;
      // on bit patterns, as eps > 0; nothing is below a threshold that is NaN
      const long long eb = __double_as_longlong(td.eps);
      bool ok = sis >= NS || (t >= 0 && !nan && mb < eb && eb <= 0x7ff0000000000000LL);
      const double m = __longlong_as_double(__shfl_sync(0xffffffffu, mb, 4 * own));
      // no finer leaf around the family: cells of [-1, 4]^d outside [0, 3]^d
      // (looked up only for a family whose members are all candidates)
      const bool sisters = __all_sync(0xffffffffu, ok) && above;
      for (int u = lane; sisters && u < NBOX; u += 32) {
        const int q[3] = {u % 6 - 1, (u / 6) % 6 - 1, D == 3 ? u / 36 - 1 : 0};
        bool in = true;
        for (int a = 0; a < D; ++a) in &= q[a] >= 0 && q[a] <= 3;
        if (in) continue;
        int64_t cell[3] = {0, 0, 0};
        for (int a = 0; a < D; ++a) cell[a] = 2 * fc[a] + q[a];
        if (tab_get<D>(pv, td, b.lvl + 1, cell) >= 0) ok = false;
      }
      const bool all = __all_sync(0xffffffffu, ok) && above;
      const bool first = all && !__any_sync(0xffffffffu, prev);
      e = make_int2(!all || first ? 1 : 0, all && !first ? 1 : 0);
      if (lane == 0) {
        pv.mdet[s] = m;
        if (isnan(m)) set_err(pv, kErrNaN);
        pv.flag[s] = all ? -2 : 0;
        pv.emit[2 * p] = e.x;
        pv.emit[2 * p + 1] = e.y;
      }
    }
    emit_group(pv, g, nact, sh, par, e);
  }
  // SCAN: the CTA that finishes last scans the totals, which saves the separate
  // scan launch
  if constexpr (SCAN) {
    if (last_cta_all(pv.cnt)) {
      scan_groups(pv, nact);
      if (threadIdx.x == 0) pv.cnt->ctas_done = 0;
    }
  }
}

// Neighbour table (Sec. 2.2): rel[r] = (sx, sy, sz, sub), see mr.h for the order.
template <int D>
__global__ void k_neighbors(PoolView pv, const int4* rel, int R, int32_t* nbr, int8_t* dl) {
  pdl_enter();
  const int nact = pv.cnt->n_act;
  for (int64_t w = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; w < (int64_t)nact * R;
       w += (int64_t)gridDim.x * blockDim.x) {
    const int p = (int)(w / R), r = (int)(w % R);
    const BlockInfo b = load_block(pv, pv.act[p]);
    const TreeDev& td = pv.trees[b.tree];
    const int4 rr = rel[r];
    const int s[3] = {rr.x, rr.y, rr.z};
    int64_t k[3] = {0, 0, 0};
    bool corner = true;
    for (int a = 0; a < D; ++a) {
      k[a] = b.c[a] + s[a];
      corner &= s[a] != 0;
    }
    const int64_t n = (int64_t)1 << b.lvl;
    auto child = [&](int sub, int64_t ch[3]) {
      int z = 0;
      for (int a = 0; a < D; ++a) {
        int bit;
        if (s[a] != 0) bit = s[a] < 0 ? 1 : 0;
        else bit = (sub >> (z++)) & 1;
        ch[a] = 2 * pmod64(k[a], n) + bit;
      }
    };
    int found = -1, d = 0;
    if (rr.w < 0) {
      found = tab_get<D>(pv, td, b.lvl, k);
      if (found < 0) {
        int64_t pc[3] = {0, 0, 0};
        for (int a = 0; a < D; ++a) pc[a] = pmod64(k[a], n) >> 1;
        found = tab_get<D>(pv, td, b.lvl - 1, pc);
        d = -1;
        if (found < 0 && corner) {
          int64_t ch[3] = {0, 0, 0};
          child(0, ch);
          found = tab_get<D>(pv, td, b.lvl + 1, ch);
          d = 1;
        }
      }
    } else if (tab_get<D>(pv, td, b.lvl, k) < 0) {
      int64_t ch[3] = {0, 0, 0};
      child(rr.w, ch);
      found = tab_get<D>(pv, td, b.lvl + 1, ch);
      d = 1;
    }
    nbr[w] = found >= 0 ? pv.pos_of_slot[found] : -1;
    dl[w] = found >= 0 ? (int8_t)d : 0;
  }
}

template <int D>
__global__ void k_export_info(PoolView pv, mr_block_info* info, int8_t* flags, double* mdet) {
  pdl_enter();
  const int nact = pv.cnt->n_act;
  for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < nact; p += gridDim.x * blockDim.x) {
    const int s = pv.act[p];
    const BlockInfo b = load_block(pv, s);
    if (info) {
      mr_block_info o;
      o.level = b.lvl;
      o.tree = b.tree;
      o.treecode = morton<D>(b.c, b.lvl);
      for (int a = 0; a < 3; ++a) o.coords[a] = (int32_t)b.c[a];
      o.pad = 0;
      o.hilbert_key = pv.hkey[s];
      info[p] = o;
    }
    if (flags) flags[p] = pv.flag[s];
    if (mdet) mdet[p] = pv.mdet[s];
  }
}

// set_blocks: place input block i in slot i, validate, mark its finest cells.
template <int D>
__global__ void k_sb_place(PoolView pv, int64_t n, const int32_t* lvl, const int32_t* tree,
                           const int32_t* crd, int ntrees) {
  pdl_enter();
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int t = tree ? tree[i] : 0;
    if (t < 0 || t >= ntrees) { set_err(pv, kErrLayout); continue; }
    const TreeDev& td = pv.trees[t];
    const int l = lvl[i];
    if (l < td.Jmin || l > td.Jmax) { set_err(pv, kErrLayout); continue; }
    int32_t c32[3] = {0, 0, 0};
    int64_t c[3] = {0, 0, 0};
    bool bad = false;
    for (int a = 0; a < D; ++a) {
      c32[a] = crd[3 * i + a];
      c[a] = c32[a];
      bad |= c[a] < 0 || c[a] >= ((int64_t)1 << l);
    }
    if (bad) { set_err(pv, kErrLayout); continue; }
    pv.lvl[i] = (int8_t)l;
    pv.tree[i] = (int16_t)t;
    for (int a = 0; a < 3; ++a) pv.crd[3 * i + a] = c32[a];
    pv.hkey[i] = block_key<D>(c32, l, td.Jmax);
    pv.flag[i] = 0;
    pv.mdet[i] = 0.0;
    int* e = &pv.tab[td.tab_off[l] + (int64_t)morton<D>(c, l)];
    if (atomicCAS(e, -1, (int)i) != -1) set_err(pv, kErrLayout);
  }
}

// Every finest cell of every block gets +1 (coverage check: all must be 1).
template <int D>
__global__ void k_sb_cover(PoolView pv, int64_t n) {
  pdl_enter();
  for (int64_t i = blockIdx.x; i < n; i += gridDim.x) {
    const int l = pv.lvl[i];
    if (l < 0) continue;
    const TreeDev& td = pv.trees[pv.tree[i]];
    const int sh = td.Jmax - l;
    const int64_t per = (int64_t)1 << (D * sh);
    for (int64_t r = threadIdx.x; r < per; r += blockDim.x) {
      int64_t cell[3] = {0, 0, 0};
      for (int a = 0; a < D; ++a) {
        int64_t off = 0;
        for (int bb = 0; bb < sh; ++bb) off |= ((r >> (bb * D + a)) & 1) << bb;
        cell[a] = ((int64_t)pv.crd[3 * i + a] << sh) + off;
      }
      atomicAdd(&pv.cells[2 * (td.cell_off + (int64_t)morton<D>(cell, td.Jmax))], 1);
    }
  }
}

template <int D>
__global__ void k_sb_mark(PoolView pv, int64_t n) {
  pdl_enter();
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    if (pv.lvl[i] < 0) continue;
    const TreeDev& td = pv.trees[pv.tree[i]];
    pv.cells[2 * (td.cell_off + (int64_t)pv.hkey[i])] = 1;
  }
}

template <int D>
__global__ void k_sb_order(PoolView pv, int64_t n) {
  pdl_enter();
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    if (pv.lvl[i] < 0) continue;
    const TreeDev& td = pv.trees[pv.tree[i]];
    pv.act[pv.eoff[2 * (td.cell_off + (int64_t)pv.hkey[i])]] = (int32_t)i;
  }
}

// Graded-tree check: every ring cell must be covered by a leaf at l-1..l+1.
template <int D>
__global__ void k_check_graded(PoolView pv) {
  pdl_enter();
  const int nact = pv.cnt->n_act;
  for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < nact; p += gridDim.x * blockDim.x) {
    const BlockInfo b = load_block(pv, pv.act[p]);
    const TreeDev& td = pv.trees[b.tree];
    constexpr int NR = D == 3 ? 64 : 16;
    for (int r = 0; r < NR; ++r) {
      const int q[3] = {r % 4 - 1, (r / 4) % 4 - 1, r / 16 - 1};
      const int64_t nl1 = (int64_t)1 << (b.lvl + 1);
      int64_t cell[3] = {0, 0, 0}, c1[3] = {0, 0, 0}, c2[3] = {0, 0, 0};
      for (int a = 0; a < D; ++a) {
        cell[a] = pmod64(2 * b.c[a] + q[a], nl1);
        c1[a] = cell[a] >> 1;
        c2[a] = cell[a] >> 2;
      }
      if (tab_get<D>(pv, td, b.lvl + 1, cell) < 0 && tab_get<D>(pv, td, b.lvl, c1) < 0 &&
          tab_get<D>(pv, td, b.lvl - 1, c2) < 0)
        set_err(pv, kErrGraded);
    }
  }
}

}  // namespace mr
