// Device building blocks of the multiresolution step (templated on the block
// geometry).  Included by the per-dimension kernel translation units.
//
// Central idea: the pool stores only block interiors (Bs^d nodes per variable);
// every kernel that needs a block with its ghost layer builds the synchronised
// tile in shared memory directly from the neighbours' interiors ("gather").
// The paper fills ghosts in two passes (copies/injection first, then
// coarse-to-fine prediction by ascending level, Sec. 2.5).  On a graded tree
// every coarse node that a prediction stencil of a ghost node touches lies in
// a leaf of level >= l-1 that is a node there, so the second pass never needs
// another predicted value: one pass over interiors gives the same values.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

#include "mr_internal.h"

namespace mr {

// Compile-time loop: f(std::integral_constant<int, I>) for I in [A, E).
template <int A, int E, typename Fn>
__device__ __forceinline__ void static_for(Fn&& f) {
  if constexpr (A < E) {
    f(std::integral_constant<int, A>{});
    static_for<A + 1, E>(f);
  }
}

// Asynchronous global -> shared copy of one 4- or 8-byte value (cp.async):
// the value goes to shared memory without passing through registers, so a
// thread can have every copy of a tile in flight at once; cp_async_wait_all
// waits for the calling thread's copies (a barrier then publishes them).
template <typename T>
__device__ __forceinline__ void cp_async(T* smem_dst, const T* gmem_src) {
  static_assert(sizeof(T) == 4 || sizeof(T) == 8, "cp.async of 4 or 8 bytes");
  const unsigned d = (unsigned)__cvta_generic_to_shared(smem_dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(d), "l"(gmem_src), "n"(sizeof(T)) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Bulk asynchronous copy (TMA engine, cp.async.bulk) of `bytes` contiguous
// bytes from global to shared memory, completion signalled on an mbarrier
// that expects the transaction bytes.  Both addresses and the size are
// multiples of 16 bytes.  Issued by one thread.
__device__ __forceinline__ void mbar_init(uint64_t* bar, unsigned count) {
  const unsigned a = (unsigned)__cvta_generic_to_shared(bar);
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(a), "r"(count) : "memory");
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, unsigned bytes) {
  const unsigned a = (unsigned)__cvta_generic_to_shared(bar);
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(a), "r"(bytes) : "memory");
}
__device__ __forceinline__ void bulk_g2s(void* smem_dst, const void* gmem_src, unsigned bytes, uint64_t* bar) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(smem_dst);
  const unsigned b = (unsigned)__cvta_generic_to_shared(bar);
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(d), "l"(gmem_src), "r"(bytes), "r"(b) : "memory");
}
// Waits for the mbarrier phase with the given parity to complete, at most
// `limit` polls; false if it did not (the caller reports a timeout).
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, unsigned parity, int limit) {
  const unsigned a = (unsigned)__cvta_generic_to_shared(bar);
  for (int it = 0; it < limit; ++it) {
    unsigned done = 0;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
        : "=r"(done) : "r"(a), "r"(parity) : "memory");
    if (done) return true;
    if (it > 64) __nanosleep(256);
  }
  return false;
}

// float(d), rounded to nearest even, on the integer pipes: a conversion takes the
// FP64 pipe, which yields two results per clock and SM on GB300.  The rare results
// (not a normal number) stay on the integer pipes as well: a conversion in that branch
// would be evaluated for every value (skew stage, 16384 blocks of 17^2 x 4: 880 -> 846
// us per step; with f32_to_f64 2D advection, 65536 blocks, FP64 state: 241 -> 172 per
// launch).
__device__ __forceinline__ float f64_to_f32(double d) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(d);
  const unsigned hi = (unsigned)(u >> 32), sign = hi & 0x80000000u;
  const unsigned e = (hi >> 20) & 0x7ffu;
  const unsigned long long w = u & 0x7fffffffffffffffULL;
  unsigned m;
  if (e - 897u <= 253u) {  // exponent in [-126, 127]
    m = (unsigned)((w + 0x0fffffffULL + ((w >> 29) & 1ULL)) >> 29) - (896u << 23);
  } else if (e >= 1151u) {  // infinite, NaN or too large
    m = w > 0x7ff0000000000000ULL ? 0x7fffffffu : 0x7f800000u;
  } else if (e < 873u) {  // below half the smallest subnormal number
    m = 0;
  } else {
    const unsigned s = 926u - e;  // in units of 2^-149
    const unsigned long long f = (u & 0x000fffffffffffffULL) | 0x0010000000000000ULL;
    m = (unsigned)((f + ((1ULL << (s - 1)) - 1) + ((f >> s) & 1ULL)) >> s);
  }
  return __uint_as_float(m | sign);
}
// double(f), exact, likewise.
__device__ __forceinline__ double f32_to_f64(float f) {
  const unsigned u = __float_as_uint(f), sign = u & 0x80000000u, e = (u >> 23) & 0xffu, m = u & 0x7fffffu;
  if (e - 1u <= 253u) return __hiloint2double((int)(sign | (((u & 0x7fffffffu) >> 3) + (896u << 20))), (int)(u << 29));
  unsigned long long r;
  if (e) {
    r = 0x7ff0000000000000ULL | ((unsigned long long)m << 29);
  } else if (m == 0) {
    r = 0;
  } else {
    const int p = 31 - __clz((int)m);  // m 2^-149, leading bit p
    r = ((unsigned long long)(p + 874) << 52) | (((unsigned long long)m << (52 - p)) & 0x000fffffffffffffULL);
  }
  return __longlong_as_double((long long)(r | ((unsigned long long)sign << 32)));
}
// Stage value in the state's type.
template <typename TS, typename TC>
__device__ __forceinline__ TS to_state(TC v) {
  if constexpr (sizeof(TC) == 4 && sizeof(TS) == 8) return f32_to_f64(v);
  else return (TS)v;
}
// Value in the tile's type.
template <typename TT, typename TS>
__device__ __forceinline__ TT to_tile(TS v) {
  if constexpr (sizeof(TS) == 8 && sizeof(TT) == 4) return f64_to_f32(v);
  else return (TT)v;
}
// Neither infinite nor NaN, likewise on the bit pattern (3D details, 2584 FP64 blocks:
// 514 -> 470 us; 4096 blocks of 33^2 112 -> 92).
__device__ __forceinline__ bool finite(float v) { return (__float_as_uint(v) & 0x7f800000u) != 0x7f800000u; }
__device__ __forceinline__ bool finite(double v) { return (__double2hiint(v) & 0x7ff00000) != 0x7ff00000; }
// a != b of two finite or infinite values, doubles on their bit patterns (as above).
__device__ __forceinline__ bool differs(float a, float b) { return a != b; }
__device__ __forceinline__ bool differs(double a, double b) {
  const unsigned long long x = (unsigned long long)__double_as_longlong(a), z = (unsigned long long)__double_as_longlong(b);
  return x != z && ((x | z) << 1) != 0;  // +0 equals -0; equal NaN patterns need no store
}

// The state y after its edge nodes were stored through another pointer to it (src),
// past a barrier: both are __restrict__ kernel arguments, so without this the
// compiler may take loads of y before those stores, or through the read-only path.
template <typename T>
__device__ __forceinline__ const T* committed(const T* y, const void* src) {
  asm volatile("" : "+l"(y) : "l"(src) : "memory");
  return y;
}

// Thread groups that cooperate on one block: the whole CTA, or one warp.
struct CtaGroup {
  __device__ __forceinline__ int rank() const { return threadIdx.x; }
  __device__ __forceinline__ int size() const { return blockDim.x; }
  __device__ __forceinline__ void sync() const { __syncthreads(); }
};
struct WarpGroup {
  __device__ __forceinline__ int rank() const { return threadIdx.x & 31; }
  __device__ __forceinline__ int size() const { return 32; }
  __device__ __forceinline__ void sync() const { __syncwarp(); }
};

// a modulo n, n a power of two (blocks per axis at a level, lattice intervals): the
// low bits of a, also for negative a.
__device__ __forceinline__ int64_t pmod64(int64_t a, int64_t n) { return a & (n - 1); }
// The low 16 (D = 2) or 10 (D = 3) bits of x, D - 1 zero bits between them.
template <int D>
__device__ __forceinline__ uint32_t spread_bits(uint32_t x) {
  if constexpr (D == 2) {
    x = (x | (x << 8)) & 0x00ff00ffu;
    x = (x | (x << 4)) & 0x0f0f0f0fu;
    x = (x | (x << 2)) & 0x33333333u;
    x = (x | (x << 1)) & 0x55555555u;
  } else {
    x = (x | (x << 16)) & 0x030000ffu;
    x = (x | (x << 8)) & 0x0300f00fu;
    x = (x | (x << 4)) & 0x030c30c3u;
    x = (x | (x << 2)) & 0x09249249u;
  }
  return x;
}
// Morton index of a cell = treecode digits (Sec. 2.2), x bit lowest.  Levels reach
// 11 (2D) and 8 (3D), so the index has at most 24 bits.
template <int D>
__device__ __forceinline__ uint64_t morton(const int64_t c[3], int lvl) {
  static_assert(kMaxLevel <= 11, "2 x 11 bits in 2D");
  const uint32_t m = (1u << lvl) - 1u;
  uint32_t t = spread_bits<D>((uint32_t)c[0] & m) | (spread_bits<D>((uint32_t)c[1] & m) << 1);
  if constexpr (D == 3) t |= spread_bits<D>((uint32_t)c[2] & m) << 2;
  return t;
}

// Hilbert index (J. Skilling, AIP Conf. Proc. 707, 381 (2004)): inverse undo of
// the axis exchanges, Gray encoding, then bit interleave of the transpose.
template <int D>
__device__ __forceinline__ uint64_t hilbert(const int64_t cell[3], int bits) {
  if (bits == 0) return 0;
  uint32_t X[3] = {(uint32_t)cell[0], (uint32_t)cell[1], D == 3 ? (uint32_t)cell[2] : 0u};
  const uint32_t M = 1u << (bits - 1);
  for (uint32_t Q = M; Q > 1; Q >>= 1) {
    const uint32_t P = Q - 1;
#pragma unroll
    for (int i = 0; i < D; ++i) {
      if (X[i] & Q) {
        X[0] ^= P;
      } else {
        uint32_t t = (X[0] ^ X[i]) & P;
        X[0] ^= t;
        X[i] ^= t;
      }
    }
  }
#pragma unroll
  for (int i = 1; i < D; ++i) X[i] ^= X[i - 1];
  uint32_t t = 0;
  for (uint32_t Q = M; Q > 1; Q >>= 1)
    if (X[D - 1] & Q) t ^= Q - 1;
#pragma unroll
  for (int i = 0; i < D; ++i) X[i] ^= t;
  uint64_t h = 0;
  for (int b = bits - 1; b >= 0; --b)
#pragma unroll
    for (int i = 0; i < D; ++i) h = (h << 1) | ((X[i] >> b) & 1u);
  return h;
}

template <int D>
__device__ __forceinline__ uint64_t block_key(const int32_t* c, int lvl, int Jmax) {
  int64_t cell[3] = {0, 0, 0};
  for (int a = 0; a < D; ++a) cell[a] = (int64_t)c[a] << (Jmax - lvl);
  return hilbert<D>(cell, Jmax);
}

// Slot of the leaf with block coordinates c at level m (periodic wrap: morton
// keeps the low m bits), or -1.
template <int D>
__device__ __forceinline__ int tab_get(const PoolView& pv, const TreeDev& td, int m,
                                       const int64_t c[3]) {
  if (m < td.Jmin || m > td.Jmax) return -1;
  return pv.tab[td.tab_off[m] + (int64_t)morton<D>(c, m)];
}

template <int D, int B>
struct Geo {
  static constexpr int G = kG;
  static constexpr int T = B + 2 * G;
  static constexpr int TZ = D == 3 ? T : 1;
  static constexpr int GZ = D == 3 ? G : 0;
  static constexpr int BZ = D == 3 ? B : 1;
  static constexpr int TILE = T * T * TZ;
  static constexpr int NI = B * B * BZ;
  static constexpr int NR = D == 3 ? 64 : 16;  // ring of level l+1 cells, [-1,2]^d
  static constexpr int NCH = 1 << D;
  static_assert(G + 2 < (B - 1) / 2, "prediction stencils of ghosts must stay in the ring");
  // coarse box: level l-1 nodes around the block that prediction stencils of
  // ghost nodes can touch, coarse index n in [CLO, CLO + CB) relative to the
  // block origin
  static constexpr int CLO = -(G / 2) - 1;
  static constexpr int CB = (B - 1) / 2 + G + 3;
  static constexpr int CBOX = CB * CB * (D == 3 ? CB : 1);
  __device__ static __forceinline__ int tix(int i, int j, int k) {
    return ((k + GZ) * T + (j + G)) * T + (i + G);
  }
  __device__ static __forceinline__ int lin(int i, int j, int k) { return (k * B + j) * B + i; }
};

// Part of the tile a consumer reads: the box of ghost width W (W <= G) and the
// coarse nodes its prediction stencils touch, CLO..CLO+CB-1 per axis.
template <int D, int B, int W>
struct Box {
  static_assert(W >= 1 && W <= kG, "ghost width");
  static constexpr int S = B + 2 * W;
  static constexpr int NPTS = S * S * (D == 3 ? S : 1);
  static constexpr int TILE = NPTS;  // tile of this width: S^d nodes, x fastest
  static constexpr int CLO = -((W + 1) / 2) - 1;
  static constexpr int CB = (B - 1) / 2 + 2 * ((W + 1) / 2) + 3;
  static constexpr int CBOX = CB * CB * (D == 3 ? CB : 1);
  // scratch of the separable prediction (2D), per variable: X[ny][x] (coarse y, fine x)
  static constexpr int SCR = CB * S;
  __device__ static __forceinline__ int cix(int i, int j, int k) {
    return ((D == 3 ? k - CLO : 0) * CB + (j - CLO)) * CB + (i - CLO);
  }
  __device__ static __forceinline__ int tix(int i, int j, int k) {
    return (((D == 3 ? k + W : 0)) * S + (j + W)) * S + (i + W);
  }
};

struct BlockInfo {
  int slot, lvl, tree;
  int64_t c[3];
};

__device__ __forceinline__ BlockInfo load_block(const PoolView& pv, int slot) {
  BlockInfo b;
  b.slot = slot;
  b.lvl = pv.lvl[slot];
  b.tree = pv.tree[slot];
  for (int a = 0; a < 3; ++a) b.c[a] = pv.crd[3 * slot + a];
  return b;
}

__device__ __forceinline__ void set_err(const PoolView& pv, int bits) {
  atomicOr(&pv.cnt->err, bits);
}

// Polls after which a wait for a bulk copy is given up (a test sets 0).
#ifndef MR_WAIT_POLLS
#define MR_WAIT_POLLS (1 << 20)
#endif
// Waits for the bulk copies of the mbarrier's phase.  A copy that does not land is
// reported, not waited for without end: false, and the caller leaves the kernel (the
// barrier's phase is still open, and its block has no values), after a second bounded
// wait, so that no copy is in flight to shared memory that another CTA may get.
__device__ __forceinline__ bool bulk_landed(const PoolView& pv, uint64_t* bar, unsigned parity) {
  if (mbar_wait(bar, parity, MR_WAIT_POLLS)) return true;
  set_err(pv, kErrTimeout);
  mbar_wait(bar, parity, 1 << 20);
  return false;
}

// Ring map: for every level-(l+1) cell q in [-1,2]^d around the block (its own
// 2^d child cells included) the leaf covering it, searched at l+1, l, l-1,
// with the leaf's origin relative to the block origin in level-(l+1) node
// units (periodic images resolved once here, so per-point work needs no
// modulo).  These cells carry exactly the 16 (2D) / 74 (3D) relations of
// Sec. 2.2.  A cell covered by no leaf in that range means a non-graded tree.
//
// Region table (filled when some ring leaf is not at the block's level): along
// each axis a level-l node index x relative to the block origin falls into one
// of 7 classes -- inside ring cell -1 (x < 0), on the face x = 0 between cells
// -1 and 0, inside cell 0, on the face x = H, inside cell 1, on the face x = 2H,
// inside cell 2 (H = (Bs - 1) / 2).  All nodes of one class box (7^d boxes)
// have the same leaves containing them, in the same position (inside, or on
// the same faces), hence the same owner: the owner is searched once per box,
// and each node only offsets into it.
template <int D>
struct RingD {
  static constexpr int NREG = D == 3 ? 343 : 49;
  int slot[64];
  int org[64][3];
  int8_t lvl[64];
  int finer;    // some leaf one level finer touches the block
  int coarser;  // some leaf one level coarser touches the block
  int mixed;    // some ring leaf is not at the block's level
  // classes (bit c of 7 per axis: x, y << 7, z << 14) of the class boxes owned
  // by a coarser leaf: the tile nodes predicted from the coarse lattice lie
  // in their union, so the separable prediction passes are confined to it
  int cmask;
  // per class box: owner slot (-1: none), owner level, owner origin
  // (level-(l+1) node units, relative to the block origin) x | y << 16, z
  int4 reg[NREG];
};
template <int D>
constexpr int kRingBytesD = (int)((sizeof(RingD<D>) + 15) / 16 * 16);
static_assert(RingD<2>::NREG + 1 == reg_entries(2) && RingD<3>::NREG + 1 == reg_entries(3), "table size");

template <int D, int B, typename G = CtaGroup>
__device__ void build_ring(const PoolView& pv, const TreeDev& td, const BlockInfo& b, RingD<D>& R) {
  const G g{};
  using Gm = Geo<D, B>;
  if (g.rank() == 0) R.finer = R.coarser = R.mixed = R.cmask = 0;
  g.sync();
  for (int r = g.rank(); r < Gm::NR; r += g.size()) {
    const int q[3] = {r % 4 - 1, (r / 4) % 4 - 1, r / 16 - 1};
    bool inside = true;
    for (int a = 0; a < D; ++a) inside &= (q[a] == 0 || q[a] == 1);
    if (inside) {
      R.slot[r] = b.slot;
      R.lvl[r] = (int8_t)b.lvl;
      for (int a = 0; a < 3; ++a) R.org[r][a] = 0;
      continue;
    }
    const int64_t nl1 = (int64_t)1 << (b.lvl + 1);
    int64_t cell[3] = {0, 0, 0}, c1[3] = {0, 0, 0}, c2[3] = {0, 0, 0};
    int un[3] = {0, 0, 0};
    for (int a = 0; a < D; ++a) {
      un[a] = (int)(2 * b.c[a] + q[a]);
      cell[a] = (int64_t)(un[a]) & (nl1 - 1);
      c1[a] = cell[a] >> 1;
      c2[a] = cell[a] >> 2;
    }
    // the three candidate levels are looked up together (one memory round trip)
    const int sf = tab_get<D>(pv, td, b.lvl + 1, cell), se = tab_get<D>(pv, td, b.lvl, c1),
              sc = tab_get<D>(pv, td, b.lvl - 1, c2);
    int s = sf, m = b.lvl + 1;
    if (s < 0) { s = se; m = b.lvl; }
    if (s < 0) { s = sc; m = b.lvl - 1; }
    if (s < 0) {
      set_err(pv, kErrGraded);
      m = -1;
    }
    if (m == b.lvl + 1) R.finer = 1;  // benign races: all writers store 1
    if (m == b.lvl - 1) R.coarser = 1;
    if (m != b.lvl) R.mixed = 1;
    const int sh = b.lvl + 1 - m;
    for (int a = 0; a < 3; ++a) {
      const int oc = a < D && m >= 0 ? ((un[a] >> sh) << sh) - (int)(2 * b.c[a]) : 0;
      R.org[r][a] = oc * (B - 1);
    }
    R.slot[r] = s;
    R.lvl[r] = (int8_t)m;
  }
}

// Owner of a point: among the leaves whose closed cell contains the point (found
// through the ring), the finest; among equal levels the one in which the point
// is the upper edge node on the fewest leading axes (combo order).  Point given
// in level-(l+1) node units relative to the block origin.  off[] receives the
// point's offset inside the owner, again in level-(l+1) units.
struct Own {
  int slot, m, combo;
  int off[3];
};

template <int B>
struct Log2B {
  static constexpr int value = B == 17 ? 4 : (B == 33 ? 5 : -1);
};

template <int D, int B>
__device__ __forceinline__ bool owner(const BlockInfo& b, const int h[3], int min_m, const RingD<D>& R,
                                      Own& o) {
  constexpr int P = Log2B<B>::value;
  static_assert(P > 0, "Bs - 1 must be a power of two");
  int c0[3] = {0, 0, 0};
  bool onb[3] = {false, false, false};
  bool any = false;
#pragma unroll
  for (int a = 0; a < D; ++a) {
    c0[a] = h[a] >> P;
    onb[a] = (h[a] & (B - 2)) == 0;
    any |= onb[a];
  }
  // Candidate A: the ring cell holding the point at its lower edge or inside.
  // In its leaf the point is never the upper edge node, so A has the smallest
  // combo; it is the owner unless another candidate is finer.
  const int rA = (c0[0] + 1) + 4 * (c0[1] + 1) + 16 * (D == 3 ? c0[2] + 1 : 0);
  const int mA = R.lvl[rA];
  int mmax = R.slot[rA] >= 0 ? mA : -1;
  if (any) {
#pragma unroll
    for (int combo = 1; combo < (1 << D); ++combo) {
      bool ok = true;
      int r = 0, mul = 1;
#pragma unroll
      for (int a = 0; a < D; ++a) {
        const int bit = (combo >> a) & 1;
        if (bit && !onb[a]) ok = false;
        const int q = c0[a] - bit;
        if (q < -1) ok = false;
        r += (q + 1) * mul;
        mul *= 4;
      }
      if (ok && R.slot[r] >= 0 && R.lvl[r] > mmax) mmax = R.lvl[r];
    }
  }
  if (mmax < 0 || mmax < min_m) {
    o.m = -1;
    return false;
  }
  const int l1 = b.lvl + 1;
  if (mA == mmax && R.slot[rA] >= 0) {
    o.m = mA;
    o.combo = 0;
    o.slot = R.slot[rA];
#pragma unroll
    for (int a = 0; a < 3; ++a) o.off[a] = a < D ? h[a] - R.org[rA][a] : 0;
    return true;
  }
  // a finer leaf shares the point: smallest combo among the finest candidates
  o.m = -1;
  o.combo = 1 << 30;
#pragma unroll
  for (int combo = 1; combo < (1 << D); ++combo) {
    bool ok = true;
    int r = 0, mul = 1;
#pragma unroll
    for (int a = 0; a < D; ++a) {
      const int bit = (combo >> a) & 1;
      if (bit && !onb[a]) ok = false;
      const int q = c0[a] - bit;
      if (q < -1) ok = false;
      r += (q + 1) * mul;
      mul *= 4;
    }
    if (!ok || R.slot[r] < 0 || R.lvl[r] != mmax) continue;
    const int W = (B - 1) << (l1 - mmax);
    int oc = 0, off[3] = {0, 0, 0};
#pragma unroll
    for (int a = 0; a < D; ++a) {
      off[a] = h[a] - R.org[r][a];
      if (off[a] == W) oc |= 1 << a;
    }
    if (oc < o.combo) {
      o.m = mmax;
      o.combo = oc;
      o.slot = R.slot[r];
#pragma unroll
      for (int a = 0; a < 3; ++a) o.off[a] = off[a];
    }
  }
  return o.m >= 0;
}

// x / 16 rounded to nearest even.  FP64 on the integer pipes, which leaves four of
// the prediction's five operations to the FP64 pipe: a normal result differs in the
// exponent alone; a subnormal one (exponent field 4 or less) is shifted and
// rounded; zeros, infinities and NaN stay.  No multiplication is left in the rare
// branch: the compiler would evaluate it for every value.  Measured per step of
// 2584 blocks of 17^3 FP64: details 638 -> 594 us, refinement 220 -> 189; 736
// mothers of 33^2 x 4, FP64: refinement 140 -> 132.
__device__ __forceinline__ float sixteenth(float x) { return x * 0.0625f; }
__device__ __forceinline__ double sixteenth(double x) {
  const int hi = __double2hiint(x);
  const unsigned e = ((unsigned)hi >> 20) & 0x7ffu;
  if (e - 5u <= 2041u) return __hiloint2double(hi - (4 << 20), __double2loint(x));
  const unsigned long long u = (unsigned long long)__double_as_longlong(x), sign = u & 0x8000000000000000ULL;
  if (e == 0x7ffu || u == sign) return x;
  const unsigned long long m = (u & 0x000fffffffffffffULL) | (e ? 0x0010000000000000ULL : 0ULL);
  const int s = e ? 5 - (int)e : 4;
  return __longlong_as_double((long long)(sign | ((m + ((1ULL << (s - 1)) - 1) + ((m >> s) & 1)) >> s)));
}
template <typename T>
__device__ __forceinline__ T dd4(T fm1, T f0, T f1, T f2) {
  // 4-point interpolating-wavelet midpoint prediction (Sec. 2.3, 4th order)
  return sixteenth(T(9) * (f0 + f1) - (fm1 + f2));
}

// Coarse-lattice prediction at half-coarse position o (relative to the block
// origin) from the staged coarse box: x first, then y, then z.
template <int D, int B, int W, typename TT>
__device__ __forceinline__ TT predict_box(const TT* box, const int o[3]) {
  using Gm = Box<D, B, W>;
  int base[3] = {0, 0, 0}, ns[3] = {1, 1, 1};
#pragma unroll
  for (int a = 0; a < D; ++a) {
    const int fl = o[a] >> 1;
    if (o[a] & 1) { ns[a] = 4; base[a] = fl - 1; }
    else base[a] = fl;
  }
  TT vx[4][4];
  for (int sz = 0; sz < ns[2]; ++sz)
    for (int sy = 0; sy < ns[1]; ++sy) {
      const int y = base[1] + sy, z = base[2] + sz;
      if (ns[0] == 4) {
        const TT* r = box + Gm::cix(base[0], y, z);
        vx[sz][sy] = dd4(r[0], r[1], r[2], r[3]);
      } else {
        vx[sz][sy] = box[Gm::cix(base[0], y, z)];
      }
    }
  TT vy[4];
  for (int sz = 0; sz < ns[2]; ++sz)
    vy[sz] = ns[1] == 4 ? dd4(vx[sz][0], vx[sz][1], vx[sz][2], vx[sz][3]) : vx[sz][0];
  return ns[2] == 4 ? dd4(vy[0], vy[1], vy[2], vy[3]) : vy[0];
}

// Class (0..6) of a level-l node index x relative to the block origin, for
// -(H - 1) <= x <= 3H - 1 (H = (Bs - 1) / 2): inside ring cell -1, face 0,
// inside cell 0, face H, inside cell 1, face 2H, inside cell 2.
template <int B>
__device__ __forceinline__ int reg_class(int x) {
  constexpr int H = (B - 1) / 2;
  return (x >= 0) + (x > 0) + (x >= H) + (x > H) + (x >= 2 * H) + (x > 2 * H);
}
// A node index of class c.
template <int B>
__device__ __forceinline__ int reg_rep(int c) {
  constexpr int H = (B - 1) / 2;
  return c == 0 ? -1 : c == 1 ? 0 : c == 2 ? 1 : c == 3 ? H : c == 4 ? H + 1 : c == 5 ? 2 * H : 2 * H + 1;
}

// Owner of every class box (see RingD), found with owner() at one node of the box.
template <int D, int B, typename G>
__device__ void build_regions(const BlockInfo& b, RingD<D>& R) {
  const G g{};
  for (int r = g.rank(); r < RingD<D>::NREG; r += g.size()) {
    const int c[3] = {r % 7, (r / 7) % 7, r / 49};
    int h[3] = {0, 0, 0};
#pragma unroll
    for (int a = 0; a < D; ++a) h[a] = 2 * reg_rep<B>(c[a]);
    Own o;
    int4 e = make_int4(-1, -1, 0, 0);
    if (owner<D, B>(b, h, 0, R, o)) {
      const int ox = h[0] - o.off[0], oy = h[1] - o.off[1], oz = h[2] - o.off[2];
      e = make_int4(o.slot, o.m, (ox & 0xffff) | (oy << 16), oz);
      if (o.m < b.lvl) atomicOr(&R.cmask, (1 << c[0]) | (1 << (7 + c[1])) | (D == 3 ? 1 << (14 + c[2]) : 0));
    }
    R.reg[r] = e;
  }
}

// Class-box owner table of plan position p (built with the stage plan while
// the tree is fixed): NREG entries, then {finer, coarser, mixed}.
template <int D>
__device__ __forceinline__ int4* plan_regions(const PoolView& pv, int p) {
  return pv.regs + (int64_t)p * (RingD<D>::NREG + 1);
}
template <int D, typename G>
__device__ void store_regions(const PoolView& pv, int p, const RingD<D>& R) {
  const G g{};
  int4* dst = plan_regions<D>(pv, p);
  for (int r = g.rank(); r < RingD<D>::NREG; r += g.size()) dst[r] = R.reg[r];
  if (g.rank() == 0) dst[RingD<D>::NREG] = make_int4(R.finer, R.coarser, R.mixed, R.cmask);
}
// Loads the table of plan position p into the ring (the caller synchronises
// the group before use).
template <int D, typename G>
__device__ void load_regions(const PoolView& pv, int p, RingD<D>& R) {
  const G g{};
  const int4* src = plan_regions<D>(pv, p);
  for (int r = g.rank(); r < RingD<D>::NREG; r += g.size()) R.reg[r] = src[r];
  if (g.rank() == 0) {
    const int4 f = src[RingD<D>::NREG];
    R.finer = f.x;
    R.coarser = f.y;
    R.mixed = f.z;
    R.cmask = f.w;
  }
}

// Tile nodes (per axis, tile coordinates) that can be predicted from the
// coarse lattice: the span of the classes in mask7 (bit c = class c of
// reg_class), clipped to the tile box of ghost width W; and the coarse
// indices the separable passes read for them, clipped to the coarse box.
template <int B, int W>
struct PredBox {
  int lo[3], hi[3];    // predicted tile nodes
  int nlo[3], nhi[3];  // coarse nodes their prediction reads
  __device__ __forceinline__ PredBox(int cmask, int D) {
    constexpr int H = (B - 1) / 2;
    using Bx = Box<2, B, W>;  // CLO and CB do not depend on the dimension
    // first and last node of class c within the tile box
    auto clo = [](int c) { return c == 0 ? -W : c == 1 ? 0 : c == 2 ? 1 : c == 3 ? H : c == 4 ? H + 1 : c == 5 ? 2 * H : 2 * H + 1; };
    auto chi = [](int c) { return c == 0 ? -1 : c == 1 ? 0 : c == 2 ? H - 1 : c == 3 ? H : c == 4 ? 2 * H - 1 : c == 5 ? 2 * H : B - 1 + W; };
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const int m = (cmask >> (7 * a)) & 127;
      if (a >= D || m == 0) {
        lo[a] = hi[a] = 0;
        nlo[a] = nhi[a] = 0;
        continue;
      }
      lo[a] = clo(__ffs(m) - 1);
      hi[a] = chi(31 - __clz(m));
      nlo[a] = max(Bx::CLO, (lo[a] >> 1) - 1);
      nhi[a] = min(Bx::CLO + Bx::CB - 1, (hi[a] >> 1) + 2);
    }
  }
};

// Separable prediction over the 2D coarse box (values of nv variables in cbox), x
// first, then y: the same operations in the same order as predict_box, evaluated only
// where the predicted nodes of pb need them.  The x pass goes to scr (y per point from
// it).  Ends with a group barrier.
template <int B, int W, typename TT, typename G>
__device__ void coarse_passes(int nv, const TT* cbox, TT* scr, const PredBox<B, W>& pb) {
  const G g{};
  using Bx = Box<2, B, W>;
  // x in [lo0, hi0], coarse rows ny in [nlo1, nhi1]
  const int ex = pb.hi[0] - pb.lo[0] + 1, ey = pb.nhi[1] - pb.nlo[1] + 1;
  for (int v = 0; v < nv; ++v) {
    const TT* cb = cbox + v * Bx::CBOX;
    TT* X = scr + v * Bx::SCR;
    for (int q = g.rank(); q < ex * ey; q += g.size()) {
      const int x = q % ex + pb.lo[0], ny = (q / ex) % ey + pb.nlo[1];
      const int fl = x >> 1;
      const int at = (ny - Bx::CLO) * Bx::S + (x + W);
      X[at] = (x & 1) ? dd4(cb[Bx::cix(fl - 1, ny, 0)], cb[Bx::cix(fl, ny, 0)], cb[Bx::cix(fl + 1, ny, 0)],
                            cb[Bx::cix(fl + 2, ny, 0)])
                      : cb[Bx::cix(fl, ny, 0)];
    }
  }
  g.sync();
}

// Fills the synchronised tile (nvar x T^d, type TT) of block b from field F.
// Block-edge nodes owned by another block (a finer one, Sec. 2.2 rule 2, or an
// equal-level one that holds the node at its lower edge, which keeps redundant
// copies identical as Sec. 2.5 assumes) take the owner's value; with commit
// they are also written back into F when they differ.  cbox: scratch
// of nvar x CBOX values for the coarse lattice (used when a coarser leaf
// touches the block): every coarse node takes its owner's value, and ghost
// nodes between coarse nodes are predicted from it, in 2D in separable passes over
// scr (nvar x SCR values) if given, else node by node.
// ES: tile layout, 1 = variable after variable, 4 = the four variables of a node
// side by side.
template <int D, int B, typename TF, typename TT, int W = kG, typename G = CtaGroup, int ES = 1>
__device__ void fill_tile(const PoolView& pv, const BlockInfo& b, const TF* F, TF* Fw, TT* tile,
                          bool commit, RingD<D>& R, TT* cbox, TT* scr = nullptr, bool have_regions = false) {
  const G g{};
  using Gm = Geo<D, B>;
  using Bx = Box<D, B, W>;
  // Each thread takes U points at a time: owners and addresses first, then the
  // U loads together, then the stores, so that the loads are in flight at once.
  constexpr int U = 4;
  auto at_tile = [&](int v, int idx) { return ES == 1 ? v * Bx::TILE + idx : ES * idx + v; };
  const int nv = pv.nvar;
  const int64_t own = (int64_t)b.slot * nv * pv.vs;
  if (!R.mixed) {
    // every ring leaf has the block's level: the owner of a point is the ring
    // cell holding it from below (equal-level rule of owner()), no search
    constexpr int P = Log2B<B>::value;
    for (int q0 = g.rank(); q0 < Bx::NPTS; q0 += U * g.size()) {
      int64_t at[U];
      int idx[U], li[U];
      bool ok[U], ed[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int q = q0 + u * g.size();
        ok[u] = q < Bx::NPTS;
        const int qq = ok[u] ? q : 0;
        const int i = qq % Bx::S - W;
        const int j = (qq / Bx::S) % Bx::S - W;
        const int k = D == 3 ? qq / (Bx::S * Bx::S) - W : 0;
        idx[u] = Bx::tix(i, j, k);
        li[u] = Gm::lin(i, j, k);
        const int h[3] = {2 * i, 2 * j, 2 * k};
        int r = 0, lo[3] = {0, 0, 0};
#pragma unroll
        for (int a = 0; a < D; ++a) r += ((h[a] >> P) + 1) << (2 * a);
#pragma unroll
        for (int a = 0; a < D; ++a) lo[a] = (h[a] - R.org[r][a]) >> 1;
        const int src = R.slot[r];
        at[u] = (int64_t)src * nv * pv.vs + Gm::lin(lo[0], lo[1], lo[2]);
        // block-edge node owned by the equal-level neighbour (i or j = B-1)
        bool edge_node = true;
#pragma unroll
        for (int a = 0; a < D; ++a) edge_node &= (h[a] >= 0 && h[a] <= 2 * (B - 1));
        ed[u] = commit && src != b.slot && edge_node;
      }
      for (int v = 0; v < nv; ++v) {
        TF val[U];
#pragma unroll
        for (int u = 0; u < U; ++u) val[u] = ok[u] ? F[at[u] + (int64_t)v * pv.vs] : TF(0);
#pragma unroll
        for (int u = 0; u < U; ++u) {
          if (!ok[u]) continue;
          tile[at_tile(v, idx[u])] = to_tile<TT>(val[u]);
          if (ed[u]) {
            const int64_t me = own + (int64_t)v * pv.vs + li[u];
            if (differs(F[me], val[u])) Fw[me] = val[u];
          }
        }
      }
    }
    return;
  }
  // some ring leaf is at another level: one owner search per class box
  // (unless the table was loaded from the stage plan)
  if (!have_regions) {
    build_regions<D, B, G>(b, R);
    g.sync();
  }
  const int l1 = b.lvl + 1;
  // owner of level-l node x (relative to the block origin) and the node's
  // offset inside it in level-(l+1) units
  auto region = [&](const int x[3], int& slot, int& m, int off[3]) {
    const int r = reg_class<B>(x[0]) + 7 * reg_class<B>(x[1]) + (D == 3 ? 49 * reg_class<B>(x[2]) : 0);
    const int4 e = R.reg[r];
    slot = e.x;
    m = e.y;
    off[0] = 2 * x[0] - (int)(int16_t)(e.z & 0xffff);
    off[1] = 2 * x[1] - (e.z >> 16);
    off[2] = D == 3 ? 2 * x[2] - e.w : 0;
  };
  if (R.coarser && R.cmask) {
    const PredBox<B, W> pb(R.cmask, D);
    for (int q0 = g.rank(); q0 < Bx::CBOX; q0 += U * g.size()) {
      int64_t at[U];
      bool ok[U], good[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int idx = q0 + u * g.size();
        ok[u] = idx < Bx::CBOX;
        good[u] = false;
        at[u] = 0;
        if (!ok[u]) continue;
        const int n[3] = {idx % Bx::CB + Bx::CLO, (idx / Bx::CB) % Bx::CB + Bx::CLO,
                          D == 3 ? idx / (Bx::CB * Bx::CB) + Bx::CLO : 0};
        bool need = true;  // read by the prediction of some node of pb
#pragma unroll
        for (int a = 0; a < D; ++a) need &= n[a] >= pb.nlo[a] && n[a] <= pb.nhi[a];
        if (!need) continue;
        // coarse node n sits at level-l node 2n
        const int x[3] = {2 * n[0], 2 * n[1], 2 * n[2]};
        int slot, m, off[3];
        region(x, slot, m, off);
        if (slot < 0 || m < b.lvl - 1) {
          set_err(pv, kErrGraded);
          continue;
        }
        good[u] = true;
        const int sh = l1 - m;
        at[u] = ((int64_t)slot * nv) * pv.vs + Gm::lin(off[0] >> sh, off[1] >> sh, D == 3 ? off[2] >> sh : 0);
      }
      for (int v = 0; v < nv; ++v) {
        TF val[U];
#pragma unroll
        for (int u = 0; u < U; ++u) val[u] = good[u] ? F[at[u] + (int64_t)v * pv.vs] : TF(0);
#pragma unroll
        for (int u = 0; u < U; ++u)
          if (ok[u]) cbox[v * Bx::CBOX + q0 + u * g.size()] = good[u] ? to_tile<TT>(val[u]) : TT(0);
      }
    }
    g.sync();
    if constexpr (D == 2) {
      if (scr) coarse_passes<B, W, TT, G>(nv, cbox, scr, pb);
    }
  }
  // kinds of tile points: 0 own node, 1 block-edge node of another owner,
  // 2 ghost node that is a node of its owner, 3 ghost predicted from the coarse
  // box, 4 no owner (error, zero)
  for (int q0 = g.rank(); q0 < Bx::NPTS; q0 += U * g.size()) {
    int64_t at[U];
    int idx[U], li[U], kind[U], ijk[U][3];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int q = q0 + u * g.size();
      const int qq = q < Bx::NPTS ? q : 0;
      const int i = qq % Bx::S - W;
      const int j = (qq / Bx::S) % Bx::S - W;
      const int k = D == 3 ? qq / (Bx::S * Bx::S) - W : 0;
      ijk[u][0] = i;
      ijk[u][1] = j;
      ijk[u][2] = k;
      idx[u] = Bx::tix(i, j, k);
      li[u] = Gm::lin(i, j, k);
      at[u] = 0;
      kind[u] = 5;  // past the end
      if (q >= Bx::NPTS) continue;
      bool core = true;  // strictly inside the block: its own node
#pragma unroll
      for (int a = 0; a < D; ++a) core &= (ijk[u][a] >= 1 && ijk[u][a] <= B - 2);
      if (core) {
        kind[u] = 0;
        at[u] = own + li[u];
        continue;
      }
      int slot, m, off[3];
      region(ijk[u], slot, m, off);
      if (slot < 0) {
        set_err(pv, kErrGraded);
        kind[u] = 4;
        continue;
      }
      bool inner = true;
#pragma unroll
      for (int a = 0; a < D; ++a) inner &= (ijk[u][a] >= 0 && ijk[u][a] <= B - 1);
      const int sh = l1 - m;
      if (inner) {
        // the block's own node, or an edge node whose owner is another block
        // (a finer one, or an equal-level one holding it at its lower edge)
        if (slot == b.slot) {
          kind[u] = 0;
          at[u] = own + li[u];
        } else {
          kind[u] = 1;
          at[u] = ((int64_t)slot * nv) * pv.vs + Gm::lin(off[0] >> sh, off[1] >> sh, D == 3 ? off[2] >> sh : 0);
        }
        continue;
      }
      const bool node = ((off[0] | off[1] | off[2]) & ((1 << sh) - 1)) == 0;
      if (m >= b.lvl || node) {
        kind[u] = 2;
        at[u] = ((int64_t)slot * nv) * pv.vs + Gm::lin(off[0] >> sh, off[1] >> sh, D == 3 ? off[2] >> sh : 0);
      } else {
        if (m != b.lvl - 1) set_err(pv, kErrGraded);
        kind[u] = 3;
      }
    }
    for (int v = 0; v < nv; ++v) {
      TF val[U];
#pragma unroll
      for (int u = 0; u < U; ++u) val[u] = kind[u] <= 2 ? F[at[u] + (int64_t)v * pv.vs] : TF(0);
#pragma unroll
      for (int u = 0; u < U; ++u) {
        if (kind[u] == 5) continue;
        TT* t = tile + at_tile(v, idx[u]);
        if (kind[u] == 3) {
          if (D == 2 && scr) {
            // y from the scratch (X)
            const TT* c = scr + v * Bx::SCR + (ijk[u][0] + W);
            constexpr int st = Bx::S;
            const int e = ijk[u][1], fl = e >> 1;
            *t = (e & 1) ? dd4(c[(fl - 1 - Bx::CLO) * st], c[(fl - Bx::CLO) * st], c[(fl + 1 - Bx::CLO) * st],
                               c[(fl + 2 - Bx::CLO) * st])
                         : c[(fl - Bx::CLO) * st];
          } else {
            *t = predict_box<D, B, W, TT>(cbox + v * Bx::CBOX, ijk[u]);
          }
        } else if (kind[u] == 4) {
          *t = TT(0);
        } else {
          *t = to_tile<TT>(val[u]);
          if (kind[u] == 1 && commit) {
            const int64_t me = own + (int64_t)v * pv.vs + li[u];
            if (differs(F[me], val[u])) Fw[me] = val[u];
          }
        }
      }
    }
  }
}

// Stage plan of one active block, valid while the tree is fixed (the four RK
// stages of a step): INTS int32 per active position,
//   [0] slot, [1] level | tree << 8 | uniform << 30, [2 .. 2+D) block coordinates,
//   [2+D .. 2+D+NB) slots of the 3^d blocks at offsets (dx, dy, dz) in {-1,0,1}^d
//   (x fastest), the centre being the block itself.
// "uniform": every one of them is a leaf at the block's level, so each node of
// the ghost layer and each block-edge node has an equal-level owner, the block
// that holds it at its lower edge (Sec. 2.2, Sec. 2.5).
template <int D>
struct Plan {
  static constexpr int NB = D == 3 ? 27 : 9;
  static constexpr int INTS = D == 3 ? 32 : 16;
  static constexpr int NBO = 2 + D;  // offset of the neighbour slots
};

template <int D>
__device__ __forceinline__ BlockInfo plan_block(const int32_t* pl) {
  BlockInfo b;
  b.slot = pl[0];
  b.lvl = pl[1] & 255;
  b.tree = (pl[1] >> 8) & 0xffff;
#pragma unroll
  for (int a = 0; a < 3; ++a) b.c[a] = a < D ? pl[2 + a] : 0;
  return b;
}

template <typename T>
__device__ __forceinline__ T* smem_as(size_t offset_bytes) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  return reinterpret_cast<T*>(smem_raw + offset_bytes);
}

// Exclusive scan of n int2 pairs (in -> out) by one CTA of NT threads: PER
// consecutive pairs per thread per pass, a running carry between passes; the
// totals go to tot[0..1].  The input is read past L1 (written by other CTAs of
// the same grid).  Every thread of the CTA takes part.
template <int NT, int PER>
__device__ void cta_scan2(const int32_t* in, int32_t* out, int n, int32_t* tot) {
  __shared__ int2 wt[NT / 32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int2 carry = make_int2(0, 0);
  for (int base = 0; base < n; base += NT * PER) {
    int2 loc[PER];
    int2 s = make_int2(0, 0);
#pragma unroll
    for (int r = 0; r < PER; ++r) {
      const int i = base + threadIdx.x * PER + r;
      loc[r] = i < n ? __ldcg(reinterpret_cast<const int2*>(in) + i) : make_int2(0, 0);
      s.x += loc[r].x;
      s.y += loc[r].y;
    }
    int2 v = s;  // inclusive scan within the warp, then over the warp totals
    for (int o = 1; o < 32; o <<= 1) {
      const int x = __shfl_up_sync(0xffffffffu, v.x, o), y = __shfl_up_sync(0xffffffffu, v.y, o);
      if (lane >= o) { v.x += x; v.y += y; }
    }
    if (lane == 31) wt[w] = v;
    __syncthreads();
    if (w == 0) {
      int2 t = lane < NT / 32 ? wt[lane] : make_int2(0, 0);
      for (int o = 1; o < NT / 32; o <<= 1) {
        const int x = __shfl_up_sync(0xffffffffu, t.x, o), y = __shfl_up_sync(0xffffffffu, t.y, o);
        if (lane >= o) { t.x += x; t.y += y; }
      }
      if (lane < NT / 32) wt[lane] = t;
    }
    __syncthreads();
    if (w > 0) { v.x += wt[w - 1].x; v.y += wt[w - 1].y; }
    int2 run = make_int2(carry.x + v.x - s.x, carry.y + v.y - s.y);
#pragma unroll
    for (int r = 0; r < PER; ++r) {
      const int i = base + threadIdx.x * PER + r;
      if (i < n) { out[2 * i] = run.x; out[2 * i + 1] = run.y; }
      run.x += loc[r].x;
      run.y += loc[r].y;
    }
    carry.x += wt[NT / 32 - 1].x;
    carry.y += wt[NT / 32 - 1].y;
    __syncthreads();
  }
  if (threadIdx.x == 0 && tot) { tot[0] = carry.x; tot[1] = carry.y; }
}

// True in every thread of the CTA of the grid that finishes last; the writes
// of every other CTA of the grid are visible to it.  The caller resets
// ctas_done.
__device__ __forceinline__ bool last_cta_all(Counters* c) {
  __shared__ bool last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(&c->ctas_done, 1u) == gridDim.x - 1;
  __syncthreads();
  return last;
}

__device__ __forceinline__ void atomic_max_pos(double* addr, double v) {
  // non-negative doubles order like their bit patterns
  atomicMax(reinterpret_cast<unsigned long long*>(addr), (unsigned long long)__double_as_longlong(v));
}

}  // namespace mr
