// Launches single kernels of the library on hand-made blocks, for states that the
// public calls cannot reach (an owner table without owners, a wait that runs out), rounds
// chosen values with the library's helpers, and asks for what a kernel's launch shape
// leaves resident.  Built and called by
// tests/test_gpu_device_harness.py.
#include <vector>

#include "mr_adv2.cuh"
#include "mr_adv3.cuh"
#include "mr_det2.cuh"

using namespace mr;

namespace {

// One tree with one block (slot 0) at level `lvl`; its plan and owner table are the caller's.
struct OneBlock {
  std::vector<void*> mem;
  PoolView pv{};
  template <typename T>
  T* put(const std::vector<T>& h) {
    void* p = nullptr;
    cudaMalloc(&p, h.size() * sizeof(T));
    cudaMemcpy(p, h.data(), h.size() * sizeof(T), cudaMemcpyHostToDevice);
    mem.push_back(p);
    return (T*)p;
  }
  OneBlock(int dim, int B, int lvl, const std::vector<int32_t>& plan, const std::vector<int4>& regs) {
    int ni = 1;
    for (int a = 0; a < dim; ++a) ni *= B;
    pv.dim = dim; pv.Bs = B; pv.nvar = 1; pv.ntrees = 1; pv.cap = 1;
    pv.vs = (ni + 3) / 4 * 4;
    TreeDev td{};
    td.Jmin = 0; td.Jmax = 4; td.eps = 1.0; td.N = (int64_t)(B - 1) << 4;
    for (int l = 0; l <= kMaxLevel; ++l) td.cD[l] = td.cDf[l] = 1.0f;
    for (int a = 0; a < 3; ++a) td.rhs[a] = td.rhsf[a] = 1.0f;
    Counters c{};
    c.n_act = c.n_round = 1;
    c.first_round = 1;
    pv.trees = put(std::vector<TreeDev>{td});
    pv.cnt = put(std::vector<Counters>{c});
    pv.plan = put(plan);
    pv.regs = put(regs);
  }
  int err() {
    Counters c{};
    cudaMemcpy(&c, pv.cnt, sizeof(c), cudaMemcpyDeviceToHost);
    return c.err;
  }
  ~OneBlock() {
    for (void* p : mem) cudaFree(p);
  }
};

template <typename K, typename... A>
bool launch(K k, int threads, size_t smem, A... a) {
  cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  k<<<1, threads, smem>>>(a...);
  return cudaDeviceSynchronize() == cudaSuccess;
}

// Stage 0 of a block at level 2 whose ring no leaf covers: the owner table names no owner.
template <int D, typename TS, typename TY, int GT, int NW>
int ownerless(TS* y, int* err) {
  using PL = Plan<D>;
  std::vector<int32_t> plan(PL::INTS, -1);
  plan[0] = 0;
  plan[1] = 2;  // level 2, tree 0, not uniform
  for (int a = 0; a < D; ++a) plan[2 + a] = a & 1;
  OneBlock ob(D, 17, 2, plan, std::vector<int4>(reg_entries(D), make_int4(-1, -1, 0, 0)));
  const int n = (int)ob.pv.vs;
  TS* dy = ob.put(std::vector<TS>(y, y + n));
  TS* acc = ob.put(std::vector<TS>(n, TS(0)));
  TY* next = ob.put(std::vector<TY>(n, TY(0)));
  StageArgs sa{};
  bool ok;
  if constexpr (D == 2) {
    ok = launch(k_stage2<17, MR_RHS_ADV, TS, TY, TS, GT, NW, 0>, GT * NW, Stage2<17, TS, TY, GT, NW, 0>::BYTES, ob.pv,
                (const TS*)dy, dy, acc, next, 1, sa);
  } else {
    using SM = Stage3Smem<TY, TS>;
    ok = launch(k_stage3<TS, TY, TS, 0>, SM::NT, SM::BYTES, ob.pv, (const TS*)dy, dy, acc, next, sa);
  }
  cudaMemcpy(y, dy, n * sizeof(TS), cudaMemcpyDeviceToHost);
  *err = ob.err();
  return ok;
}

// One block at level 0, its own neighbour on every side.
template <int D>
std::vector<int32_t> periodic_plan() {
  using PL = Plan<D>;
  std::vector<int32_t> plan(PL::INTS, 0);
  plan[1] = 1 << 30;  // level 0, tree 0, uniform
  return plan;
}
// Runs stage ST (2D or 3D) or, with ST = -1, the 2D details on it; the block's fields
// in f: y, accumulator, the field read, the field written.
template <int D, int B, typename T, int GT, int NW, int ST>
int periodic(T* f, double* md, int* err) {
  OneBlock ob(D, B, 0, periodic_plan<D>(), std::vector<int4>(reg_entries(D), make_int4(-1, -1, 0, 0)));
  const int n = (int)ob.pv.vs;
  T* dev = ob.put(std::vector<T>(f, f + 4 * n));
  T *y = dev, *acc = dev + n, *src = dev + 2 * n, *next = dev + 3 * n;
  ob.pv.md = ob.put(std::vector<double>{*md});
  ob.pv.bmax = ob.put(std::vector<double>{*md});
  StageArgs sa{};
  bool ok;
  if constexpr (ST < 0) {
    ok = launch(k_details2<B, T, T, T>, Det2<B>::NT, Det2Smem<B, T, T, T>::BYTES, ob.pv, y);
  } else if constexpr (D == 2) {
    ok = launch(k_stage2<B, MR_RHS_ADV, T, T, T, GT, NW, ST>, GT * NW, Stage2<B, T, T, GT, NW, ST>::BYTES, ob.pv,
                (const T*)src, y, acc, next, 1, sa);
  } else {
    using SM = Stage3Smem<T, T>;
    ok = launch(k_stage3<T, T, T, ST>, SM::NT, SM::BYTES, ob.pv, (const T*)src, y, acc, next, sa);
  }
  cudaMemcpy(f, dev, 4 * n * sizeof(T), cudaMemcpyDeviceToHost);
  cudaMemcpy(md, ob.pv.md, sizeof(double), cudaMemcpyDeviceToHost);
  *err = ob.err();
  return ok;
}

__global__ void k_round(const double* d, float* f, double* w, double* q, int n) {
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    f[i] = f64_to_f32(d[i]);
    w[i] = f32_to_f64(f[i]);
    q[i] = sixteenth(d[i]);
  }
}
__global__ void k_widen(const float* f, double* d, int n) {
  for (int i = threadIdx.x; i < n; i += blockDim.x) d[i] = f32_to_f64(f[i]);
}

template <int B, typename TS>
int refine_occupancy() {
  using RC = RefineCfg<B, TS>;
  auto k = k_refine<B, TS>;
  cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)RC::BYTES);
  int n = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k, RC::NT, RC::BYTES);
  return n * RC::NT;
}

}  // namespace

extern "C" {

// form: 0 FP64, 1 FP32, 2 FP64 state with FP32 stages; warp: one warp per block (2D)
int ownerless_stage(int dim, int form, int warp, void* y, int* err) {
  double* d = (double*)y;
  float* f = (float*)y;
  if (dim == 2 && warp)
    return form == 0 ? ownerless<2, double, double, 32, 4>(d, err) : form == 1 ? ownerless<2, float, float, 32, 4>(f, err)
                                                                   : ownerless<2, double, float, 32, 4>(d, err);
  if (dim == 2)
    return form == 0   ? ownerless<2, double, double, 160, 1>(d, err)
           : form == 1 ? ownerless<2, float, float, 160, 1>(f, err)
                       : ownerless<2, double, float, 160, 1>(d, err);
  return form == 0 ? ownerless<3, double, double, 0, 0>(d, err) : form == 1 ? ownerless<3, float, float, 0, 0>(f, err)
                                                                : ownerless<3, double, float, 0, 0>(d, err);
}

// kernels that wait for bulk copies; f: four fields of a block (see periodic)
int periodic_block(int kernel, void* f, double* md, int* err) {
  float* s = (float*)f;
  double* d = (double*)f;
  switch (kernel) {
    case 0: return periodic<2, 17, float, 32, 4, 0>(s, md, err);
    case 1: return periodic<2, 17, float, 160, 1, 1>(s, md, err);
    case 2: return periodic<2, 33, double, 288, 1, 2>(d, md, err);
    case 3: return periodic<3, 17, float, 0, 0, 1>(s, md, err);
    case 4: return periodic<2, 17, float, 0, 0, -1>(s, md, err);
    default: return periodic<2, 33, double, 0, 0, -1>(d, md, err);
  }
}

// FP64 values d (n) rounded to FP32, widened again and divided by 16; FP32 values widened
int round_values(int n, const double* d, float* f, double* w, double* q) {
  OneBlock ob(2, 17, 0, {0}, {make_int4(0, 0, 0, 0)});
  double* dd = ob.put(std::vector<double>(d, d + n));
  float* df = ob.put(std::vector<float>(n));
  double *dw = ob.put(std::vector<double>(n)), *dq = ob.put(std::vector<double>(n));
  const bool ok = launch(k_round, 512, 0, (const double*)dd, df, dw, dq, n);
  cudaMemcpy(f, df, n * 4, cudaMemcpyDeviceToHost);
  cudaMemcpy(w, dw, n * 8, cudaMemcpyDeviceToHost);
  cudaMemcpy(q, dq, n * 8, cudaMemcpyDeviceToHost);
  return ok;
}
int widen_values(int n, const float* f, double* d) {
  OneBlock ob(2, 17, 0, {0}, {make_int4(0, 0, 0, 0)});
  float* df = ob.put(std::vector<float>(f, f + n));
  double* dd = ob.put(std::vector<double>(n));
  const bool ok = launch(k_widen, 512, 0, (const float*)df, dd, n);
  cudaMemcpy(d, dd, n * 8, cudaMemcpyDeviceToHost);
  return ok;
}

// threads per SM of the 2D refinement kernel
int refine_threads_per_sm(int Bs, int fp64) {
  if (Bs == 17) return fp64 ? refine_occupancy<17, double>() : refine_occupancy<17, float>();
  return fp64 ? refine_occupancy<33, double>() : refine_occupancy<33, float>();
}

}  // extern "C"
