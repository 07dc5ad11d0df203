// Persistent batched RK stage (FP32 operator): one cooperative launch per RK stage for
// every member of a batch, whatever its order (P = 1 .. 6).
//
// Each block of kPersistThreads threads walks the phase-A work items of all members
// (blocks of E_P consecutive elements of a member, E_P = the elements of order P that
// fill the block), meets every other block at a grid barrier, then walks the phase-B items
// of all members.  The per-item arithmetic is the single-mesh kernels' (volume_block,
// surface_block), so a member computes what it computes alone; only the blocking differs.
// The grid holds as many blocks as are resident at once (a cooperative launch), and the
// barrier's wait is bounded (about a second): on expiry the block sets the batch's error
// flag and returns.  The launches of a step form one CUDA graph, after a reset of the
// barrier's counter.
#include "dg_aux.h"
#include "dg_barrier.cuh"
#include "dg_launch.cuh"

namespace dgnn {

constexpr int kPersistThreads = 384;
// Elements per work item of order P, at most (P = 3, 16 threads per element: see persist_elems_of).
__host__ __device__ constexpr int persist_elems(int P) {
  return kPersistThreads / (use_rows4(P, sizeof(float), false) ? 16 : (P + 1) * (P + 1) * (P + 1));
}

struct PersistTable {
  BatchTable<float> tb;   // block_start: first work item of each member (the same items in both phases)
  int P[kMaxBatch];
  unsigned* bar;          // [0] arrivals at the barrier, [1] its generation
};

template <int SRC, int MODE>
__global__ void __launch_bounds__(kPersistThreads, 2) k_batch_persistent(const __grid_constant__ PersistTable pt) {
  const BatchTable<float>& tb = pt.tb;
  const int items = tb.block_start[tb.n];
  for (int item = blockIdx.x; item < items; item += gridDim.x) {
    const int i = batch_instance(tb.block_start, tb.n, item);
    const int blk = item - tb.block_start[i];
    switch (pt.P[i]) {
#define DG_PA(PP)                                                                                   \
  case PP:                                                                                          \
    volume_phase<PP, float, SRC>(blk, tb.a[i].q, tb.qs[i], tb.rv[i], tb.vt[i], tb.C[i]);            \
    break;
      DG_PA(1) DG_PA(2) DG_PA(3) DG_PA(4) DG_PA(5) DG_PA(6)
#undef DG_PA
    }
    __syncthreads();   // the next item reuses the shared memory
  }
  if (!grid_barrier_bounded(pt.bar, gridDim.x)) {
    if (threadIdx.x == 0 && tb.err[0]) atomicExch(tb.err[0], 1);
    return;
  }
  for (int item = blockIdx.x; item < items; item += gridDim.x) {
    const int i = batch_instance(tb.block_start, tb.n, item);
    const int blk = item - tb.block_start[i];
    switch (pt.P[i]) {
#define DG_PB(PP)                                                                                   \
  case PP:                                                                                          \
    surface_prologue<PP, float, false>(blk, tb.C[i].E, tb.C[i]);                                    \
    surface_block<PP, float, MODE>(blk, tb.C[i].E, tb.a[i], Forcing{}, tb.C[i], tb.rk[i]);          \
    break;
      DG_PB(1) DG_PB(2) DG_PB(3) DG_PB(4) DG_PB(5) DG_PB(6)
#undef DG_PB
    }
    __syncthreads();
  }
}

namespace {

// Shared memory of a work item of E elements of order P (the larger phase).
size_t persist_smem_p(int P, int E) {
  switch (P) {
#define DG_SM(PP) \
  case PP: return std::max(volume_smem<PP, float, false>(E, false), surface_smem_bytes<PP, float>(E));
    DG_SM(1) DG_SM(2) DG_SM(3) DG_SM(4) DG_SM(5) DG_SM(6)
#undef DG_SM
  }
  return 0;
}

// Elements per work item of order P, `elems` of them in the launch.  P = 3: a full block of rows
// (24 elements) leaves most of the chip idle on small meshes, so as many as give every block
// of the grid an item, and at least a node per thread of phase B.  us per RK3 step with 24 /
// 6 / one item per block: 8^3 83 / 49 / 54, twelve 5^3 88 / 63 / 70, 16^3 + 12^3 128 / 174 / 112.
int persist_elems_of(int P, int elems, int grid) {
  if (!use_rows4(P, sizeof(float), false)) return persist_elems(P);
  const int nodes = kPersistThreads / ((P + 1) * (P + 1) * (P + 1));
  return std::max(nodes, std::min(persist_elems(P), (elems + grid - 1) / grid));
}

using PersistKernel = void (*)(const PersistTable);

PersistKernel persist_kernel(int k) {
  return k == 0 ? k_batch_persistent<0, 2> : k == 1 ? k_batch_persistent<1, 3> : k_batch_persistent<1, 4>;
}

}  // namespace

// Constant-memory tables of this unit's kernels (see upload_const_D).
cudaError_t prepare_batch_persist_constants() { return upload_const_D(); }

bool batch_persistent_ok(int P) { return P >= 1 && P <= 6; }

cudaError_t batch_persistent_prepare(const int* orders, int n, int* grid_out) {
  size_t smem = 0;
  for (int i = 0; i < n; ++i) smem = std::max(smem, persist_smem_p(orders[i], persist_elems(orders[i])));
  int grid = 0;
  for (int k = 0; k < 3; ++k) {
    PersistKernel kern = persist_kernel(k);
    cudaError_t e = set_smem(kern, smem);
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kPersistThreads, smem);
    if (e != cudaSuccess) return e;
    int dev = 0, sms = 0;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    const int g = per_sm * sms;
    grid = (k == 0) ? g : std::min(grid, g);
  }
  if (grid < 1) return cudaErrorInvalidConfiguration;
  *grid_out = grid;
  return cudaSuccess;
}

cudaError_t batch_persistent_stage(dg_ctx* const* ctx, double* const* q, const double* dt, int n, int k,
                                   const RkStage& rk, unsigned* bar, int grid, cudaStream_t st) {
  if (n < 1 || n > kMaxBatch) return cudaErrorInvalidValue;
  PersistTable pt;
  fill_batch<float>(&pt.tb, ctx, q, dt, n, k, rk);
  // work items of E_P elements per member, whatever blocking the member uses alone
  int items = 0, elems[kMaxP + 1] = {};
  size_t smem = 0;
  for (int i = 0; i < n; ++i) {
    if (!batch_persistent_ok(ctx[i]->P)) return cudaErrorInvalidValue;
    elems[ctx[i]->P] += owned_elems(ctx[i]);
  }
  for (int i = 0; i < n; ++i) {
    const int P = ctx[i]->P, E = persist_elems_of(P, elems[P], grid);
    smem = std::max(smem, persist_smem_p(P, E));   // no more than it needs: the rest is L1
    pt.P[i] = P;
    pt.tb.C[i].E = E;
    pt.tb.block_start[i] = items;
    items += (owned_elems(ctx[i]) + E - 1) / E;
  }
  pt.tb.block_start[n] = items;
  pt.bar = bar;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(std::min(grid, items));
  cfg.blockDim = dim3(kPersistThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, persist_kernel(k), pt);
}

}  // namespace dgnn
