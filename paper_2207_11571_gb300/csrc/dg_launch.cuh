// Host launchers of the operator kernels for one operator precision T; included by
// dg_kernels_f32.cu and dg_kernels_f64.cu so that the two precisions compile in
// parallel translation units.
#pragma once

#include <algorithm>
#include <type_traits>

#include "dg_kernels.cuh"

namespace dgnn {

// Elements a launch processes: the whole mesh, or a slab's own layers.
inline int owned_elems(const dg_ctx* c) { return c->e_end - c->e_begin; }

// Where phase A of a launch of `nodes` nodes lets the next launch in.  Let in early, its blocks
// fill whichever SMs drain first instead of spreading over the chip: phase B at 9^3/P3 in FP64
// 704 -> 250 us per RK3 step with the release at the end of phase A's blocks, 9^3/P4 44.6 -> 35.6,
// 16^3/P3 50.2 -> 48.4.  Only the small blocks of a small mesh (512 nodes per SM) leave room for
// both phases, and the launch latency saved counts there: 10^3/P3 32.0 -> 29.1, 8^3/P2 23.7 -> 22.3.
template <typename T>
bool release_early(int P, long long nodes) {
  return std::is_same<T, float>::value && P <= 3 && nodes <= kSMs * 512;
}

template <typename T>
OpConst<T> make_const(const dg_ctx* c) {
  OpConst<T> k;
  k.K = c->K;
  k.E = c->geom.E;
  k.nel = c->e_end;
  k.Kz = c->Kz;
  k.e_begin = c->e_begin;
  k.N = c->N;
  const Phys& ph = c->phys;
  k.gm1 = T(ph.gamma - 1.0);
  k.rho_ref = T(ph.rho_ref);
  k.theta_ref = T(ph.theta_ref);
  k.Hc = T(ph.Hc);
  k.s2h = T(c->geom.two_over_h);
  k.winv = T(c->geom.winv);
  k.mu = T(ph.mu);
  k.lam = T(ph.lam);
  k.csd2 = T(ph.csd2);
  k.lam_t = T(ph.lam_t);
  k.les = ph.les;
  k.drho_ref = ph.rho_ref;
  k.dE_ref = ph.E_ref;
  k.early = release_early<T>(c->P, c->N);
  k.feat = c->feat_out;
  for (int i = 0; i < kMaxN1 * kMaxN1; ++i) k.D[i] = T(c->geom.D[i]);
  return k;
}

// Fills this translation unit's constant-memory derivative matrices (c_D32) on the
// current device, once per device.  Synchronous: called from dg_create, outside any
// stream capture.
static cudaError_t upload_const_D() {
  static bool done[64] = {};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev >= 0 && dev < 64 && done[dev]) return cudaSuccess;
  static float2 h[kMaxP + 1][kMaxN1 * kMaxN1];
  for (int P = 1; P <= kMaxP; ++P) {
    Basis1D b;
    if (build_basis(P, &b) != 0) return cudaErrorInvalidValue;
    for (int i = 0; i < (P + 1) * (P + 1); ++i) h[P][i] = make_float2((float)b.D[i], (float)b.D[i]);
  }
  e = cudaMemcpyToSymbol(c_D32, h, sizeof(h));
  if (e == cudaSuccess && dev >= 0 && dev < 64) done[dev] = true;
  return e;
}

// Launch with programmatic stream serialization (the kernels wait for their predecessor
// themselves, see pdl_wait in dg_kernels.cuh).
template <typename... KArgs, typename... Args>
cudaError_t launch_pdl(void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, std::forward<Args>(args)...);
}

template <typename K>
cudaError_t set_smem(K kern, size_t smem) {
  if (smem > 48 * 1024) return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  return cudaSuccess;
}

// Phase A of one mesh.  src 0: the stage state from q, written to c->qf; else: the stage
// state in c->cur.
template <int P, typename T, int SRC, bool CUBE, bool FEAT, bool SPLIT, bool BESIDE>
cudaError_t volume_launch(const dg_ctx* c, const double* q, cudaStream_t st) {
  const int E = CUBE ? kCubeElems : c->geom.E;
  const size_t smem = volume_smem<P, T, SPLIT>(E, CUBE);
  auto kern = k_volume<P, T, SRC, CUBE, FEAT, SPLIT, BESIDE>;
  cudaError_t e = set_smem(kern, smem);
  if (e != cudaSuccess) return e;
  const int h = c->K / 2;
  const int grid = CUBE ? h * h * h : (owned_elems(c) + E - 1) / E;
  return launch_pdl(kern, dim3(grid), dim3(volume_threads<P, T, SPLIT>(E)), smem, st, q, static_cast<T*>(SRC == 0 ? c->qf : c->cur),
                    static_cast<T*>(c->rv), static_cast<T*>(c->vt), make_const<T>(c));
}

// With a forcing network (features at P = 3, see nn_phase_a_features) an FP64 launch writes
// the features of the state it forms; an FP32 launch, whose state was formed with its
// features before, runs beside the network.
template <int P, typename T, int SRC, bool CUBE, bool SPLIT>
cudaError_t volume_shape(const dg_ctx* c, const double* q, cudaStream_t st) {
  constexpr bool f64 = std::is_same<T, double>::value;
  if constexpr (P == 3 && (f64 || SRC == 1)) {
    if (f64 ? c->feat_out.out != nullptr : c->beside_forcing)
      return volume_launch<P, T, SRC, CUBE, f64, SPLIT, !f64>(c, q, st);
  }
  return volume_launch<P, T, SRC, CUBE, false, SPLIT, false>(c, q, st);
}

template <int P, typename T, int SRC, bool SPLIT>
cudaError_t volume_p(const dg_ctx* c, const double* q, cudaStream_t st) {
  if constexpr (cube_ok(P) && !SPLIT) {
    if (c->geom.cube) return volume_shape<P, T, SRC, true, false>(c, q, st);
  }
  return volume_shape<P, T, SRC, false, SPLIT>(c, q, st);
}

// The stage state in a pass of its own (c->cur is then c->qf), where the order has one.
template <int P, typename T, bool SPLIT>
cudaError_t state_p(const dg_ctx* c, const double* q, bool* done, cudaStream_t st) {
  *done = use_rows4(P, sizeof(T), SPLIT);
  if constexpr (use_rows4(P, sizeof(T), SPLIT))
    return launch_pdl(k_state4<T>, dim3((c->nel + kStateElems - 1) / kStateElems), dim3(256), 0, st, q,
                      static_cast<T*>(c->qf), c->nel, make_const<T>(c));
  return cudaSuccess;
}

template <int P, typename T, bool SPLIT>
cudaError_t volume_src(const dg_ctx* c, const double* q, int src, cudaStream_t st) {
  bool formed = src != 0;
  if (!formed) {
    const cudaError_t e = state_p<P, T, SPLIT>(c, q, &formed, st);
    if (e != cudaSuccess) return e;
  }
  if constexpr (std::is_same<T, float>::value) {
    if (formed) return volume_p<P, T, 1, SPLIT>(c, q, st);
  }
  if constexpr (!use_rows4(P, sizeof(T), SPLIT)) return volume_p<P, T, 0, SPLIT>(c, q, st);
  return cudaErrorInvalidValue;
}

#define DG_FOR_EACH_P(CALL)        \
  switch (c->P) {                  \
    case 1: return CALL(1);        \
    case 2: return CALL(2);        \
    case 3: return CALL(3);        \
    case 4: return CALL(4);        \
    case 5: return CALL(5);        \
    case 6: return CALL(6);        \
    case 7: return CALL(7);        \
    case 8: return CALL(8);        \
  }                                \
  return cudaErrorInvalidValue;

template <typename T, bool SPLIT>
cudaError_t volume_t(const dg_ctx* c, const double* q, int src, cudaStream_t st) {
#define DG_V(PP) volume_src<PP, T, SPLIT>(c, q, src, st)
  DG_FOR_EACH_P(DG_V)
#undef DG_V
}

template <typename T>
cudaError_t state_t(const dg_ctx* c, const double* q, bool* done, cudaStream_t st) {
#define DG_P(PP) state_p<PP, T, false>(c, q, done, st)
  DG_FOR_EACH_P(DG_P)
#undef DG_P
}

// Operands of phase B of mode `mode` (see k_surface).
template <typename T>
SurfArgs<T> surf_args(const dg_ctx* c, double* q, double* dqdt) {
  SurfArgs<T> a;
  a.q = q;
  a.s = static_cast<const T*>(c->cur);
  a.rv = static_cast<const T*>(c->rv);
  a.vt = static_cast<const T*>(c->vt);
  a.dqdt = dqdt;
  a.g = static_cast<T*>(c->g);
  a.x = static_cast<T*>(c->qf);
  a.y = static_cast<T*>(c->qy);
  a.dlt = c->dlt;
  return a;
}

template <int P, typename T, int MODE, int E, int THREADS, bool CUBE, bool FEAT = false>
cudaError_t surface_launch(const dg_ctx* c, double* q, double* dqdt, const Forcing& f, const RkArgs<T>& rk,
                           cudaStream_t st) {
  if constexpr (P == 3 && std::is_same<T, float>::value && !FEAT && (MODE == 2 || MODE == 3 || MODE == 5)) {
    if (c->feat_out.out) return surface_launch<P, T, MODE, E, THREADS, CUBE, true>(c, q, dqdt, f, rk, st);
  }
  const size_t smem = surface_smem_bytes<P, T>(E);
  auto kern = k_surface<P, T, MODE, E, THREADS, CUBE, FEAT>;
  cudaError_t e = set_smem(kern, smem);
  if (e != cudaSuccess) return e;
  return launch_pdl(kern, dim3((owned_elems(c) + E - 1) / E), dim3(THREADS), smem, st, surf_args<T>(c, q, dqdt), f,
                    make_const<T>(c), rk);
}

// Elements and threads of phase B's blocks for n elements in a launch: f(E, THREADS) as
// integral constants.
// FP64: few elements per block at P = 2 and 3, so that the FP64 pipes of all SMs have an equal
// share.  us per RK3 step, P = 3, 2 x 96 / 8 x 128 elements x threads: 8^3 130 / 196, 11^3
// 328 / 413, 12^3 360 / 414, 16^3 811 / 867; a batch of 8^3, 6^3 and 4^3 222 / 683.
// P = 3 in FP32: the smallest block whose launch is still one wave (1024 threads per SM at
// 64 registers), so that every SM has its share of a small mesh; large meshes want many
// elements per block.  us per RK3 step with 2 x 192 / 2 x 96 / 4 x 128 / 8 x 128 elements x
// threads: 8^3 28.4 / 29.8 / 29.9 / 31.9, 14^3 44.9 / 41.0 / 42.1 / 42.7, 16^3 53.8 / 49.5 /
// 48.5 / 49.3, 32^3 345 / 295 / 294 / 290.
// P >= 6: a block per element.  Where every element has an SM to itself, a thread per node, as
// nothing else hides the block's latency (us per RK3 step against the general threads: FP32 3^3/P7
// 30.4 -> 23.1, 4^3/P6 22.7 -> 21.4, 5^3/P8 40.7 -> 29.6; FP64 5^3/P8 400 -> 316, 5^3/P6 207 -> 154);
// with two elements per SM the general threads overlap better (7^3/P8 61.0 against 69.6).
template <int N>
using Int = std::integral_constant<int, N>;
template <int P, typename T, typename F>
auto with_surf_block(int n, F f) {
  if constexpr (std::is_same<T, double>::value) {
    if constexpr (P == 3) return f(Int<2>{}, Int<96>{});
    if constexpr (P == 2) return f(Int<4>{}, Int<192>{});
  }
  if constexpr (P == 3 && std::is_same<T, float>::value) {
    constexpr int kWave = kSMs * 1024;   // threads
    if (n <= kWave / 192 * 2) return f(Int<2>{}, Int<192>{});
    if (n <= kWave / 96 * 2) return f(Int<2>{}, Int<96>{});
    if (n <= kWave / 128 * 4) return f(Int<4>{}, Int<128>{});
  }
  if constexpr (P >= 6) {
    if (n <= kSMs) return f(Int<1>{}, Int<max_threads_for(P)>{});
  }
  return f(Int<surf_elems(P)>{}, Int<surf_threads(P)>{});
}

template <int P, typename T, int MODE>
cudaError_t surface_p(const dg_ctx* c, double* q, double* dqdt, const Forcing& f, const RkArgs<T>& rk,
                      cudaStream_t st) {
  const int n = owned_elems(c);
  // FP64: cubes where they pay (two per SM at least) and tile the mesh (a slab's layers:
  // rows); the twelve internal faces' terms are formed once for both sides, to the same bits
  // as per side.  us per RK3 step, P = 3, cubes / rows: 8^3 164 / 130, 12^3 365 / 360, 16^3
  // 770 / 811.
  if constexpr (surf_cube(P, sizeof(T))) {
    if (!c->part && c->K % 2 == 0 && n >= 2 * kSMs * kCubeElems)
      return surface_launch<P, T, MODE, kCubeElems, surf_threads_cube(P), true>(c, q, dqdt, f, rk, st);
  }
  return with_surf_block<P, T>(n, [&](auto E, auto threads) {
    return surface_launch<P, T, MODE, E.value, threads.value, false>(c, q, dqdt, f, rk, st);
  });
}

// FP64 operator: modes 0 (dq/dt) and 1 (FP64 RK stage).  FP32 operator: modes 0, 2, 3, 4.
template <int P, typename T>
cudaError_t surface_mode(const dg_ctx* c, double* q, double* dqdt, const Forcing& f, int mode, const RkArgs<T>& rk,
                         cudaStream_t st) {
  if constexpr (std::is_same<T, float>::value) {
    switch (mode) {
      case 0: return surface_p<P, T, 0>(c, q, dqdt, f, rk, st);
      case 2: return surface_p<P, T, 2>(c, q, dqdt, f, rk, st);
      case 3: return surface_p<P, T, 3>(c, q, dqdt, f, rk, st);
      case 4: return surface_p<P, T, 4>(c, q, dqdt, f, rk, st);
      case 5: return surface_p<P, T, 5>(c, q, dqdt, f, rk, st);
    }
  } else {
    switch (mode) {
      case 0: return surface_p<P, T, 0>(c, q, dqdt, f, rk, st);
      case 1: return surface_p<P, T, 1>(c, q, dqdt, f, rk, st);
    }
  }
  return cudaErrorInvalidValue;
}

template <typename T>
RkArgs<T> rk_args(const RkStage& k, double dt) {
  return RkArgs<T>{T(k.A), T(k.B), T(dt), T(k.invB1), T(k.wc)};
}

template <typename T>
cudaError_t surface_t(const dg_ctx* c, double* q, double* dqdt, const Forcing& f, int mode, const RkStage& k, double dt,
                      cudaStream_t st) {
  const RkArgs<T> rk = rk_args<T>(k, dt);
#define DG_S(PP) surface_mode<PP, T>(c, q, dqdt, f, mode, rk, st)
  DG_FOR_EACH_P(DG_S)
#undef DG_S
}

// ---------------------------------------------------------------------------------------
// Batched RK stage: one phase-A and one phase-B launch for all instances of order P.
// Instances must share the operator precision T and the elements-per-block E.

// Elements per phase-B block of a launch of n elements of order P in all.
template <typename T>
int surf_block_elems(int P, int n) {
  const auto elems = [](auto E, auto) { return (int)E.value; };
  switch (P) {
    case 1: return with_surf_block<1, T>(n, elems);
    case 2: return with_surf_block<2, T>(n, elems);
    case 3: return with_surf_block<3, T>(n, elems);
    case 4: return with_surf_block<4, T>(n, elems);
    case 5: return with_surf_block<5, T>(n, elems);
    case 6: return with_surf_block<6, T>(n, elems);
    case 7: return with_surf_block<7, T>(n, elems);
  }
  return with_surf_block<8, T>(n, elems);
}

template <typename T>
void fill_batch(BatchTable<T>* tb, dg_ctx* const* ctx, double* const* q, const double* dt, int n, int k,
                const RkStage& rk) {
  tb->n = n;
  int blocks = 0, surf = 0, state = 0, elems = 0;
  long long nodes = 0;
  for (int i = 0; i < n; ++i) {
    elems += owned_elems(ctx[i]);
    nodes += ctx[i]->N;
  }
  tb->early = release_early<T>(ctx[0]->P, nodes);
  const int E = surf_block_elems<T>(ctx[0]->P, elems);
  for (int i = 0; i < n; ++i) {
    const dg_ctx* c = ctx[i];
    tb->block_start[i] = blocks;
    blocks += (owned_elems(c) + c->geom.E - 1) / c->geom.E;
    tb->surf_start[i] = surf;
    surf += (owned_elems(c) + E - 1) / E;
    tb->state_start[i] = state;
    state += (c->nel + kStateElems - 1) / kStateElems;
    tb->qs[i] = static_cast<T*>(stage_buffer(c, k));
    tb->rv[i] = static_cast<T*>(c->rv);
    tb->vt[i] = static_cast<T*>(c->vt);
    tb->a[i] = surf_args<T>(c, q[i], nullptr);
    tb->a[i].s = tb->qs[i];
    tb->rk[i] = rk_args<T>(rk, dt[i]);
    tb->C[i] = make_const<T>(c);
    tb->err[i] = c->err_dev;
  }
  tb->block_start[n] = blocks;
  tb->surf_start[n] = surf;
  tb->state_start[n] = state;
}

// The phase-B kernel of stage k.
template <int P, typename T, int E, int THREADS>
auto batch_surface(int k) {
  if constexpr (std::is_same<T, float>::value)
    return k == 0 ? k_surface_batch<P, T, 2, E, THREADS>
                  : k == 1 ? k_surface_batch<P, T, 3, E, THREADS> : k_surface_batch<P, T, 4, E, THREADS>;
  else return k_surface_batch<P, T, 1, E, THREADS>;
}

// Stage k of the RK3 step: the same source and mode sequence as the single-mesh path
// (FP32 operator: sources 0, 1, 1 and modes 2, 3, 4; FP64 operator: source 0, mode 1), and
// its rules for phase B's blocks and for the release, over all members.
template <int P, typename T>
cudaError_t batch_stage_p(const BatchTable<T>& tb, int elems, int E, int k, cudaStream_t st) {
  void (*kg)(const BatchTable<T>);
  if constexpr (std::is_same<T, float>::value) {
    if constexpr (use_rows4(P, sizeof(T), false)) kg = k_volume_batch<P, T, 1>;
    else kg = k == 0 ? k_volume_batch<P, T, 0> : k_volume_batch<P, T, 1>;
  } else {
    kg = k_volume_batch<P, T, 0>;
  }
  cudaError_t e;
  if constexpr (use_rows4(P, sizeof(T), false)) {
    if (k == 0 && (e = launch_pdl(k_state4_batch<T>, dim3(tb.state_start[tb.n]), dim3(256), 0, st, tb)) != cudaSuccess)
      return e;
  }
  if ((e = launch_pdl(kg, dim3(tb.block_start[tb.n]), dim3(volume_threads<P, T, false>(E)),
                      volume_smem<P, T, false>(E, false), st, tb)) != cudaSuccess)
    return e;
  return with_surf_block<P, T>(elems, [&](auto SE, auto threads) {
    return launch_pdl(batch_surface<P, T, SE.value, threads.value>(k), dim3(tb.surf_start[tb.n]), dim3(threads.value),
                      surface_smem_bytes<P, T>(SE.value), st, tb);
  });
}

// Dynamic shared-memory attributes of the batched kernels of order P at E elements per
// block of phase A; set before any launch (and outside stream capture).
template <int P, typename T>
cudaError_t batch_prepare_p(int elems, int E) {
  const size_t gs = volume_smem<P, T, false>(E, false);
  cudaError_t e = cudaSuccess;
  if constexpr (!use_rows4(P, sizeof(T), false)) e = set_smem(k_volume_batch<P, T, 0>, gs);
  if constexpr (std::is_same<T, float>::value) {
    if (e == cudaSuccess) e = set_smem(k_volume_batch<P, T, 1>, gs);
  }
  return with_surf_block<P, T>(elems, [&](auto SE, auto threads) {
    for (int k = 0; k < 3 && e == cudaSuccess; ++k)
      e = set_smem(batch_surface<P, T, SE.value, threads.value>(k), surface_smem_bytes<P, T>(SE.value));
    return e;
  });
}

template <typename T>
cudaError_t batch_prepare_t(int P, int elems, int E) {
  switch (P) {
    case 1: return batch_prepare_p<1, T>(elems, E);
    case 2: return batch_prepare_p<2, T>(elems, E);
    case 3: return batch_prepare_p<3, T>(elems, E);
    case 4: return batch_prepare_p<4, T>(elems, E);
    case 5: return batch_prepare_p<5, T>(elems, E);
    case 6: return batch_prepare_p<6, T>(elems, E);
    case 7: return batch_prepare_p<7, T>(elems, E);
    case 8: return batch_prepare_p<8, T>(elems, E);
  }
  return cudaErrorInvalidValue;
}

template <typename T>
cudaError_t batch_stage_t(int P, dg_ctx* const* ctx, double* const* q, const double* dt, int n, int k,
                          const RkStage& rk, cudaStream_t st) {
  if (n < 1 || n > kMaxBatch) return cudaErrorInvalidValue;
  BatchTable<T> tb;
  fill_batch<T>(&tb, ctx, q, dt, n, k, rk);
  const int E = ctx[0]->geom.E;
  int elems = 0;
  for (int i = 0; i < n; ++i) elems += owned_elems(ctx[i]);
  switch (P) {
    case 1: return batch_stage_p<1, T>(tb, elems, E, k, st);
    case 2: return batch_stage_p<2, T>(tb, elems, E, k, st);
    case 3: return batch_stage_p<3, T>(tb, elems, E, k, st);
    case 4: return batch_stage_p<4, T>(tb, elems, E, k, st);
    case 5: return batch_stage_p<5, T>(tb, elems, E, k, st);
    case 6: return batch_stage_p<6, T>(tb, elems, E, k, st);
    case 7: return batch_stage_p<7, T>(tb, elems, E, k, st);
    case 8: return batch_stage_p<8, T>(tb, elems, E, k, st);
  }
  return cudaErrorInvalidValue;
}

}  // namespace dgnn
