// Auxiliary kernels: Taylor-Green initial state (Sec. 3.1, Eq. 11), the filter G
// (Eq. 2, Sec. 2.6), FP64 integral diagnostics (Sec. 2.4, Eq. 9) and the training
// pairs of Algorithm 1 (Sec. 2.1).
#include <algorithm>
#include <cmath>

#include "dg_aux.h"
#include "dg_device.cuh"

namespace dgnn {

// ---------------------------------------------------------------- Taylor-Green vortex

__global__ void k_init_tgv(double* __restrict__ q, const double* __restrict__ pert, NodeGeom ng, double p0,
                           double gamma) {
  const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (t >= ng.N) return;
  const int n = ng.n, np = n * n * n;
  const int e = (int)(t / np), node = (int)(t - (long long)e * np);
  const int i = node % n, j = (node / n) % n, k = node / (n * n);
  const int K = ng.K;
  const int ex = e % K, ey = (e / K) % K, ez = (e / (K * K) + ng.z_off) % K;
  const double x = -M_PI + (ex + 0.5 * (ng.xi[i] + 1.0)) * ng.h;
  const double y = -M_PI + (ey + 0.5 * (ng.xi[j] + 1.0)) * ng.h;
  const double z = -M_PI + (ez + 0.5 * (ng.xi[k] + 1.0)) * ng.h;
  double sx, cx, sy, cy, sz, cz;
  sincos(x, &sx, &cx);
  sincos(y, &sy, &cy);
  sincos(z, &sz, &cz);
  const double u = sx * cy * cz, v = -cx * sy * cz;
  const double p = p0 + (cos(2.0 * x) + cos(2.0 * y)) * (cos(2.0 * z) + 2.0) / 16.0;
  double qv[5] = {1.0, u, v, 0.0, p / (gamma - 1.0) + 0.5 * (u * u + v * v)};
  for (int c = 0; c < 5; ++c) {
    double val = qv[c];
    if (pert) val += pert[c * ng.N + t];
    q[c * ng.N + t] = val;
  }
}

cudaError_t launch_init_tgv(const dg_ctx* c, double* q, const double* pert, cudaStream_t st) {
  NodeGeom ng = node_geom(c);
  const double p0 = 1.0 / (c->opts.gamma * c->Mach * c->Mach);
  const int threads = 256;
  const long long blocks = (c->N + threads - 1) / threads;
  k_init_tgv<<<(unsigned)blocks, threads, 0, st>>>(q, pert, ng, p0, c->opts.gamma);
  return cudaGetLastError();
}

// ---------------------------------------------------------------- filter G

// One block per element: for each variable, apply the 1D filter along x, y, z.
__global__ void k_project(const double* __restrict__ qh, double* __restrict__ ql, int nel, int nh, int nl,
                          long long Nh, long long Nl, const double* __restrict__ Gm) {
  __shared__ double sG[kMaxN1 * kMaxN1];
  __shared__ double a[kMaxN1 * kMaxN1 * kMaxN1];
  __shared__ double b[kMaxN1 * kMaxN1 * kMaxN1];
  const int e = blockIdx.x;
  if (e >= nel) return;
  const int nph = nh * nh * nh, npl = nl * nl * nl;
  for (int t = threadIdx.x; t < nl * nh; t += blockDim.x) sG[t] = Gm[t];
  for (int v = 0; v < 5; ++v) {
    __syncthreads();
    for (int t = threadIdx.x; t < nph; t += blockDim.x) a[t] = qh[v * Nh + (long long)e * nph + t];
    __syncthreads();
    // x pass: b[(ii, j, k)] (ii < nl, j, k < nh), x fastest
    for (int t = threadIdx.x; t < nl * nh * nh; t += blockDim.x) {
      const int ii = t % nl, j = (t / nl) % nh, k = t / (nl * nh);
      double s = 0.0;
      for (int m = 0; m < nh; ++m) s += sG[ii * nh + m] * a[m + nh * (j + nh * k)];
      b[t] = s;
    }
    __syncthreads();
    // y pass: a[(ii, jj, k)]
    for (int t = threadIdx.x; t < nl * nl * nh; t += blockDim.x) {
      const int ii = t % nl, jj = (t / nl) % nl, k = t / (nl * nl);
      double s = 0.0;
      for (int m = 0; m < nh; ++m) s += sG[jj * nh + m] * b[ii + nl * (m + nh * k)];
      a[t] = s;
    }
    __syncthreads();
    // z pass
    for (int t = threadIdx.x; t < npl; t += blockDim.x) {
      const int ii = t % nl, jj = (t / nl) % nl, kk = t / (nl * nl);
      double s = 0.0;
      for (int m = 0; m < nh; ++m) s += sG[kk * nh + m] * a[ii + nl * (jj + nl * m)];
      ql[v * Nl + (long long)e * npl + t] = s;
    }
  }
}

cudaError_t launch_project(const dg_ctx* hi, const dg_ctx* lo, const double* qh, double* ql, const double* Gdev,
                           cudaStream_t st) {
  k_project<<<hi->nel, 256, 0, st>>>(qh, ql, hi->nel, hi->n, lo->n, hi->N, lo->N, Gdev);
  return cudaGetLastError();
}

// k_project is a transform from nh to nl nodes per direction for any nh, nl <= 9 (its
// scratch holds every intermediate of either direction), so it also interpolates upwards.
cudaError_t launch_prolong(const dg_ctx* lo, const dg_ctx* hi, const double* ql, double* qh, const double* Idev,
                           cudaStream_t st) {
  k_project<<<lo->nel, 256, 0, st>>>(ql, qh, lo->nel, lo->n, hi->n, lo->N, hi->N, Idev);
  return cudaGetLastError();
}

// ---------------------------------------------------------------- diagnostics

// 1 / x by one Newton-Raphson step of third order, r (1 + e + e^2) with e = 1 - x r, from the
// FP32 reciprocal (|e| < 2^-22): three FP64 operations, the last rounding the only one that
// counts.  x outside FP32's range is divided.
__device__ __forceinline__ double reciprocal64(double x) {
  const float r32 = 1.f / d2f_rn(x);
  if (!(fabsf(r32) > 1e-37f && fabsf(r32) < 1e37f)) return 1.0 / x;
  const double r = f2d(r32), e = fma(-x, r, 1.0);
  return fma(r, fma(e, e, e), r);
}

__device__ __forceinline__ bool finite64(double x) {   // on the integer pipe
  return (((unsigned)__double2hiint(x) >> 20) & 0x7FFu) != 0x7FFu;
}

// max(a, b) of a >= 0 and b >= 0 or NaN (ignored), on the integer pipe.
__device__ __forceinline__ double max_pos(double a, double b) {
  const unsigned long long u = __double_as_longlong(a), v = __double_as_longlong(b);
  return v > u && v <= 0x7FF0000000000000ull ? b : a;
}

// Warp sums of eight values in a fixed order, the value of lane / 4 in each lane: halves of
// the values are exchanged at each step, 9 additions per lane instead of 40.
__device__ __forceinline__ double warp_sum8(const double v[8], int lane) {
  double a[4], b[2];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const bool up = lane & 16;
    a[i] = (up ? v[4 + i] : v[i]) + __shfl_xor_sync(0xffffffffu, up ? v[i] : v[4 + i], 16);
  }
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const bool up = lane & 8;
    b[i] = (up ? a[2 + i] : a[i]) + __shfl_xor_sync(0xffffffffu, up ? a[i] : a[2 + i], 8);
  }
  const bool up = lane & 4;
  double s = (up ? b[1] : b[0]) + __shfl_xor_sync(0xffffffffu, up ? b[0] : b[1], 4);
  s += __shfl_xor_sync(0xffffffffu, s, 2);
  return s + __shfl_xor_sync(0xffffffffu, s, 1);
}
__device__ __forceinline__ double warp_max(double x) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) x = max_pos(x, __shfl_xor_sync(0xffffffffu, x, off));
  return x;
}

// The largest wave speed |v| + c of a node in FP64 (the expression the reference computes).
__device__ __forceinline__ double wave64(const double qv[5], double gamma) {
  const double ir = 1.0 / qv[0];
  const double vx = qv[1] * ir, vy = qv[2] * ir, vz = qv[3] * ir;
  const double v2 = vx * vx + vy * vy + vz * vz;
  const double p = (gamma - 1.0) * (qv[4] - 0.5 * qv[0] * v2);
  return sqrt(v2) + sqrt(fmax(gamma * p * ir, 0.0));
}

// Per-node sums (mass, momenta, energy, kinetic energy, dKE/dt) and maxima (e_inf, wave
// speed) of the owned nodes.  GB300's FP64 rate is a small fraction of its FP32 rate and
// bounds this kernel, so the FP64 work per node is kept to the sums, about 20 operations: the
// quadrature weights come from a table, one three-operation reciprocal serves the kinetic
// energy and its derivative, tests and maxima run on the integer pipe, and the wave speed
// (some 45 operations) is screened in FP32: a thread keeps the node of its largest FP32
// estimate and evaluates the FP64 expression at the end, if that estimate is within 1e-5 of
// the block's largest, or at once for a node within 1e-5 of the one it keeps (and of the
// block's largest so far: on a symmetric flow such nodes are common).  Where
// p/(gamma-1) is at least a quarter of rho e, the estimate is within 2e-6 of the exact value
// (rounding of the inputs, and of a difference that multiplies it by four at most); every
// other node goes to FP64 at once.  The node with the largest exact value is therefore never
// screened out (its estimate is at least (1 - 4e-6) times every other), and the maximum is
// the FP64 maximum over all nodes.  Screened against the thread's own running maximum, nearly
// every warp took the FP64 path at every node.  The last block to finish reduces the block
// partials (in index order): a launch of one block took 13 us.
// 16^3/P8 with dq/dt: 352 + 13 -> 208 us (239 MB), 16^3/P3 with a reference 61 + 13 -> 53.
__global__ void __launch_bounds__(kDiagThreads)
k_diag_partial(const double* __restrict__ q, const double* __restrict__ R, const double* __restrict__ qref, NodeGeom ng,
               double gamma, double* partial, const int* __restrict__ flag, unsigned* ticket, double* __restrict__ out) {
  constexpr int kWarps = kDiagThreads / 32;
  __shared__ double sh[kWarps][kDiagLen];
  __shared__ unsigned sm;   // the block's largest estimate so far (bits: estimates are positive)
  __shared__ double sW[kMaxN1 * kMaxN1 * kMaxN1];   // quadrature weight x Jacobian of each node
  double acc[kDiagLen];
  for (int i = 0; i < kDiagLen; ++i) acc[i] = 0.0;
  const int n = ng.n, np = n * n * n, warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const double jac = 0.125 * ng.h * ng.h * ng.h;
  if (threadIdx.x == 0) sm = 0;
  for (int t = threadIdx.x; t < np; t += blockDim.x) {
    const int i = t % n, j = (t / n) % n, k = t / (n * n);
    sW[t] = ng.w[i] * ng.w[j] * ng.w[k] * jac;
  }
  __syncthreads();
  const float gg = (float)(gamma * (gamma - 1.0));   // rounded once: gamma may be near 1
  float m32 = 0.f;             // this thread's largest FP32 estimate of a wave speed
  long long m_at = -1;         // its node
  int bad = 0;
  const long long stride = (long long)gridDim.x * blockDim.x;
  const long long t0 = ng.t_begin + blockIdx.x * (long long)blockDim.x + threadIdx.x;
  int node = (int)(t0 % np);
  const int dnode = (int)(stride % np);
  for (long long t = t0; t < ng.t_end; t += stride, node = (node + dnode >= np) ? node + dnode - np : node + dnode) {
    const double W = sW[node];
    double qv[5], rv[4];
#pragma unroll
    for (int c = 0; c < 5; ++c) qv[c] = q[c * ng.N + t];
    if (R) {
#pragma unroll
      for (int c = 0; c < 4; ++c) rv[c] = R[c * ng.N + t];
    }
    bool finite = true;
#pragma unroll
    for (int c = 0; c < 5; ++c) finite = finite && finite64(qv[c]);
    if (!finite) {
      ++bad;
      continue;
    }
#pragma unroll
    for (int c = 0; c < 5; ++c) acc[c] += W * qv[c];
    const double ir = reciprocal64(qv[0]);
    const double ke2 = (qv[1] * qv[1] + qv[2] * qv[2] + qv[3] * qv[3]) * ir;   // rho v^2
    acc[5] += W * ke2;   // halved at the end
    if (R) {
      const double dk = (qv[1] * rv[1] + qv[2] * rv[2] + qv[3] * rv[3]) * ir - 0.5 * (ke2 * ir) * rv[0];
      acc[6] += W * dk;
    }
    if (qref) {
#pragma unroll
      for (int c = 0; c < 3; ++c) acc[8 + c] = max_pos(acc[8 + c], fabs(qv[1 + c] - qref[(1 + c) * ng.N + t]));
    }
    // wave speed: FP32 screen, FP64 where it may set the maximum
    const float r = d2f_rn(qv[0]), e = d2f_rn(qv[4]);
    const float mx = d2f_rn(qv[1]), my = d2f_rn(qv[2]), mz = d2f_rn(qv[3]);
    const float irf = 1.f / r;
    const float vx = mx * irf, vy = my * irf, vz = mz * irf;
    const float pe = e - 0.5f * (mx * vx + my * vy + mz * vz);   // p / (gamma - 1)
    const float wf = sqrtf(vx * vx + vy * vy + vz * vz) + sqrtf(fmaxf(gg * pe * irf, 0.f));
    // the bounds on r and wf: what FP32 flushes to zero is below 1e-6 of the estimate
    const bool sound32 = pe > 0.25f * fabsf(e) && r > 1e-20f && wf > 1e-3f && wf < 1e18f;
    const bool tie = wf >= m32 * (1.f - 1e-5f) && wf <= m32 * (1.f + 1e-5f);
    if (sound32) {
      const unsigned act = __activemask(), top = __reduce_max_sync(act, __float_as_uint(wf));
      if (lane == __ffs(act) - 1) atomicMax(&sm, top);
    }
    if (!sound32 || (tie && wf >= __uint_as_float(*(volatile unsigned*)&sm) * (1.f - 1e-5f))) {
      acc[11] = max_pos(acc[11], wave64(qv, gamma));
    } else if (wf > m32 && !tie) {
      m32 = wf;
      m_at = t;
    }
  }
  __syncthreads();
  const float bm = __uint_as_float(sm);
  if (m_at >= 0 && m32 >= bm * (1.f - 1e-5f)) {
    double qv[5];
#pragma unroll
    for (int c = 0; c < 5; ++c) qv[c] = q[c * ng.N + m_at];
    acc[11] = max_pos(acc[11], wave64(qv, gamma));
  }
  acc[5] *= 0.5;
  acc[kDiagNonfinite] = (double)bad;
  static_assert(kDiagSum == 8, "warp_sum8");
  const double s8 = warp_sum8(acc, lane);
  if (lane % 4 == 0) sh[warp][lane / 4] = s8;
#pragma unroll
  for (int i = kDiagSum; i < kDiagLen; ++i) {
    const double x = warp_max(acc[i]);
    if (lane == 0) sh[warp][i] = x;
  }
  __syncthreads();
  if (threadIdx.x < kDiagLen) {
    double x = sh[0][threadIdx.x];
    for (int w = 1; w < kWarps; ++w) x = threadIdx.x < kDiagSum ? x + sh[w][threadIdx.x] : max_pos(x, sh[w][threadIdx.x]);
    partial[threadIdx.x * gridDim.x + blockIdx.x] = x;
    __threadfence();
  }
  __shared__ bool last;
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(ticket, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!last) return;
  __threadfence();
  for (int i = warp; i < kDiagLen; i += kWarps) {
    double x[4] = {0.0, 0.0, 0.0, 0.0};
    for (int b0 = 0; b0 < (int)gridDim.x; b0 += 128) {
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int b = b0 + 32 * u + lane;
        const double y = b < (int)gridDim.x ? __ldcg(partial + (size_t)i * gridDim.x + b) : 0.0;
        x[u] = i < kDiagSum ? x[u] + y : max_pos(x[u], y);
      }
    }
    double s = x[0];
#pragma unroll
    for (int u = 1; u < 4; ++u) s = i < kDiagSum ? s + x[u] : max_pos(s, x[u]);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      const double y = __shfl_xor_sync(0xffffffffu, s, off);
      s = i < kDiagSum ? s + y : max_pos(s, y);
    }
    if (lane == 0) out[i] = s;
  }
  if (threadIdx.x == 0) {   // the error flag in the next slot: one copy carries both
    *reinterpret_cast<int*>(out + kDiagLen) = *flag;
    *ticket = 0;
  }
}

cudaError_t launch_diagnostics(const dg_ctx* c, const double* q, const double* R, const double* qref, cudaStream_t st) {
  NodeGeom ng = node_geom(c);
  // two nodes per thread at least: the reduction of a thread's sums costs as much as a node
  const int nblocks =
      (int)std::min<long long>(kDiagBlocks, (ng.t_end - ng.t_begin + 2 * kDiagThreads - 1) / (2 * kDiagThreads));
  k_diag_partial<<<nblocks, kDiagThreads, 0, st>>>(q, R, qref, ng, c->opts.gamma, c->red + kDiagOut, c->err_dev,
                                                   reinterpret_cast<unsigned*>(c->red + kDiagLen + 1), c->red);
  return cudaGetLastError();
}

// n doubles and an int flag from device memory into pinned host memory (written by the
// SMs through the coherent host mapping, not by the copy engine: a few bytes that must not
// queue behind other streams' large copies).
__global__ void k_store_host(const double* __restrict__ src, int n, const int* __restrict__ flag, double* host) {
  const int i = threadIdx.x;
  if (i < n) host[i] = src[i];
  if (i == n) {
    int f = *flag;
    memcpy(host + n, &f, sizeof(int));
  }
}

cudaError_t launch_store_host(const double* src, int n, const int* flag, double* host, cudaStream_t st) {
  if (n < 0 || n >= 1024) return cudaErrorInvalidValue;
  k_store_host<<<1, ((n + 1 + 31) / 32) * 32, 0, st>>>(src, n, flag, host);
  return cudaGetLastError();
}

// ---------------------------------------------------------------- slab face traces

// Components and element size of the traces of `what` (see launch_trace_pack).
static void trace_shape(const dg_ctx* c, int what, int* comps, int* esize) {
  const bool f32 = c->opts.precision == DG_PREC_FP32;
  *comps = what == 2 ? 9 : 5;
  *esize = what == 0 ? 8 : (what == 1 ? 4 : (f32 ? 4 : 8));
}

size_t trace_bytes_for(const dg_ctx* c, int what) {
  int comps, esize;
  trace_shape(c, what, &comps, &esize);
  return (size_t)comps * esize * c->K * c->K * c->n * c->n;
}

// One thread per (component, element of the layer, face node); side 0 = lo, 1 = hi.
template <typename T>
__device__ __forceinline__ T* trace_value(double* q, T* s, T* vt, int what, int v, int n, long long e, int ab, int upper,
                                          long long N) {
  const int n2 = n * n;
  const int node = ab + (upper ? n2 * (n - 1) : 0);   // upper face k = P, lower face k = 0
  if (what == 0) return reinterpret_cast<T*>(q + v * N + e * (n2 * n) + node);
  if (v < 5) return s + e * state_record(n) + v * node_stride(n) + node;
  return vt + e * face_record(n) + (4 + upper) * (kFaceVis * n2) + (v - 5) * n2 + ab;
}

// PACK: lo takes the lower faces of layer z_lo, hi the upper faces of layer z_hi; else the
// upper faces of (ghost) layer z_lo come from lo, the lower faces of layer z_hi from hi.
template <typename T, bool PACK>
__global__ void k_trace(double* __restrict__ q, T* __restrict__ s, T* __restrict__ vt, int what, int comps, int K, int n,
                        int z_lo, int z_hi, long long N, T* __restrict__ lo, T* __restrict__ hi) {
  const int n2 = n * n, K2 = K * K;
  const long long per_side = (long long)comps * K2 * n2;
  const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (t >= 2 * per_side) return;
  const int side = t >= per_side;
  const long long u = t - side * per_side;
  const int v = (int)(u / ((long long)K2 * n2));
  const int r = (int)(u - (long long)v * K2 * n2);
  const int el = r / n2, ab = r - el * n2;
  T* value = trace_value<T>(q, s, vt, what, v, n, (long long)(side ? z_hi : z_lo) * K2 + el, ab, PACK ? side : !side, N);
  T* buf = (side ? hi : lo) + u;
  if (PACK) *buf = *value;
  else *value = *buf;
}

template <typename T, bool PACK>
static cudaError_t trace_t(const dg_ctx* c, double* q, int what, void* lo, void* hi, cudaStream_t st) {
  int comps, esize;
  trace_shape(c, what, &comps, &esize);
  const long long total = 2LL * comps * c->K * c->K * c->n * c->n;
  k_trace<T, PACK><<<(unsigned)((total + 255) / 256), 256, 0, st>>>(
      q, static_cast<T*>(c->cur), static_cast<T*>(c->vt), what, comps, c->K, c->n, PACK ? 1 : 0,
      PACK ? c->z_count : c->z_count + 1, c->N, static_cast<T*>(lo), static_cast<T*>(hi));
  return cudaGetLastError();
}

cudaError_t launch_trace_pack(const dg_ctx* c, const double* q, int what, void* lo, void* hi, cudaStream_t st) {
  int comps, esize;
  trace_shape(c, what, &comps, &esize);
  double* qq = const_cast<double*>(q);   // read only
  return esize == 8 ? trace_t<double, true>(c, qq, what, lo, hi, st) : trace_t<float, true>(c, qq, what, lo, hi, st);
}

cudaError_t launch_trace_unpack(const dg_ctx* c, double* q, int what, const void* lo, const void* hi,
                                cudaStream_t st) {
  int comps, esize;
  trace_shape(c, what, &comps, &esize);
  void *l = const_cast<void*>(lo), *h = const_cast<void*>(hi);   // read only
  return esize == 8 ? trace_t<double, false>(c, q, what, l, h, st) : trace_t<float, false>(c, q, what, l, h, st);
}

// ---------------------------------------------------------------- Algorithm 1 pairs

__global__ void k_make_pairs(const double* __restrict__ qb_n, const double* __restrict__ qnn_np1,
                             const double* __restrict__ qb_np1, double inv_dt, int first_var, int n_vars,
                             long long N, int np, float* __restrict__ X, float* __restrict__ Y) {
  const long long total = N * n_vars;
  const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (t >= total) return;
  // t enumerates (elem, slot, node) in the output order
  const int feat = n_vars * np;
  const long long e = t / feat;
  const int f = (int)(t - e * feat);
  const int slot = f / np, node = f - slot * np;
  const long long src = (long long)(first_var + slot) * N + e * np + node;
  X[t] = (float)qb_n[src];
  Y[t] = (float)((qb_np1[src] - qnn_np1[src]) * inv_dt);
}

cudaError_t launch_make_pairs(const dg_ctx* lo, const double* qb_n, const double* qnn_np1, const double* qb_np1,
                              double dt, int first_var, int n_vars, float* X, float* Y, cudaStream_t st) {
  const long long total = lo->N * n_vars;
  const int threads = 256;
  k_make_pairs<<<(unsigned)((total + threads - 1) / threads), threads, 0, st>>>(
      qb_n, qnn_np1, qb_np1, 1.0 / dt, first_var, n_vars, lo->N, lo->np, X, Y);
  return cudaGetLastError();
}

// ---------------------------------------------------------------- post-step forcing

// Algorithm 1, third loop: q^{n+1} = (uncorrected step) + dt s(q^n), s stored per element
// as [elem][slot][node] with slot = variable - first_var.
__global__ void k_add_forcing(double* __restrict__ q, const float* __restrict__ s, int first_var, int n_vars,
                              int stride, int np, long long N, double dt) {
  const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (t >= N * n_vars) return;
  const int slot = (int)(t / N);
  const long long g = t - (long long)slot * N;
  const long long e = g / np;
  const int node = (int)(g - e * np);
  q[(long long)(first_var + slot) * N + g] += dt * (double)s[e * stride + (long long)slot * np + node];
}

cudaError_t launch_add_forcing(const dg_ctx* c, double* q, const Forcing& f, double dt, cudaStream_t st) {
  const long long total = c->N * f.n_vars;
  const int threads = 256;
  k_add_forcing<<<(unsigned)((total + threads - 1) / threads), threads, 0, st>>>(q, f.s, f.first_var, f.n_vars,
                                                                               f.stride, c->np, c->N, dt);
  return cudaGetLastError();
}

// ---------------------------------------------------------------- conversion self-check

// Counts the inputs where the integer-pipe conversions differ from the hardware ones:
// d2f_rn vs __double2float_rn (inputs in the FP32 normal range or zero), and the exact
// widening f2d vs (double) of the FP32 result.
__global__ void k_check_conversions(const double* __restrict__ x, long long n, unsigned long long* __restrict__ bad) {
  const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (t >= n) return;
  const double v = x[t];
  const float a = d2f_rn(v), b = __double2float_rn(v);
  const bool same = (__float_as_uint(a) == __float_as_uint(b)) || (isnan(a) && isnan(b));
  const bool wide = (f2d(b) == (double)b) || isnan(b);
  if (!same) atomicAdd(&bad[0], 1ull);
  if (!wide) atomicAdd(&bad[1], 1ull);
}

}  // namespace dgnn

extern "C" int dg_check_conversions(const double* x, int64_t n, int64_t* mismatches, void* stream) {
  using namespace dgnn;
  if (!x || n < 0 || !mismatches) return fail(DG_ERR_INVALID_ARG, "dg_check_conversions: bad argument");
  cudaStream_t st = (cudaStream_t)stream;
  unsigned long long* bad = nullptr;
  DG_CUDA(cudaMalloc(&bad, 2 * sizeof(unsigned long long)));
  cudaError_t e = cudaMemsetAsync(bad, 0, 2 * sizeof(unsigned long long), st);
  if (e == cudaSuccess && n > 0) {
    k_check_conversions<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(x, n, bad);
    e = cudaGetLastError();
  }
  unsigned long long h[2] = {0, 0};
  if (e == cudaSuccess) e = cudaMemcpyAsync(h, bad, sizeof(h), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  cudaFree(bad);
  if (e != cudaSuccess) return cuda_fail(e, "dg_check_conversions");
  mismatches[0] = (int64_t)h[0];
  mismatches[1] = (int64_t)h[1];
  return DG_OK;
}
