// The two phases of one evaluation of the DGSEM operator p(q) (Sec. 2, Eq. 3):
//
//  phase A (k_volume): BR1 lifted gradient of (v1, v2, v3, theta)
//     G_d = (2/h) [ D_d U + (U^ - U)|right / w_P - (U^ - U)|left / w_0 ],  U^ central,
//     the viscous stresses and heat flux of Appendix A (Eq. A.3), optionally with the
//     Smagorinsky viscosity, and from them the whole volume term of the element,
//     -(2/h) sum_d D_d (f^a_d - f^nu_d).  Writes the volume term (5 values per node), the
//     viscous flux normal to each face (4 values per face node) and, from an FP64 state,
//     the stage state in operator precision.
//  phase B (k_surface): Roe + central-BR1 interface fluxes and their lifting (strong
//     form), optional forcing s (Eq. 4), then dq/dt or one stage of the low-storage RK3.
//
// A node's viscous quantities enter the operator twice: in its own element's volume term
// and, on a face, in the interface flux.  Forming the volume term where the stresses are
// formed therefore leaves only the face values to hand over: 20 + 96/n bytes per node
// and way in FP32 instead of the 36 of all nine viscous quantities, and the state's
// primitives and fluxes are formed once.
//
// RK3 in the FP32 operator: the state q stays FP64 and is read and written once per
// step.  The stages work on FP32 stage states in two alternating buffers: phase A of
// stage 1 forms s1 = q - reference in qf, phase B of stage 1 writes s2 = s1 + d1 to qy and
// the increment d1 to dlt, phase B of stage 2 writes s3 = s1 + d2 over s1 in qf (phase B
// reads neighbours from qy only) and folds what stage 3 needs, d2 + B3 A3 g2, into dlt;
// stage 3 adds dlt + B3 dt R to q in FP64.  In the FP64 operator every stage updates q in
// FP64 (the plain 2N scheme) and qf holds the stage's copy of q.
//
// Workspace layout: element-major records [elem][component][node] (node stride padded to a
// multiple of 4 values), face values [elem][face][component][face node], face = 2 d + side.
// Every component of a node or face node is then at a compile-time offset from one address.
//
// Phase A: a block owns E consecutive elements (or, at P <= 3 on even K, a 2 x 2 x 2 cube
// of elements whose twelve internal faces need no halo), one thread per node (P = 3 in FP32:
// per row of four).  Phase B: a block owns a few elements, the more the larger the mesh; its
// interface terms are dense work items, one per (element, face, face node), so that every
// lane does useful Roe work, and its nodes add the lifted results in a fixed order.  All
// constants arrive in the operator precision (OpConst): in the FP32 operator no FP64
// arithmetic or conversion runs per node except where the FP64 state is read or written.
#pragma once

#include <cuda_bf16.h>

#include <type_traits>

#include "dg_device.cuh"

namespace dgnn {

// Programmatic dependent launch between the operator's launches: a kernel waits until its
// predecessor in the stream has completed and its writes are visible, and lets its
// successor be launched (which happens once every block of this grid has said so: where
// along a block that pays is in make_const), so the next launch's start overlaps its tail.  Kernels launched
// without the attribute pass the wait at once.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_release() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Maximum threads per phase-A block for order P (one node per thread, E elements per block).
__host__ __device__ constexpr int max_threads_for(int P) {
  return P == 1 ? 256 : P <= 4 ? 512 : P == 5 ? 448 : P == 6 ? 352 : P == 7 ? 512 : 736;
}

// Mesh, basis and physics constants in the operator precision T.
// Elements processed: [e_begin, nel) of a local mesh of K x K x Kz elements (a whole
// periodic mesh: e_begin = 0, nel = K^3, Kz = K; a slab of element layers with one ghost
// layer on each side: e_begin = K^2, nel = K^2 (Kz - 1), and the ghost layers hold the
// neighbouring slabs' face data).
template <typename T>
struct OpConst {
  int K, E, nel;
  int Kz, e_begin;
  long long N;
  T gm1, rho_ref, theta_ref, Hc;  // reference-shifted state (zero references in FP64)
  T s2h;                          // 2 / h
  T winv;                         // 1 / w_0 = 1 / w_P
  T mu, lam, csd2, lam_t;         // transport
  int les;
  double drho_ref, dE_ref;        // references for shifting the FP64 state
  int early;                      // phase A lets the next launch in as it starts, not as it ends (release_early)
  FeatureOut feat;                // network features to write with the stage state (feat.out may be NULL)
  T D[kMaxN1 * kMaxN1];
};

// Element coordinates of the first element of the block (one set of divisions per thread).
struct BlockCoords {
  int x, y, z;
};

__device__ __forceinline__ BlockCoords block_coords(int e0, int K) {
  BlockCoords b;
  b.x = e0 % K;
  const int r = e0 / K;
  b.y = r % K;
  b.z = r / K;
  return b;
}

// Periodic +/-1 step of a coordinate in [0, K).
__device__ __forceinline__ int wrap_step(int x, int shift, int K) {
  x += shift;
  return x < 0 ? x + K : (x >= K ? x - K : x);
}


// 2 x 2 x 2 element blocks ("cubes", even K): block b covers the elements 2 c + l,
// l in {0, 1}^3, of the (K/2)^3 grid of cubes; local element hl = lx + 2 ly + 4 lz.
// Each local element has one external face per direction (on side (hl >> d) & 1) and
// shares the other with local element hl ^ (1 << d).
constexpr int kCubeElems = 8;
__host__ __device__ constexpr bool cube_ok(int P) { return P <= 3; }

__device__ __forceinline__ BlockCoords cube_coords(int b, int K) {
  const int h = K >> 1;
  BlockCoords c;
  c.x = 2 * (b % h);
  const int r = b / h;
  c.y = 2 * (r % h);
  c.z = 2 * (r / h);
  return c;
}

__device__ __forceinline__ int cube_element(const BlockCoords& c, int hl, int K) {
  return (c.x + (hl & 1)) + K * ((c.y + ((hl >> 1) & 1)) + K * (c.z + (hl >> 2)));
}


// Element across face 2 d + side of element e (periodic; Kz layers along z).
__device__ __forceinline__ int element_across(int e, int face, int K, int Kz) {
  BlockCoords c = block_coords(e, K);
  const int step = (face & 1) ? 1 : -1, d = face >> 1;
  if (d == 0) c.x = wrap_step(c.x, step, K);
  else if (d == 1) c.y = wrap_step(c.y, step, K);
  else c.z = wrap_step(c.z, step, Kz);
  return c.x + K * (c.y + K * c.z);
}

// Internal faces of a cube, u <-> (ab, p, d): face p (0..3) normal to d joins the local
// elements hlL (bit d clear) and hlL | 1 << d.
__device__ __forceinline__ int cube_left_of_pair(int p, int d) {
  return ((p >> d) << (d + 1)) | (p & ((1 << d) - 1));
}

// Node of the face normal to d at normal index m with tangential index ab.
template <int P>
__device__ __forceinline__ int face_node(int d, int m, int ab) {
  constexpr int n = P + 1;
  const int a = ab % n, b = ab / n;
  return d == 0 ? m + n * (a + n * b) : d == 1 ? a + n * (m + n * b) : a + n * (b + n * m);
}

// Tangential index of node (i, j, k) on a face normal to d.
template <int P>
__device__ __forceinline__ int face_ab(int d, const int idx[3]) {
  constexpr int n = P + 1;
  return d == 0 ? idx[1] + n * idx[2] : d == 1 ? idx[0] + n * idx[2] : idx[0] + n * idx[1];
}


// Face item t <-> (ab, face, hl), ab fastest, element slowest; face = 2 d + side.
template <int P>
struct Item {
  int ab, face, hl;
};

template <int P>
__device__ __forceinline__ Item<P> item_of(int t) {
  constexpr int n2 = (P + 1) * (P + 1);
  Item<P> it;
  it.ab = t % n2;
  const int r = t / n2;
  it.face = r % 6;
  it.hl = r / 6;
  return it;
}

template <int P>
__device__ __forceinline__ int item_index(int ab, int face, int hl) {
  constexpr int n2 = (P + 1) * (P + 1);
  return ab + n2 * (face + 6 * hl);
}

// External face items of a cube, t <-> (ab, hl, d), ab fastest, direction slowest (a warp
// shares d); the face lies on side (hl >> d) & 1 of local element hl.
template <int P>
__device__ __forceinline__ Item<P> cube_item_of(int t) {
  constexpr int n2 = (P + 1) * (P + 1);
  Item<P> it;
  it.ab = t % n2;
  const int r = t / n2;
  it.hl = r % kCubeElems;
  const int d = r / kCubeElems;
  it.face = 2 * d + ((it.hl >> d) & 1);
  return it;
}

template <int P>
__device__ __forceinline__ int cube_item_index(int ab, int d, int hl) {
  constexpr int n2 = (P + 1) * (P + 1);
  return ab + n2 * (hl + kCubeElems * d);
}

// Multiply, add and fused multiply-add with no contraction left to the compiler.
__device__ __forceinline__ float mul_(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float add_(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float fma_(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double mul_(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ double add_(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ double fma_(double a, double b, double c) { return __fma_rn(a, b, c); }

// A value (four consecutive ones) that another launch may have written after this SM last
// cached its line: read at the L2, the point of coherence, in program order.
__device__ __forceinline__ float ld_l2(const float* p) {
  float v;
  asm volatile("ld.relaxed.gpu.global.f32 %0, [%1];" : "=f"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ double ld_l2(const double* p) {
  double v;
  asm volatile("ld.relaxed.gpu.global.f64 %0, [%1];" : "=d"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void ld4_l2(const float* p, float v[4]) {
  asm volatile("ld.relaxed.gpu.global.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3])
               : "l"(p)
               : "memory");
}
// A value of the stage state, by phase A's source (see k_volume).
template <int SRC, typename T>
__device__ __forceinline__ T state_value(const T* p) {
  return SRC == 2 ? ld_l2(p) : *p;
}

// ---------------------------------------------------------------- shared-memory tiles

// Four values of a node in shared memory, read and written as vectors: FP32 one plane of
// 16-byte quads, FP64 two planes of 16-byte pairs (cnt entries each).
__device__ __forceinline__ void quad_store(float* base, int, int i, const float v[4]) {
  reinterpret_cast<float4*>(base)[i] = make_float4(v[0], v[1], v[2], v[3]);
}
__device__ __forceinline__ void quad_store(double* base, int cnt, int i, const double v[4]) {
  double2* p = reinterpret_cast<double2*>(base);
  p[i] = make_double2(v[0], v[1]);
  p[cnt + i] = make_double2(v[2], v[3]);
}
__device__ __forceinline__ void quad_load(const float* base, int, int i, float v[4]) {
  const float4 a = reinterpret_cast<const float4*>(base)[i];
  v[0] = a.x;
  v[1] = a.y;
  v[2] = a.z;
  v[3] = a.w;
}
__device__ __forceinline__ void quad_load(const double* base, int cnt, int i, double v[4]) {
  const double2* p = reinterpret_cast<const double2*>(base);
  const double2 a = p[i], b = p[cnt + i];
  v[0] = a.x;
  v[1] = a.y;
  v[2] = b.x;
  v[3] = b.y;
}

// Two FP32 multiply-adds in one instruction (each rounded as fmaf).  The FP32 rate is the
// same as fmaf's (measured 37.4 against 35.6 T multiply-adds/s), the issue slots are half.
using f32x2 = unsigned long long;
__device__ __forceinline__ void fma2(f32x2& acc, f32x2 a, f32x2 b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(a), "l"(b));
}
__device__ __forceinline__ f32x2 pack2(float a, float b) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void unpack2(f32x2 p, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(p));
}

// An entry of the derivative matrix as the contractions use it: FP32 a duplicated pair.
template <typename T>
struct DEntry {
  using type = T;
  __device__ static __forceinline__ T make(T x) { return x; }
};
template <>
struct DEntry<float> {
  using type = f32x2;
  __device__ static __forceinline__ f32x2 make(float x) { return pack2(x, x); }
};

// Running sum over a line of D entry x quad.
template <typename T>
struct QuadSum {
  T a[4] = {T(0), T(0), T(0), T(0)};
  __device__ __forceinline__ void add(T d, const T* base, int cnt, int i) {
    T v[4];
    quad_load(base, cnt, i, v);
#pragma unroll
    for (int k = 0; k < 4; ++k) a[k] += d * v[k];
  }
  __device__ __forceinline__ void get(T out[4]) const {
#pragma unroll
    for (int k = 0; k < 4; ++k) out[k] = a[k];
  }
};
template <>
struct QuadSum<float> {
  f32x2 a[2] = {0ull, 0ull};
  __device__ __forceinline__ void add(f32x2 d, const float* base, int, int i) {
    const ulonglong2 v = reinterpret_cast<const ulonglong2*>(base)[i];
    fma2(a[0], d, v.x);
    fma2(a[1], d, v.y);
  }
  __device__ __forceinline__ void get(float out[4]) const {
    unpack2(a[0], out[0], out[1]);
    unpack2(a[1], out[2], out[3]);
  }
};
__device__ __forceinline__ double d_scalar(double d) { return d; }
__device__ __forceinline__ float d_scalar(f32x2 d) {
  float a, b;
  unpack2(d, a, b);
  return a;
}

// ---------------------------------------------------------------- line contractions

// FP32 at P >= 5: the contractions run line by line, one task per (direction, pair of
// components, line) computing the derivative at every node of the line, so that each
// operand is read from shared memory once per line instead of once per output node.
template <typename T>
__host__ __device__ constexpr bool use_lines(int P) {
  return std::is_same<T, float>::value && P >= 5;
}
// Shared-memory index of a node: rows of odd length, so that the lanes of a warp reading
// consecutive x-lines fall on different banks.
__host__ __device__ constexpr int line_row(int n) { return n | 1; }
__host__ __device__ constexpr int line_nodes(int n) { return line_row(n) * n * n; }

// c_D32 holds the derivative matrices of every order as duplicated FP32 pairs, row-major, in
// constant memory (one copy per translation unit, filled by upload_const_D on the host before
// the first launch), read with compile-time indices.
__constant__ float2 c_D32[kMaxP + 1][kMaxN1 * kMaxN1];

__device__ __forceinline__ f32x2 line_sub(f32x2 a, f32x2 b) {   // a - b in one instruction: -1 x b + a
  fma2(a, 0xBF800000BF800000ull, b);
  return a;
}
__device__ __forceinline__ float line_sub(float a, float b) { return a - b; }
__device__ __forceinline__ float line_neg(float a) { return -a; }
__device__ __forceinline__ f32x2 line_neg(f32x2 a) { return a ^ 0x8000000080000000ull; }
__device__ __forceinline__ void line_fma(f32x2& acc, float2 d, f32x2 v) { fma2(acc, pack2(d.x, d.y), v); }
__device__ __forceinline__ void line_fma(float& acc, float2 d, float v) { acc = fmaf(d.x, v, acc); }

// out[node(i)] = sum_m D[i][m] f[node(m)], i = 0..P, for the line of nodes along direction
// D with tangential index ab; f and out may be the same array (the line's values are all
// read before any is written, and no other task touches the line).  D[P-i][P-m] = -D[i][m]:
// an entry, once read, serves the two mirrored rows.
//
// The sums run over the plain values.  The sums and differences f_m +- f_{P-m} would halve
// the multiply-adds, but they are rounded before D weighs them: the error of dq/dt in density
// and momenta grew up to 1.6 times (16^3/P8 RK3 step 504 us with them, 518 without).
//
// REL: D annihilates constants, so a line may be taken relative to one of its nodes.  The
// energy flux has a large common part at low Mach numbers, whose rounding the plain sum
// carries into the result; it goes relative to node 1 in the lower half and P - 1 in the
// upper, which on a coarse mesh are near enough to every row's own node (one middle node
// doubled the error of the energy on 2^3 elements at P = 8).
template <int P, int D, bool REL, typename V>
__device__ __forceinline__ void line_derivative(const V* f, V* out, int ab) {
  constexpr int n = P + 1, rs = line_row(n);
  const int a = ab % n, b = ab / n;
  const int base = D == 0 ? rs * (a + n * b) : D == 1 ? a + rs * n * b : a + rs * b;
  constexpr int st = D == 0 ? 1 : D == 1 ? rs : rs * n;
  V v[n], u[n];   // the line and its mirror image
#pragma unroll
  for (int m = 0; m < n; ++m) v[m] = f[base + m * st];
#pragma unroll
  for (int m = 0; m < n; ++m) u[m] = v[P - m];
  if (REL) {
    const V r = v[1], s = u[1];
#pragma unroll
    for (int m = 0; m < n; ++m) {
      v[m] = line_sub(v[m], r);
      u[m] = line_sub(u[m], s);
    }
  }
#pragma unroll
  for (int i = 0; i < (n + 1) / 2; ++i) {
    V lo = V(0), hi = V(0);
#pragma unroll
    for (int m = 0; m < n; ++m) {
      if ((m == i && i > 0) || (REL && m == 1)) continue;   // D[i][i] = 0 inside; v[1] = u[1] = 0
      line_fma(lo, c_D32[P][i * n + m], v[m]);
      if (2 * i < P) line_fma(hi, c_D32[P][i * n + m], u[m]);
    }
    out[base + i * st] = lo;
    if (2 * i < P) out[base + (P - i) * st] = line_neg(hi);
  }
}

template <int P, bool REL, typename V>
__device__ __forceinline__ void line_derivative_dir(int d, const V* f, V* out, int ab) {
  if (d == 0) line_derivative<P, 0, REL>(f, out, ab);
  else if (d == 1) line_derivative<P, 1, REL>(f, out, ab);
  else line_derivative<P, 2, REL>(f, out, ab);
}

template <typename T>
__device__ __forceinline__ Prim<T> prim_c(const T s[5], const OpConst<T>& C) {
  return primitives(s, C.rho_ref, C.gm1);
}

// Variable v of the stage state: the FP64 value relative to the reference, rounded once.
// The difference is volatile so that the compiler does not form it, on the slow FP64 pipe,
// for the variables without a reference too.
template <typename T>
__device__ __forceinline__ T shifted(double x, int v, const OpConst<T>& C) {
  if (v == 0 || v == 4) asm volatile("sub.rn.f64 %0, %0, %1;" : "+d"(x) : "d"(v == 0 ? C.drho_ref : C.dE_ref));
  return from_double<T>(x);
}

// Stage state of an element's node from the FP64 state q ([var][node], gi = elem n^3 + node).
template <typename T>
__device__ __forceinline__ void state_from_q(const double* __restrict__ q, long long gi, const OpConst<T>& C, T s[5]) {
  double qd[5];
#pragma unroll
  for (int v = 0; v < 5; ++v) qd[v] = q[v * C.N + gi];
  s[0] = from_double<T>(qd[0] - C.drho_ref);
  s[1] = from_double<T>(qd[1]);
  s[2] = from_double<T>(qd[2]);
  s[3] = from_double<T>(qd[3]);
  s[4] = from_double<T>(qd[4] - C.dE_ref);
}

// Effective viscosity and heat coefficient (Smagorinsky when les != 0).
template <typename T>
__device__ __forceinline__ void transport_c(const OpConst<T>& C, T rho, const T G[3][4], T* mu, T* lam) {
  T m = C.mu, l = C.lam;
  if (C.les) {
    T ss = T(0);
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
      for (int b = 0; b < 3; ++b) {
        const T s = T(0.5) * (G[b][a] + G[a][b]);
        ss += s * s;
      }
    const T mut = rho * C.csd2 * sqrt(T(2) * ss);  // IEEE square root: the argument may be zero
    m += mut;
    l += mut * C.lam_t;
  }
  *mu = m;
  *lam = l;
}

// Split form: a node's primitives for the two-point flux, (rho, v1, v2, v3, p', H) with
// H = (rho e + p) / rho (the reference pressure cancels in the split pressure term, so p'
// enters it; H needs the full enthalpy).
template <typename T>
__device__ __forceinline__ void store_split_prims(const T s[5], const Prim<T>& w, const OpConst<T>& C, T* out,
                                                  int stride) {
  out[0] = w.rho;
  out[stride] = w.v[0];
  out[2 * stride] = w.v[1];
  out[3 * stride] = w.v[2];
  out[4 * stride] = w.pp;
  out[5 * stride] = (s[4] + w.pp + C.Hc) * w.ir;
}

// Pirozzoli's kinetic-energy-preserving two-point flux in direction d from two nodes'
// primitives: m = {rho}{v_d}; (m, m {v_j} + {p'} delta_jd, m {H}).
template <typename T>
__device__ __forceinline__ void kep_flux_prims(const T a[6], const T b[6], int d, T F[5]) {
  const T m = T(0.25) * (a[0] + b[0]) * (a[1 + d] + b[1 + d]);
  F[0] = m;
#pragma unroll
  for (int k = 0; k < 3; ++k) F[1 + k] = m * (T(0.5) * (a[1 + k] + b[1 + k]));
  F[1 + d] += T(0.5) * (a[4] + b[4]);
  F[4] = m * (T(0.5) * (a[5] + b[5]));
}


// Shared memory of a phase-A block (values of T unless said otherwise), in this order:
// neighbour elements [6 E] (int), D entries [n^2] (direct contraction), then
//   direct: U quads [4][E np], halo quads [4][faces], flux quads [3][4][E np] and energy
//           fluxes [3][E np] (quads need 16-byte alignment), split form: primitives [6][E np];
//   lines:  U pairs [2][E ln], halo pairs [2][faces], derivatives and then fluxes pairs
//           [6][E ln], energy fluxes [3][E ln], split form: primitives [6][E np].
template <int P, typename T>
__host__ __device__ constexpr size_t volume_smem_bytes(int E, int faces, bool split) {
  constexpr int n = P + 1, n2 = n * n, np = n2 * n, ln = line_nodes(n);
  const size_t head = ((6 * E + 3) & ~3) * sizeof(int);
  const size_t prims = split ? (size_t)6 * E * np : 0;
  if (use_lines<T>(P)) return head + sizeof(float) * ((size_t)E * ln * (4 + 12 + 3) + 4 * (size_t)faces + prims);
  return head + sizeof(typename DEntry<T>::type) * ((n2 + 1) & ~1) + sizeof(T) * ((size_t)E * np * (4 + 15) + 4 * (size_t)faces + prims);
}

// Phase A of block `blk` of one mesh (the body of k_volume and k_volume_batch).
// SRC 0: the stage state is formed from the FP64 state q and written to qf; SRC 1: it is
// read from qf; SRC 2: the same, at the L2 (BESIDE, see k_volume).  CUBE: the block is a 2 x 2 x 2 cube of elements; the halo holds only the
// external faces, internal faces take the neighbour's values from the own tile.  FEAT:
// also write the forcing network's input features (C.feat; FP64, P = 3).  SPLIT: the Euler part of the
// volume term in the kinetic-energy-preserving split form, 2 sum_m D_im F#(q_i, q_m) along
// each line with Pirozzoli's two-point flux F# (mass flux {rho}{v_d}; momentum m {v_j} +
// {p'} delta_jd; energy m {H}), from a tile of primitives; the viscous part keeps the
// standard form.
template <int P, typename T, int SRC, bool CUBE = false, bool FEAT = false, bool SPLIT = false>
__device__ __forceinline__ void volume_block(int blk, const double* __restrict__ q, T* qf,
                                             T* __restrict__ rv, T* __restrict__ vt, const OpConst<T>& C) {
  constexpr int n = P + 1, n2 = n * n, np = n2 * n, ns = node_stride(n);
  constexpr bool kLines = use_lines<T>(P);
  constexpr int tn = kLines ? line_nodes(n) : np;   // tile entries per element
  using DT = typename DEntry<T>::type;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int E = CUBE ? kCubeElems : C.E;
  const int tileN = E * tn;
  const int haloN = CUBE ? 3 * kCubeElems * n2 : E * 6 * n2;
  int* sNb = reinterpret_cast<int*>(smem_raw);                      // element across each face
  DT* sD = reinterpret_cast<DT*>(sNb + ((6 * E + 3) & ~3));         // direct contraction only
  T* sU = kLines ? reinterpret_cast<T*>(sD) : reinterpret_cast<T*>(sD + ((n2 + 1) & ~1));
  T* sH = sU + 4 * tileN;                                           // neighbours' gradient variables
  T* sF = sH + 4 * haloN;
  const int e0 = C.e_begin + blk * E;
  const BlockCoords bc = CUBE ? cube_coords(blk, C.K) : BlockCoords{0, 0, 0};

  const int le = threadIdx.x / np;
  const int node = threadIdx.x - le * np;
  const int e = CUBE ? cube_element(bc, le, C.K) : e0 + le;
  const bool active = CUBE ? (le < kCubeElems) : (le < E) && (e < C.nel);
  T* qe = qf + (size_t)e * state_record(n) + node;

  T s[5];
  if (active) {
    if (SRC == 0) {
      state_from_q(q, (long long)e * np + node, C, s);
#pragma unroll
      for (int v = 0; v < 5; ++v) qe[v * ns] = s[v];
    } else {
#pragma unroll
      for (int v = 0; v < 5; ++v) s[v] = state_value<SRC>(qe + v * ns);
    }
  }
  // set-up that the own loads' latency covers
  for (int t = threadIdx.x; t < 6 * E; t += blockDim.x) {
    const int hl = t / 6, eh = CUBE ? cube_element(bc, hl, C.K) : e0 + hl;
    sNb[t] = element_across(eh, t - 6 * hl, C.K, C.Kz);
  }
  if (!kLines)
    for (int t = threadIdx.x; t < n2; t += blockDim.x) sD[t] = DEntry<T>::make(C.D[t]);
  __syncthreads();

  // halo: gradient variables of the neighbours' face nodes
  for (int t = threadIdx.x; t < haloN; t += blockDim.x) {
    const Item<P> it = CUBE ? cube_item_of<P>(t) : item_of<P>(t);
    if (!CUBE && e0 + it.hl >= C.nel) continue;
    const int enb = sNb[6 * it.hl + it.face];
    const int fn = face_node<P>(it.face >> 1, (it.face & 1) ? 0 : P, it.ab);
    T sn[5], Un[4];
    if (SRC == 0) {
      state_from_q(q, (long long)enb * np + fn, C, sn);
    } else {
      const T* qn = qf + (size_t)enb * state_record(n) + fn;
#pragma unroll
      for (int v = 0; v < 5; ++v) sn[v] = state_value<SRC>(qn + v * ns);
    }
    const Prim<T> wn = prim_c(sn, C);
    gradient_vars(sn, wn, C.theta_ref, Un);
    if constexpr (kLines) {
      f32x2* h = reinterpret_cast<f32x2*>(sH);
      h[t] = pack2(Un[0], Un[1]);
      h[haloN + t] = pack2(Un[2], Un[3]);
    } else {
      quad_store(sH, haloN, t, Un);
    }
  }

  const int idx[3] = {node % n, (node / n) % n, node / n2};
  const int ti = kLines ? le * tn + node + (node / n) * (line_row(n) - n) : le * np + node;  // own tile entry
  T U[4];
  Prim<T> w;
  if (active) {
    if (FEAT) {
      // the forcing network's input features of this node, from the stage state: the same
      // arithmetic as the separate feature kernels of the network
      __nv_bfloat16* fo = static_cast<__nv_bfloat16*>(C.feat.out) + (long long)e * C.feat.ld + node;
#pragma unroll
      for (int v = 0; v < 5; ++v) {
        const int slot = v - C.feat.first_var;
        if (slot < 0 || slot >= C.feat.n_vars) continue;
        const int f = slot * np + node;
        const float x = d2f_rn(double(s[v]) - C.feat.mean64[f]) / C.feat.sd[f];
        fo[slot * np] = __float2bfloat16_rn(x);
      }
    }
    w = prim_c(s, C);
    gradient_vars(s, w, C.theta_ref, U);
    if constexpr (kLines) {
      f32x2* u2 = reinterpret_cast<f32x2*>(sU);
      u2[ti] = pack2(U[0], U[1]);
      u2[tileN + ti] = pack2(U[2], U[3]);
    } else {
      quad_store(sU, tileN, ti, U);
    }
  }
  __syncthreads();

  T G[3][4];
  DT Dr[3][kLines ? 1 : n];
  constexpr int stride[3] = {1, n, n2};
  if constexpr (kLines) {
    f32x2* u2 = reinterpret_cast<f32x2*>(sU);
    f32x2* g2 = reinterpret_cast<f32x2*>(sF);
    for (int task = threadIdx.x; task < E * 6 * n2; task += blockDim.x) {
      const int r = task / n2, ab = task - r * n2, hl = r / 6, dp = r - 6 * hl;   // dp = 2 d + pair
      line_derivative_dir<P, false>(dp >> 1, u2 + (dp & 1) * tileN + hl * tn, g2 + dp * tileN + hl * tn, ab);
    }
    __syncthreads();
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      if (!active) continue;
      unpack2(g2[(2 * d) * tileN + ti], G[d][0], G[d][1]);
      unpack2(g2[(2 * d + 1) * tileN + ti], G[d][2], G[d][3]);
    }
  } else if (active) {
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const DT* Drow = sD + idx[d] * n;
      const int base = ti - idx[d] * stride[d];
      QuadSum<T> sum;
#pragma unroll
      for (int m = 0; m < n; ++m) {
        Dr[d][m] = Drow[m];
        sum.add(Dr[d][m], sU, tileN, base + m * stride[d]);
      }
      sum.get(G[d]);
    }
  }

  T vis[9];
  if (active) {
    const T lift = C.s2h * C.winv * T(0.5);
#pragma unroll
    for (int d = 0; d < 3; ++d) {
#pragma unroll
      for (int a = 0; a < 4; ++a) G[d][a] *= C.s2h;
      // interface lifting with the central U^ = (U + U_nb) / 2
      const bool right = (idx[d] == P), left = (idx[d] == 0);
      if (right || left) {
        const int ab = face_ab<P>(d, idx);
        const T sgn = right ? lift : -lift;
        T Un[4];
        if (CUBE && (right ? 1 : 0) != ((le >> d) & 1)) {   // internal face: the neighbour's tile entry
          const int o = (le ^ (1 << d)) * np + face_node<P>(d, right ? 0 : P, ab);
          quad_load(sU, tileN, o, Un);
        } else {
          const int o = CUBE ? cube_item_index<P>(ab, d, le) : item_index<P>(ab, 2 * d + (right ? 1 : 0), le);
          if constexpr (kLines) {
            const f32x2* h = reinterpret_cast<const f32x2*>(sH);
            unpack2(h[o], Un[0], Un[1]);
            unpack2(h[haloN + o], Un[2], Un[3]);
          } else {
            quad_load(sH, haloN, o, Un);
          }
        }
#pragma unroll
        for (int a = 0; a < 4; ++a) G[d][a] += sgn * (Un[a] - U[a]);
      }
    }
    T mu, lam;
    transport_c(C, w.rho, G, &mu, &lam);
    const T div = G[0][0] + G[1][1] + G[2][2];
    const T t23 = T(2.0 / 3.0) * mu * div;
    // G[d][a] = d u_a / d x_d, tau_ab = mu (du_a/dx_b + du_b/dx_a) - 2/3 mu div delta_ab
    vis[0] = T(2) * mu * G[0][0] - t23;
    vis[1] = T(2) * mu * G[1][1] - t23;
    vis[2] = T(2) * mu * G[2][2] - t23;
    vis[3] = mu * (G[1][0] + G[0][1]);
    vis[4] = mu * (G[2][0] + G[0][2]);
    vis[5] = mu * (G[2][1] + G[1][2]);
    vis[6] = lam * G[0][3];
    vis[7] = lam * G[1][3];
    vis[8] = lam * G[2][3];
    // viscous flux normal to each face the node lies on, in the face's frame (see face_terms):
    // (tau_nn, s tau_nt1, s tau_nt2, s k theta_n) with s = +1 on the right, -1 on the left
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const bool right = (idx[d] == P), left = (idx[d] == 0);
      if (!(right || left)) continue;
      const T sg = right ? T(1) : T(-1);
      T* o = vt + (size_t)e * face_record(n) + (2 * d + (right ? 1 : 0)) * (kFaceVis * n2) + face_ab<P>(d, idx);
      const int t1 = (d + 1) % 3, t2 = (d + 2) % 3;
      o[0] = vis[d];
      o[n2] = sg * vis[sym_index(t1, d)];
      o[2 * n2] = sg * vis[sym_index(t2, d)];
      o[3 * n2] = sg * vis[6 + d];
    }
    // volume fluxes of the three directions
    T* sW = sF + 15 * tileN;
    if (SPLIT) store_split_prims(s, w, C, sW + le * np + node, E * np);
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      T F[5], fv[5];
      viscous_flux(vis, w.v, d, fv);
      if (SPLIT) {
#pragma unroll
        for (int c = 0; c < 5; ++c) F[c] = -fv[c];
      } else {
        euler_flux(s, w, C.Hc, d, F);
#pragma unroll
        for (int c = 0; c < 5; ++c) F[c] -= fv[c];
      }
      if constexpr (kLines) {
        // over this node's own derivative entries, already read
        f32x2* f2 = reinterpret_cast<f32x2*>(sF);
        f2[(2 * d) * tileN + ti] = pack2(F[0], F[1]);
        f2[(2 * d + 1) * tileN + ti] = pack2(F[2], F[3]);
        sF[(12 + d) * tileN + ti] = F[4];
      } else {
        quad_store(sF + 4 * d * tileN, tileN, ti, F);
        sF[(12 + d) * tileN + ti] = F[4];
      }
    }
  }
  __syncthreads();

  T R[5] = {T(0), T(0), T(0), T(0), T(0)};
  if constexpr (kLines) {
    f32x2* f2 = reinterpret_cast<f32x2*>(sF);
    T* f1 = sF + 12 * tileN;
    for (int task = threadIdx.x; task < E * 9 * n2; task += blockDim.x) {
      const int r = task / n2, ab = task - r * n2, hl = r / 9, k = r - 9 * hl;
      if (k < 6) line_derivative_dir<P, false>(k >> 1, f2 + k * tileN + hl * tn, f2 + k * tileN + hl * tn, ab);
      else line_derivative_dir<P, true>(k - 6, f1 + (k - 6) * tileN + hl * tn, f1 + (k - 6) * tileN + hl * tn, ab);
    }
    __syncthreads();
    if (!active) return;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      T a[5];
      unpack2(f2[(2 * d) * tileN + ti], a[0], a[1]);
      unpack2(f2[(2 * d + 1) * tileN + ti], a[2], a[3]);
      a[4] = f1[d * tileN + ti];
#pragma unroll
      for (int c = 0; c < 5; ++c) R[c] -= C.s2h * a[c];
    }
  } else {
    if (!active) return;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const int base = ti - idx[d] * stride[d];
      QuadSum<T> sum;
      T a[5];
      a[4] = T(0);
#pragma unroll
      for (int m = 0; m < n; ++m) {
        sum.add(Dr[d][m], sF + 4 * d * tileN, tileN, base + m * stride[d]);
        a[4] += d_scalar(Dr[d][m]) * sF[(12 + d) * tileN + base + m * stride[d]];
      }
      sum.get(a);
#pragma unroll
      for (int c = 0; c < 5; ++c) R[c] -= C.s2h * a[c];
    }
  }
  if (SPLIT) {
    const T* sW = sF + 15 * tileN;
    const int wN = E * np, wi0 = le * np + node;
    T wi[6];
#pragma unroll
    for (int k = 0; k < 6; ++k) wi[k] = sW[k * wN + wi0];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const int base = wi0 - idx[d] * stride[d];
      T acc[5] = {T(0), T(0), T(0), T(0), T(0)};
#pragma unroll
      for (int m = 0; m < n; ++m) {
        const int o = base + m * stride[d];
        T wm[6];
#pragma unroll
        for (int k = 0; k < 6; ++k) wm[k] = sW[k * wN + o];
        T F[5];
        kep_flux_prims(wi, wm, d, F);
        const T dm = kLines ? C.D[idx[d] * n + m] : d_scalar(Dr[d][kLines ? 0 : m]);
#pragma unroll
        for (int c = 0; c < 5; ++c) acc[c] += dm * F[c];
      }
#pragma unroll
      for (int c = 0; c < 5; ++c) R[c] -= C.s2h * (T(2) * acc[c]);
    }
  }
  T* re = rv + (size_t)e * state_record(n) + node;
#pragma unroll
  for (int v = 0; v < 5; ++v) re[v * ns] = R[v];
}

// ---------------------------------------------------------------- phase A at P = 3, FP32
//
// n = 4 makes a row of nodes along x one 16-byte vector, so a thread owns a row: its
// x-derivatives stay in registers, its y- and z-derivatives read whole rows, and every
// global and shared access moves four nodes.  An element is 16 threads of one warp, and
// its 16 halo rows along y and z (4 faces of 4 rows) are one per thread, so the kernel needs
// warp-level synchronisation only.  Against one node per thread (k_volume at P = 3 as the
// other orders have it) shared-memory traffic, which bounded that, falls from 133 to 80
// floats per node and warp instructions to less than half.
__host__ __device__ constexpr bool use_rows4(int P, int tsize, bool split) { return P == 3 && tsize == 4 && !split; }

// Four consecutive values as two pairs.
struct Row {
  f32x2 lo, hi;
};
__device__ __forceinline__ Row row_load(const float* p) {
  const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(p);
  return Row{v.x, v.y};
}
__device__ __forceinline__ void row_unpack(const Row& r, float v[4]) {
  unpack2(r.lo, v[0], v[1]);
  unpack2(r.hi, v[2], v[3]);
}
__device__ __forceinline__ void row_store(float* p, const float v[4]) {
  *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
}
__device__ __forceinline__ void row_read(const float* p, float v[4]) {
  const float4 a = *reinterpret_cast<const float4*>(p);
  v[0] = a.x;
  v[1] = a.y;
  v[2] = a.z;
  v[3] = a.w;
}
// sum_m d[m] row_m over a line of four rows: row 0 the thread's own, the others at base + at[...]
// (m: the exclusive-or of their positions along the line).  Farthest row first, own row last:
// of the orders that an exclusive-or gives, the one no less accurate than along the line.
__device__ __forceinline__ void rows_contract(const Row& own, const float* base, const int at[3], const f32x2 d[4],
                                              float out[4]) {
  Row acc{0ull, 0ull};
#pragma unroll
  for (int m = 3; m >= 0; --m) {
    const Row r = m ? row_load(base + at[m - 1]) : own;
    fma2(acc.lo, d[m], r.lo);
    fma2(acc.hi, d[m], r.hi);
  }
  row_unpack(acc, out);
}

// Four consecutive FP64 values (two 16-byte loads where the address allows).
__device__ __forceinline__ void row_read64(const double* p, bool wide, double v[4]) {
  if (wide) {
    const double2 a = reinterpret_cast<const double2*>(p)[0], b = reinterpret_cast<const double2*>(p)[1];
    v[0] = a.x;
    v[1] = a.y;
    v[2] = b.x;
    v[3] = b.y;
  } else {
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i] = p[i];
  }
}

// Stage state of the row of four nodes at node index `node` of element e.
template <int SRC>
__device__ __forceinline__ void state_row(const double* __restrict__ q, const float* qf, int e, int node, bool wide,
                                          const OpConst<float>& C, float s[5][4]) {
#pragma unroll
  for (int v = 0; v < 5; ++v) {
    if (SRC == 0) {
      double d[4];
      row_read64(q + v * C.N + (long long)e * 64 + node, wide, d);
#pragma unroll
      for (int i = 0; i < 4; ++i) s[v][i] = shifted(d[i], v, C);
    } else if (SRC == 2) {
      ld4_l2(qf + (size_t)e * state_record(4) + v * 64 + node, s[v]);
    } else {
      row_read(qf + (size_t)e * state_record(4) + v * 64 + node, s[v]);
    }
  }
}

// The stage state s1 from the FP64 state, one thread per node, in a pass of its own ahead of a
// volume4_block<1> launch.  Formed in that launch, a state is converted 2.5 times (own row
// and neighbours' faces) with the FP64 pipe 63 % busy; one pass moves 60 bytes per node and
// converts once (32^3 RK3 step 331 -> 306 us, 16^3 58.2 -> 54.1, 8^3 29.7 -> 27.1; a thread per
// row of four nodes here: 16^3 58.6).  At the other orders, whose kernels hide the
// conversions, it does not pay (16^3/P8 516 -> 521 us).
// It also writes the forcing network's input features (C.feat), the same arithmetic as the
// separate feature kernels of the network.
__device__ __forceinline__ void feature_store(const FeatureOut& f, int e, int np, int node, int v, float s) {
  const int slot = v - f.first_var;
  if (slot < 0 || slot >= f.n_vars) return;
  const int i = slot * np + node;
  static_cast<__nv_bfloat16*>(f.out)[(long long)e * f.ld + i] = __float2bfloat16_rn((s - f.shift32[i]) / f.sd[i]);
}
// A row of four nodes at P = 3 (every array 16-byte aligned: n^3 = 64 features per variable).
__device__ __forceinline__ void feature_row(const FeatureOut& f, int e, int node, int v, const float s[4]) {
  const int slot = v - f.first_var;
  if (slot < 0 || slot >= f.n_vars) return;
  const int i = slot * 64 + node;
  float sh[4], sd[4], x[4];
  row_read(f.shift32 + i, sh);
  row_read(f.sd + i, sd);
#pragma unroll
  for (int m = 0; m < 4; ++m) x[m] = (s[m] - sh[m]) / sd[m];
  const __nv_bfloat162 lo = __floats2bfloat162_rn(x[0], x[1]), hi = __floats2bfloat162_rn(x[2], x[3]);
  *reinterpret_cast<uint2*>(static_cast<__nv_bfloat16*>(f.out) + (long long)e * f.ld + i) =
      make_uint2(*reinterpret_cast<const unsigned*>(&lo), *reinterpret_cast<const unsigned*>(&hi));
}

constexpr int kStateElems = 4;   // per block of 256 threads
__device__ __forceinline__ void state4_block(int blk, const double* __restrict__ q, float* __restrict__ qf, int nel,
                                             const OpConst<float>& C) {
  const int e = blk * kStateElems + (threadIdx.x >> 6), node = threadIdx.x & 63;
  if (e >= nel) return;
  float s[5];
  state_from_q(q, (long long)e * 64 + node, C, s);
#pragma unroll
  for (int v = 0; v < 5; ++v) qf[(size_t)e * state_record(4) + v * 64 + node] = s[v];
  if (C.feat.out != nullptr) {
#pragma unroll
    for (int v = 0; v < 5; ++v) feature_store(C.feat, e, 64, node, v, s[v]);
  }
}

template <typename T>   // float only
__global__ void __launch_bounds__(256) k_state4(const double* __restrict__ q, T* __restrict__ qf, int nel,
                                                const OpConst<T> C) {
  pdl_wait();
  pdl_release();
  state4_block(blockIdx.x, q, qf, nel, C);
}

constexpr int kRows4Floats = 18 * 64;   // shared floats per element: U, halo rows (4 + 4), y- and z-fluxes (10)

template <int SRC, bool CUBE>
__device__ __forceinline__ void volume4_block(int blk, const double* __restrict__ q, float* qf, float* __restrict__ rv,
                                              float* __restrict__ vt, const OpConst<float>& C) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int E = CUBE ? kCubeElems : C.E;
  const int le = threadIdx.x >> 4, r = threadIdx.x & 15, j = r & 3, k = r >> 2;
  const int e = CUBE ? cube_element(cube_coords(blk, C.K), le, C.K) : C.e_begin + blk * E + le;
  // an element's 16 threads are half a warp: with an odd number of elements the other half idles
  const bool active = le < E && e < C.nel;
  const unsigned half = 0xffffu << (threadIdx.x & 16);
  if (!active) return;
  float* sU = reinterpret_cast<float*>(smem_raw) + le * kRows4Floats;   // [4][16 rows][4]
  float* sH = sU + 4 * 64;                                              // [4][16 halo rows][4]
  float* sF = sU + 8 * 64;                                              // [2][5][16 rows][4]
  const bool wide = (reinterpret_cast<size_t>(q) & 15) == 0;

  // own row; halo row r: faces y-, y+ (r / 4 = 0, 1; row k = r % 4), then z-, z+ (row j = r % 4);
  // the x faces' one node on each side
  const int hside = (r >> 2) & 1, hz = r >> 3;
  const int hrow = hz ? (r & 3) + (hside ? 0 : 12) : (hside ? 0 : 3) + 4 * (r & 3);
  const BlockCoords bc = block_coords(e, C.K);
  const int base_y = C.K * (bc.y + C.K * bc.z);
  const int exl = wrap_step(bc.x, -1, C.K) + base_y, exr = wrap_step(bc.x, 1, C.K) + base_y;
  const int hstep = hside ? 1 : -1;
  const int eh = hz ? bc.x + C.K * (bc.y + C.K * wrap_step(bc.z, hstep, C.Kz))
                    : bc.x + C.K * (wrap_step(bc.y, hstep, C.K) + C.K * bc.z);

  float s[5][4];
  state_row<SRC>(q, qf, e, 4 * r, wide, C, s);
  float UL[4], UR[4];
  {
    float hs[5][4], xl[5], xr[5];
    state_row<SRC>(q, qf, eh, 4 * hrow, wide, C, hs);
    if (SRC == 0) {
      state_from_q(q, (long long)exl * 64 + 4 * r + 3, C, xl);
      state_from_q(q, (long long)exr * 64 + 4 * r, C, xr);
    } else {
#pragma unroll
      for (int v = 0; v < 5; ++v) xl[v] = state_value<SRC>(qf + (size_t)exl * state_record(4) + v * 64 + 4 * r + 3);
#pragma unroll
      for (int v = 0; v < 5; ++v) xr[v] = state_value<SRC>(qf + (size_t)exr * state_record(4) + v * 64 + 4 * r);
    }
    float hU[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float t[5] = {hs[0][i], hs[1][i], hs[2][i], hs[3][i], hs[4][i]};
      float u[4];
      gradient_vars(t, prim_c(t, C), C.theta_ref, u);
#pragma unroll
      for (int a = 0; a < 4; ++a) hU[a][i] = u[a];
    }
#pragma unroll
    for (int a = 0; a < 4; ++a) row_store(sH + a * 64 + 4 * r, hU[a]);
    gradient_vars(xl, prim_c(xl, C), C.theta_ref, UL);
    gradient_vars(xr, prim_c(xr, C), C.theta_ref, UR);
  }
  float U[4][4], pp[4], rho[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float t[5] = {s[0][i], s[1][i], s[2][i], s[3][i], s[4][i]};
    const Prim<float> w = prim_c(t, C);
    float u[4];
    gradient_vars(t, w, C.theta_ref, u);
#pragma unroll
    for (int a = 0; a < 4; ++a) U[a][i] = u[a];
    pp[i] = w.pp;
    rho[i] = w.rho;
  }
#pragma unroll
  for (int a = 0; a < 4; ++a) row_store(sU + a * 64 + 4 * r, U[a]);
  if (SRC == 0) {
#pragma unroll
    for (int v = 0; v < 5; ++v) row_store(qf + (size_t)e * state_record(4) + v * 64 + 4 * r, s[v]);
  }
  // the other rows of this row's y- and z-line (j ^ m, k ^ m) and their matrix entries
  f32x2 Dy[4], Dz[4];
  int yat[3], zat[3];
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    const float dy = C.D[4 * j + (j ^ m)], dz = C.D[4 * k + (k ^ m)];
    Dy[m] = pack2(dy, dy);
    Dz[m] = pack2(dz, dz);
    if (m) {
      yat[m - 1] = 4 * ((j ^ m) + 4 * k);
      zat[m - 1] = 4 * (j + 4 * (k ^ m));
    }
  }
  __syncwarp(half);

  // BR1 gradient G[d][a][node], lifted with the central U^ = (U + U_nb) / 2
  float G[3][4][4];
  const float lift = C.s2h * C.winv * 0.5f;
#pragma unroll
  for (int a = 0; a < 4; ++a) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      float g = 0.f;
#pragma unroll
      for (int m = 0; m < 4; ++m) g += C.D[4 * i + m] * U[a][m];
      G[0][a][i] = mul_(C.s2h, g);
    }
    G[0][a][0] = fma_(-lift, UL[a] - U[a][0], G[0][a][0]);
    G[0][a][3] = fma_(lift, UR[a] - U[a][3], G[0][a][3]);
    const Row own{pack2(U[a][0], U[a][1]), pack2(U[a][2], U[a][3])};
    rows_contract(own, sU + a * 64, yat, Dy, G[1][a]);
    rows_contract(own, sU + a * 64, zat, Dz, G[2][a]);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      G[1][a][i] = mul_(C.s2h, G[1][a][i]);
      G[2][a][i] = mul_(C.s2h, G[2][a][i]);
    }
  }
  if (j == 0 || j == 3) {
    const float sg = j ? lift : -lift;
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      float nb[4];
      row_read(sH + a * 64 + 4 * ((j ? 4 : 0) + k), nb);
#pragma unroll
      for (int i = 0; i < 4; ++i) G[1][a][i] = fma_(sg, nb[i] - U[a][i], G[1][a][i]);
    }
  }
  if (k == 0 || k == 3) {
    const float sg = k ? lift : -lift;
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      float nb[4];
      row_read(sH + a * 64 + 4 * (8 + (k ? 4 : 0) + j), nb);
#pragma unroll
      for (int i = 0; i < 4; ++i) G[2][a][i] = fma_(sg, nb[i] - U[a][i], G[2][a][i]);
    }
  }

  // viscous quantities (xx, yy, zz, xy, xz, yz, k th_x, k th_y, k th_z)
  float vis[9][4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    float g[3][4];
#pragma unroll
    for (int d = 0; d < 3; ++d)
#pragma unroll
      for (int a = 0; a < 4; ++a) g[d][a] = G[d][a][i];
    float mu, lam;
    transport_c(C, rho[i], g, &mu, &lam);
    const float t23 = float(2.0 / 3.0) * mu * (g[0][0] + g[1][1] + g[2][2]);
    vis[0][i] = 2.f * mu * g[0][0] - t23;
    vis[1][i] = 2.f * mu * g[1][1] - t23;
    vis[2][i] = 2.f * mu * g[2][2] - t23;
    vis[3][i] = mu * (g[1][0] + g[0][1]);
    vis[4][i] = mu * (g[2][0] + g[0][2]);
    vis[5][i] = mu * (g[2][1] + g[1][2]);
    vis[6][i] = lam * g[0][3];
    vis[7][i] = lam * g[1][3];
    vis[8][i] = lam * g[2][3];
  }
  // face-normal viscous fluxes in the faces' frames (see volume_block)
  float* ve = vt + (size_t)e * face_record(4);
  ve[r] = vis[0][0];                        // x-: tau_xx, -tau_xy, -tau_xz, -k th_x
  ve[16 + r] = -vis[3][0];
  ve[32 + r] = -vis[4][0];
  ve[48 + r] = -vis[6][0];
  ve[64 + r] = vis[0][3];                   // x+
  ve[80 + r] = vis[3][3];
  ve[96 + r] = vis[4][3];
  ve[112 + r] = vis[6][3];
  if (j == 0 || j == 3) {                   // y: tau_yy, tau_yz, tau_yx, k th_y
    const float sg = j ? 1.f : -1.f;
    float* o = ve + (j ? 192 : 128) + 4 * k;
    float t[3][4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      t[0][i] = sg * vis[5][i];
      t[1][i] = sg * vis[3][i];
      t[2][i] = sg * vis[7][i];
    }
    row_store(o, vis[1]);
    row_store(o + 16, t[0]);
    row_store(o + 32, t[1]);
    row_store(o + 48, t[2]);
  }
  if (k == 0 || k == 3) {                   // z: tau_zz, tau_zx, tau_zy, k th_z
    const float sg = k ? 1.f : -1.f;
    float* o = ve + (k ? 320 : 256) + 4 * j;
    float t[3][4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      t[0][i] = sg * vis[4][i];
      t[1][i] = sg * vis[5][i];
      t[2][i] = sg * vis[8][i];
    }
    row_store(o, vis[2]);
    row_store(o + 16, t[0]);
    row_store(o + 32, t[1]);
    row_store(o + 48, t[2]);
  }

  // volume fluxes: x contracted in registers, y and z through shared memory
  float R[5][4];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    float F[5][4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float t[5] = {s[0][i], s[1][i], s[2][i], s[3][i], s[4][i]};
      Prim<float> w;
      w.v[0] = U[0][i];
      w.v[1] = U[1][i];
      w.v[2] = U[2][i];
      w.pp = pp[i];
      float f[5], fv[5], vi[9];
#pragma unroll
      for (int c = 0; c < 9; ++c) vi[c] = vis[c][i];
      euler_flux(t, w, C.Hc, d, f);
      viscous_flux(vi, w.v, d, fv);
#pragma unroll
      for (int c = 0; c < 5; ++c) F[c][i] = f[c] - fv[c];
    }
#pragma unroll
    for (int c = 0; c < 5; ++c) {
      if (d == 0) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          float g = 0.f;
#pragma unroll
          for (int m = 0; m < 4; ++m) g = fma_(C.D[4 * i + m], F[c][m], g);
          R[c][i] = mul_(-C.s2h, g);
        }
      } else {
        row_store(sF + (5 * (d - 1) + c) * 64 + 4 * r, F[c]);
      }
    }
  }
  __syncwarp(half);
  // Each line is summed before it is scaled and added: D's large entries make every partial
  // sum several times the derivative, and R must not be rounded at that size.
  float* re = rv + (size_t)e * state_record(4) + 4 * r;
#pragma unroll
  for (int c = 0; c < 5; ++c) {
    const float* fy = sF + c * 64;
    const float* fz = fy + 5 * 64;
    float g[4];
    rows_contract(row_load(fy + 4 * r), fy, yat, Dy, g);
#pragma unroll
    for (int i = 0; i < 4; ++i) R[c][i] = fma_(-C.s2h, g[i], R[c][i]);
    rows_contract(row_load(fz + 4 * r), fz, zat, Dz, g);
#pragma unroll
    for (int i = 0; i < 4; ++i) R[c][i] = fma_(-C.s2h, g[i], R[c][i]);
    row_store(re + c * 64, R[c]);
  }
}

// Threads, shared memory and register budget of a phase-A block of E elements.
template <int P, typename T, bool SPLIT>
__host__ __device__ constexpr int volume_threads(int E) {
  const int t = use_rows4(P, sizeof(T), SPLIT) ? 16 * E : E * (P + 1) * (P + 1) * (P + 1);
  return (t + 31) / 32 * 32;
}
template <int P, typename T, bool SPLIT>
__host__ __device__ constexpr size_t volume_smem(int E, bool cube) {
  return use_rows4(P, sizeof(T), SPLIT)
             ? sizeof(float) * (size_t)kRows4Floats * E
             : volume_smem_bytes<P, T>(E, (cube ? 3 : 6) * E * (P + 1) * (P + 1), SPLIT);
}
template <int P, typename T, bool SPLIT>
__host__ __device__ constexpr int volume_max_threads() {
  return use_rows4(P, sizeof(T), SPLIT) ? 128 : max_threads_for(P);
}
template <int P, typename T, bool SPLIT>
__host__ __device__ constexpr int volume_min_blocks() {
  return use_rows4(P, sizeof(T), SPLIT) ? 4 : sizeof(T) == 8 ? 1 : P == 1 ? 4 : P == 6 ? 3 : 2;
}

template <int P, typename T, int SRC, bool CUBE = false, bool FEAT = false, bool SPLIT = false>
__device__ __forceinline__ void volume_phase(int blk, const double* __restrict__ q, T* qf, T* __restrict__ rv,
                                             T* __restrict__ vt, const OpConst<T>& C) {
  if constexpr (use_rows4(P, sizeof(T), SPLIT)) volume4_block<SRC, CUBE>(blk, q, qf, rv, vt, C);
  else volume_block<P, T, SRC, CUBE, FEAT, SPLIT>(blk, q, qf, rv, vt, C);
}

// BESIDE: launched after the forcing network of the same stage state, to run beside it on the
// SMs it leaves idle.  The network releases this launch after its own wait, so the stage state
// was complete, and at the L2, before any block here starts.  This launch has waited for
// nothing itself, and this SM's L1 may hold lines of the former contents: the fence pairs with the
// network's ahead of its release, and the state is read past the L1, by loads the compiler can
// neither move above the fence nor take for read-only.  Everything else read here is a kernel
// parameter.  The wait for the network comes last: the next launch, which waits for this one
// only, must be one that waits before it touches memory (phase B).
template <int P, typename T, int SRC, bool CUBE = false, bool FEAT = false, bool SPLIT = false, bool BESIDE = false>
__global__ void __launch_bounds__(volume_max_threads<P, T, SPLIT>(), volume_min_blocks<P, T, SPLIT>())
k_volume(const double* __restrict__ q, T* qf, T* __restrict__ rv, T* __restrict__ vt, const OpConst<T> C) {
  static_assert(!BESIDE || SRC == 1, "beside the network the stage state exists");
  if (BESIDE) asm volatile("fence.acq_rel.gpu;" ::: "memory");
  else pdl_wait();
  if (C.early) pdl_release();
  volume_phase<P, T, BESIDE ? 2 : SRC, CUBE, FEAT, SPLIT>(blockIdx.x, q, qf, rv, vt, C);
  pdl_release();
  if (BESIDE) pdl_wait();
}

// ---------------------------------------------------------------- phase B

// Per-launch RK data of phase B in the arithmetic of the update.
template <typename R>
struct RkArgs {
  R A, B, dt;   // Williamson coefficients of the stage and the step size
  R invB1;      // 1 / B of stage 1 (the FP32 increment scheme recovers g1 = dlt1 / B1)
  R wc;         // B A of stage 3: the share of g2 in the final increment
};

// Operands of phase B on one mesh.
template <typename T>
struct SurfArgs {
  double* q;          // FP64 state
  const T* s;         // stage state of this stage
  const T* rv;        // volume term
  const T* vt;        // face-normal viscous fluxes
  double* dqdt;       // MODE 0
  T* g;               // MODE 1: RK register
  T* x;               // MODE 2: s1 (read); MODE 3: s1, replaced by s3
  T* y;               // MODE 2: s2, MODE 5: the next step's s1 (written)
  float* dlt;         // MODES 2 to 5: increment (see the head of this file)
};

// The FP32 increment scheme, one value.  Stage 1: g1 = dt R, d1 = B1 g1, s2 = s1 + d1.
// Stage 2: g2 = A2 g1 + dt R with g1 = d1 / B1, d2 = d1 + B2 g2, s3 = s1 + d2, and
// w = d2 + B3 A3 g2, all that stage 3 needs of them.  Stage 3: d3 = d2 + B3 (A3 g2 + dt R).
template <typename T>
__device__ __forceinline__ void rk_stage1(const RkArgs<T>& rk, T R, T s1, T& d1, T& s2) {
  d1 = mul_(rk.B, mul_(rk.dt, R));
  s2 = add_(s1, d1);
}
template <typename T>
__device__ __forceinline__ void rk_stage2(const RkArgs<T>& rk, T R, T s1, T d1, T& w, T& s3) {
  const T g2 = fma_(rk.A, mul_(d1, rk.invB1), mul_(rk.dt, R));
  const T d2 = fma_(rk.B, g2, d1);
  s3 = add_(s1, d2);
  w = fma_(rk.wc, g2, d2);
}
template <typename T>
__device__ __forceinline__ T rk_stage3(const RkArgs<T>& rk, T R, T w) {
  return fma_(rk.B, mul_(rk.dt, R), w);
}

// Square root and its square's inverse of c2 = c^2, from one reciprocal square root (FP32:
// the approximate instruction).
__device__ __forceinline__ void sound(float c2, float* c, float* inv_c2) {
  const float r = rsqrtf(c2);
  *c = c2 * r;
  *inv_c2 = r * r;
}
__device__ __forceinline__ void sound(double c2, double* c, double* inv_c2) {
  const double r = rsqrt(c2);
  *c = mul_(c2, r);
  *inv_c2 = mul_(r, r);
}

// One side of an interface in the face's frame: normal component first, pointing out of
// the element the frame belongs to.
template <typename T>
struct FaceState {
  T s[5];     // rho', m_n, m_t1, m_t2, e (reference-shifted)
  T rho, ir, vn, v1, v2, pp, h;   // h = rho e + p
};

template <typename T>
__device__ __forceinline__ void face_state(FaceState<T>& f, const OpConst<T>& C) {
  f.vn = mul_(f.s[1], f.ir);
  f.v1 = mul_(f.s[2], f.ir);
  f.v2 = mul_(f.s[3], f.ir);
  const T mv = fma_(f.s[1], f.vn, fma_(f.s[2], f.v1, mul_(f.s[3], f.v2)));
  f.pp = mul_(C.gm1, fma_(T(-0.5), mv, f.s[4]));
  f.h = add_(add_(f.s[4], f.pp), C.Hc);
}

// Densities of both sides of a face, their reciprocals, rt = sqrt(rho_o rho_b) and
// wd = 1 / (sqrt rho_o + sqrt rho_b)^2 = 1 / (rho_o + rho_b + 2 rt).  FP64: one division
// serves all three reciprocals (the FP64 pipe bounds that operator).
// Negative densities on both sides have a positive product: the root is then taken of one of
// them, so that a flow that has left the physical states gives NaN and not plausible fluxes.
__device__ __forceinline__ void face_densities(FaceState<float>& o, FaceState<float>& b, float rho_ref, float& rt,
                                               float& wd) {
  o.rho = add_(o.s[0], rho_ref);
  b.rho = add_(b.s[0], rho_ref);
  o.ir = drcp(o.rho);
  b.ir = drcp(b.rho);
  rt = dsqrt(o.rho < 0.f ? o.rho : mul_(o.rho, b.rho));
  wd = drcp(fma_(2.f, rt, add_(o.rho, b.rho)));
}
__device__ __forceinline__ void face_densities(FaceState<double>& o, FaceState<double>& b, double rho_ref, double& rt,
                                               double& wd) {
  o.rho = add_(o.s[0], rho_ref);
  b.rho = add_(b.s[0], rho_ref);
  const double pr = mul_(o.rho, b.rho);
  rt = sqrt(o.rho < 0.0 ? o.rho : pr);
  const double den = fma_(2.0, rt, add_(o.rho, b.rho));
  const double inv = 1.0 / mul_(pr, den), ipr = mul_(inv, den);
  wd = mul_(inv, pr);
  o.ir = mul_(b.rho, ipr);
  b.ir = mul_(o.rho, ipr);
}

// Interface terms of one face node in the frame of the own element (o) looking at its
// neighbour (b): with the outward fluxes f and f^nu, A = (f_b - f_o)/2 + (f^nu_o - f^nu_b)/2
// and B = |A~|(q_b - q_o)/2, so that f* - f = A - B on the own side.  to, tb: the viscous
// values each element stored for its side (volume_block), each in its own frame.
//
// The right and left element of a face evaluate the same expressions in mirrored frames
// (normal components change sign, own and neighbour exchange roles), and every expression
// here is exactly even or odd under that exchange: sums over the two sides are formed
// without contraction, the acoustic strengths enter as a1 + a5 and a5 - a1.  Both
// sides of a face therefore get the same flux to the last bit, without selecting left
// and right states.
//
// The Roe averages (sqrt rho_o u_o + sqrt rho_b u_b) / (sqrt rho_o + sqrt rho_b) are taken
// with numerator and denominator multiplied by the latter: (m_o + m_b + rt (u_o + u_b)) wd,
// which needs one square root instead of two.
template <typename T>
__device__ __forceinline__ void face_terms(FaceState<T>& o, FaceState<T>& b, const T to[4], const T tb[4],
                                           const OpConst<T>& C, T A[5], T B[5]) {
  const T half = T(0.5);
  T rt, wd;
  face_densities(o, b, C.rho_ref, rt, wd);
  face_state(o, C);
  face_state(b, C);
  const T un = mul_(fma_(rt, add_(o.vn, b.vn), add_(o.s[1], b.s[1])), wd);
  const T u1 = mul_(fma_(rt, add_(o.v1, b.v1), add_(o.s[2], b.s[2])), wd);
  const T u2 = mul_(fma_(rt, add_(o.v2, b.v2), add_(o.s[3], b.s[3])), wd);
  const T H = mul_(fma_(rt, add_(mul_(o.h, o.ir), mul_(b.h, b.ir)), add_(o.h, b.h)), wd);
  const T ke = mul_(half, fma_(un, un, fma_(u1, u1, mul_(u2, u2))));
  T c, ic2;
  sound(mul_(C.gm1, add_(H, -ke)), &c, &ic2);
  const T dr = add_(b.s[0], -o.s[0]), dp = add_(b.pp, -o.pp), dn = add_(b.vn, -o.vn);
  const T hc = mul_(half, ic2), x = mul_(rt, c);
  const T l1 = mul_(fabs(add_(un, -c)), mul_(fma_(-x, dn, dp), hc));
  const T l5 = mul_(fabs(add_(un, c)), mul_(fma_(x, dn, dp), hc));
  const T l2 = fabs(un), a2 = fma_(-dp, ic2, dr);
  const T ls = add_(l1, l5), ld = mul_(add_(l5, -l1), c);
  const T h1 = mul_(rt, add_(b.v1, -o.v1)), h2 = mul_(rt, add_(b.v2, -o.v2));   // shear waves
  B[0] = mul_(half, fma_(l2, a2, ls));
  B[1] = mul_(half, fma_(ls, un, fma_(l2, mul_(a2, un), ld)));
  B[2] = mul_(half, fma_(ls, u1, mul_(l2, fma_(a2, u1, h1))));
  B[3] = mul_(half, fma_(ls, u2, mul_(l2, fma_(a2, u2, h2))));
  B[4] = mul_(half, fma_(ls, H, fma_(ld, un, mul_(l2, fma_(a2, ke, fma_(u1, h1, mul_(u2, h2)))))));
  // outward fluxes; the neighbour stored its viscous values in its own frame
  const T eo = fma_(o.vn, to[0], fma_(o.v1, to[1], fma_(o.v2, to[2], to[3])));
  const T eb = fma_(b.vn, tb[0], -fma_(b.v1, tb[1], fma_(b.v2, tb[2], tb[3])));
  A[0] = mul_(half, add_(b.s[1], -o.s[1]));
  A[1] = mul_(half, add_(add_(fma_(b.s[1], b.vn, b.pp), -fma_(o.s[1], o.vn, o.pp)), add_(to[0], -tb[0])));
  A[2] = mul_(half, add_(add_(mul_(b.s[2], b.vn), -mul_(o.s[2], o.vn)), add_(to[1], tb[1])));
  A[3] = mul_(half, add_(add_(mul_(b.s[3], b.vn), -mul_(o.s[3], o.vn)), add_(to[2], tb[2])));
  // the energy flux is rounded with its viscous part in it, as the volume term rounds it: the
  // rounding of the own flux (a large number at low Mach numbers) then enters both alike and
  // partly cancels; rounded apart, the error of the FP32 energy grew by 2 to 4 % at P = 1, 2, 4
  A[4] = mul_(half, add_(fma_(b.vn, b.h, -eb), -fma_(o.vn, o.h, -eo)));
}

// Loads one side of a face item: the stage state at node fn of element record se and the
// viscous values at ve, in the frame with outward sign sg (the state's normal momentum).
template <int P, typename T>
__device__ __forceinline__ void load_side(const T* __restrict__ se, int fn, int d, T sg, T s[5]) {
  constexpr int ns = node_stride(P + 1);
  const int d1 = d == 2 ? 0 : d + 1, d2 = d == 0 ? 2 : d - 1;
  const T* p = se + fn;
  s[0] = p[0];
  s[1] = sg * p[(1 + d) * ns];
  s[2] = p[(1 + d1) * ns];
  s[3] = p[(1 + d2) * ns];
  s[4] = p[4 * ns];
}

// Elements and threads of a phase-B block (rows of elements).
__host__ __device__ constexpr int surf_elems(int P) {
  return P == 1 ? 16 : P == 2 ? 8 : P == 3 ? 8 : P == 4 ? 2 : 1;
}
__host__ __device__ constexpr int surf_threads(int P) {
  return P == 1 ? 128 : P == 2 ? 224 : P == 3 ? 128 : P == 4 ? 160 : P == 5 ? 224 : P == 6 ? 192 : P == 7 ? 128 : 256;
}
__host__ __device__ constexpr int surf_threads_cube(int P) { return P == 1 ? 96 : 192; }
// Orders whose phase-B blocks may be cubes (on a whole mesh of even K): the cube's 36 face
// evaluations instead of 48 pay where those bound the launch, on the FP64 pipe; in FP32 rows
// win (16^3/P3: 48.5 against 52.4 us per RK3 step).
__host__ __device__ constexpr bool surf_cube(int P, int tsize) { return tsize == 8 && P <= 3; }
// Blocks per SM the phase-B kernel is compiled for: 64 registers per thread in FP32, 128 in FP64.
__host__ __device__ constexpr int surf_min_blocks(int threads, int tsize) {
  const int blocks = (tsize == 8 ? 512 : 1024) / threads;
  return blocks > 0 ? blocks : 1;
}

// Shared memory of a phase-B block: neighbour elements [6 E] (int), lifted interface terms
// [5][E 6 n^2].
template <int P, typename T>
__host__ __device__ constexpr size_t surface_smem_bytes(int E) {
  return ((6 * E + 3) & ~3) * sizeof(int) + sizeof(T) * 5 * E * 6 * (P + 1) * (P + 1);
}

// MODE 0: dqdt = R.  MODE 1: FP64 RK stage (g = A g + dt R; q += B g).
// MODES 2, 3, 4: FP32 increment scheme, stages 1, 2, 3; MODE 5: stage 3 that also writes the
// next step's s1 (to y: neighbours still read s3 in x).
// Phase B of block `blk` of one mesh, E elements (the body of k_surface and k_surface_batch).
// prologue: work that may run before the previous launch has completed.
template <int P, typename T, bool CUBE>
__device__ __forceinline__ void surface_prologue(int blk, int E, const OpConst<T>& C) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  int* sNb = reinterpret_cast<int*>(smem_raw);
  const int e0 = C.e_begin + blk * E;
  const BlockCoords bc = CUBE ? cube_coords(blk, C.K) : BlockCoords{0, 0, 0};
  for (int t = threadIdx.x; t < 6 * E; t += blockDim.x) {
    const int hl = t / 6, eh = CUBE ? cube_element(bc, hl, C.K) : e0 + hl;
    sNb[t] = element_across(eh, t - 6 * hl, C.K, C.Kz);
  }
  __syncthreads();
}

template <int P, typename T, int MODE, bool CUBE = false, bool FEAT = false>
__device__ __forceinline__ void surface_block(int blk, int E, const SurfArgs<T>& a, const Forcing& fc,
                                              const OpConst<T>& C, const RkArgs<T>& rk) {
  constexpr int n = P + 1, n2 = n * n, np = n2 * n, ns = node_stride(n);
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int* sNb = reinterpret_cast<const int*>(smem_raw);
  T* sS = reinterpret_cast<T*>(smem_raw + ((6 * E + 3) & ~3) * sizeof(int));   // [5][E 6 n2]
  const int faceN = E * 6 * n2;
  const int e0 = C.e_begin + blk * E;
  const BlockCoords bc = CUBE ? cube_coords(blk, C.K) : BlockCoords{0, 0, 0};
  const T lift = C.s2h * C.winv;

  // interface terms; in a cube the external faces first, then one item per internal face
  // node for both sides
  const int extN = CUBE ? 3 * kCubeElems * n2 : faceN;
  const int nItems = CUBE ? extN + 12 * n2 : faceN;
  for (int t = threadIdx.x; t < nItems; t += blockDim.x) {
    Item<P> it;
    if (!CUBE) {
      it = item_of<P>(t);
      if (e0 + it.hl >= C.nel) continue;
    } else if (t < extN) {
      it = cube_item_of<P>(t);
    } else {   // internal face node: the left element's right side
      const int u = t - extN, r = u / n2, d = r >> 2;
      it.ab = u - r * n2;
      it.hl = cube_left_of_pair(r & 3, d);
      it.face = 2 * d + 1;
    }
    const int d = it.face >> 1;
    const bool right = it.face & 1;
    const T sg = right ? T(1) : T(-1);
    const int e = CUBE ? cube_element(bc, it.hl, C.K) : e0 + it.hl;
    const int enb = sNb[6 * it.hl + it.face];
    const int st = d == 0 ? 1 : d == 1 ? n : n2;
    const int f0 = face_node<P>(d, 0, it.ab);
    FaceState<T> o, b;
    T to[4], tb[4];
    load_side<P>(a.s + (size_t)e * state_record(n), right ? f0 + P * st : f0, d, sg, o.s);
    load_side<P>(a.s + (size_t)enb * state_record(n), right ? f0 : f0 + P * st, d, sg, b.s);
    const T* vo = a.vt + (size_t)e * face_record(n) + it.face * (kFaceVis * n2) + it.ab;
    const T* vb = a.vt + (size_t)enb * face_record(n) + (it.face ^ 1) * (kFaceVis * n2) + it.ab;
#pragma unroll
    for (int i = 0; i < 4; ++i) to[i] = vo[i * n2];
#pragma unroll
    for (int i = 0; i < 4; ++i) tb[i] = vb[i * n2];
    T A[5], B[5];
    face_terms(o, b, to, tb, C, A, B);
    // lifted terms -(2/h)/w (f* - f) back in mesh components
    const int cn = (1 + d) * faceN, c1 = (1 + (d == 2 ? 0 : d + 1)) * faceN, c2 = (1 + (d == 0 ? 2 : d - 1)) * faceN;
    T* out = sS + item_index<P>(it.ab, it.face, it.hl);
    out[0] = mul_(-lift, add_(A[0], -B[0]));
    out[cn] = mul_(-lift * sg, add_(A[1], -B[1]));
    out[c1] = mul_(-lift, add_(A[2], -B[2]));
    out[c2] = mul_(-lift, add_(A[3], -B[3]));
    out[4 * faceN] = mul_(-lift, add_(A[4], -B[4]));
    if (CUBE && t >= extN) {
      // the right element's left side: A and B of the mirrored frame
      T* ob = sS + item_index<P>(it.ab, it.face ^ 1, it.hl | (1 << d));
      ob[0] = mul_(-lift, add_(A[0], B[0]));
      ob[cn] = mul_(lift, add_(-A[1], -B[1]));
      ob[c1] = mul_(-lift, add_(A[2], B[2]));
      ob[c2] = mul_(-lift, add_(A[3], B[3]));
      ob[4 * faceN] = mul_(-lift, add_(A[4], B[4]));
    }
  }
  __syncthreads();

  if constexpr (P == 3 && sizeof(T) == 4) {
    // a thread owns a row of four nodes along x: every access is a 16-byte vector
    const bool wide = (reinterpret_cast<size_t>(MODE == 0 ? a.dqdt : a.q) & 15) == 0;
    for (int t = threadIdx.x; t < E * 16; t += blockDim.x) {
      const int le = t >> 4, r = t & 15, j = r & 3, k = r >> 2;
      const int e = CUBE ? cube_element(bc, le, C.K) : e0 + le;
      if (!CUBE && e >= C.nel) break;
      const size_t o = (size_t)e * state_record(n) + 4 * r;
      const long long g = (long long)e * 64 + 4 * r;
      float R[5][4];
#pragma unroll
      for (int c = 0; c < 5; ++c) row_read(a.rv + o + c * 64, R[c]);
      // the lifted interface terms in a fixed order (x, y, z)
      const float* ss = sS + le * 96;
#pragma unroll
      for (int c = 0; c < 5; ++c) {
        R[c][0] += ss[c * faceN + r];
        R[c][3] += ss[c * faceN + 16 + r];
      }
      if (j == 0 || j == 3) {
#pragma unroll
        for (int c = 0; c < 5; ++c) {
          float l[4];
          row_read(ss + c * faceN + (j ? 48 : 32) + 4 * k, l);
#pragma unroll
          for (int i = 0; i < 4; ++i) R[c][i] += l[i];
        }
      }
      if (k == 0 || k == 3) {
#pragma unroll
        for (int c = 0; c < 5; ++c) {
          float l[4];
          row_read(ss + c * faceN + (k ? 80 : 64) + 4 * j, l);
#pragma unroll
          for (int i = 0; i < 4; ++i) R[c][i] += l[i];
        }
      }
      if (fc.s != nullptr) {
        const float* fs = fc.s + (long long)e * fc.stride + 4 * r;
#pragma unroll
        for (int c = 0; c < 5; ++c) {
          const int slot = c - fc.first_var;
          if (slot < 0 || slot >= fc.n_vars) continue;
#pragma unroll
          for (int i = 0; i < 4; ++i) R[c][i] += fs[slot * 64 + i];
        }
      }
#pragma unroll
      for (int c = 0; c < 5; ++c) {
        double q1[4];
        float u[4], v[4], x1[4], g1[4];
        if (MODE == 2 || MODE == 3) row_read(a.x + o + c * 64, x1);
        if (MODE >= 3) row_read(a.dlt + o + c * 64, g1);
        if (MODE >= 4) row_read64(a.q + c * C.N + g, wide, q1);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          if (MODE == 0) q1[i] = double(R[c][i]);
          else if (MODE == 2) rk_stage1(rk, R[c][i], x1[i], u[i], v[i]);
          else if (MODE == 3) rk_stage2(rk, R[c][i], x1[i], g1[i], u[i], v[i]);
          else q1[i] += f2d(rk_stage3(rk, R[c][i], g1[i]));
        }
        if (MODE == 2 || MODE == 3) {
          row_store(a.dlt + o + c * 64, u);
          row_store((MODE == 2 ? a.y : a.x) + o + c * 64, v);
          if constexpr (FEAT) feature_row(C.feat, e, 4 * r, c, v);
        } else {
          double* out = (MODE == 0 ? a.dqdt : a.q) + c * C.N + g;
          if (wide) {
            reinterpret_cast<double2*>(out)[0] = make_double2(q1[0], q1[1]);
            reinterpret_cast<double2*>(out)[1] = make_double2(q1[2], q1[3]);
          } else {
#pragma unroll
            for (int i = 0; i < 4; ++i) out[i] = q1[i];
          }
          if (MODE == 5) {
#pragma unroll
            for (int i = 0; i < 4; ++i) u[i] = shifted(q1[i], c, C);
            row_store(a.y + o + c * 64, u);
            if constexpr (FEAT) feature_row(C.feat, e, 4 * r, c, u);
          }
        }
      }
    }
  } else {
  for (int t = threadIdx.x; t < E * np; t += blockDim.x) {
    const int le = t / np, node = t - le * np;
    const int e = CUBE ? cube_element(bc, le, C.K) : e0 + le;
    if (!CUBE && e >= C.nel) break;
    const size_t o = (size_t)e * state_record(n) + node;
    const long long g = (long long)e * np + node;
    T R[5], g1[5], x1[5];
    double q1[5];
#pragma unroll
    for (int c = 0; c < 5; ++c) R[c] = a.rv[o + c * ns];
    if (MODE == 2 || MODE == 3) {
#pragma unroll
      for (int c = 0; c < 5; ++c) x1[c] = a.x[o + c * ns];
    }
    if (MODE >= 3) {
#pragma unroll
      for (int c = 0; c < 5; ++c) g1[c] = T(a.dlt[o + c * ns]);
    }
    if (MODE == 1) {
#pragma unroll
      for (int c = 0; c < 5; ++c) g1[c] = rk.A == T(0) ? T(0) : a.g[o + c * ns];
    }
    if (MODE == 1 || MODE >= 4) {
#pragma unroll
      for (int c = 0; c < 5; ++c) q1[c] = a.q[c * C.N + g];
    }
    const int idx[3] = {node % n, (node / n) % n, node / n2};
    // the lifted interface terms in a fixed order (x, y, z)
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const bool right = (idx[d] == P), left = (idx[d] == 0);
      if (!(right || left)) continue;
      const int h = item_index<P>(face_ab<P>(d, idx), 2 * d + (right ? 1 : 0), le);
#pragma unroll
      for (int c = 0; c < 5; ++c) R[c] += sS[c * faceN + h];
    }
    if (fc.s != nullptr) {
      const float* fs = fc.s + (long long)e * fc.stride + node;
#pragma unroll
      for (int c = 0; c < 5; ++c) {
        const int slot = c - fc.first_var;
        if (slot >= 0 && slot < fc.n_vars) R[c] += T(fs[slot * np]);
      }
    }
#pragma unroll
    for (int c = 0; c < 5; ++c) {
      if (MODE == 0) {
        a.dqdt[c * C.N + g] = double(R[c]);
      } else if (MODE == 1) {   // FP64 operator: plain 2N update of the FP64 state
        T gnew = mul_(rk.dt, R[c]);
        if (rk.A != T(0)) gnew = fma_(rk.A, g1[c], gnew);
        a.g[o + c * ns] = gnew;
        a.q[c * C.N + g] = fma_(double(rk.B), double(gnew), q1[c]);
      } else if (MODE == 2) {
        T d1, s2;
        rk_stage1(rk, R[c], x1[c], d1, s2);
        a.dlt[o + c * ns] = float(d1);
        a.y[o + c * ns] = s2;
      } else if (MODE == 3) {
        T w, s3;
        rk_stage2(rk, R[c], x1[c], g1[c], w, s3);
        a.x[o + c * ns] = s3;
        a.dlt[o + c * ns] = float(w);
      } else {
        const double qn = q1[c] + f2d(float(rk_stage3(rk, R[c], g1[c])));
        a.q[c * C.N + g] = qn;
        if (MODE == 5) a.y[o + c * ns] = shifted(qn, c, C);
      }
    }
  }
  }
}

// E elements per block (kCubeElems with CUBE), THREADS threads.  FEAT: also writes the network
// features of the stage state it forms (MODES 2, 3, 5; P = 3).
template <int P, typename T, int MODE, int E, int THREADS, bool CUBE, bool FEAT>
__global__ void __launch_bounds__(THREADS, surf_min_blocks(THREADS, sizeof(T)))
k_surface(SurfArgs<T> a, Forcing fc, const OpConst<T> C, RkArgs<T> rk) {
  // last block first: phase A has just written the end of the mesh, which is still in L2
  const int blk = gridDim.x - 1 - blockIdx.x;
  surface_prologue<P, T, CUBE>(blk, E, C);
  pdl_wait();
  surface_block<P, T, MODE, CUBE, FEAT>(blk, E, a, fc, C, rk);
  pdl_release();
}

// ---------------------------------------------------------------------------------------
// Batched launches: independent meshes of the same order P (different K, Re, closure,
// dt) share one launch.  Block b belongs to the instance whose block range holds it; the
// table travels as one kernel parameter, so its per-instance constants are read from the
// constant bank like the single-mesh kernels' own.
constexpr int kMaxBatch = 16;

template <typename T>
struct BatchTable {
  int n;                             // instances in this launch
  int early;                         // phase A lets the next launch in as it starts, not as it ends
  int block_start[kMaxBatch + 1];    // first phase-A block of each instance; block_start[n] = grid
  int surf_start[kMaxBatch + 1];     // the same for phase B
  int state_start[kMaxBatch + 1];    // the same for the state pass (P = 3, FP32)
  T* qs[kMaxBatch];                  // stage state of this stage
  T* rv[kMaxBatch];                  // volume term
  T* vt[kMaxBatch];                  // face-normal viscous fluxes
  SurfArgs<T> a[kMaxBatch];
  RkArgs<T> rk[kMaxBatch];
  OpConst<T> C[kMaxBatch];
  int* err[kMaxBatch];               // device error flag of the instance (may be NULL)
};

__device__ __forceinline__ int batch_instance(const int* start, int n, int b) {
  int i = 0;
  while (i + 1 < n && b >= start[i + 1]) ++i;
  return i;
}

template <typename T>   // float only
__global__ void __launch_bounds__(256) k_state4_batch(const __grid_constant__ BatchTable<T> tb) {
  pdl_wait();
  pdl_release();
  const int i = batch_instance(tb.state_start, tb.n, blockIdx.x);
  state4_block(blockIdx.x - tb.state_start[i], tb.a[i].q, tb.qs[i], tb.C[i].nel, tb.C[i]);
}

template <int P, typename T, int SRC>
__global__ void __launch_bounds__(volume_max_threads<P, T, false>(), volume_min_blocks<P, T, false>())
k_volume_batch(const __grid_constant__ BatchTable<T> tb) {
  pdl_wait();
  if (tb.early) pdl_release();
  const int i = batch_instance(tb.block_start, tb.n, blockIdx.x);
  volume_phase<P, T, SRC>(blockIdx.x - tb.block_start[i], tb.a[i].q, tb.qs[i], tb.rv[i], tb.vt[i], tb.C[i]);
  pdl_release();
}

template <int P, typename T, int MODE, int E, int THREADS>
__global__ void __launch_bounds__(THREADS, surf_min_blocks(THREADS, sizeof(T)))
k_surface_batch(const __grid_constant__ BatchTable<T> tb) {
  const int b = gridDim.x - 1 - blockIdx.x;
  const int i = batch_instance(tb.surf_start, tb.n, b);
  const int blk = b - tb.surf_start[i];
  surface_prologue<P, T, false>(blk, E, tb.C[i]);
  pdl_wait();
  surface_block<P, T, MODE>(blk, E, tb.a[i], Forcing{}, tb.C[i], tb.rk[i]);
  pdl_release();
}

}  // namespace dgnn
