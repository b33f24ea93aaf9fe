// Device kernels of the DG shallow-water right-hand side, the multirate
// Adams-Bashforth update and the limiters (CUDA, sm_103a).
//
// This file holds what the stage kernels share (traces, fluxes, Adams-Bashforth weights),
// the limiter kernels and the pieces of the kernel-split ablation, where one thread owns
// one element: its nodal state stays in registers, and the reference operators are
// staged once per CTA in shared memory. The stage kernels themselves are in
// kernels_team.cuh (SIMT, a team of lanes per element) and kernels_tc.cuh (tensor
// cores). Nodal arrays are node-major planes (node i of element e at plane[i * KS + e]),
// so a warp's loads and stores of one node cover consecutive elements: whole sectors,
// and nearly so for the neighbour traces of a mesh numbered with locality.
//
// Formulation. The state is stored as (eta, hu, hv) with the free surface
// eta = h + B. The momentum fluxes and the source are written about the datum
// eta = 0 ("pre-balanced"): with the cubature exact to degree 3N-1 and the face
// Gauss rule exact to degree 3N, the static parts g B^2/2 of the volume flux,
// g B grad B of the source and g (B^-)^2/2 of the face flux cancel element by
// element (divergence theorem), so dropping them gives the same semi-discrete
// R(Q) as Section 3 / Eq. well_balance in exact arithmetic while avoiding the
// cancellation of g h^2/2 against g h grad B in floating point:
//   volume:  F = (hu, hu u + p, hu v), G = (hv, hv u, hv v + p), p = g/2 eta (h - B),
//            S = (0, -g eta B_x, -g eta B_y);
//   faces:   pressure term of the well-balanced flux (own side "-")
//            g/2 eta^- (h^- - B^-) + g/4 (h*^+ - h*^-)(h*^+ + h*^-),
//            h*^{+-} = max(0, eta^{+-} - max(B^+, B^-)).
// Element reference split. With eta = eta0 + eta' and B = B0 + B' (eta0, B0 the
// element's values at its node 0), the pressure g/2 eta (eta - 2B) is a constant
// plus terms linear in eta' and B' with constant coefficients plus
// p'' = g/2 eta' (eta' - 2B'). For a constant or such a linear term P (a
// polynomial of degree N) the volume term plus the own-side face term is exactly
// the strong derivative -dP/dx (integration by parts, exact integration); with the
// source's -g eta0 grad B' the linear terms sum to -g h0 grad eta, h0 = eta0 - B0.
// So with p'' in the volume and face pressures, the source -g eta' grad B' and
// -g h0 (r_x Dr + s_x Ds) eta (and the y analogue) once, nothing large is left. The stage
// kernels go one step further where the rules are exact (kernels_team.cuh): pressure,
// source and this term together are the projection of -g h grad eta; the inexact schemes
// and the kernel-split ablation keep the parts.
// At ocean depths the pressure is ~1e5 where R is ~1, and on a beach a film of
// millimetres sits on a bed metres above the datum: the rewrite removes both
// cancellations, and a lake at rest at any level gives R = 0 exactly. Where both
// sides of a face are wet the jump h*^+ - h*^- is computed as eta^+ - eta^-,
// which it equals, instead of as a difference of two large depths.
// In the ablation, dry elements (the positivity pass's flag) take the depth form instead:
// p_d = g/2 h'^2 and source -g h' grad B', h' = eta' - B'. It differs from
// p'', -g eta' grad B' by the static pair -g/2 B'^2, -g B' grad B', whose volume,
// own-side face and source terms cancel exactly; with it a uniform film on a
// slope (h' = 0) has no cancelling terms left, as a lake at rest (eta' = 0) has
// none in the surface form. With md = 1 for the depth form, 0 for the surface
// form: p = g/2 (eta' - md B')(eta' - (2 - md) B'), source -g (eta' - md B') grad B'.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "kernel_types.hpp"

namespace swe {

// --------------------------------------------------------------------------
// small helpers

__device__ __forceinline__ int level_of(const Sched& sc, int e) {
  int l = 1;
#pragma unroll
  for (int t = 1; t < kMaxLevels; ++t)
    if (t < sc.L && e >= sc.off[t]) l = t + 1;
  return l;
}

template <typename T>
struct Vec16;
template <>
struct Vec16<float> {
  using type = float4;
  static constexpr int n = 4;
  __device__ __forceinline__ static void unpack(const float4& v, float* o) {
    o[0] = v.x; o[1] = v.y; o[2] = v.z; o[3] = v.w;
  }
  __device__ __forceinline__ static float4 pack(const float* o) { return make_float4(o[0], o[1], o[2], o[3]); }
};
template <>
struct Vec16<double> {
  using type = double2;
  static constexpr int n = 2;
  __device__ __forceinline__ static void unpack(const double2& v, double* o) { o[0] = v.x; o[1] = v.y; }
  __device__ __forceinline__ static double2 pack(const double* o) { return make_double2(o[0], o[1]); }
};

// Load LEN (multiple of 16 bytes) consecutive values.
template <typename T, int LEN>
__device__ __forceinline__ void load_row(const T* __restrict__ p, T (&o)[LEN]) {
  using V = Vec16<T>;
  const typename V::type* pv = reinterpret_cast<const typename V::type*>(p);
#pragma unroll
  for (int k = 0; k < LEN / V::n; ++k) V::unpack(pv[k], &o[k * V::n]);
}

template <typename T, int LEN>
__device__ __forceinline__ void load_row_global(const T* __restrict__ p, T (&o)[LEN]) {
  using V = Vec16<T>;
  const typename V::type* pv = reinterpret_cast<const typename V::type*>(p);
#pragma unroll
  for (int k = 0; k < LEN / V::n; ++k) V::unpack(__ldg(pv + k), &o[k * V::n]);
}

template <typename T, int LEN>
__device__ __forceinline__ void load_row_m(const T* p, T (&o)[LEN]) {
  using V = Vec16<T>;
  const typename V::type* pv = reinterpret_cast<const typename V::type*>(p);
#pragma unroll
  for (int k = 0; k < LEN / V::n; ++k) V::unpack(pv[k], &o[k * V::n]);
}

// Node-major element access: node i of the element at p is p[i * ks]. LEN >= NP
// registers; the padding entries read as zero.
template <typename T, int NP, int LEN>
__device__ __forceinline__ void load_nodes(const T* __restrict__ p, size_t ks, T (&o)[LEN]) {
#pragma unroll
  for (int i = 0; i < LEN; ++i) o[i] = i < NP ? __ldg(p + i * ks) : T(0);
}

template <typename T, int NP, int LEN>
__device__ __forceinline__ void store_nodes(T* __restrict__ p, size_t ks, const T (&o)[LEN]) {
#pragma unroll
  for (int i = 0; i < NP; ++i) p[i * ks] = o[i];
}

// Reciprocal and square root: hardware approximations in FP32 (about 1-2 ulp, no
// slow-path branches), correctly rounded in FP64.
__device__ __forceinline__ float recip(float x) { return __fdividef(1.0f, x); }
__device__ __forceinline__ double recip(double x) { return 1.0 / x; }
// sqrt of x >= 0; the floor keeps x = 0 at 0 (0 * finite) instead of 0 * inf
__device__ __forceinline__ float sqrt_nn(float x) { return x * rsqrtf(fmaxf(x, 1e-30f)); }
__device__ __forceinline__ double sqrt_nn(double x) { return sqrt(x); }
__device__ __forceinline__ float rsqrt_t(float x) { return rsqrtf(x); }
__device__ __forceinline__ double rsqrt_t(double x) { return 1.0 / sqrt(x); }

// a b + c in one rounding. Every product that meets a sum in the stage and limiter bodies
// is written with it (or with fma2): left to the compiler, a b + c d is fused on either
// side, and the separate launch and the batch kernel would round differently.
__device__ __forceinline__ float mad(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double mad(double a, double b, double c) { return __fma_rn(a, b, c); }
// Hardware reciprocal and inverse square root without the scaling that the plain calls
// spend on subnormal arguments (three more instructions each): depths above the dry
// threshold (Phys::hvel_f is a normal number) and squared speeds are normal numbers. FP64:
// the correctly rounded ones.
__device__ __forceinline__ float recip_fast(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ double recip_fast(double x) { return 1.0 / x; }
__device__ __forceinline__ float rsqrt_fast(float x) {
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ double rsqrt_fast(double x) { return rsqrt_t(x); }
// |u| + sqrt(x), x >= 0 (FP32: the square root as in sqrt_nn)
__device__ __forceinline__ float speed(float u, float x) { return mad(x, rsqrt_fast(fmaxf(x, 1e-30f)), fabsf(u)); }
__device__ __forceinline__ double speed(double u, double x) { return fabs(u) + sqrt(x); }


// Cache hints: start a line's trip from memory early, without holding registers.
// Only addresses inside live buffers are ever passed.
__device__ __forceinline__ void prefetch_l2(const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }

// Programmatic dependent launch. The kernels of a substep run one after the other on one
// stream; each lets the next one's CTAs start (dependents_may_launch), at its own start or
// when its warps are done with their elements (`early`), and itself reads only what no
// kernel writes (operators) before wait_for_previous, which returns when the kernel before
// it has completed and its stores are visible. Every kernel launched with launch_dependent (launch.hpp) calls it.
__device__ __forceinline__ void dependents_may_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void wait_for_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Loads of the arrays the kernels write (state, Adams-Bashforth history, half-step
// records, means, dry flags, P1 values): ordinary coherent global loads, never the
// read-only data path. Inside the persistent batch kernel other CTAs of the same
// launch wrote these arrays in earlier phases, and an ordinary load after the
// acquire of the phase counter sees their stores. The separate launches use the
// same loads, so both compile the stage and limiter bodies to the same code and a
// scenario's result is the same, bit for bit, alone and in a batch.
template <typename T>
__device__ __forceinline__ T ldm(const T* p) {
  return *p;
}

template <typename T>
__device__ __forceinline__ T tmax(T a, T b) { return a > b ? a : b; }
template <typename T>
__device__ __forceinline__ T tmin(T a, T b) { return a < b ? a : b; }

// Adams-Bashforth weights (equal steps) for R^(0), R^(-1), R^(-2), in the
// kernel's precision (no FP64 work on the FP32 path).
template <typename T>
__device__ __forceinline__ void ab_weights(int depth, T w[3]) {
  if (depth <= 1) { w[0] = T(1); w[1] = T(0); w[2] = T(0); }
  else if (depth == 2) { w[0] = T(1.5); w[1] = T(-0.5); w[2] = T(0); }
  else { w[0] = T(23) / T(12); w[1] = T(-16) / T(12); w[2] = T(5) / T(12); }
}

// Integral over [0, theta] of the Lagrange interpolant of R at tau = 0, -1, -2.
template <typename T>
__device__ __forceinline__ void ab_partial_weights(int depth, T t, T w[3]) {
  if (depth <= 1) { w[0] = t; w[1] = T(0); w[2] = T(0); }
  else if (depth == 2) { w[0] = t + T(0.5) * t * t; w[1] = T(-0.5) * t * t; w[2] = T(0); }
  else {
    const T t2 = t * t, t3 = t2 * t;
    w[0] = t3 / T(6) + T(0.75) * t2 + t;
    w[1] = -(t3 / T(3) + t2);
    w[2] = t3 / T(6) + T(0.25) * t2;
  }
}

__device__ __forceinline__ float level_dt(const Sched& sc, int l, float) { return sc.dtl_f[l - 1]; }
__device__ __forceinline__ double level_dt(const Sched& sc, int l, double) { return sc.dtl_d[l - 1]; }
__device__ __forceinline__ float eps_of(const Phys& ph, float) { return ph.eps_f; }
__device__ __forceinline__ double eps_of(const Phys& ph, double) { return ph.eps; }

__device__ __forceinline__ float phys_g(const Phys& ph, float) { return ph.g_f; }
__device__ __forceinline__ double phys_g(const Phys& ph, double) { return ph.g; }
__device__ __forceinline__ float phys_hvel(const Phys& ph, float) { return ph.hvel_f; }
__device__ __forceinline__ double phys_hvel(const Phys& ph, double) { return ph.hvel; }
__device__ __forceinline__ float phys_ff(const Phys& ph, int c, float) {
  return c == 0 ? ph.ff_h_f : (c == 1 ? ph.ff_hu_f : ph.ff_hv_f);
}
__device__ __forceinline__ double phys_ff(const Phys& ph, int c, double) {
  return c == 0 ? ph.ff_h : (c == 1 ? ph.ff_hu : ph.ff_hv);
}

__device__ __forceinline__ float phys_h0(const Phys& ph, float) { return ph.h0_f; }
__device__ __forceinline__ double phys_h0(const Phys& ph, double) { return ph.h0; }
__device__ __forceinline__ float phys_M(const Phys& ph, float) { return ph.tvb_M_f; }
__device__ __forceinline__ double phys_M(const Phys& ph, double) { return ph.tvb_M; }
__device__ __forceinline__ float phys_nu(const Phys& ph, float) { return ph.tvb_nu_f; }
__device__ __forceinline__ double phys_nu(const Phys& ph, double) { return ph.tvb_nu; }

__host__ __device__ constexpr int face_node(int N, int f, int m) {
  // node index of position m along face f (from vertex f to f+1), lattice order
  return f == 0 ? m : (f == 1 ? m * (N + 1) - m * (m - 1) / 2 + (N - m)
                               : (N - m) * (N + 1) - (N - m) * (N - m - 1) / 2);
}

__device__ __forceinline__ int face_node_rt(int N, int f, int m) { return face_node(N, f, m); }

// Stage the first S entries of the operator block into shared memory (all threads
// of the CTA): the whole block for the kernel-split ablation, the per-element
// operators [0, TAIL) for the positivity kernel and the ablation's traces.
template <typename T, int N, int S = OpLayout<N>::SIZE>
__device__ __forceinline__ void stage_ops(T* sops, const T* __restrict__ gops) {
  using V = Vec16<T>;
  const typename V::type* src = reinterpret_cast<const typename V::type*>(gops);
  typename V::type* dst = reinterpret_cast<typename V::type*>(sops);
  for (int i = threadIdx.x; i < S / V::n; i += blockDim.x) dst[i] = __ldg(src + i);
  __syncthreads();
}

// --------------------------------------------------------------------------
// the well-balanced local Lax-Friedrichs flux (pre-balanced form), own side "-"

// Traces at a face point relative to the face's reference point (Ef, Bf): surface
// e = eta - Ef, bed b = B - Bf, and the momenta.
template <typename T>
struct Trace {
  T e, hu, hv, b;
};

// (nx, ny) unit outward normal, (vx, vy) = (sJ/J) (nx, ny), hs = sJ/J / 2; the
// returned fluxes are already scaled by sJ/J for the lift. hg = g/2, qg = g/4.
// hf = Ef - Bf, the depth at the face's reference point, so depths are
// hf + (e - b) without cancelling two large values. epm, bpm: eta^- and B^-
// relative to the element's own eta0, B0; the own-side pressure is p'' or p_d by
// md (element reference split above).
template <typename T>
__device__ __forceinline__ void wb_flux(const Trace<T>& m, const Trace<T>& p, T hf, T epm, T bpm, T md, T nx,
                                        T ny, T vx, T vy, T hs, T g, T hg, T qg, T hvel, T& f0, T& f1, T& f2) {
  const T hm = hf + (m.e - m.b), hp = hf + (p.e - p.b);
  const T im = hm > hvel ? recip(hm) : T(0), ip = hp > hvel ? recip(hp) : T(0);
  const T um = m.hu * im, vm = m.hv * im;
  const T up = p.hu * ip, vp = p.hv * ip;
  const T bmax = tmax(m.b, p.b);
  // hydrostatically reconstructed depths and the normal mass fluxes they carry
  const T sm = tmax(T(0), hf + (m.e - bmax)), sp = tmax(T(0), hf + (p.e - bmax));
  const T unm = um * nx + vm * ny, unp = up * nx + vp * ny;
  const T lam = tmax(fabs(unm) + sqrt_nn(g * sm), fabs(unp) + sqrt_nn(g * sp));
  const T Fm = sm * unm, Fp = sp * unp;
  const T ds = (sm > T(0) && sp > T(0)) ? p.e - m.e : sp - sm;
  const T pres = hg * (epm - md * bpm) * (epm - (T(2) - md) * bpm) + qg * ds * (sp + sm);
  f0 = hs * ((Fm + Fp) - lam * ds);
  f1 = hs * ((Fm * um + Fp * up) - lam * (sp * up - sm * um)) + pres * vx;
  f2 = hs * ((Fm * vm + Fp * vp) - lam * (sp * vp - sm * vm)) + pres * vy;
}

// --------------------------------------------------------------------------
// positivity-preserving limiter (Algorithm 3) on an element held in registers.
// Trigger test, means and rescale in FP64 when the element needs limiting;
// returns the dry classification and the element means (eta, hu, hv).

template <typename T, int N>
__device__ __forceinline__ int positivity(T (&eta)[Dims<N>::NPP], T (&hu)[Dims<N>::NPP],
                                          T (&hv)[Dims<N>::NPP], const T (&bb)[Dims<N>::NPP],
                                          const T* __restrict__ sops, double Bbar, T rx, T ry, T sx,
                                          T sy, const Phys& ph, double* injected, T mean_out[3]) {
  using D = Dims<N>;
  using O = OpLayout<N>;
  const T* mw = sops + O::MW;
  T hmin = eta[0] - bb[0];
#pragma unroll
  for (int jn = 1; jn < D::NP; ++jn) hmin = tmin(hmin, eta[jn] - bb[jn]);
  const bool trig = ph.pp && (hmin <= eps_of(ph, T(0)));
  if (!trig) {
    T me = 0, mu = 0, mv = 0;
#pragma unroll
    for (int jn = 0; jn < D::NP; ++jn) {
      me += mw[jn] * eta[jn];
      mu += mw[jn] * hu[jn];
      mv += mw[jn] * hv[jn];
    }
    mean_out[0] = me; mean_out[1] = mu; mean_out[2] = mv;
    return 0;
  }
  double hbar = 0.0, hub = 0.0, hvb = 0.0;
#pragma unroll
  for (int jn = 0; jn < D::NP; ++jn) {
    const double w = (double)mw[jn];
    hbar += w * ((double)eta[jn] - (double)bb[jn]);
    hub += w * (double)hu[jn];
    hvb += w * (double)hv[jn];
  }
  const double h0 = ph.h0;
  if (hbar < 1.01 * h0) {  // dry (the 1% margin keeps a reset element dry under rounding)
    const double hn = ph.dry_mode ? hbar : h0;
#pragma unroll
    for (int jn = 0; jn < D::NP; ++jn) {
      eta[jn] = (T)(hn + (double)bb[jn]);
      hu[jn] = T(0);
      hv[jn] = T(0);
    }
    const double area = 2.0 / ((double)rx * (double)sy - (double)ry * (double)sx);
    *injected += area * (hn - hbar);
    mean_out[0] = (T)(hn + Bbar); mean_out[1] = T(0); mean_out[2] = T(0);
    return 1;
  }
  // P1 projection at the vertices (FP64), theta rescale toward the mean
  const T* t1 = sops + O::T1;
  double vh[3], vu[3], vv[3];
#pragma unroll
  for (int v = 0; v < 3; ++v) {
    double a = 0, b = 0, c = 0;
#pragma unroll
    for (int jn = 0; jn < D::NP; ++jn) {
      const double w = (double)t1[v * D::NPP + jn];
      a += w * ((double)eta[jn] - (double)bb[jn]);
      b += w * (double)hu[jn];
      c += w * (double)hv[jn];
    }
    vh[v] = a; vu[v] = b; vv[v] = c;
  }
  const double h1min = fmin(vh[0], fmin(vh[1], vh[2]));
  const double den = hbar - h1min;
  const double theta = den > 0.0 ? fmin(1.0, (hbar - h0) / den) : 1.0;
  const T* bary = sops + O::BARY;
#pragma unroll
  for (int jn = 0; jn < D::NP; ++jn) {
    const double l0 = bary[jn * 4 + 0], l1 = bary[jn * 4 + 1], l2 = bary[jn * 4 + 2];
    const double h1 = l0 * vh[0] + l1 * vh[1] + l2 * vh[2];
    const double u1 = l0 * vu[0] + l1 * vu[1] + l2 * vu[2];
    const double w1 = l0 * vv[0] + l1 * vv[1] + l2 * vv[2];
    eta[jn] = (T)(theta * (h1 - hbar) + hbar + (double)bb[jn]);
    hu[jn] = (T)(theta * (u1 - hub) + hub);
    hv[jn] = (T)(theta * (w1 - hvb) + hvb);
  }
  mean_out[0] = (T)(hbar + Bbar); mean_out[1] = (T)hub; mean_out[2] = (T)hvb;
  return 0;
}

// Vertex values of Pi1 (eta, hu, hv) for the TVB limiter (Section 5.3), stored
// as planes p1[(3 field + vertex) * KS + e] by whoever last committed the state.
template <typename T, int N>
__device__ __forceinline__ void store_p1(T* __restrict__ p1, size_t ks, const T* __restrict__ sops,
                                         const T (&eta)[Dims<N>::NPP], const T (&hu)[Dims<N>::NPP],
                                         const T (&hv)[Dims<N>::NPP]) {
  using D = Dims<N>;
  const T* t1 = sops + OpLayout<N>::T1;
#pragma unroll
  for (int v = 0; v < 3; ++v) {
    T s0 = 0, s1 = 0, s2 = 0;
#pragma unroll
    for (int jn = 0; jn < D::NP; ++jn) {
      const T w = t1[v * D::NPP + jn];
      s0 += w * eta[jn];
      s1 += w * hu[jn];
      s2 += w * hv[jn];
    }
    p1[(0 + v) * ks] = s0;
    p1[(3 + v) * ks] = s1;
    p1[(6 + v) * ks] = s2;
  }
}

// The reference part of the pressure and source in strong form (element
// reference split above): R_hu -= g h0 (r_x Dr + s_x Ds)(eta - eta0),
// R_hv -= g h0 (r_y Dr + s_y Ds)(eta - eta0), h0 = eta0 - B0 the depth at node 0.
template <typename T, int N>
__device__ __forceinline__ void add_reference_pressure(const T* __restrict__ sops, const T (&eta)[Dims<N>::NPP],
                                                       const T (&bb)[Dims<N>::NPP], T g, T rx, T ry, T sx,
                                                       T sy, T (&R1)[Dims<N>::NP], T (&R2)[Dims<N>::NP]) {
  using D = Dims<N>;
  using O = OpLayout<N>;
  constexpr int NP = D::NP, NPP = D::NPP;
  T d[NPP];
#pragma unroll
  for (int j = 0; j < NPP; ++j) d[j] = j < NP ? eta[j] - eta[0] : T(0);
  const T gb = -g * (eta[0] - bb[0]);
#pragma unroll
  for (int i = 0; i < NP; ++i) {
    T dr[NPP], ds[NPP];
    load_row<T, NPP>(sops + O::DR + i * NPP, dr);
    load_row<T, NPP>(sops + O::DS + i * NPP, ds);
    T er = 0, es = 0;
#pragma unroll
    for (int j = 0; j < NP; ++j) {
      er += dr[j] * d[j];
      es += ds[j] * d[j];
    }
    R1[i] += gb * (rx * er + sx * es);
    R2[i] += gb * (ry * er + sy * es);
  }
}

// --------------------------------------------------------------------------
// Volume term N(Q) (Section 7.1) of one element, accumulated into R: interpolate
// to the cubature points, volume flux and source there, project back.
template <typename T, int N>
__device__ __forceinline__ void volume_term(const T* __restrict__ sops, const T (&eta)[Dims<N>::NPP],
                                            const T (&hu)[Dims<N>::NPP], const T (&hv)[Dims<N>::NPP],
                                            const T (&bb)[Dims<N>::NPP], T rx, T ry, T sx, T sy, T md, T g,
                                            T hvel, T (&R0)[Dims<N>::NP], T (&R1)[Dims<N>::NP],
                                            T (&R2)[Dims<N>::NP]) {
  using D = Dims<N>;
  using O = OpLayout<N>;
  constexpr int NP = D::NP, NPP = D::NPP, NCUB = D::NCUB;
  const T hg = T(0.5) * g;
#pragma unroll 1
  for (int c = 0; c < NCUB; ++c) {
    T ic[NPP], icr[NPP], ics[NPP];
    load_row<T, NPP>(sops + O::IC + c * NPP, ic);
    load_row<T, NPP>(sops + O::ICR + c * NPP, icr);
    load_row<T, NPP>(sops + O::ICS + c * NPP, ics);
    // ec, bc, brc, bsc: of eta - eta0 and B - B0 (element reference split)
    T ec = 0, huc = 0, hvc = 0, bc = 0, brc = 0, bsc = 0;
#pragma unroll
    for (int jn = 0; jn < NP; ++jn) {
      const T ep = eta[jn] - eta[0], bp = bb[jn] - bb[0];
      ec += ic[jn] * ep;
      huc += ic[jn] * hu[jn];
      hvc += ic[jn] * hv[jn];
      bc += ic[jn] * bp;
      brc += icr[jn] * bp;
      bsc += ics[jn] * bp;
    }
    const T hc = (eta[0] - bb[0]) + (ec - bc);
    const T ih = hc > hvel ? recip(hc) : T(0);
    const T u = huc * ih, v = hvc * ih;
    // cF1 = rx F + ry G and cF2 = sx F + sy G, with the momentum rows written
    // through the mass row: rx (hu u + p) + ry hv u = u (rx hu + ry hv) + rx p;
    // p = p'' (element reference split)
    const T ep = ec - md * bc;
    const T pr = hg * ep * (ec - (T(2) - md) * bc);
    const T a0 = rx * huc + ry * hvc, b0 = sx * huc + sy * hvc;
    const T a1 = u * a0 + rx * pr, a2 = v * a0 + ry * pr;
    const T b1 = u * b0 + sx * pr, b2 = v * b0 + sy * pr;
    const T gm = -g * ep;
    const T S1 = gm * (rx * brc + sx * bsc), S2 = gm * (ry * brc + sy * bsc);
    T prt[NPP], pst[NPP], pt[NPP];
    load_row<T, NPP>(sops + O::PRT + c * NPP, prt);
    load_row<T, NPP>(sops + O::PST + c * NPP, pst);
    load_row<T, NPP>(sops + O::PT + c * NPP, pt);
#pragma unroll
    for (int i = 0; i < NP; ++i) {
      R0[i] += prt[i] * a0 + pst[i] * b0;
      R1[i] += prt[i] * a1 + pst[i] * b1 + pt[i] * S1;
      R2[i] += prt[i] * a2 + pst[i] * b2 + pt[i] * S2;
    }
  }
}

// --------------------------------------------------------------------------
// positivity limiter on the current state (initial limiting, swe_limit)

template <typename T, int N>
__global__ void __launch_bounds__(kBlock) k_positivity(LimitParams<T> p) {
  using D = Dims<N>;
  constexpr int NP = D::NP, NPP = D::NPP;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* sops = reinterpret_cast<T*>(smem_raw);
  stage_ops<T, N, OpLayout<N>::TAIL>(sops, p.s.ops);
  const Sched& sc = p.sc;
  const long long k = (*p.s.macro) * (1LL << (sc.L - 1)) + p.j;
  const size_t ks = (size_t)sc.KS, fstride = (size_t)NP * ks, bstride = 3 * fstride;
  double injected = 0.0;
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < p.nactive; e += gridDim.x * blockDim.x) {
    const int lev = level_of(sc, e);
    const long long a = k >> (lev - 1);
    const int cur = (int)((a + p.post_stage) & 1);
    const size_t eo = (size_t)e;
    T* q = p.s.q + cur * bstride;
    T eta[NPP], hu[NPP], hv[NPP], bb[NPP];
    load_nodes<T, NP, NPP>(q + eo, ks, eta);
    load_nodes<T, NP, NPP>(q + fstride + eo, ks, hu);
    load_nodes<T, NP, NPP>(q + 2 * fstride + eo, ks, hv);
    load_nodes<T, NP, NPP>(p.s.B + eo, ks, bb);
    const T rx = p.s.geo[4 * e], ry = p.s.geo[4 * e + 1], sx = p.s.geo[4 * e + 2], sy = p.s.geo[4 * e + 3];
    T mean[3];
    const int dryf = positivity<T, N>(eta, hu, hv, bb, sops, p.s.Bbar[e], rx, ry, sx, sy, p.ph, &injected, mean);
    store_nodes<T, NP, NPP>(q + eo, ks, eta);
    store_nodes<T, NP, NPP>(q + fstride + eo, ks, hu);
    store_nodes<T, NP, NPP>(q + 2 * fstride + eo, ks, hv);
    store_p1<T, N>(p.s.p1 + eo, ks, sops, eta, hu, hv);
    p.s.means[4 * (size_t)e + 0] = mean[0];
    p.s.means[4 * (size_t)e + 1] = mean[1];
    p.s.means[4 * (size_t)e + 2] = mean[2];
    p.s.dry[e] = (uint8_t)dryf;
    if (!(isfinite((double)mean[0]) && isfinite((double)mean[1]) && isfinite((double)mean[2])))
      atomicOr(p.s.flags, 1);
  }
  if (injected != 0.0) atomicAdd(p.s.acc, injected);
}

// --------------------------------------------------------------------------
// TVB limiter with the positivity modification (Section 5.3), P1 part of
// (eta, hu, hv), characteristic variables, midpoint deltas.

template <typename T>
__device__ __forceinline__ T minmod_tvb(T a, T b, T thr, bool& changed) {
  if (fabs(a) <= thr) return a;
  T r;
  if (a > 0 && b > 0) r = a < b ? a : b;
  else if (a < 0 && b < 0) r = a > b ? a : b;
  else r = T(0);
  if (r != a) changed = true;
  return r;
}

__device__ __forceinline__ float sqrt_fast(float x) { return x * rsqrt_fast(x); }
__device__ __forceinline__ double sqrt_fast(double x) { return sqrt(x); }

// The TVB limiter with the positivity modification on element e (k: the finest
// substep count of the schedule); returns without change for an element that is dry,
// has a dry neighbour or needs no limiting. ops: the operator block (shared or global
// memory; only an element that is limited reads it).
//
// What bounds it: the latency of its two dependent trips to memory (connectivity, then
// the neighbours' means) and of the arithmetic between them; small launches hardly fill
// a warp per scheduler. So the characteristic variables use the eigenvectors' closed-form
// inverse (one reciprocal per element instead of a 3 x 3 inverse per edge), the kernel
// stages nothing in shared memory, and the body is inlined with its parameters in the
// constant bank (as an out-of-line function it read them through generic loads). us per
// macro step before and after: 2,048 elements, N = 2 95 -> 83; 45k, N = 3 209 -> 197;
// 500k, N = 4 1285 -> 1254; FP64, 40k, N = 4 4785 -> 4665.
template <typename T, int N>
__device__ __forceinline__ void tvb_element(const ScnParams<T>& p, int post_stage, const T* ops, int e, long long k) {
  using D = Dims<N>;
  using O = OpLayout<N>;
  constexpr int NP = D::NP;
  const Sched& sc = p.sc;
  const T g = phys_g(p.ph, T(0)), h0 = phys_h0(p.ph, T(0));
  // Every load is issued before the first branch on loaded data (an element that is
  // dry or has a dry neighbour is skipped afterwards), so the latencies overlap.
  const int4 cn = __ldg(p.s.conn + e);
  const int de = ldm(p.s.dry + e);
  const int nbs[3] = {cn.x, cn.y, cn.z};
  const int lev = level_of(sc, e);
  const long long a = k >> (lev - 1);
  const int cur = (int)((a + post_stage) & 1);
  const size_t ks = (size_t)sc.KS, fstride = (size_t)NP * ks, bstride = 3 * fstride, eo = (size_t)e;
  T* q = p.s.q + cur * bstride + eo;
  // 16-byte rows: geometry, element means (eta, hu, hv, -) as stored by the
  // positivity pass, the neighbour-mean weights
  T gm[4], u0[4], tg[8];
  load_row_global<T, 4>(p.s.geo + 4 * eo, gm);
  load_row_m<T, 4>(p.s.means + 4 * eo, u0);
  load_row_global<T, 8>(p.s.tvbg + 8 * eo, tg);
  // P1 part: vertex values of Pi1 q for eta, hu, hv (stored with the committed state)
  T vq[3][3];
#pragma unroll
  for (int v = 0; v < 3; ++v) {
    vq[0][v] = ldm(p.s.p1 + (0 + v) * ks + eo);
    vq[1][v] = ldm(p.s.p1 + (3 + v) * ks + eo);
    vq[2][v] = ldm(p.s.p1 + (6 + v) * ks + eo);
  }
  const double Bbar_d = __ldg(p.s.Bbar + eo);
  // neighbour means and dry flags
  T un[3][4];
  int dn = 0;
#pragma unroll
  for (int f = 0; f < 3; ++f) {
    const int nb = nbs[f] < 0 ? e : nbs[f];   // a boundary face reads its own element's (replaced below)
    dn |= nbs[f] < 0 ? 0 : (int)ldm(p.s.dry + nb);
    load_row_m<T, 4>(p.s.means + 4 * (size_t)nb, un[f]);
  }
  if (de || dn) return;
  const T rx = gm[0], ry = gm[1], sx = gm[2], sy = gm[3];
  const T Bbar = (T)Bbar_d;
  // a far-field face sees the far-field state over the own mean bed; a wall face
  // mirrors the normal momentum of the own mean
#pragma unroll
  for (int f = 0; f < 3; ++f) {
    if (nbs[f] >= 0) continue;
    if (nbs[f] == kFarField) {
      un[f][0] = phys_ff(p.ph, 0, T(0)) + Bbar;
      un[f][1] = phys_ff(p.ph, 1, T(0));
      un[f][2] = phys_ff(p.ph, 2, T(0));
    } else {
      const T vxn = f == 0 ? -sx : (f == 1 ? rx + sx : -rx);
      const T vyn = f == 0 ? -sy : (f == 1 ? ry + sy : -ry);
      const T inv = rsqrt_fast(mad(vxn, vxn, vyn * vyn));
      const T nx = vxn * inv, ny = vyn * inv;
      const T mn = T(-2) * mad(u0[1], nx, u0[2] * ny);
      un[f][1] = mad(mn, nx, u0[1]);
      un[f][2] = mad(mn, ny, u0[2]);
    }
  }
  // physical midpoint-minus-centroid vectors from the affine map, up to the Jacobian
  const T Jd = recip_fast(mad(rx, sy, -(ry * sx)));
  const T dr[3] = {T(1) / 3, T(1) / 3, T(-2) / 3}, ds[3] = {T(-2) / 3, T(1) / 3, T(1) / 3};
  const T hb = u0[0] - Bbar;
  const T cb = sqrt_fast(g * hb), icb = recip_fast(cb), ihb = recip_fast(hb);
  const T ub = u0[1] * ihb, vb0 = u0[2] * ihb;
  const T floor = T(1e-6) * mad(sqrt_nn(mad(u0[1], u0[1], u0[2] * u0[2])), icb, hb);
  const T M = phys_M(p.ph, T(0)), nu = phys_nu(p.ph, T(0));
  bool changed = false;
  T dl[3][3];  // limited deltas, [edge][field]
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const int jj = (cn.w >> (6 + 2 * i)) & 3;
    const T al = tg[2 * i], be = tg[2 * i + 1];
    T dt_[3], dn_[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      dt_[c] = mad(T(0.5), vq[c][i] + vq[c][(i + 1) % 3], -u0[c]);
      const T uj = jj == 0 ? un[0][c] : (jj == 1 ? un[1][c] : un[2][c]);   // selects, no local array
      dn_[c] = mad(al, un[i][c] - u0[c], be * (uj - u0[c]));
    }
    const T mx = mad(sy, dr[i], -ry * ds[i]), my = mad(-sx, dr[i], rx * ds[i]);
    const T m2 = mad(mx, mx, my * my), im = rsqrt_fast(m2);
    const T nx = mx * im, ny = my * im, dist = Jd * (m2 * im);
    // characteristic variables: gravity waves (-, +) and shear of the linearised flux
    // Jacobian in the direction (nx, ny)
    auto waves = [&](const T (&d)[3], T (&w)[3]) {
      const T d1 = mad(-ub, d[0], d[1]), d2 = mad(-vb0, d[0], d[2]);
      const T un_ = mad(d1, nx, d2 * ny) * icb;
      w[0] = T(0.5) * (d[0] - un_);
      w[1] = mad(d2, nx, -d1 * ny);
      w[2] = T(0.5) * (d[0] + un_);
    };
    T wt[3], wn[3], wl[3];
    waves(dt_, wt);
    waves(dn_, wn);
    const T thr0 = mad(M * dist, dist, floor);
#pragma unroll
    for (int c = 0; c < 3; ++c) wl[c] = minmod_tvb<T>(wt[c], nu * wn[c], c == 1 ? thr0 * cb : thr0, changed);
    const T sum = wl[0] + wl[2], dif = cb * (wl[2] - wl[0]);
    dl[i][0] = sum;
    dl[i][1] = mad(ub, sum, mad(dif, nx, -ny * wl[1]));
    dl[i][2] = mad(vb0, sum, mad(dif, ny, nx * wl[1]));
  }
  if (!changed) return;
  T vb[3], bb[NP];   // Pi1 B at the vertices, the nodal bed
#pragma unroll
  for (int v = 0; v < 3; ++v) vb[v] = __ldg(p.s.vb + v * ks + eo);
#pragma unroll
  for (int jn = 0; jn < NP; ++jn) bb[jn] = __ldg(p.s.B + eo + jn * ks);
  // redistribution: deltas of each field sum to zero
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    T pos = 0, neg = 0;
#pragma unroll
    for (int i = 0; i < 3; ++i) { pos += tmax(dl[i][c], T(0)); neg += tmax(-dl[i][c], T(0)); }
    const T tp = pos > 0 ? tmin(T(1), neg / pos) : T(1);
    const T tn = neg > 0 ? tmin(T(1), pos / neg) : T(1);
#pragma unroll
    for (int i = 0; i < 3; ++i) dl[i][c] = mad(tp, tmax(dl[i][c], T(0)), -(tn * tmax(-dl[i][c], T(0))));
  }
  // depth deltas = eta deltas minus those of Pi1 B; positivity modification (Eq. modified_TVB)
  T dh[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) dh[i] = dl[i][0] - mad(T(0.5), vb[i] + vb[(i + 1) % 3], -Bbar);
  // vertex deltas of a field from its midpoint deltas
  auto vertices = [](const T (&d)[3], T (&S)[3]) {
    S[0] = d[0] + d[2] - d[1];
    S[1] = d[1] + d[0] - d[2];
    S[2] = d[2] + d[1] - d[0];
  };
  T S[3];
  vertices(dh, S);
  const T smin = tmin(S[0], tmin(S[1], S[2]));
  if (hb + smin < h0) {
    const T dbar = (dh[0] + dh[1] + dh[2]) / T(3);
    const T den = dbar - smin;
    T th = den > 0 ? (hb + dbar - h0) / den : T(1);
    th = tmin(T(1), tmax(T(0), th));
#pragma unroll
    for (int i = 0; i < 3; ++i) dh[i] = mad(th, dh[i] - dbar, dbar);
    vertices(dh, S);
  }
  const T du[3] = {dl[0][1], dl[1][1], dl[2][1]}, dv[3] = {dl[0][2], dl[1][2], dl[2][2]};
  T Su[3], Sv[3];
  vertices(du, Su);
  vertices(dv, Sv);
  // the P1 rebuild at the nodes, about the means: eta = eta-bar + sum_v l_v S_v + (B -
  // B-bar) with S_v the vertex deltas. The stored barycentric weights sum to one only to
  // rounding, so sum_v l_v (h-bar + S_v) would scale every rebuilt element's mean by that
  // sum; about the mean the rounding is of the size of the deltas, not of the depth.
#pragma unroll
  for (int jn = 0; jn < NP; ++jn) {
    const T l0 = ops[O::BARY + 4 * jn], l1 = ops[O::BARY + 4 * jn + 1], l2 = ops[O::BARY + 4 * jn + 2];
    q[jn * ks] = u0[0] + mad(l0, S[0], mad(l1, S[1], l2 * S[2])) + (bb[jn] - Bbar);
    q[fstride + jn * ks] = u0[1] + mad(l0, Su[0], mad(l1, Su[1], l2 * Su[2]));
    q[2 * fstride + jn * ks] = u0[2] + mad(l0, Sv[0], mad(l1, Sv[1], l2 * Sv[2]));
  }
}

// Elements e0, e0 + step, ... below e1 of the TVB limiter (post_stage: 1 limits the
// just-committed state, 0 the current one); the separate launch and the persistent batch
// kernel both inline it.
template <typename T, int N>
__device__ __forceinline__ void tvb_range(const ScnParams<T>& p, int post_stage, const T* ops, int e0, int step, int e1,
                                          long long k) {
  for (int e = e0; e < e1; e += step) tvb_element<T, N>(p, post_stage, ops, e, k);
}

template <typename T, int N>
__global__ void __launch_bounds__(kBlock, sizeof(T) == 4 ? 6 : 3) k_tvb(const __grid_constant__ LimitParams<T> p) {
  if (p.early) dependents_may_launch();
  wait_for_previous();
  const long long k = (*p.s.macro) * (1LL << (p.sc.L - 1)) + p.j;
  tvb_range<T, N>(p, p.post_stage, p.s.ops, blockIdx.x * blockDim.x + threadIdx.x, gridDim.x * blockDim.x, p.nactive,
                  k);
  if (!p.early) dependents_may_launch();
}

}  // namespace swe
