// SIMT stage kernel (FP32 and FP64 tiers): a team of L lanes works on each element.
//
// A warp holds a tile of E = 32 / L elements; lane = el + E * part. The element's
// state, its face traces and its fluxes pass between the lanes of the team through
// the warp's shared tile, and each phase deals its own items to the lanes:
//   gather    nodes of the own state (NB = NPP / L consecutive nodes per lane) and, one
//             lane per face, the neighbour's face nodes and the face's geometry
//   surface   FP32: the face's lane keeps its traces in registers and walks its Gauss
//             points (the shared-memory pipe bounds that tier). FP64: one lane per Gauss
//             point, traces through the tile (the FP64 pipe bounds it, and no lane idles)
//   volume    one lane per cubature point, L points at a time: interpolation and flux
//   project   FP32: each lane projects its own points onto all nodes, and the team's
//             partial sums meet in the tile once (a third fewer shared-memory reads than
//             passing every point's flux). FP64: the fluxes of L points pass through the
//             tile and each lane projects them onto its NB nodes
//   commit    one lane per NB nodes: mass operator, lift, Adams-Bashforth commit; the
//             limiter's reductions over the nodes are butterflies over the team
// Every item is computed once, so a team does the work of one thread per element and
// no more, with 1/L of its registers (three values of R for NB nodes instead of all)
// and 1/L of its serial chain: a mesh that cannot fill the GPU with one element per
// thread is L times faster through a step, and a large one runs twice the warps.
//
// Two exact rewrites of the volume term (polynomial identities under the rules of
// degree 3N - 1 and 3N, Dims::EXACT; see the formulation in kernels.cuh):
//   pressure and source  the weak pressure p'', its own-side face term, the source
//             -g eta' grad B' and the strong reference term -g h0 grad eta add up to
//             the projection of -g h grad eta, which has no cancelling parts at all
//             (eta = const gives zero). FP32 projects -g h' grad eta and adds the
//             reference term as a nodal product (Team::NODAL). So only h, hu, hv and the
//             two derivatives of eta are interpolated (five rows instead of six), two rows
//             per momentum carry advection alone and the faces keep only the pressure jump.
//   mass      hu and hv are polynomials of degree N, so their projection is one
//             nodal operator M^-1 D^T M (all schemes: degree 2N - 1 products): two
//             NP-long rows instead of two NCUB-long ones.
// The schemes with inexact rules keep p'', the source and the strong term.
//
// What bounds it. FP64: the FP64 pipe (two lanes per SM and clock: a warp instruction
// takes 16 clocks of an SM and holds its warp for 64), so what counts is the number of
// FP64 instructions, 12.3 k per 32 elements at N = 4 (16.9 k with one thread per element
// and the six-row form). FP32: the shared-memory pipe (operators arrive at 128 bytes per
// clock whether they are broadcast or not), then issue slots.
// Measured (GB300, whole calls), one thread per element before, and now, with the overlap
// of launches and the limiter's shorter form, which give the third case half its gain:
//   FP64, N = 2, 512 elements, 100 single-rate steps           14.45 -> 2.55 ms
//   FP64, N = 4, 40,185 elements, 2 macro steps of 4 levels    16.95 -> 9.47 ms (94 % of the
//     FP64 pipe's issue slots in an all-active launch)
//   FP32, N = 3, 20,480 elements, 25 limited steps              1.50 -> 1.17 ms
//   FP32, N = 5, 75,077 elements, one R                        139.5 -> 115.5 us
// Where it is the slower one: FP32 on large sets, since a warp has an eighth of the elements
// in flight over a trip to memory that one thread per element has. At N = 2 and 3 these take
// kernels_solo.cuh. ms per macro step of 4 levels at 500k elements, one thread per element
// before, and now: N = 4 1.873 and 1.946, order 2N 1.524 and 1.714, collocation 1.297 and
// 1.427 (N = 5 3.699 and 3.382). Tried at N = 2, 500k elements, 0.776 to 0.792 ms: L2
// prefetches a tile ahead (0.728, but 125k 0.185 to 0.193), the history of all three fields
// at once (0.716; the tensor-core kernel, which shares the commit, 1.23 to 1.30 at N = 4),
// the next tile's connectivity in registers (0.776), three CTAs per SM (0.710).
#pragma once

#include "kernels.cuh"

namespace swe {

// ---- pairs of values: FP32 pairs run as packed instructions (one issue slot for
// two multiply-adds, the same rounding as two scalar ones), FP64 pairs as two
template <typename T>
struct PairOf;
template <>
struct PairOf<float> {
  using type = float2;
};
template <>
struct PairOf<double> {
  using type = double2;
};
template <typename T>
using Pair = typename PairOf<T>::type;

__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ double2 fma2(double2 a, double2 b, double2 c) {
  return make_double2(fma(a.x, b.x, c.x), fma(a.y, b.y, c.y));
}
__device__ __forceinline__ double2 mul2(double2 a, double2 b) { return make_double2(a.x * b.x, a.y * b.y); }
__device__ __forceinline__ double2 add2(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 pair(float x, float y) { return make_float2(x, y); }
__device__ __forceinline__ double2 pair(double x, double y) { return make_double2(x, y); }
__device__ __forceinline__ float2 dup(float x) { return make_float2(x, x); }
__device__ __forceinline__ double2 dup(double x) { return make_double2(x, x); }
// s + a.x b.x + a.y b.y, one after the other. The derivative sums use it: their weights
// alternate in sign, so the two halves of a packed sum grow large with opposite signs and
// their difference keeps the rounding of both (R of a bed that varies, FP32 against FP64,
// rms: 1.1 to 1.75 times that of the plain order, most at N = 5).
template <typename P, typename T>
__device__ __forceinline__ T dot2(P a, P b, T s) {
  return mad(a.y, b.y, mad(a.x, b.x, s));
}
template <typename P>
__device__ __forceinline__ auto hsum(P a) { return a.x + a.y; }
// four consecutive values (16-byte aligned) as two pairs
__device__ __forceinline__ void load4(const float* p, float2 (&o)[2]) {
  const float4 v = *reinterpret_cast<const float4*>(p);
  o[0] = make_float2(v.x, v.y);
  o[1] = make_float2(v.z, v.w);
}
__device__ __forceinline__ void load4(const double* p, double2 (&o)[2]) {
  o[0] = reinterpret_cast<const double2*>(p)[0];
  o[1] = reinterpret_cast<const double2*>(p)[1];
}

// 1/hm and 1/hp of the two sides of a face point (0 where the depth is not above hvel).
// FP64: a division each, correctly rounded over the whole range. Both from one division,
// r = 1/(hm hp), 1/hm = r hp, would spare ten FP64 instructions per point (at most 0.5 % of
// a macro step), but is off by up to 1.8 ulp and lost where the product underflows.
template <typename T>
__device__ __forceinline__ void recip_both(T hm, T hp, T hvel, T& im, T& ip) {
  im = hm > hvel ? recip_fast(hm) : T(0);
  ip = hp > hvel ? recip_fast(hp) : T(0);
}

// Asynchronous copy of S operator entries to shared memory (16 bytes per request): the
// copies of all threads are in flight at once, and the first tile's gathers overlap
// them. team_ops_ready() waits for them and for the other threads of the CTA.
template <typename T, int S>
__device__ __forceinline__ void team_copy(T* dst_, const T* src_) {
  static_assert(S * sizeof(T) % 16 == 0, "whole 16-byte requests");
  const unsigned dst = (unsigned)__cvta_generic_to_shared(dst_);
  const char* src = reinterpret_cast<const char*>(src_);
  for (int i = threadIdx.x * 16; i < (int)(S * sizeof(T)); i += blockDim.x * 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + i), "l"(src + i) : "memory");
}
__device__ __forceinline__ void team_copy_ready() {   // the copies of this warp's lanes
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncwarp();
}
__device__ __forceinline__ void team_ops_ready() {
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();
}

// Lanes per element and the warp's shared tile. FP64 at N = 2 has a variant with sixteen
// lanes (kWide; its small meshes are bound by the chain of one element: an FP64
// instruction holds its warp for 64 cycles; team_wide in kernels_order.inc chooses),
// everything else takes four: NB * L then equals NPP at every order and a quarter-warp's
// 16-byte reads of eight elements cover all banks (every element stride is an odd multiple
// of 16 bytes).
template <typename T, int N>
struct Team {
  using D = Dims<N>;
  static constexpr bool FP64 = sizeof(T) == 8;
  static constexpr int L = (N & kWide) ? 16 : 4;
  static constexpr int E = 32 / L;
  static constexpr int NB = D::NPP >= L ? D::NPP / L : 1;   // lanes past NPP have no nodes
  static constexpr int NCH = (D::NCUB + L - 1) / L;   // chunks of L cubature points
  static constexpr int QP = OpLayout<N>::QP;          // face points padded to fours
  static constexpr int V = 16 / sizeof(T);            // values per 16 bytes
  static constexpr int odd(int n) { return (n / V) % 2 ? n : n + V; }   // stride of n values, n % V == 0
  // rows of NPP nodes: eta, hu, hv, B; FP64 also keeps what the interpolation reads
  // (h' or B', and eta', relative to node 0) and the two mass fluxes
  static constexpr int ROWS = FP64 ? 8 : 4;
  static constexpr int OS = odd(ROWS * D::NPP);
  static constexpr int FS = odd(3 * D::NFP * 8);      // FP64: [3 faces][NFP nodes][4 fields] (own, neighbour)
  static constexpr int GS = odd(3 * 8);               // FP64: [3 faces] Ef, Bf, nx, ny, hs, kind, vx, vy
  // FP64: [6 fluxes][L points] of one chunk; FP32: [L lanes][2 momenta][NPP nodes]
  static constexpr int WS = odd(FP64 ? 6 * L : 2 * L * D::NPP);
  static constexpr int XS = odd(3 * QP);              // [3 fields][QP points] surface fluxes
  static constexpr int OWN = 0;
  static constexpr int FACE = OWN + E * OS;
  static constexpr int GEO = FACE + (FP64 ? E * FS : 0);
  static constexpr int VF = GEO + (FP64 ? E * GS : 0);
  static constexpr int FX = VF + E * WS;
  static constexpr int WARP = FX + E * XS;            // values per warp
  // The reference term -g h0 grad eta (h0: the depth at node 0), the leading one at depth: a
  // nodal product, or evaluated at the points. FP32 keeps it nodal (the points of
  // collocation are the nodes): through the points it is rounded there and again by the
  // projection. Rounding of R on a bed that varies, rms over hu and hv against the nodal
  // form: 1.16 at N = 1, 1.18 at 2, 1.07 at 3, 1.06 at 4, 1.01 at 5; order-2N rules 1.14,
  // 1.15, 1.12, 1.07 at N = 2 to 5. It costs (ms per macro step of 125k elements, points
  // and nodal) 0.182 and 0.185, 0.339 and 0.345, 0.497 and 0.514, 0.959 and 0.971 at N = 2
  // to 5, 0.447 and 0.457 with order-2N rules at N = 4. FP64 with exact rules: no growth
  // against extended precision, and one product less.
  static constexpr bool NODAL = FP64 ? !D::EXACT : !D::COLLOC;
  // operators staged per CTA: [0, PRE), then the projection block
  static constexpr int PRE = NODAL ? OpLayout<N>::PRT : OpLayout<N>::DR;
  static constexpr int PJ = FP64 ? OpLayout<N>::PROJ4 : OpLayout<N>::PRT;
  static constexpr int NPJ = FP64 ? OpLayout<N>::LGT - OpLayout<N>::PROJ4 : 3 * D::NCUB * D::NPP;
  static constexpr int OPS = PRE + NPJ;
  static constexpr int bytes(int warps) { return (OPS + warps * WARP) * (int)sizeof(T); }
  // warps per CTA when the mesh fills the GPU: eight (two per scheduler), four where
  // their tiles would not fit on an SM (227 KB)
  // (FP32 at N = 3 and 4: six, so that two CTAs have 168 registers instead of 128, which
  // spill: ms per macro step of 125k elements, reference term at the points, at eight and at
  // six, cubature N = 3 0.357 and 0.336, N = 4 0.556 and 0.495; one CTA of eight 0.412 and
  // 0.567)
  static constexpr int MAXW = !FP64 && (D::N == 3 || D::N == 4) ? 6 : (bytes(8) <= 227 * 1024 ? 8 : 4);
  // FP32 up to N = 4 runs two CTAs per SM, the others one
  static constexpr int MINB = !FP64 && D::N <= 4 ? 2 : 1;
};

// Start the copy of the operators a CTA keeps in shared memory.
template <typename T, int N>
__device__ __forceinline__ void team_ops_begin(T* smem, const T* gops) {
  using C = Team<T, N>;
  team_copy<T, C::PRE>(smem, gops);
  team_copy<T, C::NPJ>(smem + C::PRE, gops + C::PJ);
  asm volatile("cp.async.commit_group;" ::: "memory");
}

// State of one lane between the gather and the compute half of a tile.
template <typename T>
struct TeamLane {
  int e, lev;
  bool valid, finer;
  long long a;
  T rx, ry, sx, sy;
};

// The neighbour of a face as the lane of that face sees it: its face nodes in the
// NEIGHBOUR's own order (its trace at this element's Gauss point g is its own point
// NG-1-g, evaluated with the same operands in the same order as the neighbour evaluates
// it) and the pair's face reference, node 0 of the lower-numbered element. Both sides of
// a face then see bit-identical traces and take the same wet/dry and velocity decisions,
// and the mass flux is exactly antisymmetric.
template <typename T, int NFP>
struct TeamFace {
  int nb;          // neighbour, kWall or kFarField
  T v[4][NFP];     // eta, hu, hv, B
  bool lower;      // the face reference is the neighbour's node 0
  T E, B;          // then its values
};

template <typename T, int N>
__device__ __forceinline__ void team_load_face(const StageParams<T>& p, const int4& cn, int e, int f, long long k,
                                               TeamFace<T, Dims<N>::NFP>& o) {
  using D = Dims<N>;
  constexpr int NP = D::NP, NPP = D::NPP, NFP = D::NFP;
  const Sched& sc = p.sc;
  const size_t ks = (size_t)sc.KS, fstride = (size_t)NP * ks, bstride = 3 * fstride;
  o.nb = f == 0 ? cn.x : (f == 1 ? cn.y : cn.z);
  // across a boundary face the lane reads its own element: the values are replaced by the
  // ghost state, and no lane needs a select
  const int nb = o.nb < 0 ? e : o.nb;
  const int fn = (cn.w >> (2 * f)) & 3;
  const int ln = ((cn.w >> (13 + 3 * f)) & 7) + 1;
  const long long an = k >> (ln - 1);
  const long long pern = 1LL << (ln - 1);
  const long long phase = k & (pern - 1);
  const bool half = 2 * phase == pern;   // the half-step record of a coarser neighbour
  const T* qn = half ? p.s.qmid + (size_t)nb * 3 * NPP : p.s.q + (size_t)(an & 1) * bstride + nb;
  // 32-bit node offsets (NP KS words of a plane set are always below 2^32 here: the
  // workspace of a larger mesh would not fit the card), one wide add per access
  const unsigned sn = half ? 1u : (unsigned)sc.KS;
  const size_t sf = half ? (size_t)NPP : fstride;
  const T *q1 = qn + sf, *q2 = q1 + sf, *qb = p.s.B + nb;
#pragma unroll
  for (int m = 0; m < NFP; ++m) {
    const unsigned jn = (unsigned)face_node_rt(D::N, fn, m);
    const unsigned idx = jn * sn;
    o.v[0][m] = ldm(qn + idx);
    o.v[1][m] = ldm(q1 + idx);
    o.v[2][m] = ldm(q2 + idx);
    o.v[3][m] = __ldg(qb + jn * (unsigned)sc.KS);
  }
  o.lower = phase == 0 && nb < e;
  if (o.lower) {
    o.E = ldm(qn);
    o.B = __ldg(qb);
  }
  if (phase != 0 && !half) {   // other fractions: Adams-Bashforth polynomial at t_k
    const int depth = an + 1 < 3 ? (int)(an + 1) : 3;
    T w[3];
    ab_partial_weights<T>(depth, (T)phase / (T)pern, w);
    const T dtn = level_dt(sc, ln, T(0));
    for (int s = 0; s < depth; ++s) {
      const T ws = dtn * (s == 0 ? w[0] : (s == 1 ? w[1] : w[2]));
      const T* rs = p.s.ring + (size_t)((an - s) % 3) * bstride + nb;
#pragma unroll
      for (int m = 0; m < NFP; ++m) {
        const size_t idx = (size_t)face_node_rt(D::N, fn, m) * ks;
        o.v[0][m] = mad(ws, ldm(rs + idx), o.v[0][m]);
        o.v[1][m] = mad(ws, ldm(rs + fstride + idx), o.v[1][m]);
        o.v[2][m] = mad(ws, ldm(rs + 2 * fstride + idx), o.v[2][m]);
      }
    }
  }
}

// Well-balanced flux (Section 5.1) of a face point from its traces (own, neighbour)
// relative to the face reference, as wb_flux in kernels.cuh, with the two sides in
// pairs; scaled by sJ/J. E0, B0: the element's node 0 (own-side p'', inexact rules).
template <typename T, int N>
__device__ __forceinline__ void team_flux(const Phys& ph, int kind, T Ef, T Bf, T E0, T B0, T nx, T ny, T hs, T vx,
                                          T vy, Pair<T> te, Pair<T> tu, Pair<T> tv, Pair<T> tb, T& f0, T& f1, T& f2) {
  using D = Dims<N>;
  const T g = phys_g(ph, T(0)), hvel = phys_hvel(ph, T(0)), qg = T(0.25) * g;
  const T hf = Ef - Bf;
  if (kind < 0) {
    if (kind == kFarField) {   // the constant state over the continued bed
      te.y = phys_ff(ph, 0, T(0)) - hf + tb.x;
      tu.y = phys_ff(ph, 1, T(0));
      tv.y = phys_ff(ph, 2, T(0));
    } else {                   // reflecting wall: mirror the normal momentum
      const T mn = T(-2) * mad(tu.x, nx, tv.x * ny);
      te.y = te.x;
      tu.y = mad(mn, nx, tu.x);
      tv.y = mad(mn, ny, tv.x);
    }
    tb.y = tb.x;
  }
  const Pair<T> h = add2(dup(hf), add2(te, pair(-tb.x, -tb.y)));
  T im, ip;
  recip_both(h.x, h.y, hvel, im, ip);
  const Pair<T> iv = pair(im, ip);
  const Pair<T> u = mul2(tu, iv), v = mul2(tv, iv);
  const T bmax = tmax(tb.x, tb.y);
  const Pair<T> st = add2(dup(hf), add2(te, dup(-bmax)));
  const Pair<T> s = pair(tmax(T(0), st.x), tmax(T(0), st.y));
  const Pair<T> un = fma2(v, dup(ny), mul2(u, dup(nx)));
  const Pair<T> gs = mul2(dup(g), s);
  const T lam = tmax(speed(un.x, gs.x), speed(un.y, gs.y));
  const Pair<T> F = mul2(s, un);
  const T ds = (s.x > T(0) && s.y > T(0)) ? te.y - te.x : s.y - s.x;
  T pres = qg * ds * (s.y + s.x);
  if constexpr (!D::EXACT) {   // own-side p'' (element reference split)
    const T epm = te.x + (Ef - E0), bpm = tb.x + (Bf - B0);
    pres = mad(T(0.5) * g * epm, epm - T(2) * bpm, pres);
  }
  const Pair<T> su = mul2(s, u), sv = mul2(s, v);
  f0 = hs * mad(-lam, ds, F.x + F.y);
  f1 = mad(hs, mad(-lam, su.y - su.x, mad(F.x, u.x, F.y * u.y)), pres * vx);
  f2 = mad(hs, mad(-lam, sv.y - sv.x, mad(F.x, v.x, F.y * v.y)), pres * vy);
}

// Outward normal times sJ/J of face f from the affine factors.
template <typename T>
__device__ __forceinline__ void face_normal(int f, T rx, T ry, T sx, T sy, T& vx, T& vy) {
  vx = f == 0 ? -sx : (f == 1 ? rx + sx : -rx);
  vy = f == 0 ? -sy : (f == 1 ? ry + sy : -ry);
}

// Gather and surface fluxes of a tile. `first`: the CTA's operators are still on their
// way (waited for once the loads of the first tile are in flight).
template <typename T, int N>
__device__ __forceinline__ void team_gather(const StageParams<T>& p, const T* sops, T* __restrict__ sw, int tile,
                                            int ntiles, int nactive, long long k, bool first, TeamLane<T>& t) {
  using D = Dims<N>;
  using C = Team<T, N>;
  using O = OpLayout<N>;
  constexpr int NP = D::NP, NPP = D::NPP, NFP = D::NFP, NG = D::NG, E = C::E, NB = C::NB;
  const Sched& sc = p.sc;
  const int lane = threadIdx.x & 31, el = lane % E, part = lane / E;
  const size_t ks = (size_t)sc.KS, fstride = (size_t)NP * ks, bstride = 3 * fstride;
  // lanes past the last active element repeat it (and store nothing)
  t.valid = tile < ntiles && tile * E + el < nactive;
  const int e = t.valid ? tile * E + el : nactive - 1;
  t.e = e;
  T own[4][NB];
#pragma unroll
  for (int f = 0; f < 4; ++f)
#pragma unroll
    for (int n = 0; n < NB; ++n) own[f][n] = T(0);
  TeamFace<T, NFP> fc;
  if (tile < ntiles) {
    const int4 cn = __ldg(p.s.conn + e);
    t.finer = (cn.w >> 12) & 1;
    if (part < 3) team_load_face<T, N>(p, cn, e, part, k, fc);
    t.lev = level_of(sc, e);
    t.a = k >> (t.lev - 1);
    const T* q = p.s.q + (size_t)(t.a & 1) * bstride + e;
#pragma unroll
    for (int n = 0; n < NB; ++n) {
      const int i = part * NB + n;
      if (i < NP) {
        own[0][n] = ldm(q + i * ks);
        own[1][n] = ldm(q + fstride + i * ks);
        own[2][n] = ldm(q + 2 * fstride + i * ks);
        own[3][n] = __ldg(p.s.B + e + i * ks);
      }
    }
    T gm[4];
    load_row_global<T, 4>(p.s.geo + 4 * (size_t)e, gm);
    t.rx = gm[0]; t.ry = gm[1]; t.sx = gm[2]; t.sy = gm[3];
  }
  if (first) team_ops_ready();
  if (tile >= ntiles) return;
  T* so = sw + C::OWN + el * C::OS;
  if (C::L * NB == NPP || part < NPP) {
#pragma unroll
    for (int f = 0; f < 4; ++f)
#pragma unroll
      for (int n = 0; n < NB; ++n) so[f * NPP + part * NB + n] = own[f][n];
    if constexpr (C::FP64) {   // the mass fluxes rx hu + ry hv and sx hu + sy hv
#pragma unroll
      for (int n = 0; n < NB; ++n) {
        so[6 * NPP + part * NB + n] = mad(t.rx, own[1][n], t.ry * own[2][n]);
        so[7 * NPP + part * NB + n] = mad(t.sx, own[1][n], t.sy * own[2][n]);
      }
    }
  }
  __syncwarp();
  const T E0 = so[0], B0 = so[3 * NPP];
  if constexpr (C::FP64) {   // rows 4, 5: h' (exact rules) or B', and eta', zero in the padding
    if (C::L * NB == NPP || part < NPP) {
#pragma unroll
      for (int n = 0; n < NB; ++n) {
        const int i = part * NB + n;
        const T de = i < NP ? own[0][n] - E0 : T(0), db = i < NP ? own[3][n] - B0 : T(0);
        so[4 * NPP + i] = D::EXACT ? de - db : db;
        so[5 * NPP + i] = de;
      }
    }
  }
  T* sx = sw + C::FX + el * C::XS;
  if (part < 3) {
    const int f = part;
    const T Ef = fc.lower ? fc.E : E0, Bf = fc.lower ? fc.B : B0;
    T vx, vy;
    face_normal(f, t.rx, t.ry, t.sx, t.sy, vx, vy);
    const T v2 = mad(vx, vx, vy * vy), iv = rsqrt_t(v2);
    const T nx = vx * iv, ny = vy * iv, hs = T(0.5) * v2 * iv;
    Pair<T> tr[NFP][4];   // (own, neighbour) relative to the face reference
#pragma unroll
    for (int m = 0; m < NFP; ++m) {
      const T* o = so + face_node_rt(D::N, f, m);
      tr[m][0] = add2(pair(o[0], fc.v[0][m]), dup(-Ef));
      tr[m][1] = pair(o[NPP], fc.v[1][m]);
      tr[m][2] = pair(o[2 * NPP], fc.v[2][m]);
      tr[m][3] = add2(pair(o[3 * NPP], fc.v[3][m]), dup(-Bf));
    }
    if constexpr (C::FP64) {
      Pair<T>* sf = reinterpret_cast<Pair<T>*>(sw + C::FACE + el * C::FS) + f * NFP * 4;
#pragma unroll
      for (int m = 0; m < NFP; ++m)
#pragma unroll
        for (int c = 0; c < 4; ++c) sf[4 * m + c] = tr[m][c];
      T* sg = sw + C::GEO + el * C::GS + f * 8;
      sg[0] = Ef;
      sg[1] = Bf;
      sg[2] = nx;
      sg[3] = ny;
      sg[4] = hs;
      sg[5] = fc.nb >= 0 ? T(0) : T(fc.nb);   // kind: 0 interior, kWall, kFarField
      sg[6] = vx;
      sg[7] = vy;
    } else {
#pragma unroll 1
      for (int gq = 0; gq < NG; ++gq) {
        const T* w = sops + O::I1P + 2 * gq * D::NFPP;
        Pair<T> te = dup(T(0)), tu = te, tv = te, tb = te;
#pragma unroll
        for (int m = 0; m < NFP; m += 2) {
          Pair<T> wp[2];
          load4(w + 2 * m, wp);
#pragma unroll
          for (int c = 0; c < 2; ++c) {
            if (m + c >= NFP) continue;
            te = fma2(wp[c], tr[m + c][0], te);
            tu = fma2(wp[c], tr[m + c][1], tu);
            tv = fma2(wp[c], tr[m + c][2], tv);
            tb = fma2(wp[c], tr[m + c][3], tb);
          }
        }
        T f0, f1, f2;
        team_flux<T, N>(p.ph, fc.nb, Ef, Bf, E0, B0, nx, ny, hs, vx, vy, te, tu, tv, tb, f0, f1, f2);
        const int q = f * NG + gq;
        sx[0 * C::QP + q] = f0;
        sx[1 * C::QP + q] = f1;
        sx[2 * C::QP + q] = f2;
      }
    }
  } else if constexpr (!C::FP64) {   // the padding of the lift's groups of four points
    for (int q = 3 * NG; q < C::QP; ++q) sx[q] = sx[C::QP + q] = sx[2 * C::QP + q] = T(0);
  }
  __syncwarp();
  if constexpr (C::FP64) {
    const T* sf = sw + C::FACE + el * C::FS;
    const T* sgeo = sw + C::GEO + el * C::GS;
#pragma unroll 1
    for (int q = part; q < C::QP; q += C::L) {
      T f0 = T(0), f1 = T(0), f2 = T(0);
      if (q < 3 * NG) {
        const int f = q / NG, gq = q - f * NG;
        const Pair<T>* tr = reinterpret_cast<const Pair<T>*>(sf) + f * NFP * 4;
        const Pair<T>* w = reinterpret_cast<const Pair<T>*>(sops + O::I1P) + gq * D::NFPP;
        Pair<T> te = dup(T(0)), tu = te, tv = te, tb = te;
#pragma unroll
        for (int m = 0; m < NFP; ++m) {
          te = fma2(w[m], tr[4 * m + 0], te);
          tu = fma2(w[m], tr[4 * m + 1], tu);
          tv = fma2(w[m], tr[4 * m + 2], tv);
          tb = fma2(w[m], tr[4 * m + 3], tb);
        }
        Pair<T> r[4][2];
        load4(sgeo + f * 8, r[0]);
        load4(sgeo + f * 8 + 4, r[1]);
        team_flux<T, N>(p.ph, (int)r[1][0].y, r[0][0].x, r[0][0].y, E0, B0, r[0][1].x, r[0][1].y, r[1][0].x,
                        r[1][1].x, r[1][1].y, te, tu, tv, tb, f0, f1, f2);
      }
      sx[0 * C::QP + q] = f0;
      sx[1 * C::QP + q] = f1;
      sx[2 * C::QP + q] = f2;
    }
    __syncwarp();
  }
}

// The volume term, the mass operator and the lift, accumulated into R of the lane's
// nodes part * NB + n.
template <typename T, int N>
__device__ __forceinline__ void team_rhs(const StageParams<T>& p, const T* sops, const T* spj,
                                         T* __restrict__ sw, const TeamLane<T>& t, T E0, T B0, T (&R)[3][Team<T, N>::NB]) {
  using D = Dims<N>;
  using O = OpLayout<N>;
  using C = Team<T, N>;
  constexpr int NP = D::NP, NPP = D::NPP, NCUB = D::NCUB, E = C::E, NB = C::NB, L = C::L, H = NPP / 2;
  constexpr bool kRegs = sizeof(T) == 4;   // FP32 keeps the interpolated rows in registers
  constexpr bool kNodal = C::NODAL;
  // FP32 collocation: the points are the nodes, so each lane takes its own nodes as its
  // points. Interpolation and the source's projection are then the identity (nothing to
  // multiply), and the reference term, a nodal product, shares the rows read for the bed:
  // 124 instead of 188 operator reads per lane at N = 4, one R of 125k elements
  // 0.095 -> 0.078 ms (0.091 with one thread per element).
  constexpr bool kOwn = kRegs && D::COLLOC;
  // FP64 collocation uses the same identities on the team's common points: a lane's point is
  // read from the tile, and the source comes back to the lane of its node. ms per macro step
  // with the points interpolated and projected as of the other schemes, and so: N = 2, 80k
  // elements 2.66 and 2.46 (2.47 with one thread per element), 20k elements N = 2 0.91 and
  // 0.85, N = 4 1.76 and 1.49, N = 5 3.02 and 2.43.
  constexpr bool kIdent = D::COLLOC;
  const int lane = threadIdx.x & 31, el = lane % E, part = lane / E;
  const int i0 = L * NB == NPP || part < NPP ? part * NB : 0;   // a lane past NPP repeats node 0 (unused)
  const T g = phys_g(p.ph, T(0)), hvel = phys_hvel(p.ph, T(0));
  const T* so = sw + C::OWN + el * C::OS;
  const T h0 = E0 - B0;
  const T rx = t.rx, ry = t.ry, sx = t.sx, sy = t.sy;
  // s0: h' (exact rules) or B'; s1: eta'; s2, s3: hu, hv
  Pair<T> s0[kRegs ? H : 1], s1[kRegs ? H : 1], s2[kRegs ? H : 1], s3[kRegs ? H : 1];
  if constexpr (kRegs) {
#pragma unroll
    for (int j = 0; j < NPP; j += 4) {
      Pair<T> ev[2], uv[2], vv[2], bv[2];
      load4(so + j, ev);
      if constexpr (!kOwn) {
        load4(so + NPP + j, uv);
        load4(so + 2 * NPP + j, vv);
      }
      load4(so + 3 * NPP + j, bv);
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        const int jj = j / 2 + c;
        Pair<T> de = add2(ev[c], dup(-E0)), db = add2(bv[c], dup(-B0));
        if (2 * jj >= NP) de.x = db.x = T(0);
        if (2 * jj + 1 >= NP) de.y = db.y = T(0);
        s1[jj] = de;
        s0[jj] = D::EXACT ? add2(de, pair(-db.x, -db.y)) : db;
        if constexpr (!kOwn) {
          s2[jj] = uv[c];
          s3[jj] = vv[c];
        }
      }
    }
  }
  Pair<T> A[3][NB];
#pragma unroll
  for (int f = 0; f < 3; ++f)
#pragma unroll
    for (int n = 0; n < NB; ++n) A[f][n] = dup(T(0));
  Pair<T> M[2][kRegs ? H : 1];   // FP32: the lane's points projected onto all nodes (hu, hv)
#pragma unroll
  for (int f = 0; f < 2; ++f)
#pragma unroll
    for (int j = 0; j < (kRegs ? H : 1); ++j) M[f][j] = dup(T(0));
  T own[2][kIdent ? NB : 1];   // collocation: source (FP32: and reference term) of the lane's nodes
#pragma unroll
  for (int f = 0; f < 2; ++f)
#pragma unroll
    for (int n = 0; n < (kIdent ? NB : 1); ++n) own[f][n] = T(0);

#pragma unroll 1
  for (int ch = 0; ch < C::NCH; ++ch) {
    // interpolation to the lane's point (padding points repeat the last one; FP64 has
    // zero projection weights for them)
    const int c0 = kOwn ? i0 + ch : ch * L + part, c = c0 < NCUB ? c0 : NCUB - 1;
    const T* ic = sops + O::IC + c * NPP;
    const T* icr = sops + O::ICR + c * NPP;
    const T* ics = sops + O::ICS + c * NPP;
    Pair<T> a0 = dup(T(0)), a1 = a0, a2 = a0, a3 = a0;
    T dr = T(0), ds = T(0), er = T(0), es = T(0);
#pragma unroll
    for (int j = 0; j < NPP; j += 4) {
      Pair<T> w[2], wr[2], ws[2];
      if constexpr (!kIdent) load4(ic + j, w);
      load4(icr + j, wr);
      load4(ics + j, ws);
      Pair<T> x0[2], x1[2], x2[2], x3[2];
      if constexpr (kRegs) {
#pragma unroll
        for (int cc = 0; cc < 2; ++cc) {
          x0[cc] = s0[j / 2 + cc]; x1[cc] = s1[j / 2 + cc];
          if constexpr (!kOwn) { x2[cc] = s2[j / 2 + cc]; x3[cc] = s3[j / 2 + cc]; }
        }
      } else {
        load4(so + 4 * NPP + j, x0);
        if constexpr (!kIdent) {
          load4(so + 5 * NPP + j, x1);
          load4(so + NPP + j, x2);
          load4(so + 2 * NPP + j, x3);
        }
      }
#pragma unroll
      for (int cc = 0; cc < 2; ++cc) {
        if (j + 2 * cc >= NP) continue;
        if constexpr (kIdent) {
          dr = dot2(wr[cc], x0[cc], dr);
          ds = dot2(ws[cc], x0[cc], ds);
          if constexpr (kOwn) {
            er = dot2(wr[cc], x1[cc], er);
            es = dot2(ws[cc], x1[cc], es);
          }
          continue;
        }
        a0 = fma2(w[cc], x0[cc], a0);
        a2 = fma2(w[cc], x2[cc], a2);
        a3 = fma2(w[cc], x3[cc], a3);
        if constexpr (D::EXACT) {
          dr = dot2(wr[cc], x1[cc], dr);
          ds = dot2(ws[cc], x1[cc], ds);
        } else {
          a1 = fma2(w[cc], x1[cc], a1);
          dr = dot2(wr[cc], x0[cc], dr);
          ds = dot2(ws[cc], x0[cc], ds);
        }
      }
    }
    const T huc = kIdent ? so[NPP + c] : hsum(a2), hvc = kIdent ? so[2 * NPP + c] : hsum(a3);
    T hc, F[6];   // rows: Pr (hu, hv), Ps (hu, hv), P (hu, hv)
    const T am = mad(rx, huc, ry * hvc), bm = mad(sx, huc, sy * hvc);
    if constexpr (D::EXACT) {
      hc = h0 + hsum(a0);
      const T ih = hc > hvel ? recip_fast(hc) : T(0);
      const T u = huc * ih, v = hvc * ih;
      F[0] = u * am; F[1] = v * am; F[2] = u * bm; F[3] = v * bm;
      const T gm = -g * (kNodal ? hsum(a0) : hc);   // without or with the reference term
      F[4] = gm * mad(rx, dr, sx * ds);
      F[5] = gm * mad(ry, dr, sy * ds);
    } else {
      const T ec = kIdent ? so[c] - E0 : hsum(a1), bc = kIdent ? so[3 * NPP + c] - B0 : hsum(a0);
      hc = h0 + (ec - bc);
      const T ih = hc > hvel ? recip_fast(hc) : T(0);
      const T u = huc * ih, v = hvc * ih, gm = -g * ec;
      const T pr = T(0.5) * g * ec * (ec - T(2) * bc);
      F[0] = mad(u, am, rx * pr); F[1] = mad(v, am, ry * pr); F[2] = mad(u, bm, sx * pr); F[3] = mad(v, bm, sy * pr);
      F[4] = gm * mad(rx, dr, sx * ds);
      F[5] = gm * mad(ry, dr, sy * ds);
      if constexpr (kOwn) {
        const T gb = -g * h0;
        F[4] = mad(gb, mad(rx, er, sx * es), F[4]);
        F[5] = mad(gb, mad(ry, er, sy * es), F[5]);
      }
    }
    if constexpr (kRegs) {   // onto all nodes, padding points excluded
      if (c0 < NCUB) {
#pragma unroll
        for (int op = 0; op < (kOwn ? 2 : 3); ++op) {
          const Pair<T> fu = dup(F[2 * op]), fv = dup(F[2 * op + 1]);
          const T* pj = spj + (op * NCUB + c) * NPP;
#pragma unroll
          for (int j = 0; j < NPP; j += 4) {
            Pair<T> w[2];
            load4(pj + j, w);
#pragma unroll
            for (int cc = 0; cc < 2; ++cc) {
              if (j + 2 * cc >= NP) continue;
              M[0][j / 2 + cc] = fma2(w[cc], fu, M[0][j / 2 + cc]);
              M[1][j / 2 + cc] = fma2(w[cc], fv, M[1][j / 2 + cc]);
            }
          }
        }
        if constexpr (kOwn) {
#pragma unroll
          for (int n = 0; n < NB; ++n) {
            own[0][n] = n == ch ? F[4] : own[0][n];
            own[1][n] = n == ch ? F[5] : own[1][n];
          }
        }
      }
    } else {
      T* vf = sw + C::VF + el * C::WS;
#pragma unroll
      for (int q = 0; q < 6; ++q) vf[q * L + part] = F[q];
      __syncwarp();
#pragma unroll 1
      for (int gg = 0; gg < L / 4; ++gg) {
        if (ch * (L / 4) + gg >= O::G4) break;
        Pair<T> x[6][2];
#pragma unroll
        for (int q = 0; q < 6; ++q) load4(vf + q * L + 4 * gg, x[q]);
        const T* pj = spj + (size_t)((ch * (L / 4) + gg) * 3 * NPP + i0) * 4;
#pragma unroll
        for (int n = 0; n < NB; ++n)
#pragma unroll
          for (int op = 0; op < (kIdent ? 2 : 3); ++op) {
            Pair<T> w[2];
            load4(pj + (op * NPP + n) * 4, w);
#pragma unroll
            for (int cc = 0; cc < 2; ++cc) {
              A[1][n] = fma2(w[cc], x[2 * op][cc], A[1][n]);
              A[2][n] = fma2(w[cc], x[2 * op + 1][cc], A[2][n]);
            }
          }
      }
      if constexpr (kIdent) {   // the source at the lane's nodes among these points
#pragma unroll
        for (int n = 0; n < NB; ++n)
          if (i0 + n < NP && (i0 + n) / L == ch) {
            own[0][n] = vf[4 * L + (i0 + n) % L];
            own[1][n] = vf[5 * L + (i0 + n) % L];
          }
      }
      __syncwarp();
    }
  }
  if constexpr (kRegs) {   // the team's partial sums, collected by the lanes of the nodes
    T* vf = sw + C::VF + el * C::WS;
#pragma unroll
    for (int f = 0; f < 2; ++f)
#pragma unroll
      for (int j = 0; j < NPP; j += 4)
        *reinterpret_cast<float4*>(vf + (part * 2 + f) * NPP + j) =
            make_float4(M[f][j / 2].x, M[f][j / 2].y, M[f][j / 2 + 1].x, M[f][j / 2 + 1].y);
    __syncwarp();
#pragma unroll
    for (int f = 0; f < 2; ++f)
#pragma unroll
      for (int n = 0; n < NB; ++n) {
        const T* v = vf + f * NPP + i0 + n;
        A[1 + f][n] = pair(v[0] + v[2 * NPP], v[4 * NPP] + v[6 * NPP]);
      }
  }
  // mass: R_h += WR (rx hu + ry hv) + WS (sx hu + sy hv)
#pragma unroll
  for (int j = 0; j < NPP; j += 4) {
    Pair<T> xa[2], xb[2];
    if constexpr (kRegs) {
      Pair<T> hu[2], hv[2];
      if constexpr (kOwn) {
        load4(so + NPP + j, hu);
        load4(so + 2 * NPP + j, hv);
      } else {
#pragma unroll
        for (int cc = 0; cc < 2; ++cc) {
          hu[cc] = s2[j / 2 + cc];
          hv[cc] = s3[j / 2 + cc];
        }
      }
#pragma unroll
      for (int cc = 0; cc < 2; ++cc) {
        xa[cc] = fma2(dup(ry), hv[cc], mul2(dup(rx), hu[cc]));
        xb[cc] = fma2(dup(sy), hv[cc], mul2(dup(sx), hu[cc]));
      }
    } else {
      load4(so + 6 * NPP + j, xa);
      load4(so + 7 * NPP + j, xb);
    }
#pragma unroll
    for (int n = 0; n < NB; ++n) {
      Pair<T> wa[2], wb[2];
      load4(sops + O::WR + (i0 + n) * NPP + j, wa);
      load4(sops + O::WS + (i0 + n) * NPP + j, wb);
#pragma unroll
      for (int cc = 0; cc < 2; ++cc) {
        if (j + 2 * cc >= NP) continue;
        A[0][n] = fma2(wa[cc], xa[cc], A[0][n]);
        A[0][n] = fma2(wb[cc], xb[cc], A[0][n]);
      }
    }
  }
  // lift: R -= L^g F, four face points at a time (LIFT4 holds -L^g)
  const T* fx = sw + C::FX + el * C::XS;
#pragma unroll 1
  for (int q = 0; q < C::QP; q += 4) {
    Pair<T> x[3][2];
#pragma unroll
    for (int f = 0; f < 3; ++f) load4(fx + f * C::QP + q, x[f]);
    const T* lf = sops + O::LIFT4 + (size_t)(q * NPP + i0 * 4);
#pragma unroll
    for (int n = 0; n < NB; ++n) {
      Pair<T> w[2];
      load4(lf + n * 4, w);
#pragma unroll
      for (int f = 0; f < 3; ++f)
#pragma unroll
        for (int cc = 0; cc < 2; ++cc) A[f][n] = fma2(w[cc], x[f][cc], A[f][n]);
    }
  }
#pragma unroll
  for (int f = 0; f < 3; ++f)
#pragma unroll
    for (int n = 0; n < NB; ++n) R[f][n] = f > 0 && kIdent ? hsum(A[f][n]) + own[f > 0 ? f - 1 : 0][kIdent ? n : 0] : hsum(A[f][n]);
  if constexpr (kNodal) {   // strong-form reference pressure (element reference split)
    const T gb = -g * h0;
#pragma unroll
    for (int n = 0; n < NB; ++n) {
      T er = T(0), es = T(0);
#pragma unroll
      for (int j = 0; j < NPP; j += 4) {
        Pair<T> wr[2], ws[2], x[2];
        load4(sops + O::DR + (i0 + n) * NPP + j, wr);
        load4(sops + O::DS + (i0 + n) * NPP + j, ws);
        if constexpr (kRegs) {
          x[0] = s1[j / 2];
          x[1] = s1[j / 2 + 1];
        } else {
          load4(so + 5 * NPP + j, x);
        }
#pragma unroll
        for (int cc = 0; cc < 2; ++cc) {
          if (j + 2 * cc >= NP) continue;
          er = dot2(wr[cc], x[cc], er);
          es = dot2(ws[cc], x[cc], es);
        }
      }
      R[1][n] = mad(gb, mad(rx, er, sx * es), R[1][n]);
      R[2][n] = mad(gb, mad(ry, er, sy * es), R[2][n]);
    }
  }
}

// Sum (or minimum) over the lanes of a team of L lanes, E elements apart: every lane
// gets the same value (a + b and b + a round alike).
template <int L, typename T>
__device__ __forceinline__ T team_sum(T v) {
#pragma unroll
  for (int m = 32 / L; m < 32; m *= 2) v += __shfl_xor_sync(0xffffffffu, v, m);
  return v;
}
template <int L, typename T>
__device__ __forceinline__ T team_min(T v) {
#pragma unroll
  for (int m = 32 / L; m < 32; m *= 2) v = tmin(v, __shfl_xor_sync(0xffffffffu, v, m));
  return v;
}

// s[f] = sum over the lane's NB nodes of w q[f], f = eta, hu, hv (`on` false: zero).
// Even NB: two nodes per packed instruction.
template <typename T, int NB>
__device__ __forceinline__ void node_sums(const T* w, bool on, const T (&q)[4][NB], T (&s)[3]) {
  if constexpr (NB % 2 == 0) {
    Pair<T> acc[3] = {dup(T(0)), dup(T(0)), dup(T(0))};
#pragma unroll
    for (int n = 0; n < NB; n += 2) {
      const Pair<T> x = *reinterpret_cast<const Pair<T>*>(w + n);
#pragma unroll
      for (int f = 0; f < 3; ++f) acc[f] = fma2(x, pair(q[f][n], q[f][n + 1]), acc[f]);
    }
#pragma unroll
    for (int f = 0; f < 3; ++f) s[f] = on ? hsum(acc[f]) : T(0);
  } else {
#pragma unroll
    for (int n = 0; n < NB; ++n) {
      const T x = on ? w[n] : T(0);
#pragma unroll
      for (int f = 0; f < 3; ++f) s[f] = mad(x, q[f][n], s[f]);
    }
  }
}

// a mod 3 of a non-negative activation count: 2^32 = 1 (mod 3), so the halves add up and
// one 32-bit remainder does
__device__ __forceinline__ int ring_slot3(long long a) {
  return (int)(((unsigned)a % 3u + (unsigned)((unsigned long long)a >> 32) % 3u) % 3u);
}

// Adams-Bashforth commit (Algorithm 1) and positivity limiter (Algorithm 3) of an
// element whose nodes part * NB + n sit with lane (el, part) of a team of L lanes
// (mode 0), or the R output in the caller's layout (mode 1). q: the state at the
// lane's nodes (eta, hu, hv, B). All 32 lanes call it; lanes with valid = false store
// nothing. kComp: compensated state update, as described at swe_params.compensated:
// each field's increments are summed first and added to the state with the rounding
// error of the previous update taken back.
template <typename T, int N, int L, int NB, bool kComp>
__device__ __forceinline__ void team_commit(const StageParams<T>& p, const T* sops, bool valid, bool finer, int e,
                                            int part, int lev, long long a, T (&q)[4][NB], const T (&R)[3][NB], T rx, T ry,
                                            T sx, T sy, double* injected) {
  using D = Dims<N>;
  using O = OpLayout<N>;
  constexpr int NP = D::NP, NPP = D::NPP;
  const Sched& sc = p.sc;
  const size_t ks = (size_t)sc.KS, fstride = (size_t)NP * ks, bstride = 3 * fstride, eo = (size_t)e;
  constexpr bool kAll = L * NB == NPP;   // else lanes past NPP have no nodes
  const int i0 = part * NB, ir = kAll || i0 < NPP ? i0 : 0;   // ir: a row to read in the operators
  if (p.mode == 1) {   // R only, caller layout
    if (valid) {
      const size_t ce = (size_t)p.perm[e] * NP, Kn = (size_t)sc.K * NP;
#pragma unroll
      for (int f = 0; f < 3; ++f)
#pragma unroll
        for (int n = 0; n < NB; ++n)
          if (i0 + n < NP) p.out[f * Kn + ce + i0 + n] = R[f][n];
    }
    return;
  }
  if (valid) {
    const int depth = a + 1 < 3 ? (int)(a + 1) : 3;
    T wab[3], wh[3];
    ab_weights<T>(depth, wab);
    ab_partial_weights<T>(depth, T(0.5), wh);
    const T dtl = level_dt(sc, lev, T(0));
    const T c0 = dtl * wab[0], c1 = dtl * wab[1], c2 = dtl * wab[2];
    const T m0 = dtl * wh[0], m1 = dtl * wh[1], m2 = dtl * wh[2];
    // finer: an element with a finer neighbour also stores the Adams-Bashforth polynomial
    // of this step at its middle, q(t_a + dt/2) (Section 4), for that neighbour's next substep
    const unsigned ks4 = (unsigned)sc.KS;
    const size_t eb = eo + (size_t)((unsigned)i0 * ks4);   // the lane's first node in a field's planes
    const int s0 = ring_slot3(a), s1 = s0 == 0 ? 2 : s0 - 1, s2 = s1 == 0 ? 2 : s1 - 1;
    T* w0 = p.s.ring + (size_t)s0 * bstride + eb;
    const T* p1 = p.s.ring + (size_t)s1 * bstride + eb;
    const T* p2 = p.s.ring + (size_t)s2 * bstride + eb;
    T* cp = kComp ? p.s.comp + eb : nullptr;
    T* qm = p.s.qmid + eo * 3 * NPP + i0;
#pragma unroll
    for (int f = 0; f < 3; ++f) {   // one field's history at a time in registers
      T r1[NB], r2[NB], ce[kComp ? NB : 1];
#pragma unroll
      for (int n = 0; n < NB; ++n) {
        const unsigned o = n * ks4;
        const bool in = kAll && NB * (L - 1) + n < NP ? true : i0 + n < NP;
        r1[n] = depth > 1 && in ? ldm(p1 + o) : T(0);
        r2[n] = depth > 2 && in ? ldm(p2 + o) : T(0);
        if constexpr (kComp) ce[n] = in ? ldm(cp + o) : T(0);
      }
#pragma unroll
      for (int n = 0; n < NB; ++n)
        if (kAll && NB * (L - 1) + n < NP ? true : i0 + n < NP) w0[n * ks4] = R[f][n];
      if (finer) {
#pragma unroll
        for (int n = 0; n < NB; ++n)
          if (kAll || i0 + n < NPP)
            qm[f * NPP + n] = mad(m2, r2[n], mad(m1, r1[n], mad(m0, R[f][n], q[f][n])));
      }
#pragma unroll
      for (int n = 0; n < NB; ++n) {
        if constexpr (kComp) {   // y = d - c, t = q + y, and the new error c = (t - q) - y
          const T y = mad(c2, r2[n], mad(c1, r1[n], c0 * R[f][n])) - ce[n];
          const T s = q[f][n] + y;
          if (i0 + n < NP) cp[n * ks4] = (s - q[f][n]) - y;
          q[f][n] = s;
        } else {
          q[f][n] = mad(c2, r2[n], mad(c1, r1[n], mad(c0, R[f][n], q[f][n])));
        }
      }
      w0 += fstride;
      p1 += fstride;
      p2 += fstride;
      if constexpr (kComp) cp += fstride;
    }
  }

  // ---- positivity limiter (Algorithm 3), trigger per element ----
  const Phys& ph = p.ph;
  T hmin = q[0][0] - q[3][0];
  {
    bool first = true;
#pragma unroll
    for (int n = 0; n < NB; ++n) {
      if (i0 + n >= NP) continue;
      const T h = q[0][n] - q[3][n];
      hmin = first ? h : tmin(hmin, h);
      first = false;
    }
    if (i0 >= NP) hmin = T(3.0e38);   // a lane without nodes
  }
  hmin = team_min<L>(hmin);
  const bool trig = valid && ph.pp && (hmin <= eps_of(ph, T(0)));
  T me[3];
  int dryf = 0;
  {
    T s[3] = {T(0), T(0), T(0)};
    node_sums<T, NB>(sops + O::MW + ir, kAll || i0 < NPP, q, s);   // zero weights in the padding
#pragma unroll
    for (int f = 0; f < 3; ++f) me[f] = team_sum<L>(s[f]);
  }
  if (__any_sync(0xffffffffu, trig)) {
    // The mean depth in FP64 decides; a dry element needs no more, and only where some
    // element of the warp is wet are the P1 sums taken (FP64 instructions hold a warp
    // for 64 cycles each). Every lane takes part in the sums.
    const double h0 = ph.h0;
    // The two lane counts of FP64 at N = 2 add up the same tree: P partial sums, a
    // product each.
    constexpr int P = sizeof(T) == 8 && D::N == 2 ? 2 : 1;
    auto total = [](const double (&x)[P]) { return team_sum<L>(P == 2 ? x[0] + x[P - 1] : x[0]); };
    double hs[P] = {};
#pragma unroll
    for (int n = 0; n < NB; ++n)
      if (i0 + n < NP)
        hs[n % P] = mad((double)sops[O::MW + ir + n], (double)q[0][n] - (double)q[3][n], hs[n % P]);
    const double hb = total(hs);
    const bool isdry = hb < 1.01 * h0;   // the 1% margin keeps a reset element dry under rounding
    if (__any_sync(0xffffffffu, trig && !isdry)) {
      double us[P] = {}, vs[P] = {}, sh[3][P] = {}, su[3][P] = {}, sv[3][P] = {};
#pragma unroll
      for (int n = 0; n < NB; ++n) {
        if (i0 + n >= NP) continue;
        const double w = (double)sops[O::MW + ir + n];
        const double h = (double)q[0][n] - (double)q[3][n], u = (double)q[1][n], v = (double)q[2][n];
        us[n % P] = mad(w, u, us[n % P]);
        vs[n % P] = mad(w, v, vs[n % P]);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          const double x = (double)sops[O::T1 + k * NPP + ir + n];
          sh[k][n % P] = mad(x, h, sh[k][n % P]);
          su[k][n % P] = mad(x, u, su[k][n % P]);
          sv[k][n % P] = mad(x, v, sv[k][n % P]);
        }
      }
      const double ub = total(us), vb = total(vs);
      double vh[3], vu[3], vv[3];
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        vh[k] = total(sh[k]);
        vu[k] = total(su[k]);
        vv[k] = total(sv[k]);
      }
      if (trig && !isdry) {   // theta rescale of the P1 part toward the mean
        const double den = hb - fmin(vh[0], fmin(vh[1], vh[2]));
        const double theta = den > 0.0 ? fmin(1.0, (hb - h0) / den) : 1.0;
#pragma unroll
        for (int n = 0; n < NB; ++n) {
          if (i0 + n >= NP) continue;
          const T* ba = sops + O::BARY + (i0 + n) * 4;
          const double l0 = ba[0], l1 = ba[1], l2 = ba[2];
          q[0][n] = (T)(mad(theta, mad(l0, vh[0], mad(l1, vh[1], l2 * vh[2])) - hb, hb) + (double)q[3][n]);
          q[1][n] = (T)mad(theta, mad(l0, vu[0], mad(l1, vu[1], l2 * vu[2])) - ub, ub);
          q[2][n] = (T)mad(theta, mad(l0, vv[0], mad(l1, vv[1], l2 * vv[2])) - vb, vb);
        }
        me[0] = (T)(hb + __ldg(p.s.Bbar + e));
        me[1] = (T)ub;
        me[2] = (T)vb;
      }
    }
    if (trig && isdry) {
      const double hn = ph.dry_mode ? hb : h0;
#pragma unroll
      for (int n = 0; n < NB; ++n) {
        q[0][n] = (T)(hn + (double)q[3][n]);
        q[1][n] = q[2][n] = T(0);
      }
      if (part == 0) {
        const double area = 2.0 / mad((double)rx, (double)sy, -((double)ry * (double)sx));
        *injected = mad(area, hn - hb, *injected);
      }
      me[0] = (T)(hn + __ldg(p.s.Bbar + e));
      me[1] = me[2] = T(0);
      dryf = 1;
    }
  }
  // vertex values of Pi1 (eta, hu, hv) for the TVB limiter (Section 5.3)
  T v1[3][3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    T s[3] = {T(0), T(0), T(0)};
    node_sums<T, NB>(sops + O::T1 + k * NPP + ir, kAll || i0 < NPP, q, s);
#pragma unroll
    for (int f = 0; f < 3; ++f) v1[f][k] = team_sum<L>(s[f]);
  }
  if (!valid) return;
  T* qd = p.s.q + (size_t)((a + 1) & 1) * bstride + eo + (size_t)((unsigned)i0 * (unsigned)sc.KS);
#pragma unroll
  for (int f = 0; f < 3; ++f) {
#pragma unroll
    for (int n = 0; n < NB; ++n)
      if (kAll && NB * (L - 1) + n < NP ? true : i0 + n < NP) qd[n * (unsigned)sc.KS] = q[f][n];
    qd += fstride;
  }
  // the element's small records, dealt to the lanes of the team: lane f < 3 (with two
  // lanes, lane 0 also field 1) stores field f
#pragma unroll
  for (int f = 0; f < 3; ++f) {
    if (part != (L >= 3 ? f : f / 2)) continue;
    p.s.means[4 * eo + f] = me[f];
#pragma unroll
    for (int k = 0; k < 3; ++k) p.s.p1[(size_t)(3 * f + k) * ks + eo] = v1[f][k];
  }
  if (part == L - 1) p.s.dry[e] = (uint8_t)dryf;
  if (part == 0 && !(isfinite(me[0]) && isfinite(me[1]) && isfinite(me[2])))
    atomicOr(p.s.flags, 1);
}

// The rest of a tile: volume, projection, commit.
template <typename T, int N, bool kComp>
__device__ __forceinline__ void team_compute(const StageParams<T>& p, const T* sops, const T* spj,
                                             T* __restrict__ sw, const TeamLane<T>& t, double* injected) {
  using C = Team<T, N>;
  constexpr int NPP = Dims<N>::NPP, NB = C::NB;
  const int lane = threadIdx.x & 31, el = lane % C::E, part = lane / C::E;
  const T* so = sw + C::OWN + el * C::OS;
  const T E0 = so[0], B0 = so[3 * NPP];
  const int ir = C::L * NB == NPP || part < NPP ? part * NB : 0;
  T R[3][NB], q[4][NB];
  team_rhs<T, N>(p, sops, spj, sw, t, E0, B0, R);
#pragma unroll
  for (int f = 0; f < 4; ++f)
#pragma unroll
    for (int n = 0; n < NB; ++n) q[f][n] = so[f * NPP + ir + n];
  team_commit<T, N, C::L, NB, kComp>(p, sops, t.valid, t.finer, t.e, part, t.lev, t.a, q, R, t.rx, t.ry, t.sx, t.sy, injected);
  __syncwarp();   // the tile's rows are read before the next gather overwrites them
}

// Tiles t0, t0 + step, ... below t1 (one warp); the separate launch and the persistent
// batch kernel both inline it. Returns the mass the positivity limiter's dry resets
// injected.
template <typename T, int N, bool kComp = false>
__device__ __forceinline__ double team_range(const StageParams<T>& __restrict__ p, const T* __restrict__ sops,
                                             const T* __restrict__ spj, T* __restrict__ sw, int t0, int step, int t1, int nactive, long long k) {
  double injected = 0.0;
  TeamLane<T> t;
  for (int tile = t0; tile < t1; tile += step) {
    team_gather<T, N>(p, sops, sw, tile, t1, nactive, k, false, t);
    team_compute<T, N, kComp>(p, sops, spj, sw, t, &injected);
  }
  return injected;
}

// kGlobalOps: the operators are read from global memory (through L1) instead of the
// CTA's shared copy (the operator-placement comparison of Section 7.4). kComp:
// compensated state update (p.s.comp). blockDim.x / 32 warps, each with its own tile.
template <typename T, int N, bool kGlobalOps = false, bool kComp = false>
__global__ void __launch_bounds__(32 * Team<T, N>::MAXW, Team<T, N>::MINB)
    k_stage(const __grid_constant__ StageParams<T> p) {
  using C = Team<T, N>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* smem = reinterpret_cast<T*>(smem_raw);
  if (p.early) dependents_may_launch();
  const T *sops = smem, *spj = smem + C::PRE;
  T* sw = smem + (threadIdx.x >> 5) * C::WARP;
  if constexpr (kGlobalOps) {
    sops = p.s.ops;
    spj = p.s.ops + C::PJ;
  } else {
    sw += C::OPS;
    team_ops_begin<T, N>(smem, p.s.ops);
  }
  wait_for_previous();
  const long long k = (*p.s.macro) * (1LL << (p.sc.L - 1)) + p.j;
  const int ntiles = (p.nactive + C::E - 1) / C::E;
  const int nw = blockDim.x >> 5, step = gridDim.x * nw;
  int tile = blockIdx.x * nw + (threadIdx.x >> 5);
  double injected = 0.0;
  for (bool first = true;; first = false) {
    TeamLane<T> t;
    // the operators' copies overlap the loads of the first tile
    team_gather<T, N>(p, sops, sw, tile, ntiles, p.nactive, k, !kGlobalOps && first, t);
    if (tile >= ntiles) break;
    team_compute<T, N, kComp>(p, sops, spj, sw, t, &injected);
    tile += step;
  }
  if (!p.early) dependents_may_launch();
  if (injected != 0.0) atomicAdd(p.s.acc, injected);
}

}  // namespace swe
