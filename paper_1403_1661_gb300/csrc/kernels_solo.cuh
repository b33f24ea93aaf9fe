// FP32 SIMT stage kernel for large active sets at N = 2 and 3: one thread per element, with
// the arithmetic of the team kernel (kernels_team.cuh) bit for bit. A thread takes the four
// lanes' parts of a team one after the other; their points' projections and the sums over
// their nodes are kept apart and added in the order of the team's exchanges.
//
// What bounds it: trips to memory and to the L2 (state, history and the neighbours' traces):
// at N = 2 and 500k elements 1.8 of 6.8 cycles per issue wait for one, and DRAM is 26 % busy.
// A warp has 32 elements in flight where the team kernel has eight, and nothing of an element
// passes through shared memory but its surface fluxes, which a thread keeps in its own column:
// the three fields' fluxes of all face points would not fit beside the state in registers,
// and the lift takes them node by node. The parts' volume sums meet in pairs (0 + 1, 2 + 3),
// so that two sets of them are live. Blocks of 128: at N = 2 four per SM (128 registers), at
// N = 3 three (168; 500k elements 0.981 ms, with two 1.029), with the rules of order 2N two,
// which spill little then (0.999 and 0.887).
// Measured (GB300), the team kernel and this one, ms per macro step of 4 levels:
//   211k elements   N = 2 0.355 and 0.262, N = 3 0.536 and 0.476, collocation 0.338 and 0.251,
//                   0.444 and 0.376, order 2N 0.350 and 0.263, 0.469 and 0.438
//   500k elements   N = 2 0.792 and 0.489, N = 3 1.180 and 0.987, collocation 0.750 and 0.459,
//                   0.971 and 0.771, order 2N 0.782 and 0.489, 1.032 and 0.920
// and one R of 500k elements: N = 2 0.114 and 0.073, N = 3 0.221 and 0.176.
// From N = 4 the state no longer fits in registers (500k, N = 4 1.946 and 1.966, order 2N
// 1.709 and 2.254), and the team kernel takes every set.
#pragma once

#include "kernels_team.cuh"

namespace swe {

template <int N>
struct Solo {
  using C = Team<float, N>;
  static constexpr int THREADS = 128;
  // Resident blocks per SM, and the blocks per SM from which a set takes this kernel. Below,
  // its threads are too few to hide an element's chain of four parts. us per single-rate step,
  // the team kernel and this one: N = 2 16k 17.6 and 22.7, 24k 18.5 and 18.5, 40k 22.6 and
  // 20.6, 64k 28.9 and 23.5, 240k 97.5 and 60.0; N = 3 64k 49.0 and 55.8, 120k 75.4 and 80.8,
  // 160k 101.7 and 96.3, 240k 143.5 and 125.2 (order 2N 126.8 and 120.3). At N = 2 one block
  // costs a 20k mesh of 4 levels 6 % (0.088 and 0.093 ms).
  static constexpr int MINB = Dims<N>::N == 2 ? 4 : Dims<N>::REDUCED ? 2 : 3;
  static constexpr int FROM = Dims<N>::N == 2 ? 2 : 7;
  static constexpr int FX = 3 * C::QP;                  // surface fluxes of a thread, in shared memory
  static constexpr int bytes() { return (C::OPS + FX * THREADS) * 4; }
};

// (s0 + s1) + (s2 + s3) of a function of the part: team_sum over four lanes
template <typename F>
__device__ __forceinline__ auto solo_sum(F&& f) {
  const auto a = f(0) + f(1);
  return a + (f(2) + f(3));
}

// sum over the NB nodes of a part of w q, in the order of node_sums
template <int NB, int NPP>
__device__ __forceinline__ float solo_nodes(const float* w, const float (&q)[NPP], int part) {
  if constexpr (NB % 2 == 0) {
    float2 acc = dup(0.f);
#pragma unroll
    for (int n = 0; n < NB; n += 2) {
      const float2 x = *reinterpret_cast<const float2*>(w + part * NB + n);
      acc = fma2(x, make_float2(q[part * NB + n], q[part * NB + n + 1]), acc);
    }
    return hsum(acc);
  } else {
    float s = 0.f;
#pragma unroll
    for (int n = 0; n < NB; ++n) s = mad(w[part * NB + n], q[part * NB + n], s);
    return s;
  }
}

template <int N, bool kComp>
__device__ __forceinline__ void solo_element(const StageParams<float>& p, const float* sops, const float* spj, float* fx,
                                             int e, long long k, double* injected) {
  using T = float;
  using D = Dims<N>;
  using O = OpLayout<N>;
  using C = Team<T, N>;
  constexpr int NP = D::NP, NPP = D::NPP, NFP = D::NFP, NG = D::NG, NCUB = D::NCUB, NB = C::NB, H = NPP / 2;
  constexpr bool kOwn = D::COLLOC, kNodal = C::NODAL;
  static_assert(C::L == 4 && NB * 4 == NPP, "the parts of a team");
  const Sched& sc = p.sc;
  const size_t ks = (size_t)sc.KS, fstride = (size_t)NP * ks, bstride = 3 * fstride, eo = (size_t)e;
  const T g = p.ph.g_f, hvel = p.ph.hvel_f;
  const int lev = level_of(sc, e);
  const long long a = k >> (lev - 1);
  const int4 cn = __ldg(p.s.conn + e);
  const T* q0 = p.s.q + (size_t)(a & 1) * bstride + eo;
  const T* qb = p.s.B + eo;
  T gm[4];
  load_row_global<T, 4>(p.s.geo + 4 * eo, gm);
  const T rx = gm[0], ry = gm[1], sx = gm[2], sy = gm[3];

  // ---- volume ----
  float2 s0[H], s1[H], s2[H], s3[H];   // h' (exact rules) or B', eta', hu, hv
  T E0, B0;
  {
    T ev[NPP], uv[NPP], vv[NPP], bv[NPP];
#pragma unroll
    for (int i = 0; i < NPP; ++i) {
      const bool in = i < NP;
      ev[i] = in ? ldm(q0 + i * ks) : T(0);
      uv[i] = in ? ldm(q0 + fstride + i * ks) : T(0);
      vv[i] = in ? ldm(q0 + 2 * fstride + i * ks) : T(0);
      bv[i] = in ? __ldg(qb + i * ks) : T(0);
    }
    E0 = ev[0];
    B0 = bv[0];
#pragma unroll
    for (int j = 0; j < H; ++j) {
      float2 de = add2(make_float2(ev[2 * j], ev[2 * j + 1]), dup(-E0)), db = add2(make_float2(bv[2 * j], bv[2 * j + 1]), dup(-B0));
      if (2 * j >= NP) de.x = db.x = 0.f;
      if (2 * j + 1 >= NP) de.y = db.y = 0.f;
      s1[j] = de;
      s0[j] = D::EXACT ? add2(de, make_float2(-db.x, -db.y)) : db;
      s2[j] = make_float2(uv[2 * j], uv[2 * j + 1]);
      s3[j] = make_float2(vv[2 * j], vv[2 * j + 1]);
    }
  }
  const T h0 = E0 - B0, gb = -g * h0;
  float2 V[2][2][H];              // [parts 0 + 1, 2 + 3][hu, hv][nodes]
  T own[2][kOwn ? NPP : 1];       // collocation: source and reference term of the nodes
#pragma unroll
  for (int pr = 0; pr < 2; ++pr) {
#pragma unroll (kOwn ? 2 : 1)
    for (int half = 0; half < 2; ++half) {
      float2 M[2][H];
#pragma unroll
      for (int f = 0; f < 2; ++f)
#pragma unroll
        for (int j = 0; j < H; ++j) M[f][j] = dup(0.f);
      const int part = 2 * pr + half;
#pragma unroll (kOwn ? NB : 1)
      for (int ch = 0; ch < C::NCH; ++ch) {
        const int c = kOwn ? part * NB + ch : ch * 4 + part;
        if (c >= NCUB) continue;
        const T* ic = sops + O::IC + c * NPP;
        const T* icr = sops + O::ICR + c * NPP;
        const T* ics = sops + O::ICS + c * NPP;
        float2 a0 = dup(0.f), a1 = a0, a2 = a0, a3 = a0;
        T dr = 0.f, ds = 0.f, er = 0.f, es = 0.f;
#pragma unroll
        for (int j = 0; j < NPP; j += 4) {
          float2 w[2], wr[2], ws[2];
          if constexpr (!kOwn) load4(ic + j, w);
          load4(icr + j, wr);
          load4(ics + j, ws);
#pragma unroll
          for (int cc = 0; cc < 2; ++cc) {
            if (j + 2 * cc >= NP) continue;
            const int jj = j / 2 + cc;
            if constexpr (kOwn) {
              dr = dot2(wr[cc], s0[jj], dr);
              ds = dot2(ws[cc], s0[jj], ds);
              er = dot2(wr[cc], s1[jj], er);
              es = dot2(ws[cc], s1[jj], es);
            } else {
              a0 = fma2(w[cc], s0[jj], a0);
              a2 = fma2(w[cc], s2[jj], a2);
              a3 = fma2(w[cc], s3[jj], a3);
              if constexpr (!D::EXACT) a1 = fma2(w[cc], s1[jj], a1);
              dr = dot2(wr[cc], D::EXACT ? s1[jj] : s0[jj], dr);
              ds = dot2(ws[cc], D::EXACT ? s1[jj] : s0[jj], ds);
            }
          }
        }
        auto at = [&](const float2 (&s)[H]) { return c % 2 ? s[kOwn ? c / 2 : 0].y : s[kOwn ? c / 2 : 0].x; };
        const T huc = kOwn ? at(s2) : hsum(a2), hvc = kOwn ? at(s3) : hsum(a3);
        T hc, F[6];
        const T am = mad(rx, huc, ry * hvc), bm = mad(sx, huc, sy * hvc);
        if constexpr (D::EXACT) {
          hc = h0 + hsum(a0);
          const T ih = hc > hvel ? recip_fast(hc) : T(0);
          const T u = huc * ih, v = hvc * ih;
          F[0] = u * am; F[1] = v * am; F[2] = u * bm; F[3] = v * bm;
          const T gq = -g * (kNodal ? hsum(a0) : hc);
          F[4] = gq * mad(rx, dr, sx * ds);
          F[5] = gq * mad(ry, dr, sy * ds);
        } else {
          const T ec = kOwn ? at(s1) : hsum(a1), bc = kOwn ? at(s0) : hsum(a0);
          hc = h0 + (ec - bc);
          const T ih = hc > hvel ? recip_fast(hc) : T(0);
          const T u = huc * ih, v = hvc * ih, gq = -g * ec;
          const T pr_ = T(0.5) * g * ec * (ec - T(2) * bc);
          F[0] = mad(u, am, rx * pr_); F[1] = mad(v, am, ry * pr_); F[2] = mad(u, bm, sx * pr_); F[3] = mad(v, bm, sy * pr_);
          F[4] = gq * mad(rx, dr, sx * ds);
          F[5] = gq * mad(ry, dr, sy * ds);
          if constexpr (kOwn) {
            F[4] = mad(gb, mad(rx, er, sx * es), F[4]);
            F[5] = mad(gb, mad(ry, er, sy * es), F[5]);
            own[0][kOwn ? c : 0] = F[4];
            own[1][kOwn ? c : 0] = F[5];
          }
        }
#pragma unroll
        for (int op = 0; op < (kOwn ? 2 : 3); ++op) {
          const float2 fu = dup(F[2 * op]), fv = dup(F[2 * op + 1]);
          const T* pj = spj + (op * NCUB + c) * NPP;
#pragma unroll
          for (int j = 0; j < NPP; j += 4) {
            float2 w[2];
            load4(pj + j, w);
#pragma unroll
            for (int cc = 0; cc < 2; ++cc) {
              if (j + 2 * cc >= NP) continue;
              M[0][j / 2 + cc] = fma2(w[cc], fu, M[0][j / 2 + cc]);
              M[1][j / 2 + cc] = fma2(w[cc], fv, M[1][j / 2 + cc]);
            }
          }
        }
      }
#pragma unroll
      for (int f = 0; f < 2; ++f)
#pragma unroll
        for (int j = 0; j < H; ++j) V[pr][f][j] = half == 0 ? M[f][j] : add2(V[pr][f][j], M[f][j]);
    }
  }

  // ---- surface fluxes, face by face, to the thread's column of shared memory ----
#pragma unroll
  for (int f = 0; f < 3; ++f) {
    TeamFace<T, NFP> fc;
    team_load_face<T, N>(p, cn, e, f, k, fc);
    const T Ef = fc.lower ? fc.E : E0, Bf = fc.lower ? fc.B : B0;
    T vx, vy;
    face_normal(f, rx, ry, sx, sy, vx, vy);
    const T v2 = mad(vx, vx, vy * vy), iv = rsqrt_t(v2);
    const T nx = vx * iv, ny = vy * iv, hs = T(0.5) * v2 * iv;
    float2 tr[NFP][4];
#pragma unroll
    for (int m = 0; m < NFP; ++m) {
      const int j = face_node(D::N, f, m);
      const T hu = j % 2 ? s2[j / 2].y : s2[j / 2].x, hv = j % 2 ? s3[j / 2].y : s3[j / 2].x;
      tr[m][0] = add2(make_float2(ldm(q0 + j * ks), fc.v[0][m]), dup(-Ef));
      tr[m][1] = make_float2(hu, fc.v[1][m]);
      tr[m][2] = make_float2(hv, fc.v[2][m]);
      tr[m][3] = add2(make_float2(__ldg(qb + j * ks), fc.v[3][m]), dup(-Bf));
    }
#pragma unroll 1
    for (int gq = 0; gq < NG; ++gq) {
      const T* w = sops + O::I1P + 2 * gq * D::NFPP;
      float2 te = dup(0.f), tu = te, tv = te, tb = te;
#pragma unroll
      for (int m = 0; m < NFP; m += 2) {
        float2 wp[2];
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
      fx[(0 * C::QP + q) * Solo<N>::THREADS] = f0;
      fx[(1 * C::QP + q) * Solo<N>::THREADS] = f1;
      fx[(2 * C::QP + q) * Solo<N>::THREADS] = f2;
    }
  }
#pragma unroll
  for (int q = 3 * NG; q < C::QP; ++q)
#pragma unroll
    for (int f = 0; f < 3; ++f) fx[(f * C::QP + q) * Solo<N>::THREADS] = 0.f;

  // ---- mass, lift and reference term, node by node ----
  T R[3][NP];
#pragma unroll
  for (int n = 0; n < NP; ++n) {
    float2 A[3];
    A[0] = dup(0.f);
#pragma unroll
    for (int f = 0; f < 2; ++f)
      A[1 + f] = n % 2 ? make_float2(V[0][f][n / 2].y, V[1][f][n / 2].y) : make_float2(V[0][f][n / 2].x, V[1][f][n / 2].x);
#pragma unroll
    for (int j = 0; j < NPP; j += 4) {
      float2 wa[2], wb[2];
      load4(sops + O::WR + n * NPP + j, wa);
      load4(sops + O::WS + n * NPP + j, wb);
#pragma unroll
      for (int cc = 0; cc < 2; ++cc) {
        if (j + 2 * cc >= NP) continue;
        const float2 hu = s2[j / 2 + cc], hv = s3[j / 2 + cc];
        const float2 xa = fma2(dup(ry), hv, mul2(dup(rx), hu)), xb = fma2(dup(sy), hv, mul2(dup(sx), hu));
        A[0] = fma2(wa[cc], xa, A[0]);
        A[0] = fma2(wb[cc], xb, A[0]);
      }
    }
#pragma unroll
    for (int q = 0; q < C::QP; q += 4) {
      float2 w[2];
      load4(sops + O::LIFT4 + q * NPP + n * 4, w);
#pragma unroll
      for (int f = 0; f < 3; ++f)
#pragma unroll
        for (int cc = 0; cc < 2; ++cc) {
          const float2 x = make_float2(fx[(f * C::QP + q + 2 * cc) * Solo<N>::THREADS],
                                       fx[(f * C::QP + q + 2 * cc + 1) * Solo<N>::THREADS]);
          A[f] = fma2(w[cc], x, A[f]);
        }
    }
#pragma unroll
    for (int f = 0; f < 3; ++f) R[f][n] = f > 0 && kOwn ? hsum(A[f]) + own[f > 0 ? f - 1 : 0][kOwn ? n : 0] : hsum(A[f]);
    if constexpr (kNodal) {
      T er = T(0), es = T(0);
#pragma unroll
      for (int j = 0; j < NPP; j += 4) {
        float2 wr[2], ws[2];
        load4(sops + O::DR + n * NPP + j, wr);
        load4(sops + O::DS + n * NPP + j, ws);
#pragma unroll
        for (int cc = 0; cc < 2; ++cc) {
          if (j + 2 * cc >= NP) continue;
          er = dot2(wr[cc], s1[j / 2 + cc], er);
          es = dot2(ws[cc], s1[j / 2 + cc], es);
        }
      }
      R[1][n] = mad(gb, mad(rx, er, sx * es), R[1][n]);
      R[2][n] = mad(gb, mad(ry, er, sy * es), R[2][n]);
    }
  }
  if (p.mode == 1) {   // R only, caller layout
    const size_t ce = (size_t)p.perm[e] * NP, Kn = (size_t)sc.K * NP;
#pragma unroll
    for (int f = 0; f < 3; ++f)
#pragma unroll
      for (int n = 0; n < NP; ++n) p.out[f * Kn + ce + n] = R[f][n];
    return;
  }

  // ---- Adams-Bashforth commit (team_commit) ----
  T q[4][NPP];
#pragma unroll
  for (int n = 0; n < NPP; ++n) {
    q[0][n] = n < NP ? ldm(q0 + n * ks) : T(0);
    q[1][n] = n % 2 ? s2[n / 2].y : s2[n / 2].x;
    q[2][n] = n % 2 ? s3[n / 2].y : s3[n / 2].x;
    q[3][n] = n < NP ? __ldg(qb + n * ks) : T(0);
  }
  {
    const int depth = a + 1 < 3 ? (int)(a + 1) : 3;
    T wab[3], wh[3];
    ab_weights<T>(depth, wab);
    ab_partial_weights<T>(depth, T(0.5), wh);
    const T dtl = level_dt(sc, lev, T(0));
    const T c0 = dtl * wab[0], c1 = dtl * wab[1], c2 = dtl * wab[2];
    const T m0 = dtl * wh[0], m1 = dtl * wh[1], m2 = dtl * wh[2];
    const int i0 = ring_slot3(a), i1 = i0 == 0 ? 2 : i0 - 1, i2 = i1 == 0 ? 2 : i1 - 1;
    const bool finer = (cn.w >> 12) & 1;
#pragma unroll
    for (int f = 0; f < 3; ++f) {
      T* w0 = p.s.ring + (size_t)i0 * bstride + f * fstride + eo;
      const T* p1 = p.s.ring + (size_t)i1 * bstride + f * fstride + eo;
      const T* p2 = p.s.ring + (size_t)i2 * bstride + f * fstride + eo;
      T* cp = kComp ? p.s.comp + f * fstride + eo : nullptr;
      T r1[NP], r2[NP], ce[kComp ? NP : 1];
#pragma unroll
      for (int n = 0; n < NP; ++n) {
        r1[n] = depth > 1 ? ldm(p1 + n * ks) : T(0);
        r2[n] = depth > 2 ? ldm(p2 + n * ks) : T(0);
        if constexpr (kComp) ce[n] = ldm(cp + n * ks);
      }
#pragma unroll
      for (int n = 0; n < NP; ++n) w0[n * ks] = R[f][n];
      if (finer) {
        T* qm = p.s.qmid + eo * 3 * NPP + f * NPP;
#pragma unroll
        for (int n = 0; n < NPP; ++n)
          qm[n] = n < NP ? mad(m2, r2[n < NP ? n : 0], mad(m1, r1[n < NP ? n : 0], mad(m0, R[f][n < NP ? n : 0], q[f][n]))) : T(0);
      }
#pragma unroll
      for (int n = 0; n < NP; ++n) {
        if constexpr (kComp) {
          const T y = mad(c2, r2[n], mad(c1, r1[n], c0 * R[f][n])) - ce[n];
          const T s = q[f][n] + y;
          cp[n * ks] = (s - q[f][n]) - y;
          q[f][n] = s;
        } else {
          q[f][n] = mad(c2, r2[n], mad(c1, r1[n], mad(c0, R[f][n], q[f][n])));
        }
      }
    }
  }

  // ---- positivity limiter (Algorithm 3) and means, in the order of the team's sums ----
  const Phys& ph = p.ph;
  T hmin = q[0][0] - q[3][0];
#pragma unroll
  for (int n = 1; n < NP; ++n) hmin = tmin(hmin, q[0][n] - q[3][n]);
  T me[3];
#pragma unroll
  for (int f = 0; f < 3; ++f)
    me[f] = solo_sum([&](int part) { return solo_nodes<NB, NPP>(sops + O::MW, q[f], part); });
  int dryf = 0;
  if (ph.pp && hmin <= eps_of(ph, T(0))) {
    const double hd = ph.h0;
    // sum over a part's nodes of w x in FP64
    auto total = [&](const T* w, auto&& x) {
      return solo_sum([&](int part) {
        double s = 0.0;
#pragma unroll
        for (int n = 0; n < NB; ++n)
          if (part * NB + n < NP) s = mad((double)w[part * NB + n], x(part * NB + n), s);
        return s;
      });
    };
    auto depth = [&](int n) { return (double)q[0][n] - (double)q[3][n]; };
    const double hb = total(sops + O::MW, depth);
    if (!(hb < 1.01 * hd)) {
      auto mu = [&](int n) { return (double)q[1][n]; };
      auto mv = [&](int n) { return (double)q[2][n]; };
      const double ub = total(sops + O::MW, mu), vb = total(sops + O::MW, mv);
      double vh[3], vu[3], vv[3];
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        vh[i] = total(sops + O::T1 + i * NPP, depth);
        vu[i] = total(sops + O::T1 + i * NPP, mu);
        vv[i] = total(sops + O::T1 + i * NPP, mv);
      }
      const double den = hb - fmin(vh[0], fmin(vh[1], vh[2]));
      const double theta = den > 0.0 ? fmin(1.0, (hb - hd) / den) : 1.0;
#pragma unroll
      for (int n = 0; n < NP; ++n) {
        const T* ba = sops + O::BARY + n * 4;
        const double l0 = ba[0], l1 = ba[1], l2 = ba[2];
        q[0][n] = (T)(mad(theta, mad(l0, vh[0], mad(l1, vh[1], l2 * vh[2])) - hb, hb) + (double)q[3][n]);
        q[1][n] = (T)mad(theta, mad(l0, vu[0], mad(l1, vu[1], l2 * vu[2])) - ub, ub);
        q[2][n] = (T)mad(theta, mad(l0, vv[0], mad(l1, vv[1], l2 * vv[2])) - vb, vb);
      }
      me[0] = (T)(hb + __ldg(p.s.Bbar + e));
      me[1] = (T)ub;
      me[2] = (T)vb;
    } else {
      const double hn = ph.dry_mode ? hb : hd;
#pragma unroll
      for (int n = 0; n < NP; ++n) {
        q[0][n] = (T)(hn + (double)q[3][n]);
        q[1][n] = q[2][n] = T(0);
      }
      const double area = 2.0 / mad((double)rx, (double)sy, -((double)ry * (double)sx));
      *injected = mad(area, hn - hb, *injected);
      me[0] = (T)(hn + __ldg(p.s.Bbar + e));
      me[1] = me[2] = T(0);
      dryf = 1;
    }
  }
  T* qd = p.s.q + (size_t)((a + 1) & 1) * bstride + eo;
#pragma unroll
  for (int f = 0; f < 3; ++f) {
#pragma unroll
    for (int n = 0; n < NP; ++n) qd[f * fstride + n * ks] = q[f][n];
    p.s.means[4 * eo + f] = me[f];
#pragma unroll
    for (int i = 0; i < 3; ++i)
      p.s.p1[(size_t)(3 * f + i) * ks + eo] =
          solo_sum([&](int part) { return solo_nodes<NB, NPP>(sops + O::T1 + i * NPP, q[f], part); });
  }
  p.s.dry[e] = (uint8_t)dryf;
  if (!(isfinite(me[0]) && isfinite(me[1]) && isfinite(me[2]))) atomicOr(p.s.flags, 1);
}

template <int N, bool kComp = false>
__global__ void __launch_bounds__(Solo<N>::THREADS, Solo<N>::MINB) k_stage_solo(const __grid_constant__ StageParams<float> p) {
  using C = Team<float, N>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float* smem = reinterpret_cast<float*>(smem_raw);
  if (p.early) dependents_may_launch();
  team_ops_begin<float, N>(smem, p.s.ops);
  team_ops_ready();
  wait_for_previous();
  const long long k = (*p.s.macro) * (1LL << (p.sc.L - 1)) + p.j;
  double injected = 0.0;
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < p.nactive; e += gridDim.x * blockDim.x)
    solo_element<N, kComp>(p, smem, smem + C::PRE, smem + C::OPS + threadIdx.x, e, k, &injected);
  if (!p.early) dependents_may_launch();
  if (injected != 0.0) atomicAdd(p.s.acc, injected);
}

}  // namespace swe
