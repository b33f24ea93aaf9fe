// Stage kernel with the volume contractions and the lift on tensor cores (FP32
// tier with split-BF16 products, Section 7.1's N(Q) = Pr cF1 + Ps cF2 + P cS and
// Section 7.2's R = N - L^g F).
//
// A warp holds a tile of 16 elements, one row of the m16 products each. Phases:
//   surface   lane (el, half): faces 0 and 1 one per lane, then face 2 with its Gauss
//             points shared by the two lanes of the element: traces and well-balanced
//             fluxes (team_flux) into the warp's flux tile
//   lift      R[16 el x Np] -= Flux[16 el x 8 pts] * L^g^T, 8 face points at a time
//   split     the state relative to node 0 as BF16 pairs hi + lo into the tile the
//             fluxes occupied, where ldmatrix reads it as A fragments
//   volume    per tile of 8 cubature points: interpolation (m16n8k16) of h, hu, hv with
//             Ic and eta with Icr, Ics; the flux on the accumulator layout, where lane
//             (g, t) holds rows g, g + 8 at points 2t, 2t + 1, which is the A layout of
//             the next product; projection with Pr, Ps, P (k16 instructions, two of the
//             split products side by side in k)
//   mass      R_h += rx WR hu + ry WR hv + sx WS hu + sy WS hv (nodal operators)
//   reference -g h0 (r_x Dr + s_x Ds) eta, the leading term at depth, in TF32 splits
//   commit    lane (el, half), half of the nodes each: team_commit
// Every BF16 product is split: a = a_hi + a_lo (operators and data) and
// a b ~ a_hi b_hi + a_hi b_lo + a_lo b_hi with FP32 accumulation (relative error of
// order 2^-16); TF32 splits 2^-21. The volume term is the form of kernels_team.cuh: with
// exact rules -P[g (h - h0) grad eta] carries pressure and source, h0 the depth at node 0
// (its product with grad eta is the reference term); the other schemes keep p'' and
// -g eta' grad B'.
//
// The operators' fragments are staged once per CTA in shared memory; results do not
// depend on the number of warps per CTA.
//
// What bounds it: latency at two to three warps per scheduler (no pipe is above 27 %,
// shared memory at half of its wavefronts; more warps cost the registers or the L1 that
// the gathers need: at N = 4 nine warps take 0.42 and ten 0.40 ms per macro step of 125k
// elements where eight take 0.34). Of a tile's 16 k clocks at N = 4, 2.8 k are the gather,
// 4.7 k the surface, 4.0 k the volume loop and 1.5 k the commit. Per 32 elements at N = 4
// it issues 8.5 k warp instructions where the form with 32-element tiles, six interpolated
// rows, eight projected fluxes and unpacked arithmetic took 11.8 k. Sixteen elements per
// tile, so that a small active set has twice the tiles and each takes half the time.
// Measured (GB300, whole calls), before and now, with the overlap of launches and the
// limiter's shorter form:
//   one R, 500,000 elements, N = 4                            0.341 -> 0.239 ms
//   45,149 elements, N = 3, 25 macro steps with transfers      6.42 -> 4.80 ms
//   2,048 elements, N = 2, 6 macro steps with transfers        0.968 -> 0.608 ms
#pragma once

#include <cuda_bf16.h>

#include "kernels.cuh"
#include "kernels_team.cuh"

namespace swe {

__device__ __forceinline__ void mma_k16(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                        uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

__device__ __forceinline__ void mma_k16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  mma_k16(d, a[0], a[1], a[2], a[3], b0, b1);
}

__device__ __forceinline__ void mma_k8(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t b0) {
  asm("mma.sync.aligned.m16n8k8.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5}, {%6}, {%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a0), "r"(a1), "r"(b0));
}

__device__ __forceinline__ void mma_tf32(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

__device__ __forceinline__ void ldmatrix4(uint32_t (&a)[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(a[0]), "=r"(a[1]), "=r"(a[2]), "=r"(a[3])
               : "r"(addr)
               : "memory");
}

// float -> (hi, lo) TF32 pair: hi rounded to 10 mantissa bits, lo the remainder
__device__ __forceinline__ void split_tf32(float x, uint32_t& hi, uint32_t& lo) {
  asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(hi) : "f"(x));
  lo = __float_as_uint(x - __uint_as_float(hi));
}

// two floats -> (hi, lo) bf16x2 pairs; the first float goes to the low half
__device__ __forceinline__ void split2(float2 x, uint32_t& hi, uint32_t& lo) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(x.x, x.y);
  hi = *reinterpret_cast<const uint32_t*>(&h);
  const float2 hf = make_float2(__uint_as_float(hi << 16), __uint_as_float(hi & 0xffff0000u));
  const float2 r = add2(x, make_float2(-hf.x, -hf.y));
  const __nv_bfloat162 l = __floats2bfloat162_rn(r.x, r.y);
  lo = *reinterpret_cast<const uint32_t*>(&l);
}

// Per-warp shared tiles. State, fluxes and R are node-major with the 16 elements
// contiguous and LS = 20 words per node: the mma fragment reads (rows g, g+8; nodes or
// points 2t, 2t+1) land on 32 distinct banks. The BF16 tile holds rows of KP values (one
// element) 2 KP + 16 bytes apart, so the eight row addresses of an ldmatrix cover all
// banks.
constexpr int LS = 20;

template <int N>
struct TcSmem {
  using D = Dims<N>;
  using C = TcDims<N>;
  static constexpr int E = 16;                            // elements per warp-tile
  static constexpr int BS = C::KP / 2 + 4;                // words per row of the BF16 tile
  static constexpr int mx(int a, int b) { return a > b ? a : b; }
  // per warp: state [4 fields][KP nodes][LS]; then, one after the other in the same
  // words, surface fluxes [3][KF][LS], the BF16 tile [4 fields][hi, lo][16][BS] and R
  // [3][NPT][LS]; geometry [16][4]
  static constexpr int STATE = 0;
  static constexpr int TILE = STATE + 4 * C::KP * LS;
  static constexpr int GEO = TILE + mx(mx(3 * C::KF * LS, 4 * 2 * E * BS), 3 * C::NPT * LS);
  static constexpr int CONN = GEO + E * 4;                // connectivity [16][4]
  static constexpr int WARP = CONN + E * 4;               // floats per warp
  static constexpr int OPS = OpLayout<N>::TAIL;           // floats of per-element operators
  static constexpr int FRAG = OPS;                        // then the operator fragments
  static constexpr int CTA = OPS + TcLayout<N>::SIZE;     // floats per CTA before the warps' tiles
  // dynamic shared memory of a CTA of `warps` warps
  static constexpr int bytes(int warps) { return (CTA + warps * WARP) * 4; }
  // warps per SM the registers are budgeted for: twelve up to N = 3 (168 registers), eight
  // at N = 4 (255; twelve spill), seven at N = 5 (their tiles and the fragments fill the
  // shared memory). A CTA has at most eight (swe_set_tc_warps)
  static constexpr int LIMIT = D::N <= 3 ? 12 : (D::N == 4 ? 8 : 7);
  // default warps per CTA (ms per macro step of a 125k-element beach, 45k at N = 5):
  // N = 2 0.180 (six 0.187, eight 0.200), N = 3 0.326 (four 0.357, three 0.364),
  // N = 4 0.340 (eight 0.350, two 0.352), N = 5 0.355 (six 0.360, four 0.401)
  static constexpr int WARPS = D::N == 3 ? 6 : (D::N == 5 ? 7 : 4);
};

// One warp-tile of 16 elements (element e = 16 tile + el). k: the finest substep count;
// nactive: elements [0, nactive) are active at this substep; next_tile: the warp's next
// tile (its planes are prefetched to L2), or -1; first: the CTA's operators are still on
// their way; have: this tile's connectivity and geometry come through the shared tile;
// sops: per-element operators followed by the fragments; sw: the warp's tiles; kComp:
// compensated state update in the commit.
template <int N, bool kComp = false>
__device__ __forceinline__ void stage_tc_warp(const StageParams<float>& p, long long k, int nactive,
                                              const float* sops, float* sw, int tile, int ntiles, int next_tile,
                                              bool first, bool have, double* injected) {
  using D = Dims<N>;
  using C = TcDims<N>;
  using TL = TcLayout<N>;
  using SM = TcSmem<N>;
  constexpr int NP = D::NP, NPP = D::NPP, NFP = D::NFP, KP = C::KP, KSTEP = C::KSTEP, CT = C::CT, NT = C::NT;
  // Gauss points a lane takes through their chains together (ms per macro step as at
  // TcSmem::WARPS): one | two at N = 2 0.190 | 0.187 (six warps), N = 3 0.317 | 0.322,
  // N = 4 0.339 | 0.341, N = 5 0.362 | 0.355
  constexpr int kPointsAtOnce = D::N == 2 || D::N == 5 ? 2 : 1;
  // both faces' gathers at once, or the second after the first face's fluxes (ms per macro
  // step of a 125k-element beach, 45k at N = 5): N = 3 0.384 and 0.358, N = 4 0.363 and 0.376,
  // N = 5 0.427 (spills) and 0.374
  constexpr bool kBothFaces = D::N == 4;
  constexpr int NG = D::NG, KT = C::KT, KF = C::KF, NPT = C::NPT, NB = NPP / 2, BS = SM::BS;
  const uint32_t* sfrag = reinterpret_cast<const uint32_t*>(sops) + SM::FRAG;
  const int lane = threadIdx.x & 31;
  const int el = lane & 15, half = lane >> 4;
  const int g = lane >> 2, t = lane & 3;
  float* st = sw + SM::STATE;
  float* sx = sw + SM::TILE;
  const Sched& sc = p.sc;
  const float gg = p.ph.g_f, hvel = p.ph.hvel_f;
  const size_t fstride = (size_t)NP * sc.KS, bstride = 3 * fstride;
  // lanes past the last active element repeat it (and store nothing)
  const bool valid = tile < ntiles && tile * 16 + el < nactive;
  const int e = valid ? tile * 16 + el : nactive - 1;
  const int lev = level_of(sc, e);
  const long long a = k >> (lev - 1);
  float4 ge;

  // ---- gather: the own nodes (half of them per lane), the first face's neighbour ----
  TeamFace<float, NFP> fc, fc2;   // the lane's first face, and face 2
  bool finer = false;
  {
    float own[4][NB];
    if (tile < ntiles) {
      // a warp's later tiles find both in the shared tile (see the end of the volume term)
      if (have) team_copy_ready();
      const int4 cn = have ? reinterpret_cast<const int4*>(sw + SM::CONN)[el] : __ldg(p.s.conn + e);
      ge = have ? reinterpret_cast<const float4*>(sw + SM::GEO)[el]
                : __ldg(reinterpret_cast<const float4*>(p.s.geo) + e);
      finer = (cn.w >> 12) & 1;
      team_load_face<float, N>(p, cn, e, half, k, fc);
      if (kBothFaces) team_load_face<float, N>(p, cn, e, 2, k, fc2);
      const unsigned ks4 = (unsigned)sc.KS, o0 = half * NB * ks4;
      const float* q0 = p.s.q + (size_t)(a & 1) * bstride + e + o0;
      const float *q1 = q0 + fstride, *q2 = q1 + fstride, *qb = p.s.B + e + o0;
#pragma unroll
      for (int n = 0; n < NB; ++n) {
        if (NB + n < NP || half * NB + n < NP) {
          own[0][n] = ldm(q0 + n * ks4);
          own[1][n] = ldm(q1 + n * ks4);
          own[2][n] = ldm(q2 + n * ks4);
          own[3][n] = __ldg(qb + n * ks4);
        }
      }
      if (!have && half == 0) {
        reinterpret_cast<int4*>(sw + SM::CONN)[el] = cn;
        reinterpret_cast<float4*>(sw + SM::GEO)[el] = ge;
      }
    }
    // this tile's older R slots and the next tile's planes start moving now (hints; the
    // first element's level stands for the tile). 64-bit offsets: the planes of three fields
    // pass 2^32 words above 97 million elements at N = 4 (one wide product per lane; a wide
    // product per plane took 0.6 % of R at N = 4 and 1.5 % of a macro step at N = 5)
    const size_t lane_ks = (size_t)(unsigned)lane * (unsigned)sc.KS;
    if (p.mode == 0 && tile < ntiles) {
      const int e0 = tile * 16;
      const long long a0 = __shfl_sync(0xffffffffu, a, 0);
      const int s0 = ring_slot3(a0);
      const float* ra = p.s.ring + (size_t)(s0 == 0 ? 2 : s0 - 1) * bstride + e0;
      const float* rb = p.s.ring + (size_t)(s0 == 2 ? 0 : s0 + 1) * bstride + e0;
#pragma unroll
      for (int pl = 0; pl < 3 * NP; pl += 32)
        if (pl + lane < 3 * NP) {
          const size_t o = lane_ks + (size_t)pl * sc.KS;
          prefetch_l2(ra + o);
          prefetch_l2(rb + o);
          if constexpr (kComp) prefetch_l2(p.s.comp + e0 + o);
        }
    }
    if (next_tile >= 0 && next_tile * 16 < nactive) {
      const int e0 = next_tile * 16;
      const long long an = k >> (level_of(sc, e0) - 1);
      const float* qn = p.s.q + (size_t)(an & 1) * bstride + e0;
      const float* bn = p.s.B + e0;
#pragma unroll
      for (int pl = 0; pl < 3 * NP; pl += 32)
        if (pl + lane < 3 * NP) prefetch_l2(qn + (size_t)pl * sc.KS + lane_ks);
      if (lane < NP) prefetch_l2(bn + lane_ks);
    }
    if (first) team_ops_ready();
    if (tile >= ntiles) return;
#pragma unroll
    for (int f = 0; f < 4; ++f)
#pragma unroll
      for (int n = 0; n < NB; ++n)
        if (NB + n < NP || half * NB + n < NP) st[(f * KP + half * NB + n) * LS + el] = own[f][n];
  }
  __syncwarp();

  // ---- surface fluxes into the tile ----
  {
    for (int q = 3 * NG + half; q < KF; q += 2)   // padding points: zero rows for the lift
      sx[(0 * KF + q) * LS + el] = sx[(1 * KF + q) * LS + el] = sx[(2 * KF + q) * LS + el] = 0.f;
    const float* my = st + el;
    const float E0 = my[0], B0 = my[3 * KP * LS];
    // the element's node-0 flux, subtracted here and from the volume fluxes (a constant
    // flux adds nothing to R), so the split products see only the variation
    const float hu0 = my[KP * LS], hv0 = my[2 * KP * LS], d0 = E0 - B0;
    const float id0 = d0 > hvel ? recip_fast(d0) : 0.f;
    const float u0 = hu0 * id0, v0 = hv0 * id0;
#pragma unroll 1
    for (int r = 0; r < 2; ++r) {
      const int f = r == 0 ? half : 2;
      const int g0 = r == 0 || half == 0 ? 0 : (NG + 1) / 2, g1 = r == 0 || half == 1 ? NG : (NG + 1) / 2;
      if (r == 1) {
        if (kBothFaces) fc = fc2;
        else team_load_face<float, N>(p, reinterpret_cast<const int4*>(sw + SM::CONN)[el], e, 2, k, fc);
      }
      const float Ef = fc.lower ? fc.E : E0, Bf = fc.lower ? fc.B : B0;
      float vx, vy;
      face_normal(f, ge.x, ge.y, ge.z, ge.w, vx, vy);
      const float v2 = mad(vx, vx, vy * vy), iv = rsqrt_fast(v2);
      const float nx = vx * iv, ny = vy * iv, hs = 0.5f * v2 * iv;
      float2 tr[NFP][4];   // (own, neighbour) relative to the face reference
#pragma unroll
      for (int m = 0; m < NFP; ++m) {
        const float* o = my + face_node_rt(D::N, f, m) * LS;
        tr[m][0] = add2(make_float2(o[0], fc.v[0][m]), dup(-Ef));
        tr[m][1] = make_float2(o[KP * LS], fc.v[1][m]);
        tr[m][2] = make_float2(o[2 * KP * LS], fc.v[2][m]);
        tr[m][3] = add2(make_float2(o[3 * KP * LS], fc.v[3][m]), dup(-Bf));
      }
      const float fr = mad(hu0, vx, hv0 * vy), fu = u0 * fr, fv = v0 * fr;
      constexpr int G = kPointsAtOnce;   // the last group may repeat the face's last point
#pragma unroll 1
      for (int gq = g0; gq < g1; gq += G) {
        float F[G][3];
#pragma unroll
        for (int i = 0; i < G; ++i) {
          const int gi = gq + i < g1 ? gq + i : g1 - 1;
          const float* w = sops + OpLayout<N>::I1P + 2 * gi * D::NFPP;
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
          team_flux<float, N>(p.ph, fc.nb, Ef, Bf, E0, B0, nx, ny, hs, vx, vy, te, tu, tv, tb, F[i][0], F[i][1], F[i][2]);
        }
#pragma unroll
        for (int i = 0; i < G; ++i) {
          const int gi = gq + i < g1 ? gq + i : g1 - 1;
          float* o = sx + (f * NG + gi) * LS + el;
          o[0] = F[i][0] - fr;
          o[KF * LS] = F[i][1] - fu;
          o[2 * KF * LS] = F[i][2] - fv;
        }
      }
    }
  }
  __syncwarp();

  // ---- lift: R -= Flux * L^g^T, k8 tiles of 8 face points ----
  const int r0 = g, r1 = g + 8;
  float Racc[3][NT][4];
#pragma unroll
  for (int f = 0; f < 3; ++f)
#pragma unroll
    for (int nt = 0; nt < NT; ++nt)
#pragma unroll
      for (int c = 0; c < 4; ++c) Racc[f][nt][c] = 0.f;
#pragma unroll
  for (int kt = 0; kt < KT; ++kt) {
    uint2 lb[NT];
#pragma unroll
    for (int nt = 0; nt < NT; ++nt)
      lb[nt] = reinterpret_cast<const uint2*>(sfrag + TL::LIFT)[(kt * NT + nt) * 32 + lane];
#pragma unroll
    for (int f = 0; f < 3; ++f) {
      const float* fq = sx + (f * KF + 8 * kt + 2 * t) * LS;
      uint32_t ah0, al0, ah1, al1;
      split2(make_float2(fq[r0], fq[LS + r0]), ah0, al0);
      split2(make_float2(fq[r1], fq[LS + r1]), ah1, al1);
#pragma unroll
      for (int nt = 0; nt < NT; ++nt) {
        mma_k16(Racc[f][nt], al0, al1, ah0, ah1, lb[nt].x, lb[nt].y);   // lo hi + hi lo
        mma_k8(Racc[f][nt], ah0, ah1, lb[nt].x);
      }
    }
  }
  __syncwarp();   // every lane has read the fluxes before the BF16 tile overwrites them

  // ---- split: the state relative to node 0 (h' or eta', hu', hv', eta' or B') ----
  {
    constexpr int KH = KP / 2;   // nodes per lane, padding included
    const float* my = st + el;
    float c0[4];
#pragma unroll
    for (int f = 0; f < 4; ++f) c0[f] = my[f * KP * LS];
    uint32_t* bt = reinterpret_cast<uint32_t*>(sx) + el * BS + half * (KH / 2);
#pragma unroll
    for (int j = 0; j < KH; j += 8) {
      uint32_t hi[4][4], lo[4][4];
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        // nodes half * KH + j + 2c, + 1; those past NP meet zero operator entries, so any
        // finite value will do (their rows hold zeros)
        const float* o = my + (half * KH + j + 2 * c) * LS;
        float2 v[4];
        if (j + 2 * c >= NP) {   // past NP in both halves
#pragma unroll
          for (int f = 0; f < 4; ++f) v[f] = make_float2(0.f, 0.f);
        } else {
          float2 x[4];
#pragma unroll
          for (int f = 0; f < 4; ++f)
            x[f] = add2(make_float2(o[f * KP * LS], o[(f * KP + 1) * LS]), dup(-c0[f]));
          v[0] = D::EXACT ? add2(x[0], make_float2(-x[3].x, -x[3].y)) : x[0];
          v[1] = x[1];
          v[2] = x[2];
          v[3] = D::EXACT ? x[0] : x[3];
        }
#pragma unroll
        for (int f = 0; f < 4; ++f) split2(v[f], hi[f][c], lo[f][c]);
      }
#pragma unroll
      for (int f = 0; f < 4; ++f) {
        *reinterpret_cast<uint4*>(bt + (2 * f) * 16 * BS + j / 2) = make_uint4(hi[f][0], hi[f][1], hi[f][2], hi[f][3]);
        *reinterpret_cast<uint4*>(bt + (2 * f + 1) * 16 * BS + j / 2) =
            make_uint4(lo[f][0], lo[f][1], lo[f][2], lo[f][3]);
      }
    }
  }
  __syncwarp();
  // ldmatrix address of this lane: row (lane & 15), k offset 8 (lane >> 4)
  const uint32_t bt0 = (uint32_t)__cvta_generic_to_shared(sx) + ((lane & 15) * BS + (lane >> 4) * 4) * 4;
  auto afrag = [&](int f, int part, int ks, uint32_t (&o)[4]) {
    ldmatrix4(o, bt0 + ((2 * f + part) * 16 * BS + ks * 8) * 4);
  };

  const float4 ge0 = reinterpret_cast<const float4*>(sw + SM::GEO)[r0];
  const float4 ge1 = reinterpret_cast<const float4*>(sw + SM::GEO)[r1];
  const float cE0 = st[r0], cE1 = st[r1];
  // ---- mass: X = W (hu', hv') per nodal operator, combined with the affine factors ----
#pragma unroll
  for (int f = 1; f < 3; ++f) {
    float X[2][NT][4];
#pragma unroll
    for (int op = 0; op < 2; ++op)
#pragma unroll
      for (int nt = 0; nt < NT; ++nt)
#pragma unroll
        for (int c = 0; c < 4; ++c) X[op][nt][c] = 0.f;
#pragma unroll
    for (int ks = 0; ks < KSTEP; ++ks) {
      uint32_t ah[4], al[4];
      afrag(f, 0, ks, ah);
      afrag(f, 1, ks, al);
#pragma unroll
      for (int op = 0; op < 2; ++op)
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
          const uint4 b = reinterpret_cast<const uint4*>(sfrag + TL::MASS)[((op * KSTEP + ks) * NT + nt) * 32 + lane];
          mma_k16(X[op][nt], al, b.x, b.y);
          mma_k16(X[op][nt], ah, b.z, b.w);
          mma_k16(X[op][nt], ah, b.x, b.y);
        }
    }
    const float wr0 = f == 1 ? ge0.x : ge0.y, wr1 = f == 1 ? ge1.x : ge1.y;
    const float ws0 = f == 1 ? ge0.z : ge0.w, ws1 = f == 1 ? ge1.z : ge1.w;
#pragma unroll
    for (int nt = 0; nt < NT; ++nt)
#pragma unroll
      for (int c = 0; c < 4; ++c)
        Racc[0][nt][c] =
            mad(c < 2 ? ws0 : ws1, X[1][nt][c], mad(c < 2 ? wr0 : wr1, X[0][nt][c], Racc[0][nt][c]));
  }

  // ---- volume: 8 cubature points at a time ----
  {
    const float2 hu0 = make_float2(st[KP * LS + r0], st[KP * LS + r1]);
    const float2 hv0 = make_float2(st[2 * KP * LS + r0], st[2 * KP * LS + r1]);
    const float2 h0 = make_float2(cE0 - st[3 * KP * LS + r0], cE1 - st[3 * KP * LS + r1]);
    float fr[2][4];   // the momentum fluxes of node 0, per row
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const float h = r ? h0.y : h0.x, mu = r ? hu0.y : hu0.x, mv = r ? hv0.y : hv0.x;
      const float4 ger = r ? ge1 : ge0;
      const float ih = h > hvel ? recip_fast(h) : 0.f;
      const float a0 = mad(ger.x, mu, ger.y * mv), b0 = mad(ger.z, mu, ger.w * mv);
      fr[r][0] = mu * ih * a0;
      fr[r][1] = mv * ih * a0;
      fr[r][2] = mu * ih * b0;
      fr[r][3] = mv * ih * b0;
    }
#pragma unroll 1
    for (int ct = 0; ct < CT; ++ct) {
      constexpr int NA = D::EXACT ? 5 : 6;   // h', hu', hv', eta_r, eta_s; or eta', hu', hv', B_r, B_s, B'
      float acc[NA][4];
#pragma unroll
      for (int o = 0; o < NA; ++o)
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[o][c] = 0.f;
#pragma unroll
      for (int ks = 0; ks < KSTEP; ++ks) {
        const uint4* ib = reinterpret_cast<const uint4*>(sfrag + TL::INTERP) + ((ct * 3) * KSTEP + ks) * 32 + lane;
        const uint4 b0 = ib[0], b1 = ib[KSTEP * 32], b2 = ib[2 * KSTEP * 32];
        uint32_t ah[4], al[4];
#pragma unroll
        for (int f = 0; f < 3; ++f) {
          afrag(f, 0, ks, ah);
          afrag(f, 1, ks, al);
          mma_k16(acc[f], al, b0.x, b0.y);
          mma_k16(acc[f], ah, b0.z, b0.w);
          mma_k16(acc[f], ah, b0.x, b0.y);
        }
        afrag(3, 0, ks, ah);
        afrag(3, 1, ks, al);
        mma_k16(acc[3], al, b1.x, b1.y);
        mma_k16(acc[4], al, b2.x, b2.y);
        mma_k16(acc[3], ah, b1.z, b1.w);
        mma_k16(acc[4], ah, b2.z, b2.w);
        mma_k16(acc[3], ah, b1.x, b1.y);
        mma_k16(acc[4], ah, b2.x, b2.y);
        if constexpr (!D::EXACT) {
          mma_k16(acc[NA - 1], al, b0.x, b0.y);
          mma_k16(acc[NA - 1], ah, b0.z, b0.w);
          mma_k16(acc[NA - 1], ah, b0.x, b0.y);
        }
      }
      // flux and source at the lane's four points, a row (two points) at a time:
      // 0..3 the advective momentum fluxes (Pr hu, hv; Ps hu, hv), 4, 5 the source
      uint32_t fh[6][2], fl[6][2];
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        const float4 ger = r ? ge1 : ge0;
        auto at = [&](int o) { return make_float2(acc[o][2 * r], acc[o][2 * r + 1]); };
        const float2 rx = dup(ger.x), ry = dup(ger.y), sxv = dup(ger.z), sy = dup(ger.w);
        const float2 mu = add2(dup(r ? hu0.y : hu0.x), at(1)), mv = add2(dup(r ? hv0.y : hv0.x), at(2));
        const float2 dh = D::EXACT ? at(0) : add2(at(0), make_float2(-acc[NA - 1][2 * r], -acc[NA - 1][2 * r + 1]));
        const float2 hc = add2(dup(r ? h0.y : h0.x), dh);
        const float2 ih = make_float2(hc.x > hvel ? recip_fast(hc.x) : 0.f, hc.y > hvel ? recip_fast(hc.y) : 0.f);
        const float2 u = mul2(mu, ih), v = mul2(mv, ih);
        const float2 am = fma2(rx, mu, mul2(ry, mv)), bm = fma2(sxv, mu, mul2(sy, mv));
        const float2 dr = at(3), ds = at(4);
        float2 F[6];
        if constexpr (D::EXACT) {
          F[0] = fma2(u, am, dup(-fr[r][0]));
          F[1] = fma2(v, am, dup(-fr[r][1]));
          F[2] = fma2(u, bm, dup(-fr[r][2]));
          F[3] = fma2(v, bm, dup(-fr[r][3]));
        } else {
          const float2 ec = at(0), bc = at(NA - 1);
          const float2 pr = mul2(mul2(dup(0.5f * gg), ec), fma2(dup(-2.f), bc, ec));
          F[0] = fma2(u, am, fma2(rx, pr, dup(-fr[r][0])));
          F[1] = fma2(v, am, fma2(ry, pr, dup(-fr[r][1])));
          F[2] = fma2(u, bm, fma2(sxv, pr, dup(-fr[r][2])));
          F[3] = fma2(v, bm, fma2(sy, pr, dup(-fr[r][3])));
        }
        const float2 gm = mul2(dup(-gg), D::EXACT ? dh : at(0));
        F[4] = mul2(gm, fma2(rx, dr, mul2(sxv, ds)));
        F[5] = mul2(gm, fma2(ry, dr, mul2(sy, ds)));
#pragma unroll
        for (int q = 0; q < 6; ++q) split2(F[q], fh[q][r], fl[q][r]);
      }
      // projection: R_hu += Pr F0 + Ps F2 + P F4, R_hv += Pr F1 + Ps F3 + P F5; the nine
      // split products of a field go in pairs through the k16 instruction
#pragma unroll
      for (int nt = 0; nt < NT; ++nt) {
        const uint2* pb = reinterpret_cast<const uint2*>(sfrag + TL::PROJ) + ((ct * NT + nt) * 3) * 32 + lane;
        const uint2 pr = pb[0], ps = pb[32], pp = pb[64];   // (hi, lo)
#pragma unroll
        for (int f = 0; f < 2; ++f) {
          float(&R)[4] = Racc[1 + f][nt];
          mma_k16(R, fl[f][0], fl[f][1], fl[2 + f][0], fl[2 + f][1], pr.x, ps.x);
          mma_k16(R, fl[4 + f][0], fl[4 + f][1], fh[f][0], fh[f][1], pp.x, pr.y);
          mma_k16(R, fh[2 + f][0], fh[2 + f][1], fh[4 + f][0], fh[4 + f][1], ps.y, pp.y);
          mma_k16(R, fh[f][0], fh[f][1], fh[2 + f][0], fh[2 + f][1], pr.x, ps.x);
          mma_k8(R, fh[4 + f][0], fh[4 + f][1], pp.x);
        }
      }
    }
    // ---- reference term: R_hu -= g h0 (rx Dr + sx Ds)(eta - eta0), R_hv alike ----
    {
      const float gh0 = -gg * h0.x, gh1 = -gg * h0.y;
      float X[2][NT][4];
#pragma unroll
      for (int op = 0; op < 2; ++op)
#pragma unroll
        for (int nt = 0; nt < NT; ++nt)
#pragma unroll
          for (int c = 0; c < 4; ++c) X[op][nt][c] = 0.f;
#pragma unroll
      for (int kk = 0; kk < KP / 8; ++kk) {
        const float* sn = st + (8 * kk + t) * LS;   // eta at node 8kk + t
        uint32_t eh[4], elo[4];
        split_tf32(sn[r0] - cE0, eh[0], elo[0]);
        split_tf32(sn[r1] - cE1, eh[1], elo[1]);
        split_tf32(sn[4 * LS + r0] - cE0, eh[2], elo[2]);
        split_tf32(sn[4 * LS + r1] - cE1, eh[3], elo[3]);
#pragma unroll
        for (int op = 0; op < 2; ++op)
#pragma unroll
          for (int nt = 0; nt < NT; ++nt) {
            const uint4 b = reinterpret_cast<const uint4*>(sfrag + TL::DIFF)[((op * (KP / 8) + kk) * NT + nt) * 32 + lane];
            mma_tf32(X[op][nt], elo, b.x, b.y);
            mma_tf32(X[op][nt], eh, b.z, b.w);
            mma_tf32(X[op][nt], eh, b.x, b.y);
          }
      }
#pragma unroll
      for (int nt = 0; nt < NT; ++nt)
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const float4 gc = c < 2 ? ge0 : ge1;
          const float gh = c < 2 ? gh0 : gh1;
          Racc[1][nt][c] = mad(gh, mad(gc.x, X[0][nt][c], gc.z * X[1][nt][c]), Racc[1][nt][c]);
          Racc[2][nt][c] = mad(gh, mad(gc.y, X[0][nt][c], gc.w * X[1][nt][c]), Racc[2][nt][c]);
        }
    }
  }
  __syncwarp();   // the BF16 tile is read before R overwrites it
  // ahead of the next tile's gather, whose neighbour loads otherwise wait for a trip to
  // memory first (ms per macro step before and after: N = 3, 125k elements 0.318 -> 0.311;
  // N = 4, 500k elements 1.253 -> 1.240; N = 5, 45k elements 0.356 -> 0.353). An L2
  // prefetch of the same lines at the tile's start costs more than it gives (1.260)
  if (next_tile >= 0) {   // the next tile's connectivity (lanes 0-15) and geometry (16-31)
    const int en = next_tile * 16 + el < nactive ? next_tile * 16 + el : nactive - 1;
    const void* src = half ? static_cast<const void*>(p.s.geo + 4 * (size_t)en) : p.s.conn + en;
    const unsigned dst = (unsigned)__cvta_generic_to_shared(sw + (half ? SM::GEO : SM::CONN) + 4 * el);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
  }
#pragma unroll
  for (int f = 0; f < 3; ++f)
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) {
      float* rn = sx + (f * NPT + 8 * nt + 2 * t) * LS;
      rn[r0] = Racc[f][nt][0];
      rn[LS + r0] = Racc[f][nt][1];
      rn[r1] = Racc[f][nt][2];
      rn[LS + r1] = Racc[f][nt][3];
    }
  __syncwarp();

  // ---- commit and positivity, two lanes per element ----
  {
    float R[3][NB], q[4][NB];
#pragma unroll
    for (int n = 0; n < NB; ++n) {
      const int i = half * NB + n;
#pragma unroll
      for (int f = 0; f < 3; ++f) R[f][n] = NB + n < NPT ? sx[(f * NPT + i) * LS + el] : 0.f;   // zero past NP
#pragma unroll
      for (int f = 0; f < 4; ++f) q[f][n] = st[(f * KP + i) * LS + el];
    }
    team_commit<float, N, 2, NB, kComp>(p, sops, valid, finer, e, half, lev, a, q, R, ge.x, ge.y, ge.z, ge.w, injected);
  }
  __syncwarp();   // the tiles are read before the next gather overwrites them
}

// The state rows past NP are read by the TF32 products (with zero operator entries):
// zeroed once, never written again.
template <int N>
__device__ __forceinline__ void stage_tc_init(float* sw) {
  using C = TcDims<N>;
  constexpr int pad = (C::KP - Dims<N>::NP) * LS;
  for (int f = 0; f < 4; ++f)
    for (int i = threadIdx.x & 31; i < pad; i += 32) sw[(f * C::KP + Dims<N>::NP) * LS + i] = 0.f;
  __syncwarp();
}

// Warp-tiles t0, t0 + step, ... below t1 (each warp calls it for its own tiles; the planes
// of its next tile are prefetched to L2); returns the mass the positivity limiter's dry
// resets injected. The separate launch and the persistent
// batch kernel both inline it (out of line the body ran 1.5 times slower: its parameters
// become memory loads).
template <int N, bool kComp = false>
__device__ __forceinline__ double stage_tc_range(const StageParams<float>& __restrict__ p, long long k,
                                              int nactive, const float* __restrict__ sops, float* sw, int t0,
                                              int step, int t1, bool first) {
  double injected = 0.0;
  int tile = t0;
  bool have = false;
  do {   // the first pass waits for the operators whether or not the warp has a tile
    const bool next = tile + step < t1;
    stage_tc_warp<N, kComp>(p, k, nactive, sops, sw, tile, t1, next ? tile + step : -1, first, have, &injected);
    first = false;
    have = next;
    tile += step;
  } while (tile < t1);
  return injected;
}

// Start the copy of a CTA's operators and fragments to shared memory.
template <int N>
__device__ __forceinline__ void tc_ops_begin(float* smem, const float* ops, const uint32_t* frag) {
  using SM = TcSmem<N>;
  team_copy<float, SM::OPS>(smem, ops);
  team_copy<float, TcLayout<N>::SIZE>(smem + SM::FRAG, reinterpret_cast<const float*>(frag));
  asm volatile("cp.async.commit_group;" ::: "memory");
}

// CTA: blockDim.x / 32 warps (1 to 8, swe_set_tc_warps), each with its own shared tiles after the CTA's
// operators. kComp: compensated state update (p.s.comp).
template <int N, bool kComp = false>
__global__ void __launch_bounds__(32 * TcSmem<N>::LIMIT, 1) k_stage_tc(const __grid_constant__ StageParams<float> p) {
  using SM = TcSmem<N>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float* sops = reinterpret_cast<float*>(smem_raw);
  if (p.early) dependents_may_launch();
  tc_ops_begin<N>(sops, p.s.ops, p.s.tcops);
  const int warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  float* sw = sops + SM::CTA + warp * SM::WARP;
  stage_tc_init<N>(sw);
  wait_for_previous();
  const long long k = (*p.s.macro) * (1LL << (p.sc.L - 1)) + p.j;
  const int ntiles = (p.nactive + SM::E - 1) / SM::E;
  const double injected =
      stage_tc_range<N, kComp>(p, k, p.nactive, sops, sw, blockIdx.x * nw + warp, gridDim.x * nw, ntiles, true);
  if (!p.early) dependents_may_launch();
  if (injected != 0.0) atomicAdd(p.s.acc, injected);
}

}  // namespace swe
