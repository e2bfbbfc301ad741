// Device helpers shared by the forward kernels (kernels.cu) and the adjoint
// kernels (adjoint_kernels.inc): ideal MHD fluxes in rationalised units (Eq. 2.2),
// the HLL solver, the Rusanov speed, MinMod, the positivity factors, and the
// face/zone index maps.
#pragma once
#include "device.cuh"

namespace geo {
namespace dev {

constexpr int TPB = 128;

template <typename R> __device__ __forceinline__ const BulkTables<R>& bulk(const DevTables& T);
template <> __device__ __forceinline__ const BulkTables<double>& bulk<double>(const DevTables& T) { return T.b64; }
template <> __device__ __forceinline__ const BulkTables<float>& bulk<float>(const DevTables& T) { return T.b32; }

// ----------------------------------------------------------------------------
// ideal MHD (Eq. 2.2 in rationalised units), in the bulk type R
// ----------------------------------------------------------------------------
template <typename R>
struct Prim {
  R rho, vx, vy, vz, p, bx, by, bz;
};

template <typename R>
__device__ __forceinline__ Prim<R> to_prim(const R* u, R g) {
  Prim<R> w;
  w.rho = u[0];
  R ir = R(1) / u[0];
  w.vx = u[1] * ir;
  w.vy = u[2] * ir;
  w.vz = u[3] * ir;
  w.bx = u[5];
  w.by = u[6];
  w.bz = u[7];
  w.p = (g - R(1)) * (u[4] - R(0.5) * w.rho * (w.vx * w.vx + w.vy * w.vy + w.vz * w.vz) -
                      R(0.5) * (w.bx * w.bx + w.by * w.by + w.bz * w.bz));
  return w;
}

// F(U).n for any vector n
template <typename R>
__device__ __forceinline__ void flux_n(const R* u, const Prim<R>& w, R nx, R ny, R nz, R* F) {
  R vn = w.vx * nx + w.vy * ny + w.vz * nz;
  R bn = w.bx * nx + w.by * ny + w.bz * nz;
  R pt = w.p + R(0.5) * (w.bx * w.bx + w.by * w.by + w.bz * w.bz);
  R vb = w.vx * w.bx + w.vy * w.by + w.vz * w.bz;
  F[0] = w.rho * vn;
  F[1] = u[1] * vn + pt * nx - w.bx * bn;
  F[2] = u[2] * vn + pt * ny - w.by * bn;
  F[3] = u[3] * vn + pt * nz - w.bz * bn;
  F[4] = (u[4] + pt) * vn - bn * vb;
  F[5] = w.bx * vn - w.vx * bn;
  F[6] = w.by * vn - w.vy * bn;
  F[7] = w.bz * vn - w.vz * bn;
}

// One side of a face for the HLL flux along the unit normal n: normal velocity and
// field, total pressure, total enthalpy, v.B and the fast speed, 1/rho formed once.
template <typename R>
struct HllSide {
  R vx, vy, vz, vn, bn, pt, H, vb, c;
};
template <typename R>
__device__ __forceinline__ HllSide<R> hll_side(const R* u, R nx, R ny, R nz, R g) {
  HllSide<R> a;
  const R ir = R(1) / u[0];
  a.vx = u[1] * ir;
  a.vy = u[2] * ir;
  a.vz = u[3] * ir;
  const R hb = R(0.5) * (u[5] * u[5] + u[6] * u[6] + u[7] * u[7]);
  const R p = (g - R(1)) * ((u[4] - hb) - R(0.5) * (u[1] * a.vx + u[2] * a.vy + u[3] * a.vz));
  a.pt = p + hb;
  a.H = u[4] + a.pt;
  a.vn = a.vx * nx + a.vy * ny + a.vz * nz;
  a.bn = u[5] * nx + u[6] * ny + u[7] * nz;
  a.vb = a.vx * u[5] + a.vy * u[6] + a.vz * u[7];
  const R a2 = g * p * ir, s = a2 + R(2) * hb * ir, bn2 = a.bn * a.bn * ir;
  a.c = sqrt(R(0.5) * (s + sqrt(fmax(s * s - R(4) * a2 * bn2, R(0)))));
  return a;
}
// acc += w F(u).n from one side's quantities
template <typename R>
__device__ __forceinline__ void hll_one_side(const R* u, const HllSide<R>& a, R nx, R ny, R nz, R w, R* acc) {
  const R wv = w * a.vn, wb = w * a.bn, wp = w * a.pt;
  acc[0] += u[0] * wv;
  acc[1] += u[1] * wv - u[5] * wb + wp * nx;
  acc[2] += u[2] * wv - u[6] * wb + wp * ny;
  acc[3] += u[3] * wv - u[7] * wb + wp * nz;
  acc[4] += a.H * wv - a.vb * wb;
  acc[5] += u[5] * wv - a.vx * wb;
  acc[6] += u[6] * wv - a.vy * wb;
  acc[7] += u[7] * wv - a.vz * wb;
}

// acc += w times the HLL flux along the unit normal (Davis wave speeds).  With
// a = w S_R / (S_R - S_L), b = -w S_L / (S_R - S_L) and d = a S_L it is
// a F_L + b F_R + d (U_R - U_L), formed from a v_n, a B_n, ... directly: about 200 FP64
// operations a point against 245 with both fluxes written out and combined (p = 4,
// 110,592 zones: 2.79 -> 2.58 ms).
template <typename R>
__device__ __forceinline__ void hll_acc(const R* uL, const R* uR, R nx, R ny, R nz, R g, R w, R* acc) {
  const HllSide<R> l = hll_side(uL, nx, ny, nz, g), r = hll_side(uR, nx, ny, nz, g);
  const R SL = fmin(l.vn - l.c, r.vn - r.c);
  const R SR = fmax(l.vn + l.c, r.vn + r.c);
  if (SL >= R(0)) {
    hll_one_side(uL, l, nx, ny, nz, w, acc);
  } else if (SR <= R(0)) {
    hll_one_side(uR, r, nx, ny, nz, w, acc);
  } else {
    const R wi = w * (R(1) / (SR - SL));
    const R a = wi * SR, b = -(wi * SL), d = a * SL;
    const R av = a * l.vn, ab = a * l.bn, bv = b * r.vn, bb = b * r.bn, p = a * l.pt + b * r.pt;
    acc[0] += av * uL[0] + bv * uR[0] + d * (uR[0] - uL[0]);
    acc[1] += av * uL[1] - ab * uL[5] + bv * uR[1] - bb * uR[5] + p * nx + d * (uR[1] - uL[1]);
    acc[2] += av * uL[2] - ab * uL[6] + bv * uR[2] - bb * uR[6] + p * ny + d * (uR[2] - uL[2]);
    acc[3] += av * uL[3] - ab * uL[7] + bv * uR[3] - bb * uR[7] + p * nz + d * (uR[3] - uL[3]);
    acc[4] += av * l.H - ab * l.vb + bv * r.H - bb * r.vb + d * (uR[4] - uL[4]);
    acc[5] += av * uL[5] - ab * l.vx + bv * uR[5] - bb * r.vx + d * (uR[5] - uL[5]);
    acc[6] += av * uL[6] - ab * l.vy + bv * uR[6] - bb * r.vy + d * (uR[6] - uL[6]);
    acc[7] += av * uL[7] - ab * l.vz + bv * uR[7] - bb * r.vz + d * (uR[7] - uL[7]);
  }
}

// One side of a face for HLLD: the state with its normal field replaced by the face's
// (velocity, pressure and tangential field kept), 1/rho formed once.
template <typename R>
struct HlldSide {
  R rho, m[3], v[3], B[3], E, un, p, pt, bn, ir;
};
template <typename R>
__device__ __forceinline__ HlldSide<R> hlld_side(const R* u, const R* n, R g) {
  HlldSide<R> a;
  a.rho = u[0];
  a.ir = R(1) / u[0];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    a.m[c] = u[1 + c];
    a.v[c] = u[1 + c] * a.ir;
    a.B[c] = u[5 + c];
  }
  a.E = u[4];
  a.un = a.v[0] * n[0] + a.v[1] * n[1] + a.v[2] * n[2];
  a.bn = a.B[0] * n[0] + a.B[1] * n[1] + a.B[2] * n[2];
  const R hb = R(0.5) * (a.B[0] * a.B[0] + a.B[1] * a.B[1] + a.B[2] * a.B[2]);
  a.p = (g - R(1)) * ((a.E - hb) - R(0.5) * (a.m[0] * a.v[0] + a.m[1] * a.v[1] + a.m[2] * a.v[2]));
  a.pt = hb;
  return a;
}
// normal field Bn: B, E and the total pressure change; returns the fast speed
template <typename R>
__device__ __forceinline__ R hlld_normal_field(HlldSide<R>& a, const R* n, R Bn, R g) {
#pragma unroll
  for (int c = 0; c < 3; ++c) a.B[c] += (Bn - a.bn) * n[c];
  const R hb = R(0.5) * (a.B[0] * a.B[0] + a.B[1] * a.B[1] + a.B[2] * a.B[2]);
  a.E += hb - a.pt;
  a.pt = a.p + hb;
  const R a2 = g * a.p * a.ir, s = a2 + R(2) * hb * a.ir, bn2 = Bn * Bn * a.ir;
  return sqrt(R(0.5) * (s + sqrt(fmax(s * s - R(4) * a2 * bn2, R(0)))));
}
// tangential velocity and field of the star state; where rho (S - u)(S - S_M) = B_n^2
// the tangential field stays unchanged
template <typename R>
__device__ __forceinline__ void hlld_star(const HlldSide<R>& a, const R* n, R Bn, R S, R d, R SM, R tol, R* vts,
                                          R* Bts) {
  const R x = d * (S - SM), Bn2 = Bn * Bn, den = x - Bn2;
  const bool ok = fabs(den) > tol * (fabs(x) + Bn2);
  const R iden = R(1) / (ok ? den : R(1));
  const R fv = ok ? Bn * (SM - a.un) * iden : R(0);
  const R fb = ok ? (d * (S - a.un) - Bn2) * iden : R(1);
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const R Bt = a.B[c] - Bn * n[c];
    vts[c] = (a.v[c] - a.un * n[c]) - fv * Bt;
    Bts[c] = Bt * fb;
  }
}

// HLLD flux along the unit normal (Miyoshi & Kusano 2005): fast waves S_L, S_R
// (Davis speeds as in hll_acc), Alfven waves S*_L, S*_R and the entropy wave S_M,
// total pressure constant in the fan; the normal field is the mean of the two
// sides' (each state keeps its pressure).  Where B_n^2 vanishes the ** states
// equal the * states.  acc += w times the flux.  Only the side that holds x/t = 0 gets
// its full star state, and each reciprocal is formed once (9 divisions instead of 21:
// p = 3 FP64, 37,518 zones: 1020 -> 664 us).
template <typename R>
__device__ __forceinline__ void hlld_acc(const R* uL0, const R* uR0, R nx, R ny, R nz, R g, R w, R* acc) {
  const R tol = sizeof(R) == 4 ? R(1e-6) : R(1e-12);
  const R n[3] = {nx, ny, nz};
  HlldSide<R> a = hlld_side(uL0, n, g), b = hlld_side(uR0, n, g);
  const R Bn = R(0.5) * (a.bn + b.bn);
  const R cL = hlld_normal_field(a, n, Bn, g), cR = hlld_normal_field(b, n, Bn, g);
  const R SL = fmin(a.un - cL, b.un - cR), SR = fmax(a.un + cL, b.un + cR);
  R dL = R(0), dR = R(0), SM = R(0), pts = R(0);
  const bool fan = !(SL > R(0) || SR <= R(0));
  if (fan) {
    dL = (SL - a.un) * a.rho;
    dR = (SR - b.un) * b.rho;
    const R idd = R(1) / (dR - dL);
    SM = (dR * b.un - dL * a.un - b.pt + a.pt) * idd;
    pts = (dR * a.pt - dL * b.pt + dL * dR * (b.un - a.un)) * idd;
  }
  // the side of the fan that holds x/t = 0
  const bool left = fan ? SM > R(0) : !(SR <= R(0));
  HlldSide<R> s;
  s.rho = left ? a.rho : b.rho;
  s.E = left ? a.E : b.E;
  s.un = left ? a.un : b.un;
  s.pt = left ? a.pt : b.pt;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    s.m[c] = left ? a.m[c] : b.m[c];
    s.v[c] = left ? a.v[c] : b.v[c];
    s.B[c] = left ? a.B[c] : b.B[c];
  }
  const R vB = s.v[0] * s.B[0] + s.v[1] * s.B[1] + s.v[2] * s.B[2];
  R F[8];
  F[0] = s.rho * s.un;
  F[4] = (s.E + s.pt) * s.un - Bn * vB;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    F[1 + c] = s.m[c] * s.un + s.pt * n[c] - s.B[c] * Bn;
    F[5 + c] = s.B[c] * s.un - s.v[c] * Bn;
  }
  if (fan) {
    R vtL[3], vtR[3], BtL[3], BtR[3];
    hlld_star(a, n, Bn, SL, dL, SM, tol, vtL, BtL);
    hlld_star(b, n, Bn, SR, dR, SM, tol, vtR, BtR);
    const R iL = R(1) / (SL - SM), iR = R(1) / (SR - SM);
    const R rL = dL * iL, rR = dR * iR, sL = sqrt(rL), sR = sqrt(rR);
    const R S = left ? SL : SR, rs = left ? rL : rR, sq = left ? sL : sR, iS = left ? iL : iR;
    R vs[3], Bs[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      vs[c] = SM * n[c] + (left ? vtL[c] : vtR[c]);
      Bs[c] = Bn * n[c] + (left ? BtL[c] : BtR[c]);
    }
    const R vBs = vs[0] * Bs[0] + vs[1] * Bs[1] + vs[2] * Bs[2];
    const R Es = ((S - s.un) * s.E - s.pt * s.un + pts * SM + Bn * (vB - vBs)) * iS;
    F[0] += S * (rs - s.rho);
    F[4] += S * (Es - s.E);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      F[1 + c] += S * (rs * vs[c] - s.m[c]);
      F[5 + c] += S * (Bs[c] - s.B[c]);
    }
    const R al = fabs(Bn) / sq, Ss = left ? SM - al : SM + al;  // this side's Alfven wave
    const bool outer = left ? Ss > R(0) : Ss <= R(0);           // between the fast and the Alfven wave
    const bool mag = Bn * Bn > tol * (pts + R(1e-300));
    if (!outer && mag) {
      const R sg = Bn > R(0) ? R(1) : R(-1), iw = R(1) / (sL + sR), ss = sL * sR * sg;
      R vBss = R(0);
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const R v2 = SM * n[c] + (sL * vtL[c] + sR * vtR[c] + (BtR[c] - BtL[c]) * sg) * iw;
        const R B2 = Bn * n[c] + (sL * BtR[c] + sR * BtL[c] + ss * (vtR[c] - vtL[c])) * iw;
        vBss += v2 * B2;
        F[1 + c] += Ss * (rs * (v2 - vs[c]));
        F[5 + c] += Ss * (B2 - Bs[c]);
      }
      F[4] += Ss * ((left ? -sq : sq) * (vBs - vBss) * sg);
    }
  }
#pragma unroll
  for (int v = 0; v < 8; ++v) acc[v] += w * F[v];
}

template <typename R>
__device__ __forceinline__ R minmod(R a, R b) {
  if (a * b > R(0)) return (a > R(0) ? R(1) : R(-1)) * fmin(fabs(a), fabs(b));
  return R(0);
}

// Positivity scaling (Zhang-Shu type) of point states toward the zone mean: the
// factor theta <= 1 keeps rho >= eps_rho and p >= eps_p at every point, using the
// concavity of p in the conserved variables for the pressure bound.
template <typename R>
__device__ __forceinline__ R pressure_of(const R* u, R g) {
  const R ir = R(1) / u[0];
  return (g - R(1)) * (u[4] - R(0.5) * (u[1] * u[1] + u[2] * u[2] + u[3] * u[3]) * ir -
                       R(0.5) * (u[5] * u[5] + u[6] * u[6] + u[7] * u[7]));
}

template <typename R>
__device__ __forceinline__ void pos_rho(const R* s, const R* mean, R eps_r, R& th_r) {
  if (s[0] < eps_r) th_r = fmin(th_r, (mean[0] - eps_r) / (mean[0] - s[0]));
}

template <typename R>
__device__ __forceinline__ void pos_p(const R* s, const R* mean, R th_r, R g, R pb, R eps_p, R& th_p) {
  R s1[8];
#pragma unroll
  for (int v = 0; v < 8; ++v) s1[v] = mean[v] + th_r * (s[v] - mean[v]);
  const R p1 = pressure_of(s1, g);
  if (p1 < eps_p) th_p = fmin(th_p, (pb - eps_p) / (pb - p1));
}

// Predictor traces, [point][zone][8]: the 8 values of point idx at Gauss time m of
// zone z are adjacent from trF_at(z, m, idx, Z) on.  One point state is one 32-byte
// sector in FP32 (two in FP64): the predictor's threads (zone, variable) store whole
// sectors, and a face or edge thread loads a state with 16-byte loads, consecutive
// zones adjacent.  With the variable outermost ([point][8][zone]) the stores of a
// block of 4 zones filled half a sector each and a state took eight 4-byte loads:
// FP32 face fluxes at p = 4 on 147,456 zones 223 -> 174 us, the predictor with
// positivity on 55,296 zones 1061 -> 1031 us.
template <int P>
__device__ __forceinline__ size_t trF_at(long long z, int m, int idx, long long Z) {
  return (static_cast<size_t>((m - 1) * Dim<P>::NQT + idx) * Z + z) * 8;
}
template <int P>
__device__ __forceinline__ size_t trE_at(long long z, int m, int idx, long long Z) {
  return (static_cast<size_t>((m - 1) * 12 * Dim<P>::NS + idx) * Z + z) * 8;
}

// 16-byte vectors of the bulk type
template <typename R> struct Chunk { static constexpr int CH = 16 / sizeof(R), NCH = 8 / CH; };

template <typename R>
__device__ __forceinline__ void ld16(const R* p, R* out) {
  if constexpr (sizeof(R) == 4) {
    const float4 q = *reinterpret_cast<const float4*>(p);
    out[0] = q.x; out[1] = q.y; out[2] = q.z; out[3] = q.w;
  } else {
    const double2 q = *reinterpret_cast<const double2*>(p);
    out[0] = q.x; out[1] = q.y;
  }
}
template <typename R>
__device__ __forceinline__ void st16(R* p, const R* in) {
  if constexpr (sizeof(R) == 4) {
    *reinterpret_cast<float4*>(p) = make_float4(in[0], in[1], in[2], in[3]);
  } else {
    *reinterpret_cast<double2*>(p) = make_double2(in[0], in[1]);
  }
}

// 16-byte loads and stores of an 8-value state (16-byte aligned)
__device__ __forceinline__ void ld8(const float* p, float* u) {
  const float4 a = reinterpret_cast<const float4*>(p)[0], b = reinterpret_cast<const float4*>(p)[1];
  u[0] = a.x; u[1] = a.y; u[2] = a.z; u[3] = a.w;
  u[4] = b.x; u[5] = b.y; u[6] = b.z; u[7] = b.w;
}
__device__ __forceinline__ void ld8(const double* p, double* u) {
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    const double2 a = reinterpret_cast<const double2*>(p)[c];
    u[2 * c] = a.x;
    u[2 * c + 1] = a.y;
  }
}
__device__ __forceinline__ void st8(float* p, const float* u) {
  reinterpret_cast<float4*>(p)[0] = make_float4(u[0], u[1], u[2], u[3]);
  reinterpret_cast<float4*>(p)[1] = make_float4(u[4], u[5], u[6], u[7]);
}
__device__ __forceinline__ void st8(double* p, const double* u) {
#pragma unroll
  for (int c = 0; c < 4; ++c) reinterpret_cast<double2*>(p)[c] = make_double2(u[2 * c], u[2 * c + 1]);
}

// column and shell of zone z (32-bit division where the index allows it)
__device__ __forceinline__ void zone_column(long long z, int nr, int& c, int& k) {
  if ((z >> 32) == 0) {
    const unsigned q = static_cast<unsigned>(z) / static_cast<unsigned>(nr);
    c = static_cast<int>(q);
    k = static_cast<int>(static_cast<unsigned>(z) - q * static_cast<unsigned>(nr));
  } else {
    c = static_cast<int>(z / nr);
    k = static_cast<int>(z % nr);
  }
}

__device__ __forceinline__ int side_of_lf(int lf) { return lf == 0 ? 3 : (lf == 1 ? 1 : (lf == 2 ? 0 : 2)); }

template <int P>
__device__ __forceinline__ int foff(int lf) {
  using Dm = Dim<P>;
  return lf < 4 ? lf * Dm::NQS : 4 * Dm::NQS + (lf - 4) * Dm::NQR;
}
template <int P>
__device__ __forceinline__ int nq_of(int lf) {
  return lf < 4 ? Dim<P>::NQS : Dim<P>::NQR;
}

// face f -> L zone / local face, R zone / local face (-1 when on the boundary),
// the zones' columns, the column and local face whose tables hold the face geometry,
// shell index k
struct FaceInfo {
  long long zL, zR;
  int lfL, lfR, cL, cR, cg, lfg, k, se;
  double gsign;  // canonical normal = gsign * outward normal of (cg, lfg)
};

__device__ __forceinline__ FaceInfo face_info(const DevTables& T, long long f) {
  FaceInfo fi;
  int nr = T.nr;
  if (f < T.F_rad) {
    int c, k;
    zone_column(f, nr + 1, c, k);
    fi.cL = fi.cR = c;
    fi.zL = (k >= 1) ? static_cast<long long>(c) * nr + k - 1 : -1;
    fi.zR = (k < nr) ? static_cast<long long>(c) * nr + k : -1;
    fi.lfL = 5;
    fi.lfR = 4;
    fi.cg = c;
    fi.lfg = 4;
    fi.gsign = -1.0;
    fi.k = k;
    fi.se = -1;
  } else {
    int se, k;
    zone_column(f - T.F_rad, nr, se, k);
    const int cL = T.se_col[2 * se], cR = T.se_col[2 * se + 1];
    fi.cL = cL;
    fi.cR = cR;
    fi.zL = static_cast<long long>(cL) * nr + k;
    fi.zR = static_cast<long long>(cR) * nr + k;
    fi.lfL = T.se_lf[2 * se];
    fi.lfR = T.se_lf[2 * se + 1];
    fi.cg = cL;
    fi.lfg = fi.lfL;
    fi.gsign = 1.0;
    fi.k = k;
    fi.se = se;
  }
  return fi;
}


}  // namespace dev
}  // namespace geo
