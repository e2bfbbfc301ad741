// Predictor schedule GEO_PRED_VAR_TEAM (a2 zone part + a3): one thread per
// serendipity node for the nonlinear fluxes, one warp per zone for the derivative
// contraction and the point values.  Included by kernels.cu inside its anonymous
// namespace.
//
// The contraction.  A serendipity field of order <= 4 is, on every face of the cube,
// the transfinite interpolant of its four edge curves.  So D^alpha F needs no matrix:
// the four edges along alpha form a ring (q = 0..3 around the axis), face q lies
// between ring edges q and q + 1, and
//   on an edge            dF is the derivative of a polynomial through its P nodes;
//   on a perpendicular    (top - bottom) plus, from the face's two ring edges, the
//   edge's inner nodes    difference of their end derivative and their secant,
//                         weighted linearly across the face.
// With even and odd parts of the edge values this takes 4 x 12 + 4 x 10 operations
// per direction and variable at P = 4 (192 multiply-adds in the sparse rows of
// D^alpha), 4 x 5 + 4 x 4 at P = 3 (96), and its coefficients are the exact small
// rationals of the element, so no table is read.  All four q run the same code on
// their own nodes: lane = q * 8 + v of the zone's warp.
//
// (P = 2: the other end of an edge is one lane bit away, three shuffles per value.)
// Per flux evaluation: the node threads store F^alpha_v (24 values) in ring order,
// lane (q, v) loads the P nodes of edge q and the 2 (P - 2) inner nodes of face q's
// perpendicular edges for the three alpha (16-byte loads at P = 4, free of bank
// conflicts), and puts dF into the same buffer, from where the node threads sum
// their three entries.  With WARP a zone's nodes and its contraction share one
// warp, so the exchange needs no block barrier; without, nodes are packed densely
// over the block's threads (P = 2, 3) and the exchanges are block barriers.
//
// Bounds (196,608 zones).  FP64: the FP64 pipe, 89 % busy at every order (fewer operations
// are the gain).  FP32: the shared memory data path and instruction issue together, 79 %
// and 65 % busy at p = 3, 69 % and 53 % at p = 4, 73 % and 71 % at p = 2.
// Measured, predictor alone, against the sparse rows on the compiled pattern of D^alpha
// (FP64 p = 4: the node team's padded rows):
//   FP32 p = 4, 147,456 zones  2446 -> 1288 us     FP64 p = 4, 110,592 zones  26.98 -> 20.95 ms
//   FP32 p = 3, 193,536 zones   705 ->  561 us     FP64 p = 3, 193,536 zones  13.23 -> 10.99 ms
//   FP32 p = 2, 1,327,104 zones 1023 -> 822 us     FP64 p = 2, 165,888 zones   1.75 ->  1.78 ms
// With positivity: FP32 p = 4 (55,296 zones) 1031 -> 688 us, FP64 p = 4 (18,432)
// 4.99 -> 3.99 ms, FP64 p = 3 (73,728) 5.90 -> 5.35 ms; at FP32 p = 3 and at p = 2 the
// node team stays ahead (419 against 427 us, 166 against 209 us).

template <int P>
struct Ring {
  using Dm = Dim<P>;
  static constexpr int PI = P - 2;        // inner nodes of an edge
  static constexpr int PS = 2 * PI;       // perpendicular inner nodes of a face: bottom, then top
  static constexpr int K = P + PS;        // nodes of one lane: its edge's, then its face's
  __host__ __device__ static constexpr int bit_b(int q) { return q == 1 || q == 2; }
  __host__ __device__ static constexpr int bit_c(int q) { return q >= 2; }
  // local edge index of ring edge q around axis a
  __host__ __device__ static constexpr int edge(int a, int q) { return 4 * a + bit_b(q) + 2 * bit_c(q); }
  // local index of the edge (bottom or top) of face q that is perpendicular to axis a;
  // it runs from ring edge q to q + 1, against its own direction for q >= 2
  __host__ __device__ static constexpr int cross_edge(int a, int q, int top) {
    const int b = a == 0 ? 1 : 0, c = a == 2 ? 1 : 2;
    const int d = (q & 1) ? c : b, o = (q & 1) ? b : c, fo = q == 1 || q == 2;
    // the fixed coordinates of an edge along d: a and o, in axis order
    return 4 * d + (a < o ? top + 2 * fo : fo + 2 * top);
  }
  // node of the t-th node thread of a zone.  P = 4 (a warp per zone): with the chunk
  // shuffle RingLayout::swz, the 8 nodes of a 16-byte access phase read their flux
  // differences from distinct bank groups in all three directions.  P = 3 (a warp
  // holds four nodes of eight zones): each four nodes have different q in all three
  // directions, so their stores fall into distinct banks.
  __host__ __device__ static constexpr int thread_node(int t) {
    constexpr unsigned char o4[32] = {2, 6, 9, 10, 17, 18, 26, 28, 0, 4, 8, 11, 16, 19, 24, 30,
                                      3, 7, 12, 15, 20, 23, 25, 31, 1, 5, 13, 14, 21, 22, 27, 29};
    constexpr unsigned char o3[20] = {0, 3, 5, 6, 1, 2, 4, 7, 8, 11, 17, 18, 9, 10, 13, 14, 12, 15, 16, 19};
    return P == 4 ? o4[t & 31] : (P == 3 ? o3[t % 20] : t);
  }
  // node of slot k of lane q
  __host__ __device__ static constexpr int node(int a, int q, int k) {
    const int b = a == 0 ? 1 : 0, c = a == 2 ? 1 : 2;
    if (k < P) {
      if (k == 0 || k == P - 1)
        return ((k != 0) << a) + (bit_b(q) << b) + (bit_c(q) << c);
      return 8 + PI * edge(a, q) + k - 1;
    }
    const int top = (k - P) / (PI > 0 ? PI : 1), j = (k - P) % (PI > 0 ? PI : 1);
    return 8 + PI * cross_edge(a, q, top) + (q < 2 ? j : PI - 1 - j);
  }
};

// execution shape per order and type.  WARP (P = 4): warp w of the block holds zone w,
// lane = node.  P = 3: a warp holds four nodes of the block's eight zones (zone
// fastest); P = 2: eight nodes of four zones.
template <int P, typename R> struct RingCfg;
template <> struct RingCfg<2, float> {
  static constexpr bool POS = false, WARP = false;
  static constexpr int ZB = 16, MINB = 14;
};
template <> struct RingCfg<3, float> {
  static constexpr bool POS = false, WARP = false;
  static constexpr int ZB = 8, MINB = 7;
};
template <> struct RingCfg<4, float> {
  static constexpr bool POS = true, WARP = true;
  static constexpr int ZB = 4, MINB = 5;
};
template <> struct RingCfg<2, double> {
  static constexpr bool POS = false, WARP = false;
  static constexpr int ZB = 16, MINB = 4;
};
template <> struct RingCfg<3, double> {
  static constexpr bool POS = true, WARP = false;
  static constexpr int ZB = 8, MINB = 3;
};
template <> struct RingCfg<4, double> {
  static constexpr bool POS = true, WARP = true;
  static constexpr int ZB = 4, MINB = 2;
};

template <int P, typename R>
struct RingLayout {
  using Dm = Dim<P>;
  using C = RingCfg<P, R>;
  static constexpr int N = Dm::N, ZB = C::ZB, NT = C::WARP ? 32 * ZB : ZB * N, NW = NT / 32;
  // row stride of one variable's nodes.  P = 4: a lane's nodes are adjacent (16-byte
  // loads), chunks at an odd chunk stride; P = 3: (k, q) order, q fastest
  static constexpr int RS = P == 4 ? (sizeof(R) == 4 ? 36 : 34) : (P == 3 ? 20 : 10);
  static constexpr int FS = 8 * RS > 32 * Ring<P>::K ? 8 * RS : 32 * Ring<P>::K;  // one direction of a zone
  static constexpr int FZ = (P == 2 ? 1 : 3) * FS + (C::WARP ? 0 : 4);            // one zone (P = 2: levels only)
  // one zone's final levels: in FP32 at P = 3 the four zones of a point task, whose
  // rows lie on multiples of 4 banks, are one bank apart
  static constexpr int FL = P == 3 ? (Dm::M - 1) * FS + 1 : FZ;
  static_assert(NT % 32 == 0, "whole warps");
  // position of (lane q, slot k) in a variable's row
  __device__ static constexpr int in_pos(int q, int k) {
    return P == 3 ? 4 * k + q : (k < P ? q * P + k : 4 * P + q * Ring<P>::PS + k - P);
  }
  // FP32, P = 4: chunk (2 q + half) of output row k sits at chunk ^ swz(k)
  __device__ static constexpr int swz(int k) {
    if (sizeof(R) == 8 || P != 4) return 0;
    return k < 4 ? (k == 0 ? 3 : (k == 1 ? 6 : (k == 2 ? 5 : 7))) : (k == 4 ? 1 : (k == 5 ? 2 : 0));
  }
  // first value of the 8-vector of (q, k); FP32: the second half sits at offset ^ 4
  __device__ static int out_pos(int q, int k) {
    if constexpr (sizeof(R) == 4) return k * 32 + ((2 * q) ^ swz(k)) * 4;
    return k * 32 + q * 8;
  }
};

template <int P, typename R>
struct RingSmem {
  using L = RingLayout<P, R>;
  using Dm = Dim<P>;
  alignas(16) R F[L::ZB * L::FZ];            // fluxes / flux differences / nodal values / final levels
  alignas(16) R in[Dm::NBIN][L::ZB];         // inputs of the divergence-free reconstruction
  alignas(16) R W[5 * Dm::NC1][L::ZB];       // fluid Taylor coefficients
  alignas(16) R Uz[8][L::ZB];                // zone means (B: the divergence-free mean)
  R fs[L::ZB];                               // dt l_0 / l_k of the zone (Eq. 5.21)
  R th[L::ZB][5];                            // positivity factors (min-reduced)
};

// with positivity: SLOTS x 4 point states of each warp, checked one per lane (the state
// stride keeps the 16-byte loads of a zone's eight states in distinct bank groups)
template <int P, typename R, bool POS>
struct RingTile {
  static constexpr int STRIDE = 32 + 16 / sizeof(R);
  static constexpr int SLOTS = P == 3 && sizeof(R) == 8 ? 4 : 8;  // within 48 KB of static shared memory
  alignas(16) R s[POS ? RingLayout<P, R>::NW : 1][POS ? SLOTS * STRIDE : 1];
};

// L consecutive values, in 16-byte vectors where they are whole ones
template <int L, typename R>
__device__ __forceinline__ void ring_load(const R* p, R* out) {
  constexpr int CH = Chunk<R>::CH;
  if constexpr (L % CH == 0) {
#pragma unroll
    for (int c = 0; c < L / CH; ++c) ld16(p + c * CH, out + c * CH);
  } else {
#pragma unroll
    for (int c = 0; c < L; ++c) out[c] = p[c];
  }
}
// the P nodes of ring edge q and the inner nodes of face q from a variable's row
template <int P, typename R>
__device__ __forceinline__ void ring_nodes(const R* row, int q, R* edge, R* inner) {
  using L = RingLayout<P, R>;
  using G = Ring<P>;
  if constexpr (P == 3) {
#pragma unroll
    for (int k = 0; k < P; ++k) edge[k] = row[L::in_pos(q, k)];
#pragma unroll
    for (int k = 0; k < G::PS; ++k) inner[k] = row[L::in_pos(q, P + k)];
  } else {
    ring_load<P>(row + L::in_pos(q, 0), edge);
    if constexpr (G::PS > 0) ring_load<G::PS>(row + L::in_pos(q, P), inner);
  }
}

// Derivative along one axis of a lane's edge nodes f[0..P) and, with the two ring
// edges of its face, of the face's perpendicular inner nodes f[P..K).  RingEdge: what a lane
// forms from its own edge, a and b of which the lane of ring edge q - 1 needs as well
// (host code too: ring_matrix checks the coefficients against the element's D^alpha).
template <typename R>
struct RingEdge {
  R u, a, b;
};
template <int P, typename R>
__host__ __device__ __forceinline__ RingEdge<R> ring_edge(const R* f) {
  RingEdge<R> e{R(0), R(0), R(0)};
  if constexpr (P == 2) {
    e.u = f[1] - f[0];
  } else if constexpr (P == 3) {
    e.u = f[2] - f[0];
    e.a = (f[0] + f[2]) - R(2) * f[1];
  } else {
    const R u = f[3] - f[0], g = (f[0] + f[3]) - (f[1] + f[2]), r = u - R(3) * (f[2] - f[1]);
    e.u = u;
    e.a = r + g;
    e.b = r - g;
  }
  return e;
}
template <int P, typename R>
__host__ __device__ __forceinline__ void ring_apply(R* f, const RingEdge<R>& e, R an, R bn) {
  if constexpr (P == 2) {
    f[0] = e.u;
    f[1] = e.u;
  } else if constexpr (P == 3) {
    const R G = e.a + an;
    const R t = f[4] - f[3];
    f[0] = e.u - R(2) * e.a;
    f[1] = e.u;
    f[2] = e.u + R(2) * e.a;
    f[3] = t - G;
    f[4] = t + G;
  } else {
    const R t1 = f[6] - f[4], t2 = f[7] - f[5];
    f[0] = e.u + R(2.25) * e.b;
    f[1] = e.u - R(0.75) * e.a;
    f[2] = e.u - R(0.75) * e.b;
    f[3] = e.u + R(2.25) * e.a;
    f[4] = (t1 + R(1.5) * e.b) + R(0.75) * bn;
    f[5] = (t2 + R(0.75) * e.b) + R(1.5) * bn;
    f[6] = (t1 + R(1.5) * e.a) + R(0.75) * an;
    f[7] = (t2 + R(0.75) * e.a) + R(1.5) * an;
  }
}
template <int P, typename R>
__device__ __forceinline__ void ring_derivative(R* f, int lane) {
  const int next = (lane + 8) & 31;  // the same variable of ring edge q + 1
  const RingEdge<R> e = ring_edge<P>(f);
  R an = R(0), bn = R(0);
  if constexpr (P > 2) an = __shfl_sync(0xffffffffu, e.a, next);
  if constexpr (P == 4) bn = __shfl_sync(0xffffffffu, e.b, next);
  ring_apply<P>(f, e, an, bn);
}

// contraction of one zone by its warp: F rows in, dF entries out, in place
template <int P, typename R>
__device__ __forceinline__ void ring_contract(R* Fz, int lane) {
  using L = RingLayout<P, R>;
  using G = Ring<P>;
  const int q = lane >> 3, v = lane & 7;
  R f[3][G::K];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    ring_nodes<P>(Fz + a * L::FS + v * L::RS, q, f[a], f[a] + P);
  }
  __syncwarp();  // every lane has its inputs: the buffer takes the outputs
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    ring_derivative<P>(f[a], lane);
    R* out = Fz + a * L::FS;
#pragma unroll
    for (int k = 0; k < G::K; ++k) {
      if constexpr (sizeof(R) == 4) out[k * 32 + (((2 * q + (v >> 2)) ^ L::swz(k)) << 2) + (v & 3)] = f[a][k];
      else out[k * 32 + lane] = f[a][k];
    }
  }
}

// Point values from ML final levels in ring order around the radial axis (levels FS
// apart), for variable v of one zone: side face q (all its points), the three edges
// radial q, bottom q, top q, and the points of both radial faces next to ring corner q
// and to face q's edge (and, shared out, the middle one).  A warp has one q and, as
// lanes, four zones x 8 variables: by the symmetry of the element all q use the same
// weights (constant bank), the point's index is uniform, and a store fills whole
// 128-byte lines of [point][zone][8].  face / edge(idx, m0, s, mine): the point's values
// at the levels m0..; with ALL every q passes every point, mine telling whose it is.
template <int P, int ML, bool ALL, typename R, typename EmitF, typename EmitE>
__device__ __forceinline__ void ring_points(const R* Fz, int q, const RefConst<P, R>& K, EmitF&& face,
                                            EmitE&& edge) {
  using L = RingLayout<P, R>;
  using G = Ring<P>;
  using Dm = Dim<P>;
  constexpr int NFN = Dm::NFN, PI = G::PI, NU = P == 4 ? 3 : 2, NV = 2;
  {
    R e0[ML][P], e1[ML][P], p0[ML][G::PS > 0 ? G::PS : 1], skip[G::PS > 0 ? G::PS : 1];
#pragma unroll
    for (int m = 0; m < ML; ++m) {
      ring_nodes<P>(Fz + m * L::FS, q, e0[m], p0[m]);
      ring_nodes<P>(Fz + m * L::FS, (q + 1) & 3, e1[m], skip);
    }
    // ---- side face q (nodes: edge q, edge q + 1, bottom and top inner nodes);
    // local face of ring face q: eta-, xi+, eta+, xi-
    const int lf = q == 0 ? 2 : (q == 1 ? 1 : (q == 2 ? 3 : 0));
    const int base = lf * Dm::NQS + (q < 2 ? 0 : (NU - 1) * NV), du = q < 2 ? NV : -NV;
#pragma unroll
    for (int a = 0; a < NU; ++a)
#pragma unroll
      for (int b = 0; b < NV; ++b) {
        const R* w = K.wS + (a * NV + b) * NFN;
        R s[ML];
#pragma unroll
        for (int m = 0; m < ML; ++m) {
          s[m] = w[0] * e0[m][0];
#pragma unroll
          for (int t = 1; t < P; ++t) s[m] += w[t] * e0[m][t];
#pragma unroll
          for (int t = 0; t < P; ++t) s[m] += w[P + t] * e1[m][t];
#pragma unroll
          for (int t = 0; t < G::PS; ++t) s[m] += w[2 * P + t] * p0[m][t];
        }
        face(base + a * du + b, 0, s, true);
      }
    // ---- edges: radial edge q, then bottom and top edge of face q
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const int z = c == 2 ? P - 1 : 0;
      const bool rev = c > 0 && q >= 2;
      const int le = c == 0 ? 8 + G::bit_b(q) + 2 * G::bit_c(q)
                            : ((q & 1) ? 4 + (q == 1) + 2 * (c - 1) : (q == 2) + 2 * (c - 1));
      const int b0 = le * Dm::NS + (rev ? Dm::NS - 1 : 0), ds = rev ? -1 : 1;
#pragma unroll
      for (int s = 0; s < Dm::NS; ++s) {
        R val[ML];
#pragma unroll
        for (int m = 0; m < ML; ++m) {
          R y[P];
#pragma unroll
          for (int t = 0; t < P; ++t)
            y[t] = c == 0 ? e0[m][t] : (t == 0 ? e0[m][z] : (t == P - 1 ? e1[m][z] : p0[m][(c - 1) * PI + t - 1]));
          if (P == 4 && s != 1) {  // Simpson's end points are nodes
            val[m] = y[s == 0 ? 0 : P - 1];
          } else {
            val[m] = K.wEd[s * P] * y[0];
#pragma unroll
            for (int t = 1; t < P; ++t) val[m] += K.wEd[s * P + t] * y[t];
          }
        }
        edge(b0 + s * ds, 0, val, true);
      }
    }
  }
  // ---- radial faces (nodes: corners q, q+1, q+2, q+3, then the inner nodes of their
  // edges), one level at a time
#pragma unroll
  for (int m = 0; m < ML; ++m) {
    R e[4][P], p[4][G::PS > 0 ? G::PS : 1];
#pragma unroll
    for (int r = 0; r < 4; ++r) ring_nodes<P>(Fz + m * L::FS, (q + r) & 3, e[r], p[r]);
#pragma unroll
    for (int top = 0; top < 2; ++top) {
      const int f0 = 4 * Dm::NQS + top * Dm::NQR;
      auto point = [&](int w3, int idx, bool mine) {
        const R* w = K.wR + w3 * NFN;
        R s[1] = {R(0)};
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          s[0] += w[r] * e[r][top * (P - 1)];
#pragma unroll
          for (int t = 0; t < PI; ++t) s[0] += w[4 + r * PI + t] * p[r][top * PI + t];
        }
        face(f0 + idx, m, s, mine);
      };
      point(0, G::bit_b(q) * (NU - 1) * NU + G::bit_c(q) * (NU - 1), true);
      if constexpr (P == 4) {
        // next to the middle of face q's edge: (1,0), (2,1), (1,2), (0,1)
        point(1, (q == 1 ? 2 : (q == 3 ? 0 : 1)) * NU + (q == 0 ? 0 : (q == 2 ? 2 : 1)), true);
        if (ALL || q == 2 * top) point(2, NU + 1, q == 2 * top);
      }
    }
  }
}

// Positivity factors of the point states held in a warp's tile (lane = zone * 8 + slot),
// min-reduced into the zones' th: pass 0 theta_rho and, for theta_rho = 1, theta_p;
// pass 1 theta_p for the zone's theta_rho.  Out of line: it is called every SLOTS points
// of the fully unrolled point code, which it would blow up beyond the instruction cache.
template <int P, typename R>
__device__ __noinline__ void ring_check(const R* my, RingSmem<P, R>& S, int held, int zl, int lane, R gam, int pass) {
  constexpr int TS = RingTile<P, R, true>::STRIDE;
  __syncwarp();
  if ((lane & 7) < held) {
    R s[8], mz[8];
    ld8(my + (lane & 7) * TS + (lane & 24), s);
#pragma unroll
    for (int e = 0; e < 8; ++e) mz[e] = S.Uz[e][zl];
    const R pb = pressure_of(mz, gam), er = fmin(R(1e-13), mz[0]), ep = fmin(R(1e-13), pb);
    R pr = R(1), pp = R(1);
    if (pass == 0) {
      pos_rho(s, mz, er, pr);
      if (pr < R(1)) smem_min_nonneg(&S.th[zl][2], pr);
    }
    pos_p(s, mz, pass == 0 ? R(1) : S.th[zl][2], gam, pb, ep, pp);
    if (pp < R(1)) smem_min_nonneg(&S.th[zl][pass == 0 ? 4 : 3], pp);
  }
  __syncwarp();
}

// STORE: also write the levels (times J) after each of the first P-1 Picard iterations to
// itS ([P-1][M-1][8][N][Z]), the linearisation points of the reverse sweep
template <int P, typename R, bool POS, bool STORE = false>
__global__ void __launch_bounds__(RingLayout<P, R>::NT, RingCfg<P, R>::MINB)
    k_ader_ring(const DevTables T, double* __restrict__ U, const double* __restrict__ phi, const R* __restrict__ Wc,
                const R* __restrict__ Bp, R* __restrict__ trF, R* __restrict__ trE, double dt, R* __restrict__ itS) {
  using Dm = Dim<P>;
  using L = RingLayout<P, R>;
  using G = Ring<P>;
  constexpr bool WARP = RingCfg<P, R>::WARP;
  constexpr int N = Dm::N, M = Dm::M, ML = M - 1, NC1 = Dm::NC1, NC = Dm::NC, NQT = Dm::NQT, NQS = Dm::NQS,
                NQR = Dm::NQR, NBIN = Dm::NBIN, ZB = L::ZB, NT = L::NT, NW = L::NW;
  __shared__ RingSmem<P, R> S;
  __shared__ RingTile<P, R, POS> tile;
  const RefConst<P, R>& K = RC<P, R>::get();
  const BulkTables<R>& BT = bulk<R>(T);
  const long long Z = T.Z, F = T.F;
  const int nr = T.nr;
  // (the warp index through a shuffle, so that the compiler keeps what follows from it,
  // the point indices and their addresses above all, in uniform registers)
  // (p = 2, 1,327,104 zones: 917 -> 877 us, p = 3, 193,536: 582 -> 561 us, FP32; at p = 4
  // it costs registers that are not there: 1288 -> 1462 us)
  const int tid = threadIdx.x, lane = tid & 31, warp = P == 4 ? tid >> 5 : __shfl_sync(0xffffffffu, tid >> 5, 0);
  const long long zbase = static_cast<long long>(blockIdx.x) * ZB;
  int c0, k0;
  zone_column(zbase, nr, c0, k0);
  // column and shell of the block's zone zl
  auto column = [&](int zl, int& c, int& k) {
    c = c0;
    k = k0 + zl;
    while (k >= nr) {
      k -= nr;
      ++c;
    }
  };
  // ---- zone inputs into shared memory, zone fastest
  for (int w = tid; w < ZB * 8 * NC1; w += NT) {
    const int zl = w % ZB, e = w / ZB;
    const long long z = zbase + zl;
    const R x = z < Z ? Wc[static_cast<size_t>(e) * Z + z] : R(0);
    if (e < 5 * NC1) {
      S.W[e][zl] = x;
    } else {
      const int d = (e - 5 * NC1) / NC1;
      S.in[e - 5 * NC1 + d + 1][zl] = x;
    }
  }
  for (int w = tid; w < ZB * 8; w += NT) {
    const int zl = w % ZB, v = w / ZB;
    const long long z = zbase + zl;
    const R x = z < Z ? static_cast<R>(U[v * Z + z]) : R(1);
    if (v < 5) S.Uz[v][zl] = x;
    else S.in[(v - 5) * NC][zl] = x;
  }
  for (int w = tid; w < ZB * (NQT + 6); w += NT) {
    const int zl = w % ZB, e = w / ZB;
    R x = R(0);
    int dst = 3 * NC + e;
    if (zbase + zl < Z) {
      int c, k;
      column(zl, c, k);
      const int lf = e >= NQT ? e - NQT : (e < 4 * NQS ? e / NQS : 4 + (e - 4 * NQS) / NQR);
      long long f;
      int sg, se = -1;
      if (lf < 4) {
        const int sd = side_of_lf(lf);
        se = T.col_side_se[4 * c + sd];
        sg = T.col_side_sgn[4 * c + sd];
        f = T.F_rad + static_cast<long long>(se) * nr + k;
      } else {
        f = static_cast<long long>(c) * (nr + 1) + k + (lf == 5 ? 1 : 0);
        sg = lf == 5 ? 1 : -1;
      }
      if (e < NQT) {
        const int q = e - foff<P>(lf);
        if (lf < 4 && sg < 0) dst = 3 * NC + foff<P>(lf) + T.se_perm[se * NQS + q];
        x = static_cast<R>(sg) * Bp[static_cast<size_t>(q) * F + f];
      } else {
        // face mean <B_perp> = Phi / A with the tabulated reciprocal area
        x = static_cast<R>(sg * phi[f] * T.iA0[6 * c + lf] * T.iq2[k]);
      }
    }
    S.in[dst][zl] = x;
  }
  if (tid < ZB) {
    int c, k;
    column(tid, c, k);
    S.fs[tid] = zbase + tid < Z ? static_cast<R>(dt / T.qpow[k]) : R(0);
#pragma unroll
    for (int t = 0; t < 5; ++t) S.th[tid][t] = R(1);
  }
  __syncthreads();
  // ---- zone-mean B (Sec. IV.b step 10)
  if constexpr (WARP) {
    // component d by warp d, the KKT row spread over its lanes
    if (warp < 3) {
      for (int z0 = 0; z0 < ZB && zbase + z0 < Z;) {
        int c, k, z1 = z0 + 1;
        column(z0, c, k);
        while (z1 < ZB && k + z1 - z0 < nr) ++z1;  // zones z0..z1-1 share the column
        const R* GM = BT.GM + (static_cast<size_t>(c) * 3 + warp) * NBIN;
        R s[ZB];
#pragma unroll
        for (int z = 0; z < ZB; ++z) s[z] = R(0);
        for (int b = lane; b < NBIN; b += 32) {
          const R gm = GM[b];
          R x[ZB];
          ring_load<ZB>(&S.in[b][0], x);
#pragma unroll
          for (int z = 0; z < ZB; ++z) s[z] += gm * x[z];
        }
#pragma unroll
        for (int z = 0; z < ZB; ++z) {
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) s[z] += __shfl_xor_sync(0xffffffffu, s[z], o);
          if (lane == 0 && z >= z0 && z < z1 && zbase + z < Z) {
            S.Uz[5 + warp][z] = s[z];
            U[(5 + warp) * Z + zbase + z] = static_cast<double>(s[z]);
          }
        }
        z0 = z1;
      }
    }
  } else if (tid < 3 * ZB) {
    const int z = tid % ZB, d = tid / ZB;
    if (zbase + z < Z) {
      int c, k;
      column(z, c, k);
      const R* GM = BT.GM + (static_cast<size_t>(c) * 3 + d) * NBIN;
      R s = R(0);
#pragma unroll 6
      for (int b = 0; b < NBIN; ++b) s += GM[b] * S.in[b][z];
      S.Uz[5 + d][z] = s;
      U[(5 + d) * Z + zbase + z] = static_cast<double>(s);
    }
  }
  // ---- node of this thread
  const int zl = WARP ? warp : (P == 3 ? tid % ZB : tid / N);
  const int i = P == 2 ? tid % N : K.tnode[WARP ? lane : tid / ZB];
  const long long z = zbase + zl;
  const bool valid = z < Z;
  int c, kz;
  column(zl, c, kz);
  const R gam = static_cast<R>(T.gamma);
  R* Fz = S.F + zl * L::FZ;
  // ---- reconstructed conserved values at the nodes (Sec. V.d steps 5-6)
  R u0[8];
  if constexpr (WARP) {
    // warp d < 3: B component d at all nodes of all zones, warp 3: the fluid, so that
    // one load of a KKT or Taylor entry serves the block's zones (of one column)
    static_assert(!WARP || NW == 4, "four warps share the nodal values");
    {
      for (int z0 = 0; z0 < ZB && zbase + z0 < Z;) {
        int cc, k, z1 = z0 + 1;
        column(z0, cc, k);
        while (z1 < ZB && k + z1 - z0 < nr) ++z1;
        if (warp < 3) {
          const R* GB = BT.GB + static_cast<size_t>(cc) * 3 * N * NBIN + warp * N + i;
          R s[ZB];
#pragma unroll
          for (int t = 0; t < ZB; ++t) s[t] = R(0);
#pragma unroll 12
          for (int b = 0; b < NBIN; ++b) {
            const R gb = GB[b * 3 * N];
            R x[ZB];
            ring_load<ZB>(&S.in[b][0], x);
#pragma unroll
            for (int t = 0; t < ZB; ++t) s[t] += gb * x[t];
          }
          for (int t = z0; t < z1; ++t)
            S.F[t * L::FZ + (5 + warp) * L::RS + i] = t == 0 ? s[0] : (t == 1 ? s[1] : (t == 2 ? s[2] : s[3]));
        } else {
          const R* TN = BT.TN + static_cast<size_t>(cc) * N * NC1 + i;
          R s[5][ZB];
#pragma unroll
          for (int v = 0; v < 5; ++v) ring_load<ZB>(&S.Uz[v][0], s[v]);
#pragma unroll 5
          for (int m = 0; m < NC1; ++m) {
            const R tn = TN[m * N];
#pragma unroll
            for (int v = 0; v < 5; ++v) {
              R x[ZB];
              ring_load<ZB>(&S.W[v * NC1 + m][0], x);
#pragma unroll
              for (int t = 0; t < ZB; ++t) s[v][t] += tn * x[t];
            }
          }
#pragma unroll
          for (int t = 0; t < ZB; ++t)
            if (t >= z0 && t < z1) {
#pragma unroll
              for (int v = 0; v < 5; ++v) S.F[t * L::FZ + v * L::RS + i] = s[v][t];
            }
        }
        z0 = z1;
      }
    }
    __syncthreads();
#pragma unroll
    for (int v = 0; v < 8; ++v) u0[v] = valid ? Fz[v * L::RS + i] : R(1);
    __syncwarp();
  } else {
    // FP32: the B components by threads (row of the KKT matrix, four zones), so that one
    // load of an entry serves four zones; FP64, bound by its pipe, keeps all threads busy
    // instead: every thread forms its own node's
    constexpr bool SHARE = sizeof(R) == 4;
    if constexpr (SHARE) {
      constexpr int ROWS = 3 * N;
      static_assert(ROWS * (ZB / 4) <= NT, "one row and four zones per thread");
      if (tid < ROWS * (ZB / 4)) {
        const int r = tid % ROWS, zq = tid / ROWS * 4;
        for (int z0 = zq; z0 < zq + 4 && zbase + z0 < Z;) {
          int cc, k, z1 = z0 + 1;
          column(z0, cc, k);
          while (z1 < zq + 4 && k + z1 - z0 < nr) ++z1;
          const R* GB = BT.GB + static_cast<size_t>(cc) * ROWS * NBIN + r;
          R s[4] = {R(0), R(0), R(0), R(0)};
#pragma unroll 12
          for (int b = 0; b < NBIN; ++b) {
            const R gb = GB[b * ROWS];
            R x[4];
            ring_load<4>(&S.in[b][zq], x);
#pragma unroll
            for (int t = 0; t < 4; ++t) s[t] += gb * x[t];
          }
#pragma unroll
          for (int t = 0; t < 4; ++t)
            if (zq + t >= z0 && zq + t < z1) S.F[(zq + t) * L::FZ + r] = s[t];
          z0 = z1;
        }
      }
    }
    if (POS || SHARE) __syncthreads();
    if (valid) {
      const R* TN = BT.TN + static_cast<size_t>(c) * N * NC1 + i;
      const R* GB = BT.GB + static_cast<size_t>(c) * 3 * N * NBIN + i;
#pragma unroll
      for (int v = 0; v < 5; ++v) u0[v] = S.Uz[v][zl];
#pragma unroll
      for (int m = 0; m < NC1; ++m) {
        const R tn = TN[m * N];
#pragma unroll
        for (int v = 0; v < 5; ++v) u0[v] += tn * S.W[v * NC1 + m][zl];
      }
      if constexpr (SHARE) {
#pragma unroll
        for (int d = 0; d < 3; ++d) u0[5 + d] = Fz[d * N + i];
      } else {
#pragma unroll
        for (int d = 0; d < 3; ++d) u0[5 + d] = R(0);
#pragma unroll 6
        for (int b = 0; b < NBIN; ++b) {
          const R x = S.in[b][zl];
#pragma unroll
          for (int d = 0; d < 3; ++d) u0[5 + d] += GB[b * 3 * N + d * N] * x;
        }
      }
    } else {
#pragma unroll
      for (int v = 0; v < 8; ++v) u0[v] = R(1);
    }
    if (SHARE) __syncthreads();  // the buffer takes the fluxes next
  }
  R Uzp[8];  // the zone mean (positivity)
  R pbar = R(0), eps_r = R(0), eps_p = R(0);
  if constexpr (POS) {
#pragma unroll
    for (int v = 0; v < 8; ++v) Uzp[v] = S.Uz[v][zl];
    pbar = pressure_of(Uzp, gam);
    eps_r = fmin(R(1e-13), Uzp[0]);
    eps_p = fmin(R(1e-13), pbar);
    R th_r = R(1), th_p = R(1);
    pos_rho(u0, Uzp, eps_r, th_r);
    if (valid && th_r < R(1)) smem_min_nonneg(&S.th[zl][0], th_r);
    if constexpr (WARP) __syncwarp(); else __syncthreads();
    th_r = S.th[zl][0];
    pos_p(u0, Uzp, th_r, gam, pbar, eps_p, th_p);
    if (valid && th_p < R(1)) smem_min_nonneg(&S.th[zl][1], th_p);
    if constexpr (WARP) __syncwarp(); else __syncthreads();
    const R th = th_r * S.th[zl][1];
    if (th < R(1)) {
#pragma unroll
      for (int v = 0; v < 8; ++v) u0[v] = Uzp[v] + th * (u0[v] - Uzp[v]);
    }
  }
  // ---- metric terms of the node, kept for all flux evaluations, and its places in
  // the ring buffers: where F^alpha goes and where dF^alpha comes from
  R iJ, g[3], Sa[9];
  team_node_metrics<P, R>(BT, c, i, valid, iJ, g, Sa);
  int fin[3], fout[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const int qk = K.rpos[a * N + i], qq = qk & 3, kk = qk >> 2;
    fin[a] = a * L::FS + L::in_pos(qq, kk);
    fout[a] = a * L::FS + L::out_pos(qq, kk);
  }
  auto barrier = [&]() {
    if constexpr (WARP) __syncwarp();
    else __syncthreads();
  };
  // one flux difference of every node: dF_i = sum_alpha D^alpha F^alpha - F(U_i) . g_i,
  // in place (the level is not needed any more: the update starts from level 1)
  auto flux_difference = [&](const R* u, R* dF) {
    R Gf[8];
    if constexpr (P == 2) {
      // trilinear element: dF^alpha is the difference along the node's edge, whose
      // other end is the node with bit alpha flipped, 8 consecutive lanes to a zone
      const Prim<R> w = to_prim(u, gam);
      flux_n(u, w, g[0], g[1], g[2], Gf);
#pragma unroll
      for (int v = 0; v < 8; ++v) Gf[v] = -Gf[v];
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        R Fa[8];
        flux_n(u, w, Sa[3 * a], Sa[3 * a + 1], Sa[3 * a + 2], Fa);
        const bool up = (i >> a) & 1;
#pragma unroll
        for (int v = 0; v < 8; ++v) {
          const R o = __shfl_xor_sync(0xffffffffu, Fa[v], 1 << a);
          Gf[v] += (up ? Fa[v] : o) - (up ? o : Fa[v]);  // operands picked, one subtraction
        }
      }
#pragma unroll
      for (int v = 0; v < 8; ++v) dF[v] = Gf[v];
      return;
    }
    {
      const Prim<R> w = to_prim(u, gam);
      flux_n(u, w, g[0], g[1], g[2], Gf);
      {
#pragma unroll
        for (int a = 0; a < 3; ++a) {
          R Fa[8];
          flux_n(u, w, Sa[3 * a], Sa[3 * a + 1], Sa[3 * a + 2], Fa);
#pragma unroll
          for (int v = 0; v < 8; ++v) Fz[fin[a] + v * L::RS] = Fa[v];
        }
      }
    }
    barrier();
    for (int t = warp; t < ZB; t += NW) ring_contract<P, R>(S.F + t * L::FZ, lane);
    barrier();
    {
#pragma unroll
      for (int v = 0; v < 8; ++v) dF[v] = -Gf[v];
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        R x[8];
        if constexpr (sizeof(R) == 4) {
          ld16(Fz + fout[a], x);
          ld16(Fz + (fout[a] ^ 4), x + 4);  // the other half of the shuffled chunk pair
        } else {
          ld8(Fz + fout[a], x);
        }
#pragma unroll
        for (int v = 0; v < 8; ++v) dF[v] += x[v];
      }
    }
    barrier();
  };
  // ---- Picard iterations (Eqs. C.34-C.36) on the conserved state itself (levels / J):
  // U_k = (U_1 - r_k1 dF_1) - sum_{m>1} r_km dF_m with r = dt l_0/(l_k J) R; in the
  // first iteration every level equals level 1, so its flux difference serves all
  const R fs = S.fs[zl] * iJ;
  R base[ML][8], Um[ML][8];
  const R j0 = valid ? BT.J0[static_cast<size_t>(c) * N + i] : R(1);
  auto keep = [&](int it) {
    if constexpr (STORE) {
      if (valid) {
#pragma unroll
        for (int k = 0; k < ML; ++k)
#pragma unroll
          for (int v = 0; v < 8; ++v)
            itS[((static_cast<size_t>(it * ML + k) * 8 + v) * N + i) * Z + z] = j0 * Um[k][v];
      }
    }
  };
  {
    R d0[8];
#pragma unroll
    for (int v = 0; v < 8; ++v) d0[v] = R(0);
    flux_difference(u0, d0);
#pragma unroll
    for (int k = 0; k < ML; ++k) {
      const R r0 = fs * K.R_[(k + 1) * M], rs = fs * K.Rs[k];
#pragma unroll
      for (int v = 0; v < 8; ++v) {
        base[k][v] = u0[v] - r0 * d0[v];
        Um[k][v] = base[k][v] - rs * d0[v];
      }
    }
  }
  keep(0);
#pragma unroll 1
  for (int it = 1; it < P; ++it) {
#pragma unroll
    for (int m = 0; m < ML; ++m) flux_difference(Um[m], Um[m]);
    R rk[ML][ML];
#pragma unroll
    for (int k = 0; k < ML; ++k)
#pragma unroll
      for (int m = 0; m < ML; ++m) rk[k][m] = fs * K.R_[(k + 1) * M + m + 1];
#pragma unroll
    for (int v = 0; v < 8; ++v) {
      R d[ML];
#pragma unroll
      for (int m = 0; m < ML; ++m) d[m] = Um[m][v];
#pragma unroll
      for (int k = 0; k < ML; ++k) {
        R s = base[k][v];
#pragma unroll
        for (int m = 0; m < ML; ++m) s -= rk[k][m] * d[m];
        Um[k][v] = s;
      }
    }
    if (it < P - 1) keep(it);
  }
  // ---- final levels J U in ring order around the radial axis
  {
#pragma unroll
    for (int m = 0; m < ML; ++m)
#pragma unroll
      for (int v = 0; v < 8; ++v) S.F[zl * L::FL + m * L::FS + (fin[2] - 2 * L::FS) + v * L::RS] = j0 * Um[m][v];
  }
  __syncthreads();
  // ---- point values: task (group of 4 zones, q) per warp, lane = zone * 8 + variable
  const int v = lane & 7;
  // (8 Z fits 32 bits: the traces of 2^29 zones exceed any GPU's memory)
  const unsigned Z8 = static_cast<unsigned>(Z) * 8u;
  const size_t ZF = static_cast<size_t>(Z8) * NQT, ZE = static_cast<size_t>(Z8) * (12 * Dm::NS);
  auto task = [&](int t, auto&& emit) {
    const int q = t & 3, zt = (t >> 2) * 4 + (lane >> 3);
    int ct, kt;
    column(zt, ct, kt);
    const bool in = zbase + zt < Z;
    if (!in) ct = c0;
    const size_t at = static_cast<size_t>(zbase + (t >> 2) * 4) * 8 + (P == 4 ? lane : 0);
    const int off = P == 4 ? 0 : lane;  // the task's 4 x 8 values, one per lane
    const R* iJF = BT.iJF + static_cast<size_t>(ct) * NQT;
    const R* iJE = BT.iJE + static_cast<size_t>(ct) * 12 * Dm::NS;
    // (1/J through the read-only path: the compiler may then keep it across the stores)
    auto put = [&](const R* iJ, R* out, size_t step, int idx, int m0, const auto& s, bool mine) {
      const R w = __ldg(iJ + idx);
      R* o = out + at + static_cast<size_t>(static_cast<unsigned>(idx)) * Z8;
#pragma unroll
      for (int m = 0; m < static_cast<int>(sizeof(s) / sizeof(R)); ++m)
        emit(in && mine, s[m] * w, o + (m0 + m) * step + off);
    };
    const R* row = S.F + zt * L::FL + v * L::RS;
    ring_points<P, ML, POS>(
        row, q, K,
        [&](int idx, int m0, const auto& s, bool mine) { put(iJF, trF, ZF, idx, m0, s, mine); },
        [&](int idx, int m0, const auto& s, bool mine) { put(iJE, trE, ZE, idx, m0, s, mine); });
  };
  static_assert(ZB % 4 == 0, "zones in fours");
  if constexpr (!POS) {
    for (int t = warp; t < ZB; t += NW)
      task(t, [&](bool in, R x, R* out) {
        if (in) *out = x;
      });
  } else {
    // the positivity scaling of the point states about the zone mean: pass 0 writes the
    // unscaled values and takes the factors theta_rho and (for theta_rho = 1) theta_p
    // over the zone's points; pass 1, for zones with theta_rho < 1, takes theta_p again;
    // pass 2, for zones with theta < 1, rewrites the values scaled.  The eight variables
    // of a point sit in eight lanes, so the states go through a tile of shared memory
    // (SLOTS points x 4 zones) and each lane checks one whole state.
#pragma unroll 1
    for (int pass = 0; pass < 3; ++pass) {
      if (pass > 0) {
        bool redo = false;
        if (tid < ZB && zbase + tid < Z) {
          if (pass == 1) redo = S.th[tid][2] < R(1);
          else redo = S.th[tid][2] * (S.th[tid][2] < R(1) ? S.th[tid][3] : S.th[tid][4]) < R(1);
        }
        if (!__syncthreads_or(redo)) continue;
      }
#pragma unroll 1
      for (int t = warp; t < ZB; t += NW) {
        const int zt = (t >> 2) * 4 + (lane >> 3);
        const R um = S.Uz[v][zt], th_r = S.th[zt][2];
        const R th = pass < 2 ? R(1) : th_r * (th_r < R(1) ? S.th[zt][3] : S.th[zt][4]);
        R* my = tile.s[warp];
        constexpr int TS = RingTile<P, R, POS>::STRIDE, SLOTS = RingTile<P, R, POS>::SLOTS;
        const bool inside = zbase + zt < Z;  // a whole octet of lanes
        if (pass < 2) {
          int held = 0;  // point states of each zone in the tile
          task(t, [&](bool in, R x, R* out) {
            my[held * TS + lane] = x;
            if (++held == SLOTS) {
              ring_check<P, R>(my, S, inside ? held : 0, zt, lane, gam, pass);
              held = 0;
            }
            if (in && pass == 0) *out = x;
          });
          ring_check<P, R>(my, S, inside ? held : 0, zt, lane, gam, pass);
        } else {
          task(t, [&](bool in, R x, R* out) {
            if (in && th < R(1)) *out = um + th * (x - um);
          });
        }
      }
      __syncthreads();
    }
  }
}
