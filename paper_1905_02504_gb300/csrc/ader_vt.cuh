// The derivative contraction as sparse rows on the compiled nonzero pattern of
// D^alpha: thread (zone, v, row group g) forms dF_{v,i} = sum_alpha sum_j D^alpha_ij
// F^alpha_{v,j} for the rows i of group g, with the F values in registers and the D
// values as constant-bank operands (Eqs. C.34-C.36).  geo_probe_contraction times it
// against the tensor-core form; the predictor uses the element's ring structure
// instead (ader_ring.cuh), with less than half the operations.
// Included by kernels.cu inside its anonymous namespace.

template <int V> using IC = std::integral_constant<int, V>;

template <int P, typename R>
struct VtLayout {
  using Dm = Dim<P>;
  static constexpr int ZB = Team<P>::ZB, N = Dm::N, CH = Chunk<R>::CH;
  // node stride of one [alpha][v] row (a multiple of the 16-byte chunk), with
  // P = 4 padded so the two variables of an 8-lane FP32 access phase sit in
  // different bank groups
  static constexpr int NP = (P == 4) ? 36 : ((N + 3) / 4) * 4;
  // zone strides padded so that the zones of one warp-wide scalar access fall
  // into distinct banks: (words per zone) = 32 / ZB modulo 32, at least 4
  static constexpr int WPE = sizeof(R) / 4;
  static constexpr int TGT = ((32 / ZB) > 4 ? (32 / ZB) : 4) / WPE;
  static constexpr int MODE = 32 / WPE;
  __host__ __device__ static constexpr int pad(int x) { return x + ((TGT - x % MODE) % MODE + MODE) % MODE; }
  static constexpr int XZ = pad(24 * NP);  // F rows / final levels per zone
  static constexpr int OZ = pad(8 * N);    // flux differences per zone
  static constexpr int G = RefPattern<P>::G;
  static constexpr int NVT = 8 * ZB * G;   // threads of the variable phase
};

// the 16-byte chunk C of F^alpha's row is used by some entry of row group G
template <int P, int A, int G, int C, int CH>
__host__ __device__ constexpr bool vt_needs_chunk() {
  using RP = RefPattern<P>;
  for (int e = RP::EG[A][G]; e < RP::EG[A][G + 1]; ++e)
    if (RP::J[A * RP::NNZ + e] / CH == C) return true;
  return false;
}

template <int P, typename R, int A, int G, int... Cs>
__device__ __forceinline__ void vt_load_row(const R* row, R* Fr, std::integer_sequence<int, Cs...>) {
  constexpr int CH = Chunk<R>::CH;
  auto one = [&](auto c) {
    if constexpr (vt_needs_chunk<P, A, G, decltype(c)::value, CH>()) ld16(row + decltype(c)::value * CH,
                                                                          Fr + decltype(c)::value * CH);
  };
  (one(IC<Cs>{}), ...);
}

// acc[i - RG[G]] += D^A_ij F_j over the entries of row group G
template <int P, typename R, int A, int G, int... Es>
__device__ __forceinline__ void vt_rows(R* acc, const R* Fr, const RefConst<P, R>& K,
                                        std::integer_sequence<int, Es...>) {
  using RP = RefPattern<P>;
  constexpr int E0 = A * RP::NNZ + RP::EG[A][G], R0 = RP::RG[G];
  ((acc[IC<RP::I[E0 + Es] - R0>::value] += K.Dpat[E0 + Es] * Fr[IC<RP::J[E0 + Es]>::value]), ...);
}

template <int P, typename R, int G, int A>
__device__ __forceinline__ void vt_direction(R* acc, const R* rowA, const RefConst<P, R>& K) {
  using RP = RefPattern<P>;
  constexpr int N = Dim<P>::N, CH = Chunk<R>::CH;
  R Fr[((N + CH - 1) / CH) * CH];
  vt_load_row<P, R, A, G>(rowA, Fr, std::make_integer_sequence<int, (N + CH - 1) / CH>{});
  vt_rows<P, R, A, G>(acc, Fr, K, std::make_integer_sequence<int, RP::EG[A][G + 1] - RP::EG[A][G]>{});
}

// variable phase of one flux evaluation for row group G: reads the F rows of
// variable v of zone zl, writes dF_{v,i} for the group's rows
template <int P, typename R, int G>
__device__ __forceinline__ void vt_contract(const R* XFz, R* XOz, int v, const RefConst<P, R>& K) {
  using RP = RefPattern<P>;
  using L = VtLayout<P, R>;
  constexpr int NRG = RP::RG[G + 1] - RP::RG[G];
  R acc[NRG];
#pragma unroll
  for (int r = 0; r < NRG; ++r) acc[r] = R(0);
  vt_direction<P, R, G, 0>(acc, XFz + (0 * 8 + v) * L::NP, K);
  vt_direction<P, R, G, 1>(acc, XFz + (1 * 8 + v) * L::NP, K);
  vt_direction<P, R, G, 2>(acc, XFz + (2 * 8 + v) * L::NP, K);
#pragma unroll
  for (int r = 0; r < NRG; ++r) XOz[v * Dim<P>::N + RP::RG[G] + r] = acc[r];
}

template <int P, typename R, int G = 0>
__device__ __forceinline__ void vt_contract_dispatch(int g, const R* XFz, R* XOz, int v, const RefConst<P, R>& K) {
  if constexpr (G < RefPattern<P>::G) {
    if (g == G) vt_contract<P, R, G>(XFz, XOz, v, K);
    else vt_contract_dispatch<P, R, G + 1>(g, XFz, XOz, v, K);
  }
}

// One out-of-line copy of the fully unrolled code of all groups.
template <int P, typename R>
__device__ __noinline__ void vt_contract_group(int g, const R* XFz, R* XOz, int v) {
  vt_contract_dispatch<P, R>(g, XFz, XOz, v, RC<P, R>::get());
}
