// Imaginary half of the split complex-step JVP (see dfr_split.cu): device
// bodies shared by the single-grid kernels (dfr_split.cu) and the batched
// ensemble kernels (ensemble.cu).
#pragma once

#include <cuda_runtime.h>

#include "check.cuh"
#include "convert.cuh"
#include "dfr_device.cuh"
#include "fixed.cuh"
#include "swepi_internal.h"

namespace swepi {

// ---------------------------------------------------------------- tangent
// The imaginary half in arithmetic type T: double (the FP64 path) or float
// (the complex64-bulk form: tables rounded from the FP64 linearisation, FP32
// accumulation).  Krylov vectors in and out stay FP64; the orthogonalisation
// dots of the epilogue are FP64 in both.
//
template <typename T, int NS>
__device__ __forceinline__ void trace_tan(const double* __restrict__ v, const float* __restrict__ v32, long long nodes,
                                          int elem, int edge, int i, const DfrConst& dc, T out[3]) {
  if constexpr (sizeof(T) == 8) {
    trace_fx<NS>(v, nodes, elem, edge, i, dc, out);
  } else {
    const long long base = (long long)elem * NS * NS;
    const float* w32 = (edge == 0 || edge == 2) ? dc.lm32 : dc.lp32;
#pragma unroll
    for (int var = 0; var < 3; ++var) {
      T acc = T(0);
#pragma unroll
      for (int k = 0; k < NS; ++k) {
        const long long idx = base + ((edge <= 1) ? (i * NS + k) : (k * NS + i)) + var * nodes;
        const float x = v32 ? __ldg(v32 + idx) : f64_to_f32_bits(__ldg(v + idx));
        acc = fmaf(w32[k], x, acc);
      }
      out[var] = acc;
    }
  }
}

template <typename T>
struct TanFaceArgs {
  const double* v;
  const float* v32;   // FP32 copy of v (complex64-bulk form), or null
  long long nodes;
  const FaceLine* lines;
  const double* fc;
  const T* lf;
  long long nfacepts;
  T* fb;
  const int* skip;
};

// imaginary half at interface point t of one grid
template <typename T, int NS>
__device__ __forceinline__ void face_tangent_body(const TanFaceArgs<T>& a, const DfrConst& dc, long long t) {
  if (t >= a.nfacepts) return;
  const int line = (int)(t / NS), i = (int)(t % NS);
  const FaceLine L = a.lines[line];
  if (!face_line_ok<NS>(L, a.nodes)) return;
  const int in = L.reversed ? NS - 1 - i : i;
  T vo[3], vn[3];
  trace_tan<T, NS>(a.v, a.v32, a.nodes, L.owner, L.owner_edge, i, dc, vo);
  trace_tan<T, NS>(a.v, a.v32, a.nodes, L.nbr, L.nbr_edge, in, dc, vn);
  const long long P = a.nfacepts;
  const T* lf = a.lf + t;
  T f[3];
#pragma unroll
  for (int mu = 0; mu < 3; ++mu) {
    T s = lf[(mu * 3) * P] * vo[0];
    s = fma(lf[(mu * 3 + 1) * P], vo[1], s);
    s = fma(lf[(mu * 3 + 2) * P], vo[2], s);
    s = fma(lf[(9 + mu * 3) * P], vn[0], s);
    s = fma(lf[(9 + mu * 3 + 1) * P], vn[1], s);
    s = fma(lf[(9 + mu * 3 + 2) * P], vn[2], s);
    f[mu] = s;
  }
  T* fo = a.fb + ((long long)L.owner * 4 + L.owner_edge) * 3 * NS + i;
  fo[0] = f[0];
  fo[NS] = f[1];
  fo[2 * NS] = f[2];
  // across panels the neighbour's components (App. C); within a panel the
  // transform is the identity and its five coefficients are not read
  if (L.handback) {
    T sig, M00, M01, M10, M11;
    if constexpr (sizeof(T) == 4) {   // FP32 copies of the hand-back coefficients after the 18 map rows
      M00 = lf[18 * P];
      M01 = lf[19 * P];
      M10 = lf[20 * P];
      M11 = lf[21 * P];
      sig = lf[22 * P];
    } else {
      const double* fc = a.fc + t;
      sig = fc[FC_SIG * P];
      M00 = fc[FC_M00 * P];
      M01 = fc[FC_M01 * P];
      M10 = fc[FC_M10 * P];
      M11 = fc[FC_M11 * P];
    }
    const T g1 = M00 * f[1] + M01 * f[2], g2 = M10 * f[1] + M11 * f[2];
    f[0] = sig * f[0];
    f[1] = g1;
    f[2] = g2;
  }
  T* fn = a.fb + ((long long)L.nbr * 4 + L.nbr_edge) * 3 * NS + in;
  fn[0] = f[0];
  fn[NS] = f[1];
  fn[2 * NS] = f[2];
}

template <typename T>
struct TanVolArgs {
  const double* v;
  long long nodes;
  long long nelem;
  const T* ln;
  const int4* le;   // FP64: exponents of the packed coefficients per element
  const T* fb;
  double* out;
  AugEpilogue ep;
};

// shared memory of one element tile
template <typename T, int NS, int EPB>
struct VolSmem {
  T sF[EPB][2][3][NS * NS];   // fluxes along xi^1 and xi^2
  T sB[EPB][4][3][NS];        // interface fluxes of the four edges
  T sD[NS][NS + 3];           // derivative matrix, padded rows: distinct banks per k
  // FP64: largest magnitude keys of the elements' fluxes (mass, momentum), by tile parity
  unsigned sE[sizeof(T) == 8 ? 2 : 1][sizeof(T) == 8 ? EPB : 1][2];
};

// derivative matrix into shared memory: in FP32 pre-multiplied by -(2/dx) *
// scale (Eq. 14 and the augmented operator's dt), so that each output is one
// chain of fused multiply-adds started from scale * source; in FP64 the packed
// integer matrix of the block fixed-point sweeps
template <typename T, int NS, int EPB, int BLOCK>
__device__ __forceinline__ void tile_dmat(const TanVolArgs<T>& a, const DfrConst& dc, VolSmem<T, NS, EPB>& sm) {
  const double dscale = -dc.two_over_dx * a.ep.scale;
  for (int t = threadIdx.x; t < NS * (NS + 2); t += BLOCK) {
    if constexpr (sizeof(T) == 4) sm.sD[t / (NS + 2)][t % (NS + 2)] = f64_to_f32_bits(dscale * dc.D[t / (NS + 2)][t % (NS + 2)]);
    else sm.sD[t / (NS + 2)][t % (NS + 2)] = dc.Dq[t / (NS + 2)][t % (NS + 2)];
  }
}

// ---- FP32 (complex64-bulk form)
// interface fluxes of the four edges of the elements eb .. eb + EPB - 1 (those
// below e_end) into shared memory
template <int NS, int EPB, int BLOCK>
__device__ __forceinline__ void tile_edges(const TanVolArgs<float>& a, VolSmem<float, NS, EPB>& sm, long long eb,
                                           long long e_end) {
  for (int t = threadIdx.x; t < EPB * 12 * NS; t += BLOCK) {
    const int e = t / (12 * NS), r = t % (12 * NS);
    const long long ge = eb + e;
    (&sm.sB[e][0][0][0])[r] = (ge < e_end) ? a.fb[ge * 12 * NS + r] : 0.f;
  }
}

// pointwise imaginary fluxes of node idx (element le of the tile, node
// `node`) into shared memory; the sources S^1, S^2 returned
template <int NS, int EPB>
__device__ __forceinline__ void tile_fluxes(const TanVolArgs<float>& a, VolSmem<float, NS, EPB>& sm, int le, int node,
                                            long long idx, float& S1, float& S2) {
  const long long N = a.nodes;
  const float v0 = f64_to_f32_bits(__ldg(a.v + idx)), v1 = f64_to_f32_bits(__ldg(a.v + idx + N));
  const float v2 = f64_to_f32_bits(__ldg(a.v + idx + 2 * N));
  const float* ln = a.ln + idx;
  const float u1 = ln[LN_U1 * N], u2 = ln[LN_U2 * N];
  const float F11 = fmaf(2.f * u1, v1, ln[LN_A11 * N] * v0);
  const float F12 = fmaf(u2, v1, fmaf(u1, v2, ln[LN_A12 * N] * v0));
  const float F22 = fmaf(2.f * u2, v2, ln[LN_A22 * N] * v0);
  S1 = fmaf(ln[LN_S11 * N], v1, fmaf(ln[LN_S12 * N], v2, ln[LN_S10 * N] * v0));
  S2 = fmaf(ln[LN_S21 * N], v1, fmaf(ln[LN_S22 * N], v2, ln[LN_S20 * N] * v0));
  sm.sF[le][0][0][node] = v1;
  sm.sF[le][0][1][node] = F11;
  sm.sF[le][0][2][node] = F12;
  sm.sF[le][1][0][node] = v2;
  sm.sF[le][1][1][node] = F12;
  sm.sF[le][1][2][node] = F22;
}

// ---- FP64: the DFR sweeps in block fixed point (fixed.cuh)
// The 6 (N_s + 2) multiply-adds per node of the two sweeps are over half of
// the kernel's FP64 operations, and the kernel is bound by the FP64 pipe.  Every line
// of an element shares a scale, so the element's fluxes (mass and momentum
// apart: their units differ) are packed once, seven conversions a node, and
// the sweeps run as integer multiply-adds.  An element that the format cannot
// hold keeps FP64 values in the same arrays and takes the FP64 chain.
// 6 x 60 x 60, p = 5, with the augmented operator and the window dots: 134 ->
// 85 us (FP64 pipe 87 -> 66 %); the product alone 129 -> 79 us with its face
// kernel, 6 x 90 x 90, p = 6: 395 -> 217 us.  Relative error against a 64-bit
// reference unchanged (3.5e-15, the reference's own).

// what one node brings to its element: its fluxes, and its share of the
// element's 12 N_s interface fluxes
template <int NS>
struct FxPoint {
  static constexpr int EC = (12 + NS - 1) / NS;   // interface values per thread
  double v1, v2, F11, F12, F22;
  double e[EC];
};

// m0, m1: largest magnitude keys of the mass and the momentum fluxes
template <int NS>
__device__ __forceinline__ void fx_edges(const double* __restrict__ fb, long long elem, int node, FxPoint<NS>& pt,
                                         unsigned& m0, unsigned& m1) {
  constexpr int NN = NS * NS;
#pragma unroll
  for (int i = 0; i < FxPoint<NS>::EC; ++i) {
    const int r = node + i * NN;
    pt.e[i] = 0.0;
    if (r < 12 * NS) {
      pt.e[i] = fb[elem * 12 * NS + r];
      const unsigned m = fx_key(pt.e[i]);
      if ((r / NS) % 3 == 0) m0 = max(m0, m);
      else m1 = max(m1, m);
    }
  }
  m0 = max(m0, max(fx_key(pt.v1), fx_key(pt.v2)));
  m1 = max(m1, max(fx_key(pt.F11), max(fx_key(pt.F12), fx_key(pt.F22))));
}

// the node's values into the tile's arrays sF [2][3][NN], sB [12 NS] of its
// element: packed where the element's keys M0, M1 allow (fixed), else as they are
template <int NS>
__device__ __forceinline__ void fx_store(double (*sF)[3][NS * NS], double* sB, int node, const FxPoint<NS>& pt,
                                         bool fixed, unsigned M0, unsigned M1) {
  constexpr int NN = NS * NS;
  const int E0 = fx_exp(M0), E1 = fx_exp(M1);
  double v1 = pt.v1, v2 = pt.v2, F11 = pt.F11, F12 = pt.F12, F22 = pt.F22;
  if (fixed) {
    v1 = fx_pack(v1, E0);
    v2 = fx_pack(v2, E0);
    F11 = fx_pack(F11, E1);
    F12 = fx_pack(F12, E1);
    F22 = fx_pack(F22, E1);
  }
  sF[0][0][node] = v1;
  sF[0][1][node] = F11;
  sF[0][2][node] = F12;
  sF[1][0][node] = v2;
  sF[1][1][node] = F12;
  sF[1][2][node] = F22;
#pragma unroll
  for (int i = 0; i < FxPoint<NS>::EC; ++i) {
    const int r = node + i * NN;
    if (r < 12 * NS) sB[r] = fixed ? fx_pack(pt.e[i], (r / NS) % 3 == 0 ? E0 : E1) : pt.e[i];
  }
}

// a scale the packed sweeps can be multiplied by through its exponent field
__device__ __forceinline__ bool fx_scale_usable(double s) {
  const int e = (__double2hiint(s) >> 20) & 0x7ff;
  return e >= 823 && e <= 1223;
}

// the two sweeps of node (k2, k1): res[mu] = dscale * (D-row k1 along xi^1 +
// D-row k2 along xi^2 + isrc[mu]) + add[mu] for mu = 1, 2 (isrc in units of the
// packed sums, where `fixed`).  E0, E1: the block exponents.  ADD:
// whether add1, add2 are added where `fixed`.  Da, Db: the packed rows in
// shared memory (each entry read once for the three variables: rows held in
// registers spilled); sB [4][3][NS].  The packed sum is converted once (one
// FP64 instruction) and scaled by dscale with the blocks' exponents added to
// its exponent field.
template <int NS, bool ADD>
__device__ __forceinline__ void fx_sweep(const double (*sF)[3][NS * NS], const double* sB, int k1, int k2,
                                         const double* Da, const double* Db, const DfrConst& dc,
                                         double dscale, bool fixed, int E0, int E1, long long isrc1, long long isrc2,
                                         double add1, double add2, double res[3]) {
  if (fixed) {
    FxAcc a[3];
#pragma unroll
    for (int l = 0; l < NS + 2; ++l) {
      const double m = Da[l];
#pragma unroll
      for (int mu = 0; mu < 3; ++mu)
        fx_mac(a[mu], l == 0 ? sB[mu * NS + k2] : (l == NS + 1 ? sB[(3 + mu) * NS + k2] : sF[0][mu][k2 * NS + l - 1]), m);
    }
#pragma unroll
    for (int l = 0; l < NS + 2; ++l) {
      const double m = Db[l];
#pragma unroll
      for (int mu = 0; mu < 3; ++mu)
        fx_mac(a[mu], l == 0 ? sB[(6 + mu) * NS + k1] : (l == NS + 1 ? sB[(9 + mu) * NS + k1] : sF[1][mu][(l - 1) * NS + k1]), m);
    }
    const int sh = __double2hiint(dscale), sl = __double2loint(dscale);
#pragma unroll
    for (int mu = 0; mu < 3; ++mu) {
      const int k = (mu == 0 ? E0 : E1) + dc.dq_exp;
      const double sc = __hiloint2double(sh + k * 1048576, sl);
      if (mu == 1) a[mu].hh += isrc1;
      if (mu == 2) a[mu].hh += isrc2;
      const double s = fx_sum(a[mu]);
      if constexpr (ADD) res[mu] = mu == 0 ? s * sc : fma(s, sc, mu == 1 ? add1 : add2);
      else res[mu] = s * sc;
    }
    return;
  }
#pragma unroll 1
  for (int mu = 0; mu < 3; ++mu) {
    double c = mu == 0 ? 0.0 : (mu == 1 ? add1 : add2);
    c = fma(dscale * dc.D[k1][0], sB[(0 * 3 + mu) * NS + k2], c);
    c = fma(dscale * dc.D[k1][NS + 1], sB[(1 * 3 + mu) * NS + k2], c);
#pragma unroll 1
    for (int l = 0; l < NS; ++l) c = fma(dscale * dc.D[k1][l + 1], sF[0][mu][k2 * NS + l], c);
    c = fma(dscale * dc.D[k2][0], sB[(2 * 3 + mu) * NS + k1], c);
    c = fma(dscale * dc.D[k2][NS + 1], sB[(3 * 3 + mu) * NS + k1], c);
#pragma unroll 1
    for (int l = 0; l < NS; ++l) c = fma(dscale * dc.D[k2][l + 1], sF[1][mu][l * NS + k1], c);
    if (mu == 0) res[0] = c;
    else if (mu == 1) res[1] = c;
    else res[2] = c;
  }
}

// ---- FP64: the point fluxes in block fixed point too
// Im sqrt(g) T^{ij} and Im S^i are sums of coefficient times v.  The
// coefficients are packed once per linearisation point (lin_node_kernel), with
// exponents per element for four classes: u for u^i, a for the A^{ij}, s for the
// S^i_j and s0 = s + a - u for the S^i_0, so that packing v^1, v^2 for the
// exponent EU = t + 2 - u and v^0 for EA = t + 2 - a puts all terms in one unit and
// the fluxes come out as block values of exponent TF = t - 1020, t the largest of
// a + e(v^0), u + e(v^i) and e(interface flux) + 1020 in the element (e: biased
// exponents; the two spare bits are the sums' headroom).  Both momentum components
// share the exponent: the weaker one's fluxes hold fewer bits, by the ratio of the
// two.  The sources, stored times -dx/2, add to the packed sweep shifted by k = De +
// u - s >= 0.  What is left for the FP64 pipe is the conversion and scaling of three
// sums a node.
// 6 x 60 x 60, p = 5: 90 -> 81 us with the augmented operator and the dots, the
// product with its face kernel 71 -> 67 us; 6 x 90 x 90, p = 6: 217 -> 188 us.
struct LinExp {
  int u, a, k, packed;
};
__device__ __forceinline__ LinExp lin_exp(const int4* __restrict__ le, long long elem) {
  const int4 x = __ldg(le + elem);
  return {x.x, x.y, x.z, x.w};
}
// a value's bid for t: its exponent plus off; zeros (and subnormals) none, and
// one past the format's range a bid past every limit
__device__ __forceinline__ unsigned fx_bid(double x, int off) {
  const int e = (__double2hiint(x) >> 20) & 0x7ff;
  return e == 0 ? 0u : (e > kFxExpMax ? 1u << 14 : (unsigned)(e + off));
}
__device__ __forceinline__ bool fx_bid_usable(unsigned t) {
  return t == 0u || (t >= 1020u + kFxExpMin && t <= 1020u + kFxExpMax);
}

// what one node brings to its element before the exponents are known
template <int NS>
struct TanPoint {
  static constexpr int EC = (12 + NS - 1) / NS;   // interface values per thread
  double v0, v1, v2;
  double e[EC];
};
template <int NS>
__device__ __forceinline__ void tan_load(const TanVolArgs<double>& a, long long elem, int node, long long idx,
                                         const LinExp& x, TanPoint<NS>& pt, unsigned& m0, unsigned& t) {
  constexpr int NN = NS * NS;
  const long long N = a.nodes;
  pt.v0 = __ldg(a.v + idx);
  pt.v1 = __ldg(a.v + idx + N);
  pt.v2 = __ldg(a.v + idx + 2 * N);
#pragma unroll
  for (int i = 0; i < TanPoint<NS>::EC; ++i) {
    const int r = node + i * NN;
    pt.e[i] = 0.0;
    if (r < 12 * NS) {
      pt.e[i] = a.fb[elem * 12 * NS + r];
      if ((r / NS) % 3 == 0) m0 = max(m0, fx_key(pt.e[i]));
      else t = max(t, fx_bid(pt.e[i], 1020));
    }
  }
  m0 = max(m0, max(fx_key(pt.v1), fx_key(pt.v2)));
  t = max(t, max(fx_bid(pt.v0, x.a), max(fx_bid(pt.v1, x.u), fx_bid(pt.v2, x.u))));
}

// the node's fluxes and interface values into the tile's arrays of its element,
// and its sources (times -dx/2): where `fixed` packed, s1 and s2 in units of the
// sweep's sums; else FP64, s1 and s2 holding their bits
template <int NS>
__device__ __forceinline__ void tan_fluxes(const TanVolArgs<double>& a, double (*sF)[3][NS * NS], double* sB, int node,
                                           long long idx, const LinExp& x, const TanPoint<NS>& pt, int De,
                                           bool fixed, unsigned M0, unsigned t, long long& s1, long long& s2) {
  constexpr int NN = NS * NS;
  const long long N = a.nodes;
  const double* ln = a.ln + idx;
  if (fixed) {
    const int E0 = fx_exp(M0), TF = t == 0u ? 1023 : (int)t - 1020;
    const double p0 = fx_pack(pt.v0, TF + 1022 - x.a);
    const double p1 = fx_pack(pt.v1, TF + 1022 - x.u), p2 = fx_pack(pt.v2, TF + 1022 - x.u);
    sF[0][0][node] = fx_pack(pt.v1, E0);
    sF[1][0][node] = fx_pack(pt.v2, E0);
    const double u1 = ln[LN_U1 * N], u2 = ln[LN_U2 * N];
    FxAcc f;
    fx_mac(f, u1, p1);
    f.hh += f.hh;
    f.mid += f.mid;
    fx_mac(f, ln[LN_A11 * N], p0);
    sF[0][1][node] = fx_repack(fx_int(f));
    f = FxAcc();
    fx_mac(f, u2, p1);
    fx_mac(f, u1, p2);
    fx_mac(f, ln[LN_A12 * N], p0);
    const double f12 = fx_repack(fx_int(f));
    sF[0][2][node] = f12;
    sF[1][1][node] = f12;
    f = FxAcc();
    fx_mac(f, u2, p2);
    f.hh += f.hh;
    f.mid += f.mid;
    fx_mac(f, ln[LN_A22 * N], p0);
    sF[1][2][node] = fx_repack(fx_int(f));
    const int k = min(x.k, 63);
    f = FxAcc();
    fx_mac(f, ln[LN_S11 * N], p1);
    fx_mac(f, ln[LN_S12 * N], p2);
    fx_mac(f, ln[LN_S10 * N], p0);
    s1 = fx_int(f) >> k;
    f = FxAcc();
    fx_mac(f, ln[LN_S21 * N], p1);
    fx_mac(f, ln[LN_S22 * N], p2);
    fx_mac(f, ln[LN_S20 * N], p0);
    s2 = fx_int(f) >> k;
#pragma unroll
    for (int i = 0; i < TanPoint<NS>::EC; ++i) {
      const int r = node + i * NN;
      if (r < 12 * NS) sB[r] = fx_pack(pt.e[i], (r / NS) % 3 == 0 ? E0 : TF);
    }
    return;
  }
  // the element keeps FP64 values: its coefficients unpacked (or, where the
  // linearisation left them so, as they are)
  auto coef = [&](int i, int E) { return x.packed ? fx_unpack(ln[i * N], E) : ln[i * N]; };
  const int es = De + x.u - x.k, es0 = De + x.a - x.k;
  const double u1 = coef(LN_U1, x.u), u2 = coef(LN_U2, x.u);
  const double f12 = fma(u2, pt.v1, fma(u1, pt.v2, coef(LN_A12, x.a) * pt.v0));
  sF[0][0][node] = pt.v1;
  sF[1][0][node] = pt.v2;
  sF[0][1][node] = fma(2.0 * u1, pt.v1, coef(LN_A11, x.a) * pt.v0);
  sF[0][2][node] = f12;
  sF[1][1][node] = f12;
  sF[1][2][node] = fma(2.0 * u2, pt.v2, coef(LN_A22, x.a) * pt.v0);
  s1 = __double_as_longlong(fma(coef(LN_S11, es), pt.v1, fma(coef(LN_S12, es), pt.v2, coef(LN_S10, es0) * pt.v0)));
  s2 = __double_as_longlong(fma(coef(LN_S21, es), pt.v1, fma(coef(LN_S22, es), pt.v2, coef(LN_S20, es0) * pt.v0)));
#pragma unroll
  for (int i = 0; i < TanPoint<NS>::EC; ++i) {
    const int r = node + i * NN;
    if (r < 12 * NS) sB[r] = pt.e[i];
  }
}

// the sweeps of the split product with the element's keys M0, t and sources s1, s2
template <int NS>
__device__ __forceinline__ void tan_sweep(const double (*sF)[3][NS * NS], const double* sB, int k1, int k2,
                                          const double* Da, const double* Db, const DfrConst& dc, double dscale,
                                          bool fixed, unsigned M0, unsigned t, long long s1, long long s2,
                                          double res[3]) {
  const int TF = t == 0u ? 1023 : (int)t - 1020;
  const double add1 = fixed ? 0.0 : dscale * __longlong_as_double(s1);
  const double add2 = fixed ? 0.0 : dscale * __longlong_as_double(s2);
  fx_sweep<NS, false>(sF, sB, k1, k2, Da, Db, dc, dscale, fixed, fx_exp(M0), TF, s1, s2, add1, add2, res);
}

// FP32: the two DFR sweeps of one node (rows Da, Db of the scaled derivative
// matrix) started from sc * source, and the b-column terms nu y_l b_l (coef32: the
// rounded nu y_l)
template <int NS, int EPB>
__device__ __forceinline__ void tile_sweep(const TanVolArgs<float>& a, const VolSmem<float, NS, EPB>& sm, int le, int k1,
                                           int k2, long long idx, const float (&Da)[NS + 2], const float (&Db)[NS + 2],
                                           float sc, float S1, float S2, const float* coef32, double res[3]) {
  const float src[3] = {0.f, S1, S2};
  float acc[3];
#pragma unroll
  for (int mu = 0; mu < 3; ++mu) {
    float c = (mu == 0) ? 0.f : sc * src[mu];
    c = fmaf(Da[0], sm.sB[le][0][mu][k2], c);
    c = fmaf(Da[NS + 1], sm.sB[le][1][mu][k2], c);
#pragma unroll
    for (int l = 0; l < NS; ++l) c = fmaf(Da[l + 1], sm.sF[le][0][mu][k2 * NS + l], c);
    c = fmaf(Db[0], sm.sB[le][2][mu][k1], c);
    c = fmaf(Db[NS + 1], sm.sB[le][3][mu][k1], c);
#pragma unroll
    for (int l = 0; l < NS; ++l) c = fmaf(Db[l + 1], sm.sF[le][1][mu][l * NS + k1], c);
    acc[mu] = c;
  }
  const long long N = a.nodes;
  const int p = a.ep.p < MAX_NB ? a.ep.p : MAX_NB;
#pragma unroll 1
  for (int l = 0; l < p; ++l) {
    const float* bl = a.ep.b32[l];
    if (!bl) continue;
#pragma unroll
    for (int mu = 0; mu < 3; ++mu) acc[mu] = fmaf(coef32[l], __ldg(bl + idx + mu * N), acc[mu]);
  }
#pragma unroll
  for (int mu = 0; mu < 3; ++mu) res[mu] = f32_to_f64_bits(acc[mu]);
}

// the complex64-bulk form's FP32 tail coefficients nu * y_l (once per block)
__device__ __forceinline__ void tile_coef32(const AugEpilogue& ep, float* coef32) {
  if (threadIdx.x < MAX_NB) {
    const int l = threadIdx.x;
    coef32[l] = (l < ep.p && ep.b32[l]) ? f64_to_f32_bits(ep.tail_in[l]) : 0.f;
  }
}

// N_s = 1 in FP64: an element is one node, nothing is shared between threads and
// each sweep has three terms, so packing 17 values a node and passing them through
// shared memory (88 bytes of spills, 47 KB) cost more than the 18 multiply-adds:
// FP64 from registers.  The product at 6 x 16 x 16, p = 0: 10.1 -> 7.8 us (FP64
// through shared memory 8.7); 6 x 64 x 64: 16.8 -> 10.1; from 6 x 128 x 128 (25.1 us)
// on it waits for memory either way (6 x 360 x 360: 153 and 156).
__device__ __forceinline__ void volume_tangent_node(const TanVolArgs<double>& a, const DfrConst& dc, long long elem,
                                                    double dscale, double res[3]) {
  const long long N = a.nodes;
  double e[12];   // interface fluxes [edge][mu], 96 bytes a thread
#pragma unroll
  for (int r = 0; r < 6; ++r) {
    const double2 x = reinterpret_cast<const double2*>(a.fb + elem * 12)[r];
    e[2 * r] = x.x;
    e[2 * r + 1] = x.y;
  }
  const double v0 = __ldg(a.v + elem), v1 = __ldg(a.v + elem + N), v2 = __ldg(a.v + elem + 2 * N);
  const double* ln = a.ln + elem;
  const double u1 = ln[LN_U1 * N], u2 = ln[LN_U2 * N];
  const double f12 = fma(u2, v1, fma(u1, v2, ln[LN_A12 * N] * v0));
  const double f1[3] = {v1, fma(2.0 * u1, v1, ln[LN_A11 * N] * v0), f12};
  const double f2[3] = {v2, f12, fma(2.0 * u2, v2, ln[LN_A22 * N] * v0)};
  const double src[3] = {0.0, fma(ln[LN_S11 * N], v1, fma(ln[LN_S12 * N], v2, ln[LN_S10 * N] * v0)),
                         fma(ln[LN_S21 * N], v1, fma(ln[LN_S22 * N], v2, ln[LN_S20 * N] * v0))};
#pragma unroll
  for (int mu = 0; mu < 3; ++mu) {
    double c = fma(dc.D[0][0], e[mu], src[mu]);
    c = fma(dc.D[0][2], e[3 + mu], c);
    c = fma(dc.D[0][1], f1[mu], c);
    c = fma(dc.D[0][0], e[6 + mu], c);
    c = fma(dc.D[0][2], e[9 + mu], c);
    res[mu] = dscale * fma(dc.D[0][1], f2[mu], c);
  }
}

// The imaginary half of the elements e0 .. e1 - 1 of one grid in tiles of EPB
// elements, by a block of BLOCK >= EPB * NS^2 threads (one per solution point, the
// rest idle), all of which call this function: share blk of nblk of the grid's
// volume work.  The window-dot terms are added up across the tiles and reduced
// once per share (per-tile block sums are FP64 adds on the slow pipe).
template <typename T, int NS, int EPB, int BLOCK, bool W3>
__device__ __forceinline__ void volume_tangent_range(const TanVolArgs<T>& a, const DfrConst& dc,
                                                     VolSmem<T, NS, EPB>& sm, long long e0, long long e1,
                                                     unsigned int blk, unsigned int nblk) {
  constexpr int NN = NS * NS;
  constexpr bool F32 = sizeof(T) == 4;
  constexpr bool NODE = !F32 && NS == 1;
  static_assert(EPB * NN <= BLOCK, "block too small for the element tile");
  if constexpr (!NODE) tile_dmat<T, NS, EPB, BLOCK>(a, dc, sm);
  __shared__ double coef[MAX_NB];
  __shared__ float coef32[MAX_NB];
  if (!F32) epilogue_coefs(a.ep, coef);
  if constexpr (F32) tile_coef32(a.ep, coef32);
  if constexpr (!F32 && !NODE)
    for (int t = threadIdx.x; t < 2 * EPB; t += BLOCK) sm.sE[0][t >> 1][t & 1] = 0u;
  __syncthreads();
  const int le = threadIdx.x / NN, node = threadIdx.x % NN;
  const int k2 = node / NS, k1 = node % NS;
  const bool lane_on = threadIdx.x < EPB * NN;
  double da = 0.0, db = 0.0, dcc = 0.0, dab = 0.0, dbc = 0.0;
  if constexpr (F32) {
    T Da[NS + 2], Db[NS + 2];
#pragma unroll
    for (int n = 0; n < NS + 2; ++n) {
      Da[n] = lane_on ? sm.sD[k1][n] : T(0);
      Db[n] = lane_on ? sm.sD[k2][n] : T(0);
    }
    const float sc = f64_to_f32_bits(a.ep.scale);
    for (long long eb = e0; eb < e1; eb += EPB) {
      const long long elem = eb + le;
      const bool active = lane_on && elem < e1;
      const long long idx = elem * NN + node;
      __syncthreads();   // the previous tile's readers are done with sF and sB
      tile_edges<NS, EPB, BLOCK>(a, sm, eb, e1);
      T S1 = T(0), S2 = T(0);
      if (active) tile_fluxes<NS, EPB>(a, sm, le, node, idx, S1, S2);
      __syncthreads();
      if (active) {
        double res[3];
        tile_sweep<NS, EPB>(a, sm, le, k1, k2, idx, Da, Db, sc, S1, S2, coef32, res);
        epilogue_node<W3, !F32>(a.ep, coef, idx, a.nodes, res, a.out, da, db, dcc, dab, dbc);
      }
    }
  } else if constexpr (NODE) {
    const double dscale = -dc.two_over_dx * a.ep.scale;
    for (long long elem = e0 + threadIdx.x; elem < e1; elem += BLOCK) {
      double res[3];
      volume_tangent_node(a, dc, elem, dscale, res);
      epilogue_node<W3, true>(a.ep, coef, elem, a.nodes, res, a.out, da, db, dcc, dab, dbc);
    }
  } else {
    const double dscale = -dc.two_over_dx * a.ep.scale;
    const bool scale_ok = fx_scale_usable(dscale);
    int par = 0;
    for (long long eb = e0; eb < e1; eb += EPB, par ^= 1) {
      const long long elem = eb + le;
      const bool active = lane_on && elem < e1;
      const long long idx = elem * NN + node;
      TanPoint<NS> pt;
      LinExp x{};
      unsigned m0 = 0u, m1 = 0u;
      if (active) {
        x = lin_exp(a.le, elem);
        tan_load<NS>(a, elem, node, idx, x, pt, m0, m1);
      }
      // this parity's keys were zeroed before the previous tile's last barrier
      fx_block_max<NN, EPB, BLOCK>(sm.sE[par], le, m0, m1);
      __syncthreads();   // the keys are complete; the previous tile's readers are done with sF and sB
      bool fixed = false;
      long long s1 = 0, s2 = 0;
      if (active) {
        m0 = sm.sE[par][le][0];
        m1 = sm.sE[par][le][1];
        fixed = x.packed && scale_ok && fx_usable(m0) && fx_bid_usable(m1);
        tan_fluxes<NS>(a, sm.sF[le], &sm.sB[le][0][0][0], node, idx, x, pt, dc.dq_exp + 1080, fixed, m0, m1, s1, s2);
      }
      for (int t = threadIdx.x; t < 2 * EPB; t += BLOCK) sm.sE[par ^ 1][t >> 1][t & 1] = 0u;
      __syncthreads();
      if (active) {
        double res[3];
        tan_sweep<NS>(sm.sF[le], &sm.sB[le][0][0][0], k1, k2, sm.sD[k1], sm.sD[k2], dc, dscale, fixed, m0, m1, s1, s2,
                      res);
        epilogue_node<W3, !F32>(a.ep, coef, idx, a.nodes, res, a.out, da, db, dcc, dab, dbc);
      }
    }
  }
  __shared__ double sred[(W3 ? 5 : 3) * BLOCK];
  epilogue_finish<BLOCK, W3>(a.ep, da, db, dcc, blk, nblk, dab, dbc, sred);
}

// The same as a persistent grid: CTA b of G takes the elements [E b / G, E (b +
// 1) / G) of E.  The even split keeps the last tiles from running on a few SMs
// alone.
template <typename T, int NS, int EPB, int BLOCK, bool W3>
__device__ __forceinline__ void volume_tangent_persistent(const TanVolArgs<T>& a, const DfrConst& dc,
                                                          VolSmem<T, NS, EPB>& sm) {
  volume_tangent_range<T, NS, EPB, BLOCK, W3>(a, dc, sm, a.nelem * blockIdx.x / gridDim.x,
                                              a.nelem * (blockIdx.x + 1) / gridDim.x, blockIdx.x, gridDim.x);
}

}  // namespace swepi
