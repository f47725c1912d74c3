// Device-side building blocks shared by the DFR kernels: the complex-step
// number type, state loads, the AUSM interface flux (App. D/E) and the trace
// extrapolation (Eq. 7 at the element ends).  See dfr.cu for the arithmetic
// conventions of the complex step.
#pragma once

#include <cuda_runtime.h>

#include "fixed.cuh"
#include "swepi_internal.h"

namespace swepi {

struct cs {
  double re, im;
};
__device__ __forceinline__ cs operator+(cs a, cs b) { return {a.re + b.re, a.im + b.im}; }
__device__ __forceinline__ cs operator-(cs a, cs b) { return {a.re - b.re, a.im - b.im}; }
__device__ __forceinline__ cs operator*(cs a, cs b) { return {a.re * b.re, fma(a.re, b.im, a.im * b.re)}; }
__device__ __forceinline__ cs operator*(double k, cs a) { return {k * a.re, k * a.im}; }
__device__ __forceinline__ cs operator+(cs a, double k) { return {a.re + k, a.im}; }
__device__ __forceinline__ cs cs_rcp(cs a) {
  double r = 1.0 / a.re;
  return {r, -a.im * r * r};
}
__device__ __forceinline__ cs cs_div(cs a, cs b) {
  double r = 1.0 / b.re;
  double qr = a.re * r;
  return {qr, (a.im - qr * b.im) * r};
}
__device__ __forceinline__ cs cs_sqrt(cs a) {
  double s = sqrt(a.re);
  return {s, a.im * (0.5 / s)};
}
__device__ __forceinline__ double re(cs a) { return a.re; }
__device__ __forceinline__ double im(cs a) { return a.im; }
__device__ __forceinline__ cs mk(double r, double i, cs*) { return {r, i}; }

// real instantiation (the RHS): same code path on plain doubles
__device__ __forceinline__ double cs_rcp(double a) { return 1.0 / a; }
__device__ __forceinline__ double cs_div(double a, double b) { return a / b; }
__device__ __forceinline__ double cs_sqrt(double a) { return sqrt(a); }
__device__ __forceinline__ double re(double a) { return a; }
__device__ __forceinline__ double im(double) { return 0.0; }
__device__ __forceinline__ double mk(double r, double, double*) { return r; }

// the part of a result the caller wants: the imaginary part for the JVP, the
// value for the RHS
__device__ __forceinline__ double part(cs a) { return a.im; }
__device__ __forceinline__ double part(double a) { return a; }

template <typename T>
__device__ __forceinline__ T load_state(const double* __restrict__ q, const double* __restrict__ v, double eps,
                                        long long i) {
  return mk(__ldg(q + i), v ? eps * __ldg(v + i) : 0.0, (T*)nullptr);
}

// ---------------------------------------------------------------- AUSM
// FP64 divisions and square roots are sequences of many FP64 instructions, so
// each side takes a single reciprocal square root: with rs = 1 / sqrt(c q^0), c =
// g_r h^dd / sqrt g, a^d = sqrt(c q^0) = c q^0 rs (corrected to the last bit by
// one residual), 1 / a^d = rs and 1 / q^0 = c rs^2 (some units in the last place off,
// where a division is correctly rounded; the results' distance from a 64-bit
// reference did not change).
struct SpeedRoot {
  double a, ia, r;   // a^d, 1 / a^d, 1 / q^0
};
__device__ __forceinline__ SpeedRoot speed_root(double q0, double c) {
  const double x = c * q0, rs = rsqrt(x);
  const double s = x * rs;
  return {fma(0.5 * rs, fma(-s, s, x), s), rs, c * rs * rs};
}
// a^d = sqrt(h^dd g_r H) (App. E) and the Froude number M = u^d / a^d.  q^d (r ia) and
// (q^d r) ia are equally accurate; which last bits they give decides accept/reject
// choices of the window-2 phi solver at long steps (6 x 60 x 60, dt = 1800 s), and the
// other one's choices led the benchmark's first start into a blown-up substep.
__device__ __forceinline__ void speed_mach(double q0, double qd, double c, double& a, double& M) {
  const SpeedRoot z = speed_root(q0, c);
  a = z.a;
  M = qd * (z.r * z.ia);
}
__device__ __forceinline__ void speed_mach(cs q0, cs qd, double c, cs& a, cs& M) {
  const SpeedRoot z = speed_root(q0.re, c);
  a = {z.a, (0.5 * c) * q0.im * z.ia};
  const double u = qd.re * z.r, ui = (qd.im - u * q0.im) * z.r;
  const double m = u * z.ia;
  M = {m, (ui - m * a.im) * z.ia};
}

// AUSM interface flux, basic splittings (reading of App. D Eq. 138-139; [41]
// Eq. 6 and 8): flux^mu = M_{1/2} a q^mu (upwind side) + beta+ P_L + beta- P_R
// with P^{mu d} = g_r h^{mu d} (q^0)^2 / (2 sqrt g), zero for mu = 0
template <typename T>
__device__ __forceinline__ void ausm_flux(const T qL[3], const T qR[3], int d, double ad, double p1, double p2,
                                          T flux[3]) {
  T ML, MR, aL, aR;
  speed_mach(qL[0], d == 1 ? qL[1] : qL[2], ad, aL, ML);
  speed_mach(qR[0], d == 1 ? qR[1] : qR[2], ad, aR, MR);
  // M+(M_L), beta+(M_L)
  T mp, bp, mm, bm;
  if (fabs(re(ML)) <= 1.0) {
    T t = ML + 1.0;
    mp = 0.25 * (t * t);
    bp = mp * (2.0 * mk(1.0, 0.0, (T*)nullptr) - ML);
  } else if (re(ML) > 0.0) {
    mp = ML;
    bp = mk(1.0, 0.0, (T*)nullptr);
  } else {
    mp = 0.0 * ML;
    bp = 0.0 * ML;
  }
  // M-(M_R), beta-(M_R)
  if (fabs(re(MR)) <= 1.0) {
    T t = MR + (-1.0);
    mm = -0.25 * (t * t);
    bm = (0.25 * (t * t)) * (MR + 2.0);
  } else if (re(MR) > 0.0) {
    mm = 0.0 * MR;
    bm = 0.0 * MR;
  } else {
    mm = MR;
    bm = mk(1.0, 0.0, (T*)nullptr);
  }
  const T Mh = mp + mm;
  const bool pos = re(Mh) > 0.0;
  const T w = Mh * (pos ? aL : aR);
  const T pres = bp * (qL[0] * qL[0]) + bm * (qR[0] * qR[0]);
  flux[0] = w * (pos ? qL[0] : qR[0]);
  flux[1] = w * (pos ? qL[1] : qR[1]) + p1 * pres;
  flux[2] = w * (pos ? qL[2] : qR[2]) + p2 * pres;
}

// One side's columns of the flux's Jacobian (what the complex step of
// ausm_flux gives for unit imaginary parts of that side's three components):
// dmh, db: d M_{1/2} / dM and d beta / dM of this side; b: its beta; W: M_{1/2}
// a^d where this side is upwind, else 0; up: the upwind side's a^d q^mu.
__device__ __forceinline__ void ausm_jacobian_side(const double q[3], int d, double M, double r, double gd,
                                                   double dmh, double db, double b, double W, const double up[3],
                                                   double p1, double p2, double J[3][3]) {
  const double g0 = -1.5 * M * r;     // dM/dq^0 (M = q^d / (q^0 a), a ~ sqrt(q^0)); gd = dM/dq^d
  const double q0sq = q[0] * q[0], hw = 0.5 * W * r, bq = 2.0 * b * q[0];
#pragma unroll
  for (int mu = 0; mu < 3; ++mu) {
    const double pm = mu == 0 ? 0.0 : (mu == 1 ? p1 : p2);
    const double c = mu == 0 ? dmh * up[0] : fma(dmh, up[mu], db * pm * q0sq);
    J[mu][0] = mu == 0 ? fma(c, g0, 1.5 * W) : fma(c, g0, fma(hw, q[mu], bq * pm));
    const double cd = c * gd;
    J[mu][1] = (d == 1 ? cd : 0.0) + (mu == 1 ? W : 0.0);
    J[mu][2] = (d == 2 ? cd : 0.0) + (mu == 2 ? W : 0.0);
  }
}

// The Jacobian of ausm_flux with respect to (qL, qR), the real parts evaluated
// once for all six columns.  (Six complex-step evaluations, one per column,
// took 343 us at 6 x 60 x 60, p = 5, bound by the FP64 pipe: every one repeats
// the square roots and reciprocals.)
__device__ __forceinline__ void ausm_jacobian(const double qL[3], const double qR[3], int d, double ad, double p1,
                                              double p2, double JL[3][3], double JR[3][3]) {
  const SpeedRoot zL = speed_root(qL[0], ad), zR = speed_root(qR[0], ad);
  const double aL = zL.a, aR = zR.a, rL = zL.r, rR = zR.r;
  const double gL = rL * zL.ia, gR = rR * zR.ia;   // dM/dq^d
  const double ML = (d == 1 ? qL[1] : qL[2]) * gL, MR = (d == 1 ? qR[1] : qR[2]) * gR;
  double mp, dmp, bp, dbp, mm, dmm, bm, dbm;
  if (fabs(ML) <= 1.0) {
    const double t = ML + 1.0;
    mp = 0.25 * t * t;
    dmp = 0.5 * t;
    bp = mp * (2.0 - ML);
    dbp = 0.75 * t * (1.0 - ML);
  } else {
    const bool up = ML > 0.0;
    mp = up ? ML : 0.0 * ML;
    dmp = bp = up ? 1.0 : 0.0;
    dbp = 0.0;
  }
  if (fabs(MR) <= 1.0) {
    const double t = MR - 1.0;
    mm = -0.25 * t * t;
    dmm = -0.5 * t;
    bm = 0.25 * t * t * (MR + 2.0);
    dbm = 0.75 * t * (MR + 1.0);
  } else {
    const bool up = MR > 0.0;
    mm = up ? 0.0 * MR : MR;
    dmm = bm = up ? 0.0 : 1.0;
    dbm = 0.0;
  }
  const double Mh = mp + mm;
  const bool pos = Mh > 0.0;
  const double au = pos ? aL : aR, W = Mh * au;
  const double up[3] = {au * (pos ? qL[0] : qR[0]), au * (pos ? qL[1] : qR[1]), au * (pos ? qL[2] : qR[2])};
  ausm_jacobian_side(qL, d, ML, rL, gL, dmp, dbp, bp, pos ? W : 0.0, up, p1, p2, JL);
  ausm_jacobian_side(qR, d, MR, rR, gR, dmm, dbm, bm, pos ? 0.0 : W, up, p1, p2, JR);
}

// ---------------------------------------------------------------- traces
// the packed trace weights of an element edge (0 W, 1 E, 2 S, 3 N)
template <int NS>
__device__ __forceinline__ void trace_weights(const DfrConst& dc, int edge, double (&wq)[NS]) {
  const bool lo = (edge & 1) == 0;
#pragma unroll
  for (int k = 0; k < NS; ++k) wq[k] = lo ? dc.lmq[k] : dc.lpq[k];
}

// traces of the three variables of x at point i of an element edge (Eq. 7 at
// the element ends), in block fixed point with the exponent of the line's N_s
// values: 36 of the split product's 59 FP64 instructions per interface point
// at N_s = 6 become six conversions (its face kernel at 6 x 60 x 60, p = 5: 34
// -> 26 us; with fewer reciprocals in the AUSM flux the face kernel of the
// right-hand side 73 -> 48 us)
template <int NS>
__device__ __forceinline__ void trace_fx(const double* __restrict__ x, long long nodes, int elem, int edge, int i,
                                         const DfrConst& dc, double out[3]) {
  const long long base = (long long)elem * NS * NS + (edge <= 1 ? i * NS : i);
  const int step = edge <= 1 ? 1 : NS;
  double wq[NS];
  trace_weights<NS>(dc, edge, wq);
#pragma unroll
  for (int var = 0; var < 3; ++var) {
    double v[NS];
#pragma unroll
    for (int k = 0; k < NS; ++k) v[k] = __ldg(x + base + k * step + var * nodes);
    out[var] = fx_dot<NS>(v, wq, dc.lq_exp, (edge & 1) == 0, dc.lm, dc.lp);
  }
}

// traces of the state (real) or of q + i eps v
template <typename T, int NS>
__device__ __forceinline__ void trace(const double* __restrict__ q, const double* __restrict__ v, double eps,
                                      long long nodes, int elem, int edge, int i, const DfrConst& dc, T out[3]) {
  double a[3], b[3] = {0.0, 0.0, 0.0};
  trace_fx<NS>(q, nodes, elem, edge, i, dc, a);
  if constexpr (sizeof(T) > sizeof(double)) {
    if (v) trace_fx<NS>(v, nodes, elem, edge, i, dc, b);
  }
#pragma unroll
  for (int k = 0; k < 3; ++k) out[k] = mk(a[k], eps * b[k], (T*)nullptr);
}

template <int NS>
struct VolShape {
  static constexpr int EPB = (256 / (NS * NS)) > 0 ? (256 / (NS * NS)) : 1;
  static constexpr int THREADS = EPB * NS * NS;
};


template <int THREADS, bool W3>
__device__ __forceinline__ void epilogue_finish(const AugEpilogue& ep, double da, double db, double dcc,
                                                unsigned int blk, unsigned int nblk, double dab, double dbc,
                                                double* sbuf);

// Epilogue of the full-evaluation volume kernels (all threads of the block call
// it; blk/nblk: this block's index and the number of blocks working on the same
// vector): out = scale * res + nu * sum_l y_l b_{p-l} (the augmented operator of
// the phi-function solver), the shift of the augmented tail, and -- when dotB is
// set -- the window dot products of the incomplete orthogonalisation (two or
// three vectors; see AugEpilogue).  W3: compiled for the window of three (dotC
// may be set); W3 = false drops that code.  The tangent kernels call its parts.
// the tail coefficients nu * y_l of the augmented operator into coef[MAX_NB]
// (shared memory; the caller synchronises before reading them)
__device__ __forceinline__ void epilogue_coefs(const AugEpilogue& ep, double* coef) {
  if (threadIdx.x < MAX_NB) {
    const int l = threadIdx.x;
    coef[l] = (l < ep.p && ep.b[l]) ? ep.nu * ep.tail_in[l] : 0.0;
  }
}

// Per-node half of the volume epilogue: o = res + sum_l coef_l b_l (B64),
// stored at out, and this node's terms of the window dots added to the
// thread's partial sums (da = z . V_{j-1}, db = z . V_j, dcc = z . V_{j-2} and
// the window's own products dab = V_j . V_{j-1}, dbc = V_j . V_{j-2}).  The
// window's products are formed here, where its vectors are read anyway: as sums
// of the scale pass they cost that pass a second read of V_j and a second
// grid-wide reduction on the critical path (6 x 30 x 30: 3 us of 21).
template <bool W3, bool B64>
__device__ __forceinline__ void epilogue_node(const AugEpilogue& ep, const double* coef, long long idx, long long N,
                                              const double res[3], double* __restrict__ out, double& da, double& db,
                                              double& dcc, double& dab, double& dbc) {
  double ob[3] = {res[0], res[1], res[2]};
  // a loop over the p columns, not an unrolled one over MAX_NB with a guard:
  // guarded-off FP64 instructions still take the FP64 pipe's issue slots
  if (B64) {
    const int p = ep.p < MAX_NB ? ep.p : MAX_NB;
#pragma unroll 1
    for (int l = 0; l < p; ++l) {
      const double* bl = ep.b[l];
      if (!bl) continue;
      const double cl = coef[l];
#pragma unroll
      for (int mu = 0; mu < 3; ++mu) ob[mu] = fma(cl, bl[idx + mu * N], ob[mu]);
    }
  }
#pragma unroll
  for (int mu = 0; mu < 3; ++mu) {
    const double o = ob[mu];
    out[idx + mu * N] = o;
    if (ep.dotB) {
      const double vb = ep.dotB[idx + mu * N];
      db = fma(o, vb, db);
      if (ep.dotA) {
        const double va = ep.dotA[idx + mu * N];
        da = fma(o, va, da);
        dab = fma(vb, va, dab);
      }
      if (W3 && ep.dotC) {
        const double vc = ep.dotC[idx + mu * N];
        dcc = fma(o, vc, dcc);
        dbc = fma(vb, vc, dbc);
      }
    }
  }
}

template <int THREADS, bool W3>
__device__ __forceinline__ void volume_epilogue(const AugEpilogue& ep, bool active, long long idx, long long N,
                                                const double res[3], double* __restrict__ out, unsigned int blk,
                                                unsigned int nblk) {
  __shared__ double coef[MAX_NB];
  epilogue_coefs(ep, coef);
  __syncthreads();
  double da = 0.0, db = 0.0, dcc = 0.0, dab = 0.0, dbc = 0.0;
  if (active) {
    double r[3];
#pragma unroll
    for (int mu = 0; mu < 3; ++mu) r[mu] = ep.scale * res[mu];
    epilogue_node<W3, true>(ep, coef, idx, N, r, out, da, db, dcc, dab, dbc);
  }
  __shared__ double sred[(W3 ? 5 : 3) * THREADS];
  epilogue_finish<THREADS, W3>(ep, da, db, dcc, blk, nblk, dab, dbc, sred);
}

// Sums of K values over the block in a fixed order, through shared scratch of
// K * THREADS doubles: every thread stores its values, warp k sums value k with
// a stride of 32 and a shuffle tree; the results are valid in thread 0.  (On
// this GPU a shuffle tree in every warp would cost each thread 5 K FP64 adds,
// more than the dots themselves.)
template <int THREADS, int K>
__device__ __forceinline__ void block_sums(double v[K], double* sbuf) {
  static_assert(THREADS >= 32 * K, "one warp per value");
  __shared__ double res[K];
#pragma unroll
  for (int k = 0; k < K; ++k) sbuf[k * THREADS + threadIdx.x] = v[k];
  __syncthreads();
  // warp k sums value k (a stride of 32, then a shuffle tree): the K sums run
  // side by side on the SM's schedulers, each in the order one warp gave it
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (w < K) {
    double a = 0.0;
    for (int i = lane; i < THREADS; i += 32) a += sbuf[w * THREADS + i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) a += __shfl_down_sync(0xffffffffu, a, o);
    if (lane == 0) res[w] = a;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
#pragma unroll
    for (int k = 0; k < K; ++k) v[k] = res[k];
  }
}

// the shift of the augmented tail (block 0)
__device__ __forceinline__ void epilogue_tail(const AugEpilogue& ep, unsigned int blk) {
  if (ep.tail_out && blk == 0 && threadIdx.x < ep.p)
    ep.tail_out[threadIdx.x] = (threadIdx.x + 1 < ep.p) ? ep.tail_in[threadIdx.x + 1] : 0.0;
}

// Second half of the volume epilogue (all threads of the block call it, with
// their partial sums over their nodes, see epilogue_node): the shift of the
// augmented tail, the tail's share of the dots, the block sums and -- in the
// last block to finish -- the modified Gram-Schmidt coefficients.  sbuf: K *
// THREADS doubles of shared scratch, K = 5 with W3, else 3.
template <int THREADS, bool W3>
__device__ __forceinline__ void epilogue_finish(const AugEpilogue& ep, double da, double db, double dcc,
                                                unsigned int blk, unsigned int nblk, double dab, double dbc,
                                                double* sbuf) {
  epilogue_tail(ep, blk);
  if (!ep.dotB) return;   // uniform over the grid
  if (blk == 0 && threadIdx.x == 0) {
    for (int l = 0; l < ep.p; ++l) {
      const double zt = (l + 1 < ep.p) ? ep.tail_in[l + 1] : 0.0;
      db = fma(zt, ep.dotB[ep.n + l], db);
      if (ep.dotA) {
        da = fma(zt, ep.dotA[ep.n + l], da);
        dab = fma(ep.dotB[ep.n + l], ep.dotA[ep.n + l], dab);
      }
      if (W3 && ep.dotC) {
        dcc = fma(zt, ep.dotC[ep.n + l], dcc);
        dbc = fma(ep.dotB[ep.n + l], ep.dotC[ep.n + l], dbc);
      }
    }
  }
  constexpr int K = W3 ? 5 : 3;
  __shared__ bool last;
  double v[5] = {da, db, dab, dcc, dbc};
  block_sums<THREADS, K>(v, sbuf);
  if (threadIdx.x == 0) {
#pragma unroll
    for (int k = 0; k < K; ++k) ep.dpart[K * blk + k] = v[k];
    __threadfence();
    const unsigned int t = atomicAdd(ep.dticket, 1u);
    last = (t == nblk - 1);
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  double u[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
  for (int k = threadIdx.x; k < (int)nblk; k += THREADS) {
#pragma unroll
    for (int i = 0; i < K; ++i) u[i] += __ldcg(ep.dpart + K * k + i);
  }
  __syncthreads();   // the scratch is reused
  block_sums<THREADS, K>(u, sbuf);
  if (threadIdx.x == 0) {
    const double a = u[0], b = u[1], vab = u[2];
    if (ep.dotA) *ep.cdot_out = vab;   // V_j . V_{j-1}: V_{j-1} . V_{j-2} of the next iteration
    // modified Gram-Schmidt coefficients, oldest vector first
    if (W3 && ep.dotC != nullptr) {
      const double h0 = u[3];                             // V_{j-2} . z
      const double h1 = a - h0 * (*ep.cprevAC);            // V_{j-1} . (z - h0 V_{j-2})
      *ep.h0_out = h0;
      *ep.h1_out = h1;
      *ep.h2_out = b - h0 * u[4] - h1 * vab;
    } else if (ep.dotA) {
      *ep.h1_out = a;
      *ep.h2_out = b - a * vab;   // V_j . (z - h1 V_{j-1})
    } else {
      *ep.h2_out = b;
    }
    *ep.dticket = 0u;
  }
}

}  // namespace swepi
