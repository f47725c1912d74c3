// Complex-step JVP split into its real and imaginary halves.
//
// Every JVP of one Krylov solve, and the remainder products of one EPI step,
// is taken at the same linearisation point q_n (Eq. 33-35).  In the
// complex-step evaluation F(q_n + i eps v) the real part of every intermediate
// (1/q^0, u^i, a^d, the Froude numbers, the AUSM splittings, ...) depends on q_n
// only, while the imaginary part is a linear function of v whose coefficients
// are those real parts.  The split path therefore evaluates the real half once
// per linearisation point and stores, per solution point and per interface
// point, the coefficients of the imaginary half:
//   lin_node_kernel   per node: u^1, u^2 and the coefficients of the imaginary
//                     parts of sqrt(g) T^{ij} (Eq. 136) and of the sources of
//                     Eq. (2) as functions of Im q, packed for block fixed point;
//   lin_face_kernel   per interface point: the 3 x 6 matrix taking the
//                     imaginary parts of the two traces to the imaginary part of
//                     the AUSM flux: what propagating unit imaginary parts
//                     through the plain kernels' AUSM code gives, with the real
//                     parts evaluated once (ausm_jacobian; the neighbour's App. C
//                     transform folded in).
// Each JVP then runs only the imaginary half, in real arithmetic:
//   face_tangent_kernel   traces of v, the 3 x 6 map, the hand-back;
//   volume_tangent_kernel pointwise imaginary fluxes and sources and the DFR
//                         sweeps (Eq. 12-14; in FP64 both as block fixed point on
//                         the integer pipe, fixed.cuh), and the augmented-operator
//                         epilogue.
// The imaginary parts are proportional to eps, so the tangent is propagated for
// v itself and the final division by eps is omitted.  Results equal the plain
// path up to rounding; no FP64 division or square root remains per JVP.
#include <cuda_runtime.h>

#include <algorithm>

#include "dfr_device.cuh"
#include "dfr_tangent.cuh"
#include "kiops_dev.h"
#include "swepi_internal.h"

namespace swepi {

namespace {

// ---------------------------------------------------------------- linearise
// The coefficients are packed for the block fixed-point products (fixed.cuh,
// dfr_tangent.cuh) with the exponents per element that their sums need: u for
// the u^i, a for the A^{ij}, s for the S^i_j, s0 for the S^i_0, with
//   s0 - s = a - u       (the terms of a source come out in one unit) and
//   k = De + u - s >= 0  (a source adds to the packed sweep after a right shift).
// u and a are the classes' own exponents, raised only where a source outweighs
// the whole sweep (which is then what the sum is rounded against); the S^i_j
// and S^i_0 take what is left, so the fluxes' coefficients keep their bits
// however small the sources' are (no Coriolis term at a panel centre).
// The sources are stored times -dx/2: the sweep's sums and they share the factor
// -2/dx.  An element with a coefficient past the format's range keeps FP64 values,
// and with N_s = 1 all of them do (volume_tangent_node).
// ln32 (complex64-bulk form): the unscaled coefficients rounded to FP32.
template <int NS>
__global__ void __launch_bounds__(VolShape<NS>::THREADS) lin_node_kernel(const double* __restrict__ q,
                                                                         const double* __restrict__ nc, long long nodes,
                                                                         double mhdx, int De, double* __restrict__ ln,
                                                                         int4* __restrict__ le,
                                                                         float* __restrict__ ln32) {
  constexpr int NN = NS * NS, EPB = VolShape<NS>::EPB, THREADS = VolShape<NS>::THREADS;
  pdl_wait();
  pdl_trigger();
  __shared__ unsigned sE[2][EPB][2];
  for (int t = threadIdx.x; t < 4 * EPB; t += THREADS) (&sE[0][0][0])[t] = 0u;
  const long long i = (long long)blockIdx.x * THREADS + threadIdx.x, N = nodes;
  const int e = threadIdx.x / NN;
  const bool active = i < nodes;
  double c[LN_COUNT];
  unsigned mu = 0u, ma = 0u, ms = 0u, ms0 = 0u;
  if (active) {
    const double q0 = q[i], q1 = q[i + N], q2 = q[i + 2 * N];
    const double r = 1.0 / q0;
    const double u1 = q1 * r, u2 = q2 * r;
    const double c11 = nc[NC_C11 * N + i], c12 = nc[NC_C12 * N + i], c22 = nc[NC_C22 * N + i];
    const double g1a = nc[NC_G1A * N + i], g1b = nc[NC_G1B * N + i];
    const double g2a = nc[NC_G2A * N + i], g2b = nc[NC_G2B * N + i];
    // Im sqrt(g)T^{ij} = u^j Im q^i + u^i Im q^j + (g_r h^ij q^0 / sqrt g - u^i u^j) Im q^0
    c[LN_U1] = u1;
    c[LN_U2] = u2;
    c[LN_A11] = 2.0 * c11 * q0 - u1 * u1;
    c[LN_A12] = 2.0 * c12 * q0 - u1 * u2;
    c[LN_A22] = 2.0 * c22 * q0 - u2 * u2;
    // Im S^i = s_i1 Im q^1 + s_i2 Im q^2 + s_i0 Im q^0 (Coriolis, Gamma^i_jk, topography terms of Eq. 2)
    c[LN_S11] = nc[NC_K11 * N + i] - 2.0 * g1a * u1 - g1b * u2;
    c[LN_S12] = nc[NC_K12 * N + i] - g1b * u1;
    c[LN_S10] = g1a * u1 * u1 + g1b * u1 * u2 + nc[NC_B1 * N + i];
    c[LN_S21] = nc[NC_K21 * N + i] - g2a * u2;
    c[LN_S22] = nc[NC_K22 * N + i] - g2a * u1 - 2.0 * g2b * u2;
    c[LN_S20] = g2a * u1 * u2 + g2b * u2 * u2 + nc[NC_B2 * N + i];
    if (ln32) {
#pragma unroll
      for (int k = 0; k < LN_COUNT; ++k) ln32[k * N + i] = (float)c[k];
    }
#pragma unroll
    for (int k = LN_S11; k < LN_COUNT; ++k) c[k] *= mhdx;
    mu = max(fx_key(c[LN_U1]), fx_key(c[LN_U2]));
    ma = max(fx_key(c[LN_A11]), max(fx_key(c[LN_A12]), fx_key(c[LN_A22])));
    ms = max(max(fx_key(c[LN_S11]), fx_key(c[LN_S12])), max(fx_key(c[LN_S21]), fx_key(c[LN_S22])));
    ms0 = max(fx_key(c[LN_S10]), fx_key(c[LN_S20]));
  }
  __syncthreads();
  fx_block_max<NN, EPB, THREADS>(sE[0], e, mu, ma);
  fx_block_max<NN, EPB, THREADS>(sE[1], e, ms, ms0);
  __syncthreads();
  if (!active) return;
  mu = sE[0][e][0];
  ma = sE[0][e][1];
  ms = sE[1][e][0];
  ms0 = sE[1][e][1];
  // an all-zero class takes the format's smallest exponent and raises no other
  const int eu = mu ? (int)(mu >> 20) : kFxExpMin, ea = ma ? (int)(ma >> 20) : kFxExpMin;
  const int es = ms ? (int)(ms >> 20) : kFxExpMin, es0 = ms0 ? (int)(ms0 >> 20) : kFxExpMin;
  const int u = max(eu, es - De), a = max(ea, es0 - De), s = max(es, es0 + u - a), s0 = s + a - u;
  // v^0 is packed for the exponent t + 2 - a, v^i for t + 2 - u, with t >= 1020 + kFxExpMin: both stay
  // large enough that a zero or subnormal entry becomes 0 (fx_pack)
  const bool packed = NS > 1 && fx_usable(mu) && fx_usable(ma) && fx_usable(ms) && fx_usable(ms0) &&
                      max(u, a) <= kFxCoefMax;
  if (threadIdx.x % NN == 0) le[i / NN] = packed ? make_int4(u, a, De + u - s, 1) : make_int4(0, 0, 0, 0);
#pragma unroll
  for (int k = 0; k < LN_COUNT; ++k) {
    const int E = k <= LN_U2 ? u : (k <= LN_A22 ? a : ((k == LN_S10 || k == LN_S20) ? s0 : s));
    ln[k * N + i] = packed ? fx_pack(c[k], E) : c[k];
  }
}

struct LinFaceArgs {
  const double* q;
  long long nodes;
  const FaceLine* lines;
  const double* fc;
  long long nfacepts;
  double* lf;   // [18][nfacepts]: owner-trace block then neighbour-trace block
};

template <int NS>
__global__ void __launch_bounds__(128) lin_face_kernel(LinFaceArgs a, DfrConst dc) {
  pdl_wait();
  pdl_trigger();
  long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= a.nfacepts) return;
  const int line = (int)(t / NS), i = (int)(t % NS);
  const FaceLine L = a.lines[line];
  if (!face_line_ok<NS>(L, a.nodes)) return;
  const int in = L.reversed ? NS - 1 - i : i;
  double qo[3], qn[3];
  trace<double, NS>(a.q, nullptr, 0.0, a.nodes, L.owner, L.owner_edge, i, dc, qo);
  trace<double, NS>(a.q, nullptr, 0.0, a.nodes, L.nbr, L.nbr_edge, in, dc, qn);
  const long long P = a.nfacepts;
  const double* fc = a.fc + t;
  const double T00 = fc[FC_T00 * P], T01 = fc[FC_T01 * P], T10 = fc[FC_T10 * P], T11 = fc[FC_T11 * P];
  const double qt[3] = {qn[0], T00 * qn[1] + T01 * qn[2], T10 * qn[1] + T11 * qn[2]};
  const double ad = fc[FC_AD * P], p1 = fc[FC_P1 * P], p2 = fc[FC_P2 * P];
  double qL[3], qR[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    qL[k] = L.owner_is_left ? qo[k] : qt[k];
    qR[k] = L.owner_is_left ? qt[k] : qo[k];
  }
  double JL[3][3], JR[3][3];
  ausm_jacobian(qL, qR, L.dir, ad, p1, p2, JL, JR);
  // columns of the owner trace and of the neighbour trace (own coordinates)
  double* out = a.lf + t;
#pragma unroll
  for (int mu = 0; mu < 3; ++mu) {
    double o[3], nb[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      o[k] = L.owner_is_left ? JL[mu][k] : JR[mu][k];
      nb[k] = L.owner_is_left ? JR[mu][k] : JL[mu][k];
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) out[(mu * 3 + k) * P] = o[k];
    // neighbour: Im q_t = blockdiag(1, T) Im q_n
    out[(9 + mu * 3 + 0) * P] = nb[0];
    out[(9 + mu * 3 + 1) * P] = nb[1] * T00 + nb[2] * T10;
    out[(9 + mu * 3 + 2) * P] = nb[1] * T01 + nb[2] * T11;
  }
}

// single-grid kernels around the shared bodies (dfr_tangent.cuh)
template <typename T, int NS>
__global__ void __launch_bounds__(128) face_tangent_kernel(TanFaceArgs<T> a, DfrConst dc) {
  pdl_wait();
  pdl_trigger();
  if (a.skip && *a.skip) return;
  face_tangent_body<T, NS>(a, dc, (long long)blockIdx.x * blockDim.x + threadIdx.x);
}

// W3: with the orthogonalisation window of three in the epilogue; a
// persistent grid (volume_ctas)
template <typename T, int NS, bool W3>
__global__ void __launch_bounds__(VolShape<NS>::THREADS, 4) volume_tangent_kernel(TanVolArgs<T> a, DfrConst dc) {
  pdl_wait();
  pdl_trigger();
  if (a.ep.skip && *a.ep.skip) return;
  __shared__ VolSmem<T, NS, VolShape<NS>::EPB> sm;
  volume_tangent_persistent<T, NS, VolShape<NS>::EPB, VolShape<NS>::THREADS, W3>(a, dc, sm);
}

// the same kernels for the device-driven solver: the Krylov iteration index and
// the augmented operator come from its device state
template <typename T, int NS>
__global__ void __launch_bounds__(128) face_tangent_dev_kernel(const KDev* __restrict__ kd, KFix f,
                                                               TanFaceArgs<T> a, DfrConst dc) {
  if (*a.skip) return;
  const long long it = kd->it;
  a.v = f.V + it * f.ldv;
  a.v32 = (sizeof(T) == 4 && f.V32) ? f.V32 + it * f.ldv : nullptr;
  face_tangent_body<T, NS>(a, dc, (long long)blockIdx.x * blockDim.x + threadIdx.x);
}

template <typename T, int NS, bool W3>
__global__ void __launch_bounds__(VolShape<NS>::THREADS, 4) volume_tangent_dev_kernel(const KDev* __restrict__ kd, KFix f,
                                                                                   TanVolArgs<T> a0, DfrConst dc) {
  __shared__ TanVolArgs<T> a;
  if (threadIdx.x == 0) {
    a = a0;
    const int it = kd->it;
    a.v = f.V + (long long)it * f.ldv;
    a.out = f.V + (long long)(it + 1) * f.ldv;
    iter_epilogue_dev(a.ep, *kd, f, it, W3, sizeof(T) == 4);
  }
  __syncthreads();
  if (*a.ep.skip) return;
  __shared__ VolSmem<T, NS, VolShape<NS>::EPB> sm;
  volume_tangent_persistent<T, NS, VolShape<NS>::EPB, VolShape<NS>::THREADS, W3>(a, dc, sm);
}

// CTAs of a persistent volume grid: as many as fit on the GPU at once (the
// kernel's occupancy x SMs), at most one per element tile, each with an even
// share of the elements.  (6 x 60 x 60, p = 5, FP64 with the window dots: 85.3
// us per launch; with 1 / 2 / 3 / 4 tiles a CTA in waves 94.5 / 88.8 / 86.3 /
// 96.4 us.  6 x 30 x 30: 29.4 us, with one tile a CTA 32.6.)  Queried once per
// kernel and device; prepare_volume_dev runs the queries of the device-driven
// solver's kernels before its stream capture.
constexpr int kMaxDevices = 64;
template <typename T, int NS, bool W3, bool DEV>
int volume_ctas(int device, long long tiles) {
  static int fit[kMaxDevices] = {};
  if (device < 0 || device >= kMaxDevices) return -1;
  if (!fit[device]) {
    int sms = 0, nb = 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device) != cudaSuccess) return -1;
    const cudaError_t e =
        DEV ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, volume_tangent_dev_kernel<T, NS, W3>,
                                                            VolShape<NS>::THREADS, 0)
            : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, volume_tangent_kernel<T, NS, W3>,
                                                            VolShape<NS>::THREADS, 0);
    if (e != cudaSuccess || nb < 1) return -1;
    fit[device] = nb * sms;
  }
  return (int)std::min<long long>(std::max<long long>(tiles, 1), fit[device]);
}

__global__ void to_float_kernel(const double* __restrict__ src, float* __restrict__ dst, long long n) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    dst[i] = (float)src[i];
}

template <int NS>
int linearize_ns(Ctx& c, const double* q, cudaStream_t s) {
  const int th = VolShape<NS>::THREADS;
  if (launch_pdl(lin_node_kernel<NS>, dim3((unsigned)((c.nodes + th - 1) / th)), dim3(th), s, q, c.d_node_coef,
                 c.nodes, -0.5 * c.dx, c.dc.dq_exp + 1080, c.d_lin_node, c.d_lin_exp,
                 c.jvp_mode == 2 ? c.d_lin_node32 : static_cast<float*>(nullptr)) != cudaSuccess)
    return SW_ECUDA;
  LinFaceArgs fa{q, c.nodes, c.d_lines, c.d_face_coef, c.nfacepts, c.d_lin_face};
  if (launch_pdl(lin_face_kernel<NS>, dim3((unsigned)((c.nfacepts + 127) / 128)), dim3(128), s, fa, c.dc) !=
      cudaSuccess)
    return SW_ECUDA;
  c.launches += 2;
  return cuda_status(cudaGetLastError());
}

// the complex64-bulk form's orthogonalisation dots are a pass of their own
template <typename T>
constexpr bool kDots = sizeof(T) == 8;

template <typename T, int NS>
int tangent_ns(Ctx& c, const double* v, double* out, const AugEpilogue& ep, const T* ln, const T* lf, T* fb,
               cudaStream_t s) {
  if (!kDots<T> && ep.dotB) return SW_EINVAL;
  const bool pf = prof_take(c, PK_FACE_JVP), pv = prof_take(c, PK_VOL_JVP);
  cudaEvent_t e0 = nullptr, e1 = nullptr, e2 = nullptr;
  if (pf) {
    e0 = prof_event(c);
    cudaEventRecord(e0, s);
  }
  TanFaceArgs<T> fa{v, sizeof(T) == 4 ? ep.v32 : nullptr, c.nodes, c.d_lines, c.d_face_coef, lf, c.nfacepts, fb,
                    ep.skip};
  if (launch_pdl(face_tangent_kernel<T, NS>, dim3((unsigned)((c.nfacepts + 127) / 128)), dim3(128), s, fa, c.dc) !=
      cudaSuccess)
    return SW_ECUDA;
  if (pf || pv) {
    e1 = prof_event(c);
    cudaEventRecord(e1, s);
  }
  TanVolArgs<T> va{v, c.nodes, c.nelem, ln, c.d_lin_exp, fb, out, ep};
  const long long vblocks = (c.nelem + VolShape<NS>::EPB - 1) / VolShape<NS>::EPB;
  int rt = 1;
  if (sizeof(T) == 4) {   // complex64-bulk form: element tiles staged by bulk copies where aligned
    rt = launch_volume_tile_f32<NS>(c, v, out, ep, s);
    if (rt < 0) return rt;
    if (rt == SW_OK) c.launches--;   // counted below
  }
  if (rt != SW_OK) {
    auto launch = [&](auto kernel, int ctas) {
      if (ctas < 1) return false;
      return launch_pdl(kernel, dim3((unsigned)ctas), dim3(VolShape<NS>::THREADS), s, va, c.dc) == cudaSuccess;
    };
    bool ok;
    if constexpr (kDots<T>) {
      ok = ep.dotC ? launch(volume_tangent_kernel<T, NS, true>, volume_ctas<T, NS, true, false>(c.device, vblocks))
                   : launch(volume_tangent_kernel<T, NS, false>, volume_ctas<T, NS, false, false>(c.device, vblocks));
    } else {
      ok = launch(volume_tangent_kernel<T, NS, false>, volume_ctas<T, NS, false, false>(c.device, vblocks));
    }
    if (!ok) return SW_ECUDA;
  }
  if (pv) {
    e2 = prof_event(c);
    cudaEventRecord(e2, s);
    prof_record(c, PK_VOL_JVP, e1, e2);
  }
  if (pf) prof_record(c, PK_FACE_JVP, e0, e1);
  c.launches += 2;
  return cuda_status(cudaGetLastError());
}

template <int NS>
int tangent_any(Ctx& c, const double* v, double* out, const AugEpilogue& ep, bool fp32, cudaStream_t s) {
  if (fp32)
    return tangent_ns<float, NS>(c, v, out, ep, c.d_lin_node32, c.d_lin_face32, reinterpret_cast<float*>(c.d_fb), s);
  return tangent_ns<double, NS>(c, v, out, ep, c.d_lin_node, c.d_lin_face, c.d_fb, s);
}

template <typename T, int NS>
int capture_iter_ns(Ctx& c, KDev* kd, const KFix& f, bool w3, int p, cudaStream_t s) {
  const bool fp32 = sizeof(T) == 4;
  const T* lf = fp32 ? reinterpret_cast<const T*>(c.d_lin_face32) : reinterpret_cast<const T*>(c.d_lin_face);
  const T* ln = fp32 ? reinterpret_cast<const T*>(c.d_lin_node32) : reinterpret_cast<const T*>(c.d_lin_node);
  T* fb = reinterpret_cast<T*>(c.d_fb);
  TanFaceArgs<T> fa{nullptr, nullptr, c.nodes, c.d_lines, c.d_face_coef, lf, c.nfacepts, fb, c.d_flags};
  face_tangent_dev_kernel<T, NS><<<(unsigned)((c.nfacepts + 127) / 128), 128, 0, s>>>(kd, f, fa, c.dc);
  c.launches++;
  if (cudaGetLastError() != cudaSuccess) return SW_ECUDA;
  if (fp32 && p <= kTileMaxB) {   // the staged kernel where the buffers allow it
    const int rt = capture_volume_tile_dev<NS>(c, kd, f, s);
    if (rt <= 0) return rt;
  }
  TanVolArgs<T> va{nullptr, c.nodes, c.nelem, ln, c.d_lin_exp, fb, nullptr, AugEpilogue{}};
  const long long vblocks = (c.nelem + VolShape<NS>::EPB - 1) / VolShape<NS>::EPB;
  auto launch = [&](auto kernel, int ctas) {
    if (ctas > 0) kernel<<<(unsigned)ctas, VolShape<NS>::THREADS, 0, s>>>(kd, f, va, c.dc);
    return ctas > 0;
  };
  bool ok;
  if constexpr (kDots<T>) {
    ok = w3 ? launch(volume_tangent_dev_kernel<T, NS, true>, volume_ctas<T, NS, true, true>(c.device, vblocks))
            : launch(volume_tangent_dev_kernel<T, NS, false>, volume_ctas<T, NS, false, true>(c.device, vblocks));
  } else {
    ok = launch(volume_tangent_dev_kernel<T, NS, false>, volume_ctas<T, NS, false, true>(c.device, vblocks));
  }
  if (!ok) return SW_ECUDA;
  c.launches++;
  return cuda_status(cudaGetLastError());
}

template <int NS>
int capture_iter_any(Ctx& c, KDev* kd, const KFix& f, bool fp32, bool w3, int p, cudaStream_t s) {
  return fp32 ? capture_iter_ns<float, NS>(c, kd, f, w3, p, s) : capture_iter_ns<double, NS>(c, kd, f, w3, p, s);
}

template <int NS>
int prepare_dev_ns(const Ctx& c, bool fp32) {
  const int a = fp32 ? volume_ctas<float, NS, false, true>(c.device, 1) : volume_ctas<double, NS, false, true>(c.device, 1);
  const int b = fp32 ? a : volume_ctas<double, NS, true, true>(c.device, 1);
  return (a < 1 || b < 1) ? SW_ECUDA : SW_OK;
}

}  // namespace

int prepare_volume_dev(const Ctx& c, bool fp32) {
  switch (c.ns) {
    case 1: return prepare_dev_ns<1>(c, fp32);
    case 2: return prepare_dev_ns<2>(c, fp32);
    case 3: return prepare_dev_ns<3>(c, fp32);
    case 4: return prepare_dev_ns<4>(c, fp32);
    case 5: return prepare_dev_ns<5>(c, fp32);
    case 6: return prepare_dev_ns<6>(c, fp32);
    case 7: return prepare_dev_ns<7>(c, fp32);
    case 8: return prepare_dev_ns<8>(c, fp32);
    default: return SW_EINVAL;
  }
}

int capture_iter_jvp(Ctx& c, KDev* kd, const KFix& f, bool fp32, bool w3, int p, cudaStream_t s) {
  switch (c.ns) {
    case 1: return capture_iter_any<1>(c, kd, f, fp32, w3, p, s);
    case 2: return capture_iter_any<2>(c, kd, f, fp32, w3, p, s);
    case 3: return capture_iter_any<3>(c, kd, f, fp32, w3, p, s);
    case 4: return capture_iter_any<4>(c, kd, f, fp32, w3, p, s);
    case 5: return capture_iter_any<5>(c, kd, f, fp32, w3, p, s);
    case 6: return capture_iter_any<6>(c, kd, f, fp32, w3, p, s);
    case 7: return capture_iter_any<7>(c, kd, f, fp32, w3, p, s);
    case 8: return capture_iter_any<8>(c, kd, f, fp32, w3, p, s);
    default: return SW_EINVAL;
  }
}

int launch_linearize(Ctx& c, const double* q, cudaStream_t s) {
  if (!c.d_lin_node && cudaMalloc(&c.d_lin_node, sizeof(double) * LN_COUNT * c.nodes) != cudaSuccess)
    return SW_ENOMEM;
  if (!c.d_lin_exp && cudaMalloc(&c.d_lin_exp, sizeof(int4) * c.nelem) != cudaSuccess) return SW_ENOMEM;
  if (c.jvp_mode == 2) {
    // complex64-bulk form: FP32 copies of the coefficient tables
    if (!c.d_lin_node32 && cudaMalloc(&c.d_lin_node32, sizeof(float) * LN_COUNT * c.nodes) != cudaSuccess)
      return SW_ENOMEM;
    if (!c.d_lin_face32 && cudaMalloc(&c.d_lin_face32, sizeof(float) * 23 * c.nfacepts) != cudaSuccess)
      return SW_ENOMEM;
    if (!c.d_v32 && cudaMalloc(&c.d_v32, sizeof(float) * c.n) != cudaSuccess) return SW_ENOMEM;
    if (int rc = ensure_flags(c)) return rc;   // where the staged kernel's bounded waits report
  }
  if (!c.d_lin_face && cudaMalloc(&c.d_lin_face, sizeof(double) * 18 * c.nfacepts) != cudaSuccess)
    return SW_ENOMEM;
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  const bool pl = prof_on(c, PK_LIN);
  if (pl) {
    e0 = prof_event(c);
    e1 = prof_event(c);
    cudaEventRecord(e0, s);
  }
  int rc;
  switch (c.ns) {
    case 1: rc = linearize_ns<1>(c, q, s); break;
    case 2: rc = linearize_ns<2>(c, q, s); break;
    case 3: rc = linearize_ns<3>(c, q, s); break;
    case 4: rc = linearize_ns<4>(c, q, s); break;
    case 5: rc = linearize_ns<5>(c, q, s); break;
    case 6: rc = linearize_ns<6>(c, q, s); break;
    case 7: rc = linearize_ns<7>(c, q, s); break;
    case 8: rc = linearize_ns<8>(c, q, s); break;
    default: return SW_EINVAL;
  }
  if (rc == SW_OK && c.jvp_mode == 2) {
    to_float_kernel<<<1024, 256, 0, s>>>(c.d_lin_face, c.d_lin_face32, 18LL * c.nfacepts);
    // M00, M01, M10, M11, sigma (consecutive rows of the face table) after the map rows
    to_float_kernel<<<1024, 256, 0, s>>>(c.d_face_coef + (long long)FC_M00 * c.nfacepts,
                                         c.d_lin_face32 + 18LL * c.nfacepts, 5LL * c.nfacepts);
    c.launches += 2;
    rc = cuda_status(cudaGetLastError());
  }
  if (pl) {
    cudaEventRecord(e1, s);
    prof_record(c, PK_LIN, e0, e1);
  }
  if (rc == SW_OK) c.linearized = true;
  return rc;
}

int launch_jvp_lin(Ctx& c, const double* v, double* out, const AugEpilogue& ep, cudaStream_t s, bool fp32) {
  if (!c.linearized) return SW_EINVAL;
  if (fp32 && !c.d_lin_node32) return SW_EINVAL;
  // the FP32 kernels take the b-column terms from their FP32 copies only
  for (int l = 0; fp32 && l < ep.p && l < MAX_NB; ++l)
    if (ep.b[l] && !ep.b32[l]) return SW_EINVAL;
  switch (c.ns) {
    case 1: return tangent_any<1>(c, v, out, ep, fp32, s);
    case 2: return tangent_any<2>(c, v, out, ep, fp32, s);
    case 3: return tangent_any<3>(c, v, out, ep, fp32, s);
    case 4: return tangent_any<4>(c, v, out, ep, fp32, s);
    case 5: return tangent_any<5>(c, v, out, ep, fp32, s);
    case 6: return tangent_any<6>(c, v, out, ep, fp32, s);
    case 7: return tangent_any<7>(c, v, out, ep, fp32, s);
    case 8: return tangent_any<8>(c, v, out, ep, fp32, s);
    default: return SW_EINVAL;
  }
}

// this translation unit's check word (bounds-checked builds; sw_check_status)
SW_CHECK_READER(check_word_split)

}  // namespace swepi
