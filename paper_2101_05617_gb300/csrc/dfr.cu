// DFR right-hand side and complex-step Jacobian-vector product on sm_103a.
//
// F(q) (Eq. 1-2 discretised by Sec. 3) is evaluated in two kernels:
//   face_flux_kernel   one thread per interface point: traces of both sides
//                      (Eq. 7 at xi = +-1), the App. C transform of the
//                      neighbour state into the owner's coordinates, the AUSM
//                      flux (App. D/E) and its hand-back to the neighbour;
//                      results go to the per-element face-flux buffer.
//   volume_kernel      one thread per solution point, a block holds whole
//                      elements: pointwise fluxes and sources (Eq. 2, 136),
//                      tangent parts staged in shared memory, the extended-node
//                      derivative sweeps (Eq. 12-14) in both directions, and an
//                      epilogue that can fold the augmented-operator terms of the
//                      Krylov solver into the output.
//
// Complex-step arithmetic (Eq. 28).  The JVP evaluates F at q + i eps v.  With
// eps = 1e-30 every imaginary part is ~1e-25 of its real part or smaller, so the
// O(eps^2) cross terms of complex products, quotients and square roots lie far
// below FP64 rounding of the real parts; the `cs` type below carries a complex
// number as (real, imaginary) and evaluates each operation without those terms:
//   (a + ib)(c + id) -> ac + i(ad + bc)
//   (a + ib)/(c + id) -> a/c + i(b - (a/c) d)/c
//   sqrt(a + ib)      -> sqrt(a) + i b / (2 sqrt(a))   (principal root, a > 0)
// Real parts are therefore the FP64 evaluation of F(q) and imaginary parts the
// first-order term, equal to the full complex result up to rounding.  Branches
// (AUSM's |M| <= 1, max/min) test the real part, ties going to the <= 0 side.
#include <cuda_runtime.h>

#include "check.cuh"
#include "dfr_device.cuh"
#include "dfr_tangent.cuh"
#include "swepi_internal.h"

namespace swepi {

// ---------------------------------------------------------------- face flux
struct FaceArgs {
  const double* q;
  const double* v;
  double eps;
  long long nodes;
  const FaceLine* lines;
  const double* fc;
  long long nfacepts;
  double* fb;
  const int* skip;
};

template <typename T, int NS>
__global__ void __launch_bounds__(128) face_flux_kernel(FaceArgs a, DfrConst dc) {
  pdl_wait();
  if (a.skip && *a.skip) return;
  long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= a.nfacepts) return;
  const int line = (int)(t / NS), i = (int)(t % NS);
  const FaceLine L = a.lines[line];
  if (!face_line_ok<NS>(L, a.nodes)) return;
  const int in = L.reversed ? NS - 1 - i : i;
  T qo[3], qn[3];
  trace<T, NS>(a.q, a.v, a.eps, a.nodes, L.owner, L.owner_edge, i, dc, qo);
  trace<T, NS>(a.q, a.v, a.eps, a.nodes, L.nbr, L.nbr_edge, in, dc, qn);
  const long long P = a.nfacepts;
  const double* fc = a.fc + t;
  const double T00 = fc[FC_T00 * P], T01 = fc[FC_T01 * P], T10 = fc[FC_T10 * P], T11 = fc[FC_T11 * P];
  T qt[3];
  qt[0] = qn[0];
  qt[1] = T00 * qn[1] + T01 * qn[2];
  qt[2] = T10 * qn[1] + T11 * qn[2];
  T fl[3];
  const double ad = fc[FC_AD * P], p1 = fc[FC_P1 * P], p2 = fc[FC_P2 * P];
  if (L.owner_is_left)
    ausm_flux<T>(qo, qt, L.dir, ad, p1, p2, fl);
  else
    ausm_flux<T>(qt, qo, L.dir, ad, p1, p2, fl);
  double f0 = part(fl[0]), f1 = part(fl[1]), f2 = part(fl[2]);
  double* fo = a.fb + ((long long)L.owner * 4 + L.owner_edge) * 3 * NS + i;
  fo[0] = f0;
  fo[NS] = f1;
  fo[2 * NS] = f2;
  if (L.handback) {   // across panels: the neighbour's components (App. C); within a panel the same flux
    const double M00 = fc[FC_M00 * P], M01 = fc[FC_M01 * P], M10 = fc[FC_M10 * P], M11 = fc[FC_M11 * P];
    const double g1 = M00 * f1 + M01 * f2, g2 = M10 * f1 + M11 * f2;
    f0 *= fc[FC_SIG * P];
    f1 = g1;
    f2 = g2;
  }
  double* fn = a.fb + ((long long)L.nbr * 4 + L.nbr_edge) * 3 * NS + in;
  fn[0] = f0;
  fn[NS] = f1;
  fn[2 * NS] = f2;
}

// ---------------------------------------------------------------- volume
struct VolArgs {
  const double* q;
  const double* v;
  double eps;
  long long nodes;
  long long nelem;
  const double* nc;
  const double* fb;
  double* out;
  AugEpilogue ep;
};

// The two sweeps are 48 of the ~75 (right-hand side) to ~120 (product) FP64
// instructions a node at N_s = 6, and the FP64 pipe bounds the kernel: they run
// as block fixed point on the integer pipe (fixed.cuh, dfr_tangent.cuh).
template <typename T, int NS, bool W3 = false>
__global__ void __launch_bounds__(VolShape<NS>::THREADS) volume_kernel(VolArgs a, DfrConst dc) {
  constexpr int EPB = VolShape<NS>::EPB;
  constexpr int NN = NS * NS;
  pdl_wait();
  if (a.ep.skip && *a.ep.skip) return;
  __shared__ VolSmem<double, NS, EPB> sm;
  for (int t = threadIdx.x; t < NS * (NS + 2); t += blockDim.x) sm.sD[t / (NS + 2)][t % (NS + 2)] = dc.Dq[t / (NS + 2)][t % (NS + 2)];
  for (int t = threadIdx.x; t < 2 * EPB; t += blockDim.x) sm.sE[0][t >> 1][t & 1] = 0u;
  const int le = threadIdx.x / NN, node = threadIdx.x % NN;
  const long long elem = (long long)blockIdx.x * EPB + le;
  const bool active = elem < a.nelem;
  const int k2 = node / NS, k1 = node % NS;
  const long long idx = elem * NN + node;

  FxPoint<NS> pt;
  double S1 = 0.0, S2 = 0.0;
  unsigned m0 = 0u, m1 = 0u;
  if (active) {
    const long long N = a.nodes;
    T q0 = load_state<T>(a.q, a.v, a.eps, idx);
    T q1 = load_state<T>(a.q, a.v, a.eps, idx + N);
    T q2 = load_state<T>(a.q, a.v, a.eps, idx + 2 * N);
    const double* nc = a.nc + idx;
    T r = cs_rcp(q0);
    T u1 = q1 * r, u2 = q2 * r;
    T q0sq = q0 * q0;
    T q1u1 = q1 * u1, q1u2 = q1 * u2, q2u2 = q2 * u2;
    // sources of Eq. (2): Coriolis, metric (Gamma^i_jk), topography
    S1 = part((nc[NC_K11 * N] * q1 + nc[NC_K12 * N] * q2) - (nc[NC_G1A * N] * q1u1 + nc[NC_G1B * N] * q1u2) +
              nc[NC_B1 * N] * q0);
    S2 = part((nc[NC_K21 * N] * q1 + nc[NC_K22 * N] * q2) - (nc[NC_G2A * N] * q1u2 + nc[NC_G2B * N] * q2u2) +
              nc[NC_B2 * N] * q0);
    pt.v1 = part(q1);
    pt.v2 = part(q2);
    pt.F11 = part(q1u1 + nc[NC_C11 * N] * q0sq);     // sqrt(g) T^{mu nu}, Eq. (136)
    pt.F12 = part(q1u2 + nc[NC_C12 * N] * q0sq);
    pt.F22 = part(q2u2 + nc[NC_C22 * N] * q0sq);
    fx_edges<NS>(a.fb, elem, node, pt, m0, m1);
  }
  __syncthreads();
  fx_block_max<NN, EPB, VolShape<NS>::THREADS>(sm.sE[0], le, m0, m1);
  __syncthreads();
  const double dscale = -dc.two_over_dx;
  bool fixed = false;
  if (active) {
    m0 = sm.sE[0][le][0];
    m1 = sm.sE[0][le][1];
    fixed = fx_usable(m0) && fx_usable(m1) && fx_scale_usable(dscale);
    fx_store<NS>(sm.sF[le], &sm.sB[le][0][0][0], node, pt, fixed, m0, m1);
  }
  __syncthreads();

  // DFR sweeps: extended flux [F(-1), f_1..f_NS, F(+1)] per line (Eq. 11-14)
  double res[3] = {0.0, 0.0, 0.0};
  if (active) {
    fx_sweep<NS, true>(sm.sF[le], &sm.sB[le][0][0][0], k1, k2, sm.sD[k1], sm.sD[k2], dc, dscale, fixed, fx_exp(m0),
                       fx_exp(m1), 0, 0, S1, S2, res);
    if (a.v) {
      const double sc = 1.0 / a.eps;
#pragma unroll
      for (int mu = 0; mu < 3; ++mu) res[mu] *= sc;
    }
  }
  volume_epilogue<VolShape<NS>::THREADS, W3>(a.ep, active, idx, a.nodes, res, a.out, blockIdx.x, gridDim.x);
}

// ---------------------------------------------------------------- launchers
template <typename T, int NS>
static int launch_ns(Ctx& c, const double* q, const double* v, double eps, double* out, const AugEpilogue& ep,
                     cudaStream_t s) {
  FaceArgs fa{q, v, eps, c.nodes, c.d_lines, c.d_face_coef, c.nfacepts, c.d_fb, ep.skip};
  int fthreads = 128;
  long long fblocks = (c.nfacepts + fthreads - 1) / fthreads;
  const bool jvp = v != nullptr;
  const int kf = jvp ? PK_FACE_JVP : PK_FACE_RHS, kv = jvp ? PK_VOL_JVP : PK_VOL_RHS;
  const bool pf = prof_take(c, kf), pv = prof_take(c, kv);
  cudaEvent_t e0 = nullptr, e1 = nullptr, e2 = nullptr;
  if (pf) {
    e0 = prof_event(c);
    cudaEventRecord(e0, s);
  }
  // Programmatic dependent launch, triggered by the CTAs' ends alone: a kernel's
  // launch overlaps its predecessor's last wave.  With the trigger at a kernel's
  // start its successor's CTAs took their places on SMs while they waited, and on
  // grids of about one wave the next kernel's CTAs were dealt two to an SM beside
  // them (6 x 20 x 20, p = 3: right-hand side 23.4 us, full product 38.2; with plain
  // launches 14.1 and 20.7, like this 13.7 and 19.9; 6 x 60 x 60, p = 5: 96 in all).
  if (launch_pdl(face_flux_kernel<T, NS>, dim3((unsigned)fblocks), dim3(fthreads), s, fa, c.dc) != cudaSuccess)
    return SW_ECUDA;
  if (pf || pv) {
    e1 = prof_event(c);
    cudaEventRecord(e1, s);
  }
  VolArgs va{q, v, eps, c.nodes, c.nelem, c.d_node_coef, c.d_fb, out, ep};
  long long vblocks = (c.nelem + VolShape<NS>::EPB - 1) / VolShape<NS>::EPB;
  const dim3 vgrid((unsigned)vblocks), vblock(VolShape<NS>::THREADS);
  const cudaError_t ev = ep.dotC ? launch_pdl(volume_kernel<T, NS, true>, vgrid, vblock, s, va, c.dc)
                                 : launch_pdl(volume_kernel<T, NS, false>, vgrid, vblock, s, va, c.dc);
  if (ev != cudaSuccess) return SW_ECUDA;
  if (pv) {
    e2 = prof_event(c);
    cudaEventRecord(e2, s);
    prof_record(c, kv, e1, e2);
  }
  if (pf) prof_record(c, kf, e0, e1);
  c.launches += 2;
  return cuda_status(cudaGetLastError());
}

template <typename T>
static int launch_any(Ctx& c, const double* q, const double* v, double eps, double* out, const AugEpilogue& ep,
                      cudaStream_t s) {
  switch (c.ns) {
    case 1: return launch_ns<T, 1>(c, q, v, eps, out, ep, s);
    case 2: return launch_ns<T, 2>(c, q, v, eps, out, ep, s);
    case 3: return launch_ns<T, 3>(c, q, v, eps, out, ep, s);
    case 4: return launch_ns<T, 4>(c, q, v, eps, out, ep, s);
    case 5: return launch_ns<T, 5>(c, q, v, eps, out, ep, s);
    case 6: return launch_ns<T, 6>(c, q, v, eps, out, ep, s);
    case 7: return launch_ns<T, 7>(c, q, v, eps, out, ep, s);
    case 8: return launch_ns<T, 8>(c, q, v, eps, out, ep, s);
    default: return SW_EINVAL;
  }
}

template <int NS>
static int launch_fb_ns(Ctx& c, const double* q, const double* v, double eps, double* out, double* fb,
                        cudaStream_t s) {
  FaceArgs fa{q, v, eps, c.nodes, c.d_lines, c.d_face_coef, c.nfacepts, fb, nullptr};
  const int fthreads = 128;
  const long long fblocks = (c.nfacepts + fthreads - 1) / fthreads;
  face_flux_kernel<cs, NS><<<(unsigned)fblocks, fthreads, 0, s>>>(fa, c.dc);
  AugEpilogue ep;
  VolArgs va{q, v, eps, c.nodes, c.nelem, c.d_node_coef, fb, out, ep};
  const long long vblocks = (c.nelem + VolShape<NS>::EPB - 1) / VolShape<NS>::EPB;
  volume_kernel<cs, NS><<<(unsigned)vblocks, VolShape<NS>::THREADS, 0, s>>>(va, c.dc);
  c.launches += 2;
  return cuda_status(cudaGetLastError());
}

int launch_jvp_fb(Ctx& c, const double* q, const double* v, double eps, double* out, double* fb,
                  cudaStream_t s) {
  switch (c.ns) {
    case 1: return launch_fb_ns<1>(c, q, v, eps, out, fb, s);
    case 2: return launch_fb_ns<2>(c, q, v, eps, out, fb, s);
    case 3: return launch_fb_ns<3>(c, q, v, eps, out, fb, s);
    case 4: return launch_fb_ns<4>(c, q, v, eps, out, fb, s);
    case 5: return launch_fb_ns<5>(c, q, v, eps, out, fb, s);
    case 6: return launch_fb_ns<6>(c, q, v, eps, out, fb, s);
    case 7: return launch_fb_ns<7>(c, q, v, eps, out, fb, s);
    case 8: return launch_fb_ns<8>(c, q, v, eps, out, fb, s);
    default: return SW_EINVAL;
  }
}

int launch_rhs(Ctx& c, const double* q, double* F, cudaStream_t s) {
  AugEpilogue ep;
  return launch_any<double>(c, q, nullptr, 1.0, F, ep, s);
}

int launch_jvp(Ctx& c, const double* q, const double* v, double eps, double* out, const AugEpilogue& ep,
               cudaStream_t s) {
  return launch_any<cs>(c, q, v, eps, out, ep, s);
}

// this translation unit's check word (bounds-checked builds; sw_check_status)
SW_CHECK_READER(check_word_dfr)

}  // namespace swepi
