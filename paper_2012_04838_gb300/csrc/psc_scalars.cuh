// Scalars of a time step that one CTA or warp takes: the forcing amplitude and
// the band energy it needs, the deterministic forcing, the CFL time step and
// the integrating-factor tables.  They run beside the transform passes rather
// than as launches of their own: the z-inverse pass of a right-hand side
// carries one extra row of CTAs whose first one takes the forcing amplitude
// (the amplitude is first read by the stage combine), and the y-forward pass of
// stage 1 one that takes the CFL reset (the maximum it needs is complete after
// the X pass, dt and the tables are first read by the combine).
#pragma once

#include "psc_common.cuh"

namespace psc {

// Visit the stored modes of the forcing band 0 < |k|^2 <= k2max, |k_i| <= kb,
// shared out over the `lanes` lanes of a warp in a fixed order: fn(index, weight).
// lanes is 32, or 8 or 16 where the CTAs of a small grid's pass hold no more.
template <class F>
__device__ __forceinline__ void for_band(const Dims& d, int kb, int k2max, int lane, int lanes, const F& fn) {
  const int side = 2 * kb + 1, nx = kb + 1;
  const int n = side * side * nx;  // < 2^29: kb <= K < 512
#pragma unroll 4
  for (int q = lane; q < n; q += lanes) {
    const int r = q / nx;
    const int kx = q - r * nx, kz = r / side - kb, ky = r % side - kb;
    const int k2 = kx * kx + ky * ky + kz * kz;
    if (k2 == 0 || k2 > k2max) continue;
    fn(((long long)(kz + d.K) * d.P + (ky + d.K)) * d.M + kx, kx == 0 ? 1.0 : 2.0);
  }
}

// Band energy E_f = sum_{0<|k|^2<=kF^2} w |u_k|^2 / (2 N^6) of the velocity `u`,
// by one warp in a fixed order; every lane returns it.
template <typename T>
__device__ __forceinline__ double band_energy(const Dims& d, const typename CT<T>::type* u, int kb, int k2max,
                                              int lane, int lanes) {
  using C = typename CT<T>::type;
  double s = 0.0;
  for_band(d, kb, k2max, lane, lanes, [&](long long i, double w) {
    const C a = u[i], b = u[d.S + i], c = u[2 * d.S + i];
    s += w * (((double)a.x * (double)a.x + (double)a.y * (double)a.y) +
              ((double)b.x * (double)b.x + (double)b.y * (double)b.y) +
              ((double)c.x * (double)c.x + (double)c.y * (double)c.y));
  });
  const unsigned mask = lanes == 32 ? 0xffffffffu : (1u << lanes) - 1u;
  for (int o = lanes / 2; o > 0; o >>= 1) s += __shfl_xor_sync(mask, s, o);
  const double n3 = (double)d.N * d.N * d.N;
  return s / (2.0 * n3 * n3);
}

// E_f of the state `in` and A = eps_inj / (2 E_f) (0 if E_f = 0).  One warp:
// the band of kF = 2 has 75 candidate modes, and what bounds this is the
// latency of their loads, so they are issued together across the lanes (one
// thread reading them in turn took 25-29 us per right-hand side at any N, the
// warp as a launch of its own 8 us).
template <typename T>
__device__ __forceinline__ void b_famp(const Dims& d, const void* in_, Ctrl* ctrl, const ForceArgs& f, int lane,
                                       int lanes = 32) {
  using C = typename CT<T>::type;
  const double ef = band_energy<T>(d, static_cast<const C*>(in_), f.kb, f.k2max, lane, lanes);
  if (lane != 0) return;
  if (f.clear_umax) ctrl->umax_bits = 0ull;
  ctrl->Ef = ef;
  if (f.step_start) ctrl->Ef_start = ef;
  // the deterministic forcing keeps the rate of its last rescaling in A
  if (f.forcing != 2) ctrl->A = (f.forcing == 1 && ef > 1e-300) ? f.eps_inj / (2.0 * ef) : 0.0;
}

// The paper's deterministic forcing (section 2.3), after the last stage of a
// step: the band 0 < |k|^2 <= kF^2 of the new state is multiplied by
// f = sqrt(Ef0 / E_f) so that it keeps the energy Ef0 it had at the start of
// the first step (Ef0 < 0: the target is taken from this step's start).  A
// records the equivalent rate ln(f) / dt.  One warp, fixed order; each lane
// rescales the modes it summed.
template <typename T>
__device__ __forceinline__ void b_hold(const Dims& d, void* u_, Ctrl* ctrl, int kb, int k2max, int lane) {
  using C = typename CT<T>::type;
  C* u = static_cast<C*>(u_);
  const double ef = band_energy<T>(d, u, kb, k2max, lane, 32);
  double ef0 = ctrl->Ef0;
  if (ef0 < 0.0) ef0 = ctrl->Ef_start;
  const double f = ef > 1e-300 ? sqrt(ef0 / ef) : 1.0;
  for_band(d, kb, k2max, lane, 32, [&](long long i, double) {
    for (int c = 0; c < 3; ++c) u[c * d.S + i] = cscale(u[c * d.S + i], (T)f);
  });
  __syncwarp();  // every lane has read Ef0
  if (lane != 0) return;
  ctrl->Ef0 = ef0;
  ctrl->A = log(f) / ctrl->dt;
  ctrl->Ef = ef * f * f;
}

// Integrating factors per axis: e(k) = exp(-nu k^2 dt / 2) (and with D), so
// that exp(-nu |k|^2 dt/2) = e(|kx|) e(|ky|) e(|kz|).  FP64 exp, stored as T.
template <typename T>
__device__ __forceinline__ void b_iftab(int K, const Ctrl* ctrl, double nu, double D, T* eu, T* ep, int k) {
  if (k > K) return;
  const double dt = ctrl->dt;
  eu[k] = (T)exp(-nu * (double)k * k * dt * 0.5);
  ep[k] = (T)exp(-D * (double)k * k * dt * 0.5);
}

// dt = cfl dx / max(|u1|+|u2|+|u3|)  (Eq. 10) on every record_every-th step
// (the step count lives on the device, so the launch sequence of a step never
// changes and can be captured in a CUDA graph); a non-finite maximum raises the
// instability flag and leaves dt unchanged.
__device__ __forceinline__ void b_cfl(Ctrl* c, double cfl, double dx, int record_every) {
  if (c->step % record_every != 0) return;
  const double m = __longlong_as_double((long long)c->umax_bits);
  if (!(m <= 1.7976931348623157e308)) {
    atomicOr(&c->err, 2);  // beside CTAs that may be raising, or polling, the time-out bit
    return;
  }
  if (m > 0.0) c->dt = cfl * dx / m;
}

// The extra first row of CTAs of a z-inverse (a.force) or y-forward (a.cfl)
// launch: its first CTA does the scalar work, thread me of nthr.
template <typename T>
__device__ __forceinline__ void lead_force(const PassArgs& a, int me, int nthr) {
  const int lanes = nthr < 32 ? nthr : 32;
  pdl_wait(a.pdl);
  if (blockIdx.x == 0 && blockIdx.z == 0 && me < lanes) b_famp<T>(a.d, a.in, a.ctrl, a.force, me, lanes);
}
template <typename T>
__device__ __forceinline__ void lead_cfl(const PassArgs& a, int me, int nthr) {
  if (blockIdx.x != 0 || blockIdx.z != 0) return;
  pdl_wait(a.pdl);
  if (me == 0) b_cfl(a.ctrl, a.cfl.cfl, a.cfl.dx, a.cfl.record_every);
  __syncthreads();
  for (int k = me; k <= a.d.K; k += nthr)
    b_iftab<T>(a.d.K, a.ctrl, a.cfl.nu, a.cfl.D, static_cast<T*>(a.cfl.eu), static_cast<T*>(a.cfl.ep), k);
}

}  // namespace psc
