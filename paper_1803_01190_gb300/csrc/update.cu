// O(N) kernels around the force sum: packing of the caller's arrays into the
// device layout, the epilogues that sum the force kernel's j-segments in a
// fixed order and apply the integrator (the paper's US kernel, section 2,
// fused with the segment sum), and the Eq. 8-10 reductions.
//
// The integrator arithmetic uses explicitly rounded operations (no fused
// multiply-add contraction) in the order the paper writes the formulas, so
// that a step differs from a plain sequential evaluation only through the
// accelerations it is given.
//
// With the spatial order the force kernels' sums come in sorted order and the
// epilogues read them through the permutation: the sums are the larger part
// of the traffic and stay coalesced, the state is touched at 32 bytes a
// particle either way, and no pass moves the sums back to input order.
#include <cuda_runtime.h>

#include "nbody_internal.cuh"

namespace nb {

template <typename real>
struct ops;
template <>
struct ops<double> {
  static __device__ __forceinline__ double add(double a, double b) { return __dadd_rn(a, b); }
  static __device__ __forceinline__ double mul(double a, double b) { return __dmul_rn(a, b); }
};
template <>
struct ops<float> {
  static __device__ __forceinline__ float add(float a, float b) { return __fadd_rn(a, b); }
  static __device__ __forceinline__ float mul(float a, float b) { return __fmul_rn(a, b); }
};

template <typename real>
__device__ __forceinline__ real4<real> mk4(real x, real y, real z, real w) {
  real4<real> v;
  v.x = x;
  v.y = y;
  v.z = z;
  v.w = w;
  return v;
}

// The epilogues work on components: thread t has component c = t mod 4 (x, y, z,
// potential or mass) of particle t / 4, all arrays being real4.  A particle's
// FP64 additions, 4 S of them and about 40 of the update, would keep one thread
// and with it a quarter of an SM busy for longer than the memory access takes
// (64 cycles a warp each; the epilogue of N = 4096 with S = 32 took 14.3 us with
// one thread per particle).  A mixed step of 2048 particles went from 51.0 to
// 48.0 us, an FP64 step of 4096 from 161.5 to 160.7; the order of the operations
// is the same.

// Component c of the sum of the S j-segment partials of the k-th particle of
// the sums, in segment order, with G and the sign of the potential applied.
template <typename real>
__device__ __forceinline__ real gather_comp(const real *part, int S, int64_t n, int64_t k, int c,
                                            real G) {
  using O = ops<real>;
  const real *p = part + 4 * k + c;
  real x = *p;
#pragma unroll 4
  for (int s = 1; s < S; s++) x = O::add(x, p[4 * (int64_t)s * n]);
  const real a = O::mul(G, x);
  return c < 3 ? a : -a;
}
template <typename real, class F>
__device__ __forceinline__ void for_components(int64_t n, const int32_t *perm, F f) {
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < 4 * n;
       t += (int64_t)gridDim.x * blockDim.x) {
    const int64_t k = t >> 2;
    f(k, perm ? (int64_t)perm[k] : k, (int)(t & 3));
  }
}

// ---------------------------------------------------------------- pack / unpack
template <typename real>
__global__ void k_pack(const double *__restrict__ pos, const double *__restrict__ vel,
                       const double *__restrict__ mass, int64_t n, real4<real> *__restrict__ posm,
                       real4<real> *__restrict__ velv, int *__restrict__ flag) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const double x = pos[3 * i], y = pos[3 * i + 1], z = pos[3 * i + 2], m = mass[i];
    double vx = 0, vy = 0, vz = 0;
    if (vel) {
      vx = vel[3 * i];
      vy = vel[3 * i + 1];
      vz = vel[3 * i + 2];
    }
    const bool ok = isfinite(x) && isfinite(y) && isfinite(z) && isfinite(m) && m >= 0.0 &&
                    isfinite(vx) && isfinite(vy) && isfinite(vz);
    if (!ok && flag) atomicOr(flag, 1);
    posm[i] = mk4<real>((real)x, (real)y, (real)z, (real)m);
    if (velv) velv[i] = mk4<real>((real)vx, (real)vy, (real)vz, (real)0);
  }
}

template <typename real>
__global__ void k_unpack_state(const real4<real> *__restrict__ posm,
                               const real4<real> *__restrict__ velv, int64_t n,
                               double *__restrict__ pos, double *__restrict__ vel) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    if (pos) {
      const real4<real> p = posm[i];
      pos[3 * i] = p.x;
      pos[3 * i + 1] = p.y;
      pos[3 * i + 2] = p.z;
    }
    if (vel) {
      const real4<real> v = velv[i];
      vel[3 * i] = v.x;
      vel[3 * i + 1] = v.y;
      vel[3 * i + 2] = v.z;
    }
  }
}

template <typename real>
__global__ void k_store_acc(const real *__restrict__ part, const int32_t *__restrict__ perm, int S,
                            int64_t n, real G, real *__restrict__ acc) {
  chain_begin();
  for_components<real>(n, perm, [&](int64_t k, int64_t i, int c) {
    acc[4 * i + c] = gather_comp<real>(part, S, n, k, c, G);
  });
}

// The sums of one evaluation straight into the caller's layout (either output
// may be NULL).
template <typename real>
__global__ void k_acc_out(const real *__restrict__ part, const int32_t *__restrict__ perm, int S,
                          int64_t n, real G, double *__restrict__ acc3,
                          double *__restrict__ pot) {
  chain_begin();
  for_components<real>(n, perm, [&](int64_t k, int64_t i, int c) {
    const real a = gather_comp<real>(part, S, n, k, c, G);
    if (c < 3) {
      if (acc3) acc3[3 * i + c] = a;
    } else if (pot) {
      pot[i] = a;
    }
  });
}

template <typename real>
__global__ void k_unpack_acc(const real4<real> *__restrict__ acc, int64_t n,
                             double *__restrict__ acc3, double *__restrict__ pot) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const real4<real> a = acc[i];
    if (acc3) {
      acc3[3 * i] = a.x;
      acc3[3 * i + 1] = a.y;
      acc3[3 * i + 2] = a.z;
    }
    if (pot) pot[i] = a.w;
  }
}

// ---------------------------------------------------------------- KDK, Eq. 5-7
// Predictor and drift for the step that starts at (r, v, a):
//   vt = v + dt a                      (Eq. 5)
//   r' = r + dt/2 (vt + v)             (Eq. 6)     -> posm_nxt (mass copied)
//   vbar = (v + vt) / 2                (first term of Eq. 7, kept for the corrector)
// one component (c = 3: the mass is copied, vbar's fourth component is 0)
template <typename real>
__device__ __forceinline__ void kdk_predict_one(int c, real dt, real hdt, real r, real v, real a,
                                                real &vbar, real &rn) {
  using O = ops<real>;
  const real t = O::add(v, O::mul(dt, a));
  rn = c < 3 ? O::add(r, O::mul(hdt, O::add(t, v))) : r;
  vbar = c < 3 ? O::mul(O::add(v, t), (real)0.5) : (real)0;
}

template <typename real>
__global__ void k_kdk_predict(int64_t n, real dt, real hdt, const real *__restrict__ posm,
                              const real *__restrict__ vel, const real *__restrict__ acc,
                              real *__restrict__ vbar, real *__restrict__ posm_nxt) {
  chain_begin();
  for_components<real>(n, nullptr, [&](int64_t, int64_t i, int c) {
    const int64_t o = 4 * i + c;
    real vb, rn;
    kdk_predict_one<real>(c, dt, hdt, posm[o], vel[o], acc[o], vb, rn);
    vbar[o] = vb;
    posm_nxt[o] = rn;
  });
}

// After the force at r(t+dt): a' = G sum(parts); corrector
//   v(t+dt) = vbar + dt/2 a'           (Eq. 7, chdt = dt/2 of the step just ended)
// then the predictor and drift of the next step, of size dt_next (the same dt
// for KDK; the next substep's for the fourth-order composition), into posm_pred.
template <typename real>
__global__ void k_kdk_correct_predict(const real *__restrict__ part,
                                      const int32_t *__restrict__ perm, int S, int64_t n, real G,
                                      real chdt, real dt, real hdt, real *__restrict__ acc,
                                      const real *__restrict__ posm_new, real *__restrict__ vel,
                                      real *__restrict__ vbar, real *__restrict__ posm_pred) {
  chain_begin();
  using O = ops<real>;
  for_components<real>(n, perm, [&](int64_t k, int64_t i, int c) {
    const int64_t o = 4 * i + c;
    const real a = gather_comp<real>(part, S, n, k, c, G);
    acc[o] = a;
    const real v = c < 3 ? O::add(vbar[o], O::mul(chdt, a)) : (real)0;
    vel[o] = v;
    real nvb, rn;
    kdk_predict_one<real>(c, dt, hdt, posm_new[o], v, a, nvb, rn);
    vbar[o] = nvb;
    posm_pred[o] = rn;
  });
}

// ---------------------------------------------------------------- RK4
// Classical Runge-Kutta on (r, v) with running sums in the order
//   r(t+dt) = r + dt/6 (((v + 2 v2) + 2 v3) + v4)
//   v(t+dt) = v + dt/6 (((a1 + 2 a2) + 2 a3) + a4)
// where v2 = v + dt/2 a1, v3 = v + dt/2 a2, v4 = v + dt a3 and the stage
// positions are r + dt/2 v, r + dt/2 v2, r + dt v3.  Stage k runs after the
// force evaluation a_k.
template <typename real>
__global__ void k_rk4_stage(const real *__restrict__ part, const int32_t *__restrict__ perm, int S,
                            int64_t n, real G, int stage, real dt, real hdt, real dt6,
                            real *__restrict__ posm0, real *__restrict__ vel0,
                            real *__restrict__ vs, real *__restrict__ sr, real *__restrict__ sv,
                            real *__restrict__ posm_stage) {
  chain_begin();
  using O = ops<real>;
  for_components<real>(n, perm, [&](int64_t k, int64_t i, int c) {
    const int64_t o = 4 * i + c;
    if (c == 3) {  // masses of the stage positions; the velocities' fourth component is 0
      if (stage < 4) posm_stage[o] = posm0[o];
      if (stage == 1 || stage == 4) (stage == 1 ? vs : vel0)[o] = (real)0;
      return;
    }
    const real a = gather_comp<real>(part, S, n, k, c, G);
    const real r0 = posm0[o], v0 = vel0[o];
    if (stage == 1) {
      const real v2 = O::add(v0, O::mul(hdt, a));
      sv[o] = a;
      sr[o] = O::add(v0, O::mul((real)2, v2));
      vs[o] = v2;
      posm_stage[o] = O::add(r0, O::mul(hdt, v0));
    } else if (stage == 2 || stage == 3) {
      const real h = stage == 2 ? hdt : dt;  // v3 = v + dt/2 a2 ; v4 = v + dt a3
      const real vp = vs[o];                 // v2 (stage 2) or v3 (stage 3)
      const real vn = O::add(v0, O::mul(h, a));
      sv[o] = O::add(sv[o], O::mul((real)2, a));
      const real w = stage == 2 ? (real)2 : (real)1;  // + 2 v3 ; + v4
      sr[o] = O::add(sr[o], O::mul(w, vn));
      vs[o] = vn;
      // stage positions r + dt/2 v2 (after a2) and r + dt v3 (after a3)
      posm_stage[o] = O::add(r0, O::mul(h, vp));
    } else {
      posm0[o] = O::add(r0, O::mul(dt6, sr[o]));
      vel0[o] = O::add(v0, O::mul(dt6, O::add(sv[o], a)));
    }
  });
}

// ---------------------------------------------------------------- Eq. 8-10
constexpr int DIAG_BT = 256;

int diag_blocks(int64_t n) {
  int64_t b = (n + DIAG_BT - 1) / DIAG_BT;
  return (int)(b < 1024 ? b : 1024);
}

// Per-block sums of (K, W, Px, Py, Pz, Lx, Ly, Lz) with
//   K = m |v|^2 / 2, W = m pot / 2 (pot carries -G sum_j m_j / |r_ij + eps|),
//   P = m v (Eq. 9), L = m r x v (Eq. 10 is L_z),
// each block striding over particles in a fixed order and reducing in a
// fixed tree: the result is deterministic for a given n.
template <typename real>
__global__ void __launch_bounds__(DIAG_BT) k_diag_blocks(const real4<real> *__restrict__ posm,
                                                         const real4<real> *__restrict__ vel,
                                                         const real4<real> *__restrict__ acc,
                                                         int64_t n, double *__restrict__ blocks) {
  __shared__ double sh[8][DIAG_BT];
  double q[8] = {0, 0, 0, 0, 0, 0, 0, 0};
  for (int64_t i = blockIdx.x * (int64_t)DIAG_BT + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * DIAG_BT) {
    const real4<real> p = posm[i];
    const real4<real> v = vel[i];
    const double m = p.w, x = p.x, y = p.y, z = p.z, vx = v.x, vy = v.y, vz = v.z;
    const double pot = acc[i].w;
    q[0] += m * (vx * vx + vy * vy + vz * vz) * 0.5;
    q[1] += m * pot * 0.5;
    q[2] += m * vx;
    q[3] += m * vy;
    q[4] += m * vz;
    q[5] += m * (y * vz - z * vy);
    q[6] += m * (z * vx - x * vz);
    q[7] += m * (x * vy - y * vx);
  }
  for (int c = 0; c < 8; c++) sh[c][threadIdx.x] = q[c];
  __syncthreads();
  for (int w = DIAG_BT / 2; w > 0; w >>= 1) {
    if (threadIdx.x < w)
      for (int c = 0; c < 8; c++) sh[c][threadIdx.x] += sh[c][threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x < 8) blocks[blockIdx.x * 8 + threadIdx.x] = sh[threadIdx.x][0];
}

// out9 = (E, K, W, Px, Py, Pz, Lx, Ly, Lz) from nb block sums, fixed order.
__global__ void __launch_bounds__(DIAG_BT) k_diag_final(const double *__restrict__ blocks, int nb,
                                                        double *__restrict__ out9) {
  __shared__ double sh[8][DIAG_BT];
  double q[8] = {0, 0, 0, 0, 0, 0, 0, 0};
  for (int b = threadIdx.x; b < nb; b += DIAG_BT)
    for (int c = 0; c < 8; c++) q[c] += blocks[b * 8 + c];
  for (int c = 0; c < 8; c++) sh[c][threadIdx.x] = q[c];
  __syncthreads();
  for (int w = DIAG_BT / 2; w > 0; w >>= 1) {
    if (threadIdx.x < w)
      for (int c = 0; c < 8; c++) sh[c][threadIdx.x] += sh[c][threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    out9[0] = sh[0][0] + sh[1][0];
    for (int c = 0; c < 8; c++) out9[1 + c] = sh[c][0];
  }
}

// ---------------------------------------------------------------- launchers
// Blocks of 64 while they spread a small system over more SMs.
static int block_for(int64_t threads) { return threads < 152 * 256 ? 64 : 256; }
static unsigned grid_for(int64_t threads) {
  const int bt = block_for(threads);
  int64_t g = (threads + bt - 1) / bt;
  if (g > 152 * 64) g = 152 * 64;
  return (unsigned)(g < 1 ? 1 : g);
}

cudaError_t launch_pack(int mode, const double *pos, const double *vel, const double *mass,
                        int64_t n, void *posm, void *velv, int *flag, cudaStream_t st) {
  if (mode == NBODY_FP32)
    k_pack<float><<<grid_for(n), block_for(n), 0, st>>>(pos, vel, mass, n, (float4 *)posm, (float4 *)velv,
                                               flag);
  else
    k_pack<double><<<grid_for(n), block_for(n), 0, st>>>(pos, vel, mass, n, (d4 *)posm, (d4 *)velv, flag);
  return cudaGetLastError();
}

cudaError_t launch_unpack_state(int mode, const void *posm, const void *velv, int64_t n,
                                double *pos, double *vel, cudaStream_t st) {
  if (mode == NBODY_FP32)
    k_unpack_state<float><<<grid_for(n), block_for(n), 0, st>>>((const float4 *)posm,
                                                       (const float4 *)velv, n, pos, vel);
  else
    k_unpack_state<double><<<grid_for(n), block_for(n), 0, st>>>((const d4 *)posm, (const d4 *)velv, n,
                                                        pos, vel);
  return cudaGetLastError();
}

cudaError_t launch_store_acc(int mode, const EpiIn &e, void *acc, cudaStream_t st) {
  const unsigned g = grid_for(4 * e.n), b = block_for(4 * e.n);
  if (mode == NBODY_FP32)
    return launch_chained(k_store_acc<float>, g, b, st, (const float *)e.part, e.perm, e.S, e.n,
                          (float)e.G, (float *)acc);
  return launch_chained(k_store_acc<double>, g, b, st, (const double *)e.part, e.perm, e.S, e.n,
                        e.G, (double *)acc);
}

cudaError_t launch_acc_out(int mode, const EpiIn &e, double *acc3, double *pot, cudaStream_t st) {
  const unsigned g = grid_for(4 * e.n), b = block_for(4 * e.n);
  if (mode == NBODY_FP32)
    return launch_chained(k_acc_out<float>, g, b, st, (const float *)e.part, e.perm, e.S, e.n,
                          (float)e.G, acc3, pot);
  return launch_chained(k_acc_out<double>, g, b, st, (const double *)e.part, e.perm, e.S, e.n, e.G,
                        acc3, pot);
}

cudaError_t launch_unpack_acc(int mode, const void *acc, int64_t n, double *acc3, double *pot,
                              cudaStream_t st) {
  if (mode == NBODY_FP32)
    k_unpack_acc<float><<<grid_for(n), block_for(n), 0, st>>>((const float4 *)acc, n, acc3, pot);
  else
    k_unpack_acc<double><<<grid_for(n), block_for(n), 0, st>>>((const d4 *)acc, n, acc3, pot);
  return cudaGetLastError();
}

cudaError_t launch_kdk_predict(int mode, int64_t n, double dt, const void *posm_cur,
                               const void *vel, const void *acc, void *vbar, void *posm_nxt,
                               cudaStream_t st) {
  const unsigned g = grid_for(4 * n), b = block_for(4 * n);
  if (mode == NBODY_FP32)
    return launch_chained(k_kdk_predict<float>, g, b, st, n, (float)dt, (float)(dt / 2),
                          (const float *)posm_cur, (const float *)vel, (const float *)acc,
                          (float *)vbar, (float *)posm_nxt);
  return launch_chained(k_kdk_predict<double>, g, b, st, n, dt, dt / 2, (const double *)posm_cur,
                        (const double *)vel, (const double *)acc, (double *)vbar,
                        (double *)posm_nxt);
}

cudaError_t launch_kdk_correct_predict(int mode, const EpiIn &e, double dt, double dt_next,
                                       void *acc, void *posm_new, void *vel, void *vbar,
                                       void *posm_pred, cudaStream_t st) {
  const unsigned g = grid_for(4 * e.n), b = block_for(4 * e.n);
  if (mode == NBODY_FP32)
    return launch_chained(k_kdk_correct_predict<float>, g, b, st, (const float *)e.part, e.perm,
                          e.S, e.n, (float)e.G, (float)(dt / 2), (float)dt_next,
                          (float)(dt_next / 2), (float *)acc, (const float *)posm_new,
                          (float *)vel, (float *)vbar, (float *)posm_pred);
  return launch_chained(k_kdk_correct_predict<double>, g, b, st, (const double *)e.part, e.perm,
                        e.S, e.n, e.G, dt / 2, dt_next, dt_next / 2, (double *)acc,
                        (const double *)posm_new, (double *)vel, (double *)vbar,
                        (double *)posm_pred);
}

cudaError_t launch_rk4_stage(int mode, const EpiIn &e, int stage, double dt, const void *posm0,
                             void *vel0, void *rk_vs, void *rk_sr, void *rk_sv, void *posm_stage,
                             cudaStream_t st) {
  const unsigned g = grid_for(4 * e.n), b = block_for(4 * e.n);
  if (mode == NBODY_FP32)
    return launch_chained(k_rk4_stage<float>, g, b, st, (const float *)e.part, e.perm, e.S, e.n,
                          (float)e.G, stage, (float)dt, (float)(dt / 2), (float)(dt / 6),
                          (float *)posm0, (float *)vel0, (float *)rk_vs, (float *)rk_sr,
                          (float *)rk_sv, (float *)posm_stage);
  return launch_chained(k_rk4_stage<double>, g, b, st, (const double *)e.part, e.perm, e.S, e.n,
                        e.G, stage, dt, dt / 2, dt / 6, (double *)posm0, (double *)vel0,
                        (double *)rk_vs, (double *)rk_sr, (double *)rk_sv, (double *)posm_stage);
}

cudaError_t launch_diag(int mode, const void *posm, const void *vel, const void *acc, int64_t n,
                        double *blocks, int nblocks, double *out9, cudaStream_t st) {
  if (mode == NBODY_FP32)
    k_diag_blocks<float><<<nblocks, DIAG_BT, 0, st>>>((const float4 *)posm, (const float4 *)vel,
                                                      (const float4 *)acc, n, blocks);
  else
    k_diag_blocks<double><<<nblocks, DIAG_BT, 0, st>>>((const d4 *)posm, (const d4 *)vel,
                                                       (const d4 *)acc, n, blocks);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  k_diag_final<<<1, DIAG_BT, 0, st>>>(blocks, nblocks, out9);
  return cudaGetLastError();
}

}  // namespace nb
