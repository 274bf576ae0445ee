// ucn_linearize (Sec. III-A, Eq. (2b)): A_i, B_i by forward-mode differentiation
// of the RK4 map in T, and d_i = RK4(x, u) - A x - B u in FP64; one thread per
// control node.
//
// In FP64 this is bound by the FP64 pipe (1/64 of the FP32 rate on GB300), and a
// tangent pass of its own for each of the nx + nu columns evaluated the dynamics
// -- six sines and cosines, the divisions -- sixteen times over.  Here
//  - several tangents share one evaluation (DualN),
//  - position and velocity columns need no pass: no model's dynamics depend on
//    position, and velocity enters linearly (p' = v, v' = ... - c v, one c for the
//    three axes): the r_j columns are unit vectors and the v_j columns hold
//    d r_j / d v_j and d v_j / d v_j of the scalar recursion -- what a pass along
//    them computes.
// Measured (GB300, 2048 quadrotors of 40..120 nodes, 164k nodes, FP64): 10.4 ms
// with a pass per column and a division per quotient, 1.83 now (1.55 with quotients
// by products with reciprocals, held over the step, whose B is 1.2 times as far off);
// the outputs alone take 0.04 ms at the copy rate.
#pragma once
#include "ucn_kernels.cuh"

namespace ucn {

// First position and velocity rows of a model (three consecutive each), and the
// velocity's linear decay rate c.
template <class M>
struct LinPart {
  static constexpr int R = IsMars14<M>::value ? 1 : 0, V = R + 3;
  static constexpr int FREE = M::NX + M::NU - 6;   // the other directions
  // direction k of them
  __host__ __device__ static constexpr int dir(int k) { return k < R ? k : k + 6; }
};
template <class M, class T>
__device__ __forceinline__ T velocity_decay(const T* prm) {
  if constexpr (IsQuad<M>::value) return prm[12];
  else return T(0);
}

// K tangent columns along the directions dirs[0..K) (a direction beyond nx + nu:
// a zero tangent).
template <class M, class T, int K>
__device__ __forceinline__ void rk4_columns(const T* prm, const Step3<T>& hs, const T* x, const T* u, const int* dirs,
                                            T (*cols)[M::NX]) {
  constexpr int NX = M::NX, NU = M::NU;
  DualN<T, K> xd[NX], ud[NU], out[NX];
#pragma unroll
  for (int j = 0; j < NX; ++j) {
    xd[j].v = x[j];
#pragma unroll
    for (int q = 0; q < K; ++q) xd[j].d[q] = T(dirs[q] == j ? 1 : 0);
  }
#pragma unroll
  for (int j = 0; j < NU; ++j) {
    ud[j].v = u[j];
#pragma unroll
    for (int q = 0; q < K; ++q) ud[j].d[q] = T(dirs[q] == NX + j ? 1 : 0);
  }
  rk4h<M, DualN<T, K>, T, T>(prm, hs.h, hs.hh, hs.h6, xd, ud, out);
#pragma unroll
  for (int j = 0; j < NX; ++j)
#pragma unroll
    for (int q = 0; q < K; ++q) cols[q][j] = out[j].d[q];
}

// Tangents per pass: as many as share the work of the value without more than a
// pass to spare.
template <class M, class T> struct LinTangents { static constexpr int value = LinPart<M>::FREE == 4 ? 4 : sizeof(T) == 8 ? 5 : 4; };

template <class M, class T>
__global__ void __launch_bounds__(128) linearize_kernel(ProblemDev P, const int* node_inst, long long total_u,
                                                        const double* xbar, const double* ubar,
                                                        double* A, double* B, double* d) {
  constexpr int NX = M::NX, NU = M::NU, K = LinTangents<M, T>::value;
  typedef LinPart<M> F;
  const long long g = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (g >= total_u) return;
  const int b = node_inst[g];
  const long long xr = P.xoff[b] + g - P.uoff[b];
  double x[NX], u[NU], prm[PRM], acc[NX];
  T xt[NX], ut[NU], prmt[PRM];
  for (int j = 0; j < NX; ++j) { x[j] = xbar[xr * NX + j]; xt[j] = (T)x[j]; }
  for (int j = 0; j < NU; ++j) { u[j] = ubar[g * NU + j]; ut[j] = (T)u[j]; }
  for (int k = 0; k < PRM; ++k) { prm[k] = derived_param<M>(P.params + b * 8, k); prmt[k] = (T)prm[k]; }
  const double h = P.dt[b];
  const Step3<T> hs = step_of<T>(h);
  double* Ag = A + g * NX * NX;
  double* Bg = B + g * NX * NU;
  rk4<M, double>(prm, h, x, u, acc);
  {
    // the r and v columns: k_v = -c v, k_r = v through the four stages
    const T c = velocity_decay<M, T>(prmt);
    T kr = T(1), kv = -c, ar = kr, av = kv, tv = T(1) + hs.hh * kv;
#pragma unroll
    for (int s = 1; s < 4; ++s) {
      kr = tv;
      kv = -c * tv;
      if (s < 3) { ar += T(2) * kr; av += T(2) * kv; tv = T(1) + (s == 1 ? hs.hh : hs.h) * kv; }
    }
    const double drv = (double)(hs.h6 * (ar + kr)), dvv = (double)(T(1) + hs.h6 * (av + kv));
#pragma unroll
    for (int r = 0; r < NX; ++r)
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        Ag[r * NX + F::R + k] = r == F::R + k ? 1.0 : 0.0;
        Ag[r * NX + F::V + k] = r == F::R + k ? drv : r == F::V + k ? dvv : 0.0;
      }
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      acc[F::R + k] -= x[F::R + k];
      acc[F::R + k] -= drv * x[F::V + k];
      acc[F::V + k] -= dvv * x[F::V + k];
    }
  }
#pragma unroll 1
  for (int k0 = 0; k0 < F::FREE; k0 += K) {
    int dirs[K];
    T cols[K][NX];
#pragma unroll
    for (int q = 0; q < K; ++q) dirs[q] = k0 + q < F::FREE ? F::dir(k0 + q) : NX + NU;
    rk4_columns<M, T, K>(prmt, hs, xt, ut, dirs, cols);
#pragma unroll
    for (int q = 0; q < K; ++q) {
      const int c = dirs[q];
      if (c < NX + NU) {
        const double v = c < NX ? xbar[xr * NX + c] : ubar[g * NU + c - NX];
        double* out = c < NX ? Ag + c : Bg + c - NX;
        const int ld = c < NX ? NX : NU;
#pragma unroll
        for (int r = 0; r < NX; ++r) {
          out[r * ld] = (double)cols[q][r];
          acc[r] -= (double)cols[q][r] * v;
        }
      }
    }
  }
  for (int r = 0; r < NX; ++r) d[g * NX + r] = acc[r];
}

}  // namespace ucn
