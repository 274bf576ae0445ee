// Fan kernel: the FP64 solve of the 12-state quadrotor with F = 8, 16 or 32 lanes
// per node and an instance over the CTAs of a thread-block cluster, for batches
// of at most one instance per SM.
//
// The FP64 pipe is what this path waits for: on GB300 one FP64 warp instruction
// takes a scheduler 64 cycles and an SM 19, whatever its active lanes (measured).
// One CTA per instance therefore leaves a single solve on one SM of 152, and a
// batch of about one instance per SM waits for its longest.  Here
//  - the lanes of a node own rows e = q, q + F, ... of xi = (x, u) and hold, in
//    registers, those rows of G = [A B] and of H^-1 and the same columns of G:
//    no matrix is read in the ADMM loop;
//  - vectors go through a staging buffer in shared memory, which every lane of
//    the node reads back as broadcasts (a shuffle would cost two instructions per
//    double);
//  - assembly and inverse (Gauss-Jordan) are shared by the lanes too; one thread
//    per node ran ~5000 FP64 instructions for them;
//  - a node's instance is split over SMs by the cluster (halo records as in
//    ucn_rows.cuh), so that its FP64 work runs on several SMs' pipes.
// Per ADMM iteration a warp issues ~50 FP64 instructions for one node (F = 32),
// ~88 for two (F = 16) or ~140 for four (F = 8), against ~275 for eight with four
// lanes per node: the more lanes the shorter, the fewer the less work in all.
// Measured (GB300, four lanes per node -> this): one quadrotor of 50 nodes, 15 x
// 200 iterations, 52.2 -> 12.96 ms (15.1 -> 3.9 us per ADMM iteration, 445 ->
// 90 us per SCP iteration outside it); 149 of 40..120 nodes, 10 x 200, 102.5 ->
// 93.1 ms.  What bounds it: the FP64 pipes at F = 8 (70% busy, counters), else
// the iteration's chain of FP64 latencies (64 cycles each) and exchanges.
#pragma once
#include "ucn_rows.cuh"

namespace ucn {

constexpr int FAN_THREADS = 256;
// Staging per node, in doubles: three vectors of 16 (stride 18: the nodes of a
// warp read different banks) and G by rows for the assembly.
constexpr int FAN_VEC = 18, FAN_G = 12 * 16, FAN_STAGE = 3 * FAN_VEC + FAN_G;

struct FanPos {
  int i, N, q;             // q: the lane's first row
  int lane, half;          // lane of the node; which half of its row (F = 32)
  bool active, hasU, later, first, last;
  bool owner;              // half 0: its row's sums and stores to other CTAs
  unsigned rank;
  int NS;
  double *t, *st;          // the node's record and staging
  double *halo0, *halo1;   // records before the first and after the last node
  RowHalo* hb;             // arrival of the neighbours' boundary values
};
// Rows per lane, and lanes that share a row (F = 32: two, half of its columns each).
template <int F>
struct FanRows {
  static constexpr int R = F == 32 ? 1 : 16 / F, SPLIT = F == 32 ? 2 : 1;
  static constexpr int C16 = 16 / SPLIT, C12 = 12 / SPLIT;
};
template <int F>
struct FanMats : FanRows<F> {
  typedef FanRows<F> S;
  double g[S::R][S::C16], gc[S::R][S::C12], h[S::R][S::C16];   // own rows of G and H^-1, own columns of G
};
template <int F>
struct FanConst {
  double kq[FanRows<F>::R], khd[FanRows<F>::R];
  double gr[3];   // the position row's part of the obstacles' Gram matrix, times rho_geo
};

// Sum over the F lanes of a node.
template <int F>
__device__ __forceinline__ double fan_sum(double v) {
#pragma unroll
  for (int o = 1; o < F; o <<= 1) v += __shfl_xor_sync(ROWS_ALL, v, o);
  return v;
}
// The lane's row (n entries, or its half of them) times v in shared memory
// (16-byte reads).
template <int F, int n>
__device__ __forceinline__ double fan_dot(const FanPos& p, const double* m, const double* v) {
  constexpr int k = n / FanRows<F>::SPLIT;
  double a = 0.0, b = 0.0;
  if constexpr (F == 32) v += k * p.half;
#pragma unroll
  for (int c = 0; c < k; c += 2) {
    const double2 w = *reinterpret_cast<const double2*>(v + c);
    a += m[c] * w.x;
    b += m[c + 1] * w.y;
  }
  a += b;
  if constexpr (F == 32) a += __shfl_xor_sync(ROWS_ALL, a, 16);
  return a;
}

// The top 21 significant bits of a double as a float, by integer instructions (a
// conversion is one of the FP64 pipe's); 0 below 2^-126, infinite above 2^128.
__device__ __forceinline__ float fan_approx(double v) {
  const int h = __double2hiint(v), e = h & 0x7fffffff;
  int m = (e - (896 << 20)) << 3;
  m = e < (897 << 20) ? 0 : e >= (1151 << 20) ? 0x7f800000 : m;
  return __int_as_float((h & 0x80000000) | m);
}

// Obstacles of the lane: projections and duals (Steps 3, 4) at the position p3,
// and the own position row's right-hand-side sum over all obstacles, sum n (rho s
// - nu).  An obstacle that is not active (nu = 0 and n^T p above its bound by
// more than the test's error) has s = n^T p and keeps nu = 0, so that its term is
// rho n n^T p: with F = 8, where a warp's FP64 work counts, the Gram row (gr, of
// all obstacles) gives it, and a round without an active one in the warp costs no
// FP64 instruction -- most rounds, as most spheres are far from a node.  full: s
// of every obstacle is stored too (the last two iterations of a call).
template <int F, bool LAST>
__device__ __forceinline__ double fan_obstacles(const FanPos& p, const Layout& L, int nobs, const double* gr,
                                                const double* p3, double rg, double irg, bool full, double* sv,
                                                double& rp) {
  if (nobs == 0) return 0.0;
  double a[3] = {0.0, 0.0, 0.0}, s3[3] = {0.0, 0.0, 0.0}, mg = 0.0;
  const double px = p3[0], py = p3[1], pz = p3[2];
  auto project = [&](int o, double nu) {   // returns with the obstacle's s, nu stored
    double* md = p.t + L.oMd + (o >> 2) * 16 + (o & 3);
    const double n0 = md[0], n1 = md[4], n2 = md[8], bd = md[12];
    const double y = n0 * px + n1 * py + n2 * pz;
    const double s = fmax(bd, y + nu * irg);
    const double d = rg * (y - s);
    double nn = nu + d, w;
    if constexpr (F == 8) {
      if (s > bd) nn = 0.0;   // (s = y + nu / rho: the sum is 0 but for rounding)
      w = -d - nn;
    } else {
      w = rg * s - nn;
    }
    if (LAST) {
      const double ds = rg * (s - p.t[L.oS + o]);
      s3[0] += n0 * ds; s3[1] += n1 * ds; s3[2] += n2 * ds;
      acc_sq_diff(rp, y, s);
    }
    p.t[L.oS + o] = s;
    p.t[L.oNus + o] = nn;
    a[0] += n0 * w; a[1] += n1 * w; a[2] += n2 * w;
  };
  bool any = true;
  if constexpr (F == 8) {
    const float fx = fan_approx(px), fy = fan_approx(py), fz = fan_approx(pz);
    const float err = 1e-4f * (fabsf(fx) + fabsf(fy) + fabsf(fz)) + 1e-30f;
    any = false;
    for (int o0 = 0; o0 < nobs; o0 += F) {
      const int o = o0 + p.lane;
      bool need = false;
      double nu = 0.0;
      if (p.active && o < nobs) {
        nu = p.t[L.oNus + o];
        const float4 n = reinterpret_cast<const float4*>(p.t + L.oMd + L.MD)[o];
        need = LAST || full || nu != 0.0 || !(n.x * fx + n.y * fy + n.z * fz > n.w + err);
      }
      if (!__any_sync(ROWS_ALL, need)) continue;
      any = true;
      if (need) project(o, nu);
    }
    mg = gr[0] * px + gr[1] * py + gr[2] * pz;   // (0 beyond the position rows)
  } else if (p.active) {
    for (int o = p.lane; o < nobs; o += F) project(o, p.t[L.oNus + o]);
  }
  if (any) {
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      a[k] = fan_sum<F>(a[k]);
      if (p.q == k) mg += a[k];
      if (LAST) {
        s3[k] = fan_sum<F>(s3[k]);
        if (p.q == k) sv[0] += s3[k];
      }
    }
  }
  return mg;
}

// One iteration of Steps 1-4 (as admm_iteration; FP64: no refinement).
template <int F, bool LAST, bool CL>
__device__ __forceinline__ void fan_iteration(const FanPos& p, const FanMats<F>& A, const FanConst<F>& K, const Layout& L,
                                              int nobs, bool full, double& mg, double re, double rd, double rg,
                                              double irg, double ired, bool head, RowHaloPhase& hp, double& rp,
                                              double& rdl, GroupX& X) {
  typedef Rec<Quad12, 2> R;
  constexpr int NX = 12, RW = FanRows<F>::R;
  double* t = p.t;
  double *vw = p.st, *vg = p.st + FAN_VEC, *vx = p.st + 2 * FAN_VEC;
  const int q = p.q;
  double xo[RW];
  // ---- Step 1
  if constexpr (CL)
    if (!head) halo_wait<8 * NX>(p.hb, hp, 1, p.last, p.lane == 0);
#pragma unroll
  for (int m = 0; m < RW; ++m) {
    const int e = q + F * m;
    if (e < NX) vw[e] = p.hasU ? t[p.NS + R::Ex2 + e] - rd * t[R::C + e] : 0.0;
  }
  __syncwarp();
#pragma unroll
  for (int m = 0; m < RW; ++m) {
    const int e = q + F * m;
    double v = fan_dot<F, 12>(p, A.gc[m], vw) + rg * t[R::Xh + e] - t[R::Nux + e] - K.kq[m];
    if (e < NX) v += re * t[R::Z + e] - t[R::Lam + e];   // (both 0 at node 0)
    if (m == 0) v += mg;
    vg[e] = v;
  }
  __syncwarp();
#pragma unroll
  for (int m = 0; m < RW; ++m) {
    xo[m] = fan_dot<F, 16>(p, A.h[m], vg);
    vx[q + F * m] = xo[m];
  }
  __syncwarp();
#pragma unroll
  for (int m = 0; m < RW; ++m) {
    const int e = q + F * m;
    const double gx = fan_dot<F, 16>(p, A.g[m], vx);
    if (e < NX && p.hasU) {
      const double d = t[R::C + e] + gx;
      t[R::Ex1 + e] = d;
      if constexpr (CL)
        if (p.last && p.owner) st_async(p.halo0 + R::Ex1 + e, p.rank + 1, d, &p.hb->bar[0]);
    }
    if (LAST && p.active) t[R::X + e] = xo[m];
  }
  split_barrier_arrive(X.bar);
  // ---- Step 3 (before Step 2: see admm_iteration) and Step 4 for nu_x, nu_u
  // (F = 32: both lanes of a row read its variables before either stores them)
  double sv[RW], dz[RW], nus[RW], old[RW];
#pragma unroll
  for (int m = 0; m < RW; ++m) {
    nus[m] = t[R::Nux + q + F * m];
    old[m] = LAST ? t[R::Xh + q + F * m] : 0.0;
  }
  if constexpr (F == 32) __syncwarp();
#pragma unroll
  for (int m = 0; m < RW; ++m) {
    const int e = q + F * m;
    sv[m] = dz[m] = 0.0;
    const double nu = nus[m];
    const double xh = clampv(xo[m] + nu * irg, t[R::Xlo + e], t[R::Xhi + e]);
    if (LAST) {
      sv[m] = rg * (xh - old[m]);
      if (p.active && p.owner) acc_sq_diff(rp, xo[m], xh);
    }
    if (p.active) {
      t[R::Xh + e] = xh;
      t[R::Nux + e] = nu + rg * (xo[m] - xh);
    }
  }
  mg = fan_obstacles<F, LAST>(p, L, nobs, K.gr, vx, rg, irg, full, sv, rp);
  split_barrier_wait(X.bar, X.ph);
  if constexpr (CL) halo_wait<8 * NX>(p.hb, hp, 0, p.first, p.lane == 0);
  // ---- Step 2: dynamic consensus, Eq. (5), then its duals (Step 4)
  if (p.later) {   // (F = 32: a warp is one node, and takes the branch whole)
    double lams[RW], mus[RW];
#pragma unroll
    for (int m = 0; m < RW; ++m) {
      const int e = q + F * m < NX ? q + F * m : 0;
      lams[m] = t[R::Lam + e];
      mus[m] = t[R::Mu + e];
      if (LAST) old[m] = t[R::Z + e];
    }
    if constexpr (F == 32) __syncwarp();
#pragma unroll
    for (int m = 0; m < RW; ++m) {
      const int e = q + F * m;
      if (e < NX) {
        const double dd = t[R::Ex1 + e - p.NS], lam = lams[m], mu = mus[m];
        const double z = (re * xo[m] + lam + rd * dd - mu) * ired;
        if (LAST) {
          dz[m] = z - old[m];
          sv[m] += re * dz[m];
          if (p.owner) {
            acc_sq_diff(rp, xo[m], z);
            acc_sq_diff(rp, z, dd);
          }
        }
        const double mun = mu + rd * (z - dd), ex = mun + rd * z;
        t[R::Z + e] = z;
        t[R::Lam + e] = lam + re * (xo[m] - z);
        t[R::Mu + e] = mun;
        t[R::Ex2 + e] = ex;
        if constexpr (CL && !LAST)
          if (p.first && p.owner) st_async(p.halo1 + R::Ex2 + e, p.rank - 1, ex, &p.hb->bar[1]);
      }
    }
  }
  if constexpr (LAST) {
    // dual residual needs rho_dyn (z_{i+1,new} - z_{i+1,old}) from the right neighbour
    if constexpr (CL) cluster_sync();
    else __syncthreads();
    if (p.later) {
#pragma unroll
      for (int m = 0; m < RW; ++m) {
        const int e = q + F * m;
        if (e < NX) {
          t[R::Ex1 + e] = rd * dz[m];
          if constexpr (CL)
            if (p.first && p.owner) st_cluster(p.halo1 + R::Ex1 + e, p.rank - 1, rd * dz[m]);
        }
      }
    }
    if constexpr (CL) cluster_sync();
    else __syncthreads();
#pragma unroll
    for (int m = 0; m < RW; ++m) {
      const int e = q + F * m;
      if (e < NX) vw[e] = p.hasU ? t[p.NS + R::Ex1 + e] : 0.0;
    }
    __syncwarp();
#pragma unroll
    for (int m = 0; m < RW; ++m) {
      const double gz = fan_dot<F, 12>(p, A.gc[m], vw);
      if (p.active && p.owner && (q + F * m < NX || p.hasU)) acc_sq(rdl, sv[m] + gz);
    }
  }
  __syncthreads();
}

// The lane's consts and boxes (as node_setup), obstacles (as node_mirror_data and
// node_reseed), G by rows and columns, H^-1; publishes mu + rho_dyn z.
template <int F, bool CL>
__device__ __forceinline__ double fan_prepare(const FanPos& p, const Node<double, 2>& nd, const Layout& L,
                                              const ProblemDev& P, const Inst<double>& I, int b, double rad, double re,
                                              double rd, double rg, FanMats<F>& A, FanConst<F>& K, InstShared& sh) {
  typedef Rec<Quad12, 2> R;
  constexpr int NX = 12, NU = 4, RW = FanRows<F>::R, C16 = FanRows<F>::C16, C12 = FanRows<F>::C12;
  const int q = p.q;
  const bool term = p.i == p.N;
  double* t = p.t;
#pragma unroll
  for (int m = 0; m < RW; ++m) {
    const int e = q + F * m;
    double kq = 0.0, khd = 1.0, lo = 0.0, hi = 0.0;   // (node N's control rows: identity, a box at 0)
    if (e < NX) {
      const double xb = nd.dat(R::Xbar, e), w = term ? P.QNd[b * NX + e] : P.Qd[b * NX + e];
      kq = w * (xb - P.xref[b * NX + e]) + (term ? P.qN[b * NX + e] : 0.0);
      khd = w + rg + (p.i > 0 ? re : 0.0);
      lo = fmax(P.xlo[b * NX + e], xb - rad) - xb;
      hi = fmin(P.xhi[b * NX + e], xb + rad) - xb;
      if (p.i == 0) lo = hi = P.xinit[b * NX + e] - xb;
      else if (term && (sh.tmask >> e & 1u)) lo = hi = P.xtarget[b * NX + e] - xb;
    } else if (p.hasU) {
      const int j = e - NX;
      const double ub = nd.dat(R::Ubar, j), w = P.Rd[b * NU + j];
      kq = w * (ub - P.uref[b * NU + j]);
      khd = w + rg;
      lo = fmax(P.ulo[b * NU + j], ub - rad) - ub;
      hi = fmin(P.uhi[b * NU + j], ub + rad) - ub;
    }
    K.kq[m] = p.active ? kq : 0.0;
    K.khd[m] = khd;
    if (p.active) {
      t[R::Xlo + e] = lo;
      t[R::Xhi + e] = hi;
    }
  }
  // obstacles and their Gram matrix (xx, xy, xz, yy, yz, zz)
  double gr[6] = {0, 0, 0, 0, 0, 0}, a[3] = {0, 0, 0}, mg = 0.0;
  if (I.nobs > 0) {
    if (p.active) {
      const double x0 = nd.dat(R::Xbar, 0), x1 = nd.dat(R::Xbar, 1), x2 = nd.dat(R::Xbar, 2);
      for (int o = p.lane; o < I.nobs; o += F) {
        const double* c = &P.obs_c[((long long)b * P.max_obs + o) * 3];
        const double d0 = x0 - c[0], d1 = x1 - c[1], d2 = x2 - c[2];
        double n0 = d0, n1 = d1, n2 = d2, nn = sqrt(d0 * d0 + d1 * d1 + d2 * d2);
        if (nn < 1e-12) { n0 = 0.0; n1 = 0.0; n2 = 1.0; nn = 1.0; }
        const double inn = 1.0 / nn;
        n0 *= inn; n1 *= inn; n2 *= inn;
        const double bd = -(n0 * d0 + n1 * d1 + n2 * d2) + P.obs_r[(long long)b * P.max_obs + o];
        double* md = t + L.oMd + (o >> 2) * 16 + (o & 3);
        md[0] = n0; md[4] = n1; md[8] = n2; md[12] = bd;
        reinterpret_cast<float4*>(t + L.oMd + L.MD)[o] = float4{(float)n0, (float)n1, (float)n2, (float)bd};
        const double s = fmax(bd, n0 * t[R::Xh] + n1 * t[R::Xh + 1] + n2 * t[R::Xh + 2]);
        t[L.oS + o] = s;
        const double w = rg * s - t[L.oNus + o];
        a[0] += n0 * w; a[1] += n1 * w; a[2] += n2 * w;
        gr[0] += n0 * n0; gr[1] += n0 * n1; gr[2] += n0 * n2; gr[3] += n1 * n1; gr[4] += n1 * n2; gr[5] += n2 * n2;
      }
    }
#pragma unroll
    for (int k = 0; k < 6; ++k) gr[k] = rg * fan_sum<F>(gr[k]);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      a[k] = fan_sum<F>(a[k]);
      if (q == k) mg = a[k];
    }
  }
  // G by rows through the staging: columns in, the own rows out
  double* G = p.st + 3 * FAN_VEC;
#pragma unroll
  for (int m = 0; m < RW; ++m)
#pragma unroll
    for (int k = 0; k < C12; ++k) G[(k + C12 * p.half) * 16 + q + F * m] = A.gc[m][k];
  __syncwarp();
#pragma unroll
  for (int m = 0; m < RW; ++m) {
    const int e = q + F * m;
#pragma unroll
    for (int c = 0; c < C16; ++c) {
      A.g[m][c] = e < NX ? G[(e < NX ? e : 0) * 16 + C16 * p.half + c] : 0.0;
      A.h[m][c] = 0.0;
    }
  }
  // H = diag + rho_dyn G^T G + Gram, own rows
#pragma unroll 2
  for (int k = 0; k < NX; ++k) {
#pragma unroll
    for (int m = 0; m < RW; ++m) {
      const double f = G[k * 16 + q + F * m];
#pragma unroll
      for (int c = 0; c < C16; ++c) A.h[m][c] += f * G[k * 16 + C16 * p.half + c];
    }
  }
#pragma unroll
  for (int m = 0; m < RW; ++m)
#pragma unroll
    for (int c = 0; c < C16; ++c) A.h[m][c] = rd * A.h[m][c] + (c + C16 * p.half == q + F * m ? K.khd[m] : 0.0);
  K.gr[0] = q == 0 ? gr[0] : q == 1 ? gr[1] : q == 2 ? gr[2] : 0.0;
  K.gr[1] = q == 0 ? gr[1] : q == 1 ? gr[3] : q == 2 ? gr[4] : 0.0;
  K.gr[2] = q == 0 ? gr[2] : q == 1 ? gr[4] : q == 2 ? gr[5] : 0.0;
#pragma unroll
  for (int c = 0; c < 3; ++c) A.h[0][c] += p.half == 0 ? K.gr[c] : 0.0;
  // inverse by Gauss-Jordan, the pivot row handed around through the staging (two
  // buffers in turn); F pivots per pass, row groups and columns rotating by F in
  // between, so that the register indexes stay fixed
  bool ok = true;
#pragma unroll 1
  for (int g = 0; g < RW; ++g) {
#pragma unroll
    for (int o = 0; o < 16 / RW; ++o) {
      constexpr int H = C16;
      double* row = p.st + (o & 1) * FAN_VEC;
      if (q == o) {
#pragma unroll
        for (int c = 0; c < H; ++c) row[c + H * p.half] = A.h[0][c];
      }
      __syncwarp();
      double piv = row[o];
      if (!(piv > 0.0)) { ok = false; piv = 1.0; }
      const double d = 1.0 / piv;
#pragma unroll
      for (int m = 0; m < RW; ++m) {
        double f = A.h[m][o % H];
        if constexpr (F == 32) f = __shfl_sync(ROWS_ALL, f, p.q + 16 * (o / H));
        const bool mine = m == 0 && q == o;
        const double fd = mine ? -d : f * d;   // the pivot row: row * d
#pragma unroll
        for (int c = 0; c < H; ++c) {
          const bool pc = c == o % H && p.half == o / H;
          const double h0 = mine || pc ? 0.0 : A.h[m][c];
          A.h[m][c] = pc ? -fd : h0 - fd * row[c + H * p.half];
        }
      }
    }
    if constexpr (RW == 2) {
#pragma unroll
      for (int c = 0; c < 8; ++c) {   // (row 0, row 1) x (columns low, high) -> swapped both ways
        const double lo0 = A.h[0][c], hi0 = A.h[0][c + 8];
        A.h[0][c] = A.h[1][c + 8];
        A.h[0][c + 8] = A.h[1][c];
        A.h[1][c] = hi0;
        A.h[1][c + 8] = lo0;
      }
    }
  }
  if (!ok) atomicOr(&sh.fail, 1);
  if (p.later) {
#pragma unroll
    for (int m = 0; m < RW; ++m) {
      const int e = q + F * m;
      if (e < NX) {
        const double v = t[R::Mu + e] + rd * t[R::Z + e];
        t[R::Ex2 + e] = v;
        if constexpr (CL)
          if (p.first && p.owner) st_cluster(p.halo1 + R::Ex2 + e, p.rank - 1, v);
      }
    }
  }
  if (!p.active) {
#pragma unroll
    for (int m = 0; m < RW; ++m)
#pragma unroll
      for (int c = 0; c < C16; ++c) A.h[m][c] = 0.0;
  }
  __syncthreads();
  return mg;
}

template <int F, bool CL_>
struct FanEngine {
  typedef Quad12 M;
  typedef double T;
  static constexpr bool GROUP = false, CL = CL_;
  typedef FanPos Pos;
  typedef FanMats<F> Mats;
  typedef FanConst<F> Const;
  typedef Rec<Quad12, 2> R;
  static constexpr int RW = FanRows<F>::R;
  __device__ static __forceinline__ Pos place(const ProblemDev& P, const Layout& L, unsigned char* smem, int b,
                                              Node<double, 2>& nd, Node<double, 2>& ndd, bool& dact) {
    Pos p;
    p.rank = CL ? cluster_rank() : 0u;
    const int base = CL ? (int)p.rank * L.chunk : 0, halo = CL ? 1 : 0;
    const int il = (int)threadIdx.x / F;
    p.N = P.N[b];
    p.lane = (int)threadIdx.x % F;
    p.q = p.lane & 15;
    p.half = F == 32 ? p.lane >> 4 : 0;
    p.owner = p.half == 0;
    p.i = base + il;
    p.active = il < L.chunk && p.i <= p.N;
    p.hasU = p.active && p.i < p.N;
    p.later = p.active && p.i >= 1;
    p.NS = L.NS;
    double* t = (double*)smem;
    p.t = t + ((p.active ? il : 0) + halo) * L.NS;
    p.st = (double*)(smem + L.oX) + il * FAN_STAGE;   // (every thread's warp has staging)
    p.first = CL && p.active && il == 0 && p.rank > 0;
    p.last = CL && p.hasU && il == L.chunk - 1;
    p.halo0 = t;
    p.halo1 = t + (L.chunk + 1) * L.NS;
    nd.t = t + (halo - base) * L.NS;
    nd.d = (double*)(smem + L.tbytes) + (halo - base) * L.DS;
    nd.c = nullptr;
    nd.S = L.S; nd.NS = L.NS; nd.DS = L.DS; nd.N = p.N;
    ndd = nd;
    nd.i = p.active ? p.i : base;
    ndd.i = base + (int)threadIdx.x;
    dact = (int)threadIdx.x < L.chunk && ndd.i <= p.N;
    return p;
  }
  // the own columns of G: one forward-mode pass per direction
  __device__ static __forceinline__ void jacobians(const Pos& p, const Node<double, 2>& nd, Mats& A, const double* prm,
                                                   const Step3<double>& hs, const Layout&) {
    double xt[12], ut[4];
#pragma unroll
    for (int j = 0; j < 12; ++j) xt[j] = nd.dat(R::Xbar, j);
#pragma unroll
    for (int j = 0; j < 4; ++j) ut[j] = p.hasU ? nd.dat(R::Ubar, j) : 1.0;
#pragma unroll 1
    for (int m = 0; m < RW; ++m) {
      double col[12];
      rk4_jvp<Quad12, double>(prm, hs, xt, ut, p.q + F * m, col);
#pragma unroll
      for (int k = 0; k < Mats::C12; ++k) {
        if constexpr (RW == 2) A.gc[0][k] = A.gc[1][k];
        const double v = F == 32 && p.half ? col[(k + 6) % 12] : col[k];
        A.gc[RW - 1][k] = p.hasU ? v : 0.0;
      }
    }
  }
  __device__ static __forceinline__ double prepare(const Pos& p, const Node<double, 2>& nd, const Layout& L,
                                                   const ProblemDev& P, const Inst<double>& I, int b, double rad,
                                                   double re, double rd, double rg, Mats& A, Const& K, InstShared& sh) {
    return fan_prepare<F, CL>(p, nd, L, P, I, b, rad, re, rd, rg, A, K, sh);
  }
  __device__ static __forceinline__ void admm(const Pos& p, const Mats& A, const Const& K, const Layout& L,
                                              const Inst<double>& I, double mg, double re, double rd, double rg,
                                              int iters, InstShared& sh, double* res, GroupShared*, GroupX& X,
                                              const ProblemDev&, RowHaloPhase& hp) {
    const double irg = 1.0 / rg, ired = 1.0 / (re + rd);
    double rp = 0.0, rdl = 0.0;
    for (int it = 0; it + 1 < iters; ++it)
      fan_iteration<F, false, CL>(p, A, K, L, I.nobs, it + 2 == iters, mg, re, rd, rg, irg, ired, it == 0, hp, rp,
                                  rdl, X);
    fan_iteration<F, true, CL>(p, A, K, L, I.nobs, true, mg, re, rd, rg, irg, ired, iters == 1, hp, rp, rdl, X);
    reduce_residuals(sh, rp, rdl, res);
  }
  __device__ static __forceinline__ void push_hat(const Pos& p) {
    if (p.first && p.owner)
#pragma unroll
      for (int m = 0; m < RW; ++m)
        if (p.q + F * m < 12) st_cluster(p.halo1 + R::Xh + p.q + F * m, p.rank - 1, p.t[R::Xh + p.q + F * m]);
  }
  __device__ static __forceinline__ void linear_model(const Pos& p, const Mats& A, const Layout&, double& lin1, double& st) {
    double* v = p.st;
#pragma unroll
    for (int m = 0; m < RW; ++m) {
      const int e = p.q + F * m;
      v[e] = p.active ? p.t[R::Xh + e] : 0.0;
      st = fmax(st, fabs(v[e]));
    }
    __syncwarp();
    double gx[RW];
#pragma unroll
    for (int m = 0; m < RW; ++m) gx[m] = fan_dot<F, 16>(p, A.g[m], v);
    if (p.hasU && p.owner) {
#pragma unroll
      for (int m = 0; m < RW; ++m) {
        const int e = p.q + F * m;
        if (e < 12) lin1 += fabs(p.t[R::C + e] - p.t[p.NS + R::Xh + e] + gx[m]);
      }
    }
  }
};

template <int F, bool CL>
__global__ void __launch_bounds__(FAN_THREADS, 1) scp_fan_kernel(ProblemDev P, Layout L, const double* x0,
                                                                 const double* u0, double* xout, double* uout,
                                                                 ucn_scp_stats* stats, int* status_out) {
  const int k = CL ? (int)blockIdx.x / L.csize : (int)blockIdx.x;
  const int b = P.order ? P.order[k] : k;
  scp_split_body<FanEngine<F, CL>>(P, L, x0, u0, xout, uout, stats, status_out, b);
}

}  // namespace ucn
