// Row kernel of the FP32 path for the quadrotors (12-state, 16 rows; quaternion,
// 17 rows): four lanes of a warp share a time node and keep its matrices in
// registers for a whole ADMM call.
//
// Lane q owns the rows e = q, q + 4, q + 8, q + 12 of xi = (x, u); a 17th row is
// carried by all four lanes alike.  It holds its rows of G = [A B] and of H^-1
// with the columns in its own order: slot s of a group of four columns is the
// column of lane q ^ s.  Then a gather of a vector (slot s <- shfl_xor(own, s))
// and the sum of partial products over the lanes (own += shfl_xor(slot s, s))
// take three shuffles per group and no selects, G^T w needs no second copy of G
// by columns, and every product is a run of two-wide FMAs over slot pairs.
//
// Why: the lane kernel that reads A, B from shared memory (four times per
// iteration) and walks each node's obstacles on three of its lanes spent an
// ADMM iteration on those reads.  Here an iteration touches shared memory for
// the node's own variables alone; the obstacles are split over the lanes with
// their right-hand side summed when the duals change, and their Gram matrix is
// summed once per SCP iteration.
//
// Measured on GB300 (fused solves, before -> with this kernel): 1023 quadrotors
// of 40..120 nodes, 10 x 200 iterations, 207 -> 37.3 ms; one of 50 nodes 8.56 ->
// 2.73 ms; 256 quaternion quadrotors of 50 nodes, 20 x 100, 27.1 -> 7.34 ms; the
// ADMM call on 511 quadrotors, 100 iterations, 8.06 -> 1.07 ms.  The error against
// FP64 is as before (medians over 64 to 128 batches 2.0e-7 to 2.4e-7).  What bounds it: latency at 8
// warps per SM -- issue slots 45% used in the ADMM loop; stalls at the two
// barriers of an iteration, instruction fetch and fixed-latency dependencies.
//
// An instance may be split over the CTAs of a thread-block cluster (CL), `chunk`
// consecutive nodes each.  Only boundary nodes talk across CTAs: they store
// their exchange vectors into the neighbour's halo records in distributed
// shared memory, asynchronously, and the neighbour's boundary node waits for the
// bytes on an mbarrier of its own; the iteration's barriers stay the CTA's (121
// nodes on two CTAs: 1.79 us per iteration with cluster barriers, 1.75 so).
#pragma once
#include "ucn_kernels.cuh"

namespace ucn {

// CTA size caps of the two register classes: up to 255 registers per thread
// (64 nodes), or 168 (96 nodes; two CTAs of 48 nodes per SM).
constexpr int ROWS_THREADS = 256, ROWS_WIDE_THREADS = 384;
constexpr unsigned ROWS_ALL = 0xffffffffu;

// Models the row kernel serves.  The 6-DOF lander is not among them: in one batch
// of 1000 in sixteen an FP32 solve of it meets a decision that rounding turns, and
// its results here were up to 5e-5 (normwise) from the one-thread kernel's.
template <class M> struct RowModel { static constexpr bool value = IsQuad<M>::value; };

// a * b + c on two floats at once (one issue slot).
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
  unsigned long long d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;"
      : "=l"(d)
      : "l"(reinterpret_cast<unsigned long long&>(a)), "l"(reinterpret_cast<unsigned long long&>(b)),
        "l"(reinterpret_cast<unsigned long long&>(c)));
  return reinterpret_cast<float2&>(d);
}
__device__ __forceinline__ float rows_xor(float v, int s) { return __shfl_xor_sync(ROWS_ALL, v, s); }
__device__ __forceinline__ float rows_from(float v, int lane) { return __shfl_sync(ROWS_ALL, v, lane, 4); }
__device__ __forceinline__ float rows_sum(float v) {
  v += rows_xor(v, 1);
  return v + rows_xor(v, 2);
}
// The q-th of four values.
__device__ __forceinline__ float sel4(float a, float b, float c, float d, int q) {
  const float lo = (q & 1) ? b : a, hi = (q & 1) ? d : c;
  return (q & 2) ? hi : lo;
}

__device__ __forceinline__ unsigned cluster_rank() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}

// Arrival of the neighbours' boundary values in the halo records: [0] Ex1 from the
// CTA before, [1] Ex2 from the one after; phases completed (every thread's copy).
// A sender is at most one iteration ahead of its receiver, and sends an exchange
// vector only when the receiver has used the last one: Ex1 of iteration k + 1
// follows the receiver's Ex2 of iteration k, which follows its use of Ex1 of k,
// and the other way round.  The last iteration of a call sends no Ex2: the next
// call's set-up does, before a cluster barrier.
struct RowHalo {
  unsigned long long bar[2];
  int fail;
};
struct RowHaloPhase {
  unsigned n[2];
};
// Waits for exchange w if this thread's node uses it (`on`), then re-arms it (one
// lane, `arm`).  Warps call it whole.
template <unsigned BYTES>
__device__ __forceinline__ void halo_wait(RowHalo* hb, RowHaloPhase& ph, int w, bool on, bool arm) {
  if (on && !tx_wait(&hb->bar[w], ph.n[w] & 1u)) hb->fail = 1;
  __syncwarp();
  if (on && arm) tx_arm(&hb->bar[w], BYTES);
  ph.n[w]++;
}
// Start of a cluster kernel, by thread 0 (a cluster barrier follows).
template <unsigned BYTES>
__device__ __forceinline__ void halo_init(RowHalo* hb) {
  hb->fail = 0;
  for (int w = 0; w < 2; ++w) {
    tx_init(&hb->bar[w]);
    tx_arm(&hb->bar[w], BYTES);
  }
}

// One thread's place: its node, its lane, and whether it takes part.
struct RowPos {
  int i, N, q;
  bool active, hasU, later;   // i <= N; i < N; 1 <= i <= N
  float* tp;                  // the lane's base in the node's record
  int NS;
  // cluster: CTA rank and whether this node is the first / last of its CTA with
  // a neighbour beyond, and the lane's base in the halo records
  unsigned rank;
  bool first, last;
  float *halo0, *halo1;       // records before the first and after the last node
  RowHalo* hb;                // arrival of the neighbours' boundary values
};

template <class M>
struct RowMats {
  static constexpr int NX = M::NX, NN = M::NX + M::NU, RX = pad4(NX) / 4;
  static constexpr bool EX = NN == 17;
  float2 g[RX][4][2], h[4][4][2];
  float gx[RX], hx[4], hxx;   // column 16 of G and H^-1 (= row 16 of H^-1)
};

// Per-SCP-iteration constants of the lane's rows: cost gradient, diagonal of H
// without the A/B Gram terms, the obstacles' Gram row (slot order).
template <class M>
struct RowConst {
  static constexpr int R = RowMats<M>::EX ? 5 : 4;
  float kq[R], khd[R];
  float gram[4];
};

// The lane's ADMM variables: in registers for the length of an ADMM call
// (REG), or in the record.  Row 16 (EX) is element 16 of the record, kept alike
// in all four lanes.
template <class M, bool REG>
struct RowState;
template <class M>
struct RowState<M, true> {
  static constexpr bool reg = true;
  typedef Rec<M, 2> R;
  static constexpr int RX = RowMats<M>::RX, RE = RowConst<M>::R;
  mutable float hv[RE], nv[RE], lv[RE], uv[RE], zv[RX], lamv[RX], muv[RX], cv[RX];
  __device__ __forceinline__ static int off(int m, int q) { return m < 4 ? 4 * m : 16 - q; }
  __device__ __forceinline__ void load(const RowPos& p) {
#pragma unroll
    for (int m = 0; m < RE; ++m) {
      const int e = off(m, p.q);
      hv[m] = p.tp[R::Xh + e]; nv[m] = p.tp[R::Nux + e]; lv[m] = p.tp[R::Xlo + e]; uv[m] = p.tp[R::Xhi + e];
    }
#pragma unroll
    for (int m = 0; m < RX; ++m) {
      zv[m] = p.tp[R::Z + 4 * m]; lamv[m] = p.tp[R::Lam + 4 * m]; muv[m] = p.tp[R::Mu + 4 * m]; cv[m] = p.tp[R::C + 4 * m];
    }
  }
  __device__ __forceinline__ void store(const RowPos& p) const {
    if (!p.active) return;
#pragma unroll
    for (int m = 0; m < RE; ++m) {
      const int e = off(m, p.q);
      p.tp[R::Xh + e] = hv[m]; p.tp[R::Nux + e] = nv[m];
    }
#pragma unroll
    for (int m = 0; m < RX; ++m) { p.tp[R::Z + 4 * m] = zv[m]; p.tp[R::Lam + 4 * m] = lamv[m]; p.tp[R::Mu + 4 * m] = muv[m]; }
  }
  __device__ __forceinline__ float hat(int m) const { return hv[m]; }
  __device__ __forceinline__ float nu(int m) const { return nv[m]; }
  __device__ __forceinline__ float lo(int m) const { return lv[m]; }
  __device__ __forceinline__ float hi(int m) const { return uv[m]; }
  __device__ __forceinline__ float z(int m) const { return zv[m]; }
  __device__ __forceinline__ float lam(int m) const { return lamv[m]; }
  __device__ __forceinline__ float mu(int m) const { return muv[m]; }
  __device__ __forceinline__ float c(int m) const { return cv[m]; }
  __device__ __forceinline__ void set_box(int m, float h, float n, bool) const { hv[m] = h; nv[m] = n; }
  __device__ __forceinline__ void set_dyn(int m, float z_, float l, float u) const { zv[m] = z_; lamv[m] = l; muv[m] = u; }
};
template <class M>
struct RowState<M, false> {
  static constexpr bool reg = false;
  typedef Rec<M, 2> R;
  static constexpr int RX = RowMats<M>::RX, RE = RowConst<M>::R;
  float* tp;
  int q;
  __device__ __forceinline__ int off(int m) const { return m < 4 ? 4 * m : 16 - q; }
  __device__ __forceinline__ void load(const RowPos& p) { tp = p.tp; q = p.q; }
  __device__ __forceinline__ void store(const RowPos&) const {}
  __device__ __forceinline__ float hat(int m) const { return tp[R::Xh + off(m)]; }
  __device__ __forceinline__ float nu(int m) const { return tp[R::Nux + off(m)]; }
  __device__ __forceinline__ float lo(int m) const { return tp[R::Xlo + off(m)]; }
  __device__ __forceinline__ float hi(int m) const { return tp[R::Xhi + off(m)]; }
  __device__ __forceinline__ float z(int m) const { return tp[R::Z + 4 * m]; }
  __device__ __forceinline__ float lam(int m) const { return tp[R::Lam + 4 * m]; }
  __device__ __forceinline__ float mu(int m) const { return tp[R::Mu + 4 * m]; }
  __device__ __forceinline__ float c(int m) const { return tp[R::C + 4 * m]; }
  // (row 16: the four lanes of a node store the same value)
  __device__ __forceinline__ void set_box(int m, float h, float n, bool on) const {
    if (on) { tp[R::Xh + off(m)] = h; tp[R::Nux + off(m)] = n; }
  }
  __device__ __forceinline__ void set_dyn(int m, float z_, float l, float u) const {
    tp[R::Z + 4 * m] = z_; tp[R::Lam + 4 * m] = l; tp[R::Mu + 4 * m] = u;
  }
};

// ------------------------------------------------------------------ products
// A vector in slot order from the lanes' own rows.
template <int RG>
__device__ __forceinline__ void rows_gather(const float* own, float2 (*v)[2]) {
#pragma unroll
  for (int m = 0; m < RG; ++m) {
    v[m][0] = {own[m], rows_xor(own[m], 1)};
    v[m][1] = {rows_xor(own[m], 2), rows_xor(own[m], 3)};
  }
}
// out[m] = row m of G times the vector v (slot order), vx its element 16.
template <class M>
__device__ __forceinline__ void rows_G(const RowMats<M>& A, const float2 (*v)[2], float vx, float* out) {
#pragma unroll
  for (int m = 0; m < RowMats<M>::RX; ++m) {
    float2 a = {0.0f, 0.0f};
    if constexpr (RowMats<M>::EX) a.x = A.gx[m] * vx;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      a = fma2(A.g[m][k][0], v[k][0], a);
      a = fma2(A.g[m][k][1], v[k][1], a);
    }
    out[m] = a.x + a.y;
  }
}
// out = G^T w (own rows; element 16 last), w the lanes' own rows of an x-vector.
template <class M>
__device__ __forceinline__ void rows_GT(const RowMats<M>& A, const float* w, float* out) {
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    float2 p0 = {0.0f, 0.0f}, p1 = {0.0f, 0.0f};
#pragma unroll
    for (int m = 0; m < RowMats<M>::RX; ++m) {
      const float2 ww = {w[m], w[m]};
      p0 = fma2(A.g[m][k][0], ww, p0);
      p1 = fma2(A.g[m][k][1], ww, p1);
    }
    out[k] = (p0.x + rows_xor(p0.y, 1)) + (rows_xor(p1.x, 2) + rows_xor(p1.y, 3));
  }
  if constexpr (RowMats<M>::EX) {
    float p = 0.0f;
#pragma unroll
    for (int m = 0; m < RowMats<M>::RX; ++m) p += A.gx[m] * w[m];
    out[4] = rows_sum(p);
  }
}
// out = H^-1 g (own rows; element 16 last), g the lanes' own rows.
template <class M>
__device__ __forceinline__ void rows_solve(const RowMats<M>& A, const float* g, float* out) {
  float2 v[4][2];
  rows_gather<4>(g, v);
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    float2 a = {0.0f, 0.0f};
    if constexpr (RowMats<M>::EX) a.x = A.hx[m] * g[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      a = fma2(A.h[m][k][0], v[k][0], a);
      a = fma2(A.h[m][k][1], v[k][1], a);
    }
    out[m] = a.x + a.y;
  }
  if constexpr (RowMats<M>::EX) {
    float p = 0.0f;
#pragma unroll
    for (int m = 0; m < 4; ++m) p += A.hx[m] * g[m];
    out[4] = rows_sum(p) + A.hxx * g[4];
  }
}

// Whether row m of the lane is a state row (all are but the last group's).
template <class M>
__device__ __forceinline__ bool rows_is_x(int m, int q) {
  return 4 * m + 3 < M::NX || (m < 4 && 4 * m + q < M::NX);
}

// ------------------------------------------------------------------ mirror sets in the ADMM loop
// Projections and duals of the lane's obstacles (Steps 3, 4) at the
// node's new position, and the sum of their right-hand-side terms n (rho s - nu)
// for the next Step 1; `mg` receives that of the lane's position row (lane q <
// 3: row q).  rp, sv as in node_mirrors (last iteration).
template <class M, bool LAST>
__device__ __forceinline__ float rows_obstacles(const RowPos& p, const Layout& L, int nobs, const float* xo, float rg,
                                                float irg, float* sv, DF& rp) {
  const float px = rows_from(xo[0], 0), py = rows_from(xo[0], 1), pz = rows_from(xo[0], 2);
  float a0 = 0.0f, a1 = 0.0f, a2 = 0.0f, s0 = 0.0f, s1 = 0.0f, s2 = 0.0f;
  if (p.active) {
    float* md = p.tp + L.oMd;
    float* ms = p.tp + L.oS;
    float* mn = p.tp + L.oNus;
    for (int o = p.q; o < nobs; o += 4, md += 16, ms += 4, mn += 4) {
      const float n0 = md[0], n1 = md[4], n2 = md[8], bd = md[12], nu = mn[0];
      const float y = n0 * px + n1 * py + n2 * pz;
      const float s = fmaxf(bd, y + nu * irg);
      const float nn = nu + rg * (y - s);
      if (LAST) {
        const float ds = rg * (s - ms[0]);
        s0 += n0 * ds; s1 += n1 * ds; s2 += n2 * ds;
        acc_sq_diff(rp, y, s);
      }
      ms[0] = s;
      mn[0] = nn;
      const float a = rg * s - nn;
      a0 += n0 * a; a1 += n1 * a; a2 += n2 * a;
    }
  }
  if (LAST) {
    s0 = rows_sum(s0); s1 = rows_sum(s1); s2 = rows_sum(s2);
    sv[0] += sel4(s0, s1, s2, 0.0f, p.q);
  }
  a0 = rows_sum(a0); a1 = rows_sum(a1); a2 = rows_sum(a2);
  return sel4(a0, a1, a2, 0.0f, p.q);
}

// ------------------------------------------------------------------ one ADMM iteration
// Steps 1-4 (Sec. III-B) as admm_iteration, lane-parallel.  Every thread calls
// it; threads without a node carry zero matrices and store nothing.  GROUP: see
// admm_iteration (12-state quadrotor).
template <class M, bool LAST, bool GROUP, bool CL, class ST>
__device__ __forceinline__ void rows_iteration(const RowPos& p, const RowMats<M>& A, const RowConst<M>& K, const ST& S,
                                               const Layout& L, const Inst<float>& I, float& mg, float re, float rd,
                                               float rg, float irg, float ired, bool head, RowHaloPhase& hp, DF& rp,
                                               DF& rdl, GroupShared* G, GroupX& X, const ProblemDev& P) {
  typedef Rec<M, 2> R;
  constexpr int RX = RowMats<M>::RX, RE = RowConst<M>::R;
  constexpr bool EX = RowMats<M>::EX;
  float* tp = p.tp;
  const int q = p.q;
  float xo[RE];
  // the constants of the lane's rows: registers, or the record where those are short
  auto at = [&](int field, int m) { return tp[field + (m < 4 ? 4 * m : 16 - q)]; };
  auto kq = [&](int m) { return ST::reg ? K.kq[m] : at(R::Kq, m); };
  auto khd = [&](int m) { return ST::reg ? K.khd[m] : at(R::Khd, m); };
  auto gram = [&](int s) { return ST::reg ? K.gram[s] : tp[R::Gr + 4 * s]; };
  // ---- Step 1
  if constexpr (CL)
    if (!head) halo_wait<4 * M::NX>(p.hb, hp, 1, p.last, q == 0);
  {
    float g[RE];
    {
      float w[RX];
#pragma unroll
      for (int m = 0; m < RX; ++m) w[m] = p.hasU ? tp[p.NS + R::Ex2 + 4 * m] - rd * S.c(m) : 0.0f;
      rows_GT<M>(A, w, g);
    }
#pragma unroll
    for (int m = 0; m < RE; ++m) {
      float v = rg * S.hat(m) - S.nu(m) - kq(m);
      if (m < RX && rows_is_x<M>(m, q)) v += re * S.z(m) - S.lam(m);   // (both 0 at node 0)
      g[m] += v;
    }
    g[0] += mg;
    rows_solve<M>(A, g, xo);
    // one refinement step: the residual with H applied from G, the diagonal and
    // the mirror Gram terms
    float2 v[4][2];
    rows_gather<4>(xo, v);
    float t[RX], r[RE];
    rows_G<M>(A, v, EX ? xo[RE - 1] : 0.0f, t);
#pragma unroll
    for (int m = 0; m < RX; ++m) t[m] *= rd;
    rows_GT<M>(A, t, r);
#pragma unroll
    for (int m = 0; m < RE; ++m) r[m] = g[m] - (khd(m) * xo[m] + r[m]);
    r[0] -= (gram(0) * v[0][0].x + gram(1) * v[0][0].y) + (gram(2) * v[0][1].x + gram(3) * v[0][1].y);
    float dx[RE];
    rows_solve<M>(A, r, dx);
#pragma unroll
    for (int m = 0; m < RE; ++m) xo[m] += dx[m];
    if constexpr (GROUP) {
      // the arguments of u_0, as early as they are known: node 0 is the first four
      // lanes; lane l hands over control l mod 4
      if (threadIdx.x < 32) {
        const double a = G->ub[q] + (double)(xo[3] + S.nu(3) * irg);
        group_publish(P, G, X, __shfl_sync(ROWS_ALL, a, (int)threadIdx.x & 3));
      }
    }
    // linearised propagation d_dyn,i = A x + B u + c_i, published to node i+1
    rows_gather<4>(xo, v);
    rows_G<M>(A, v, EX ? xo[RE - 1] : 0.0f, t);
    if (p.hasU) {
#pragma unroll
      for (int m = 0; m < RX; ++m) {
        t[m] += S.c(m);
        tp[R::Ex1 + 4 * m] = t[m];
      }
      if constexpr (CL)
        if (p.last) {
#pragma unroll
          for (int m = 0; m < RX; ++m)
            if (rows_is_x<M>(m, q)) st_async(p.halo0 + R::Ex1 + 4 * m, p.rank + 1, t[m], &p.hb->bar[0]);
        }
    }
    if (p.active && LAST) {
#pragma unroll
      for (int m = 0; m < RE; ++m) tp[R::X + (m < 4 ? 4 * m : 16 - q)] = xo[m];
    }
  }
  // Step 3 before Step 2, between the arrival (Ex1 published) and the wait
  split_barrier_arrive(X.bar);
  float sv[RE], dz[RX];
  if (LAST) {
#pragma unroll
    for (int m = 0; m < RE; ++m) sv[m] = 0.0f;
  }
  // ---- Step 3: projections onto the boxes (Eq. (7)) and Step 4 for nu_x, nu_u
  // (row 16 lies in the record for all four lanes: each reads it before any stores it)
  float nu16 = 0.0f, hat16 = 0.0f;
  if constexpr (EX) {
    nu16 = S.nu(RE - 1);
    hat16 = S.hat(RE - 1);
    __syncwarp();
  }
#pragma unroll
  for (int m = 0; m < RE; ++m) {
    const float nu = m < 4 ? S.nu(m) : nu16, arg = xo[m] + nu * irg;
    if constexpr (GROUP) {
      if (m == 3 && p.i == 0) continue;   // the consensus sets it
    }
    const float xh = clampv(arg, S.lo(m), S.hi(m));
    if (LAST) {
      // row 16 counts once; a control row at node N is zero throughout
      if (p.active && (m < 4 || q == 0)) acc_sq_diff(rp, xo[m], xh);
      sv[m] += rg * (xh - (m < 4 ? S.hat(m) : hat16));
    }
    S.set_box(m, xh, nu + rg * (xo[m] - xh), p.active);
  }
  mg = rows_obstacles<M, LAST>(p, L, I.nobs, xo, rg, irg, sv, rp);
  split_barrier_wait(X.bar, X.ph);
  if constexpr (CL) halo_wait<4 * M::NX>(p.hb, hp, 0, p.first, q == 0);
  // ---- Step 2: dynamic consensus, Eq. (5), then its duals (Step 4)
#pragma unroll
  for (int m = 0; m < RX; ++m) dz[m] = 0.0f;
  if (p.later) {
#pragma unroll
    for (int m = 0; m < RX; ++m)
      if (rows_is_x<M>(m, q)) {
        const float dd = tp[R::Ex1 + 4 * m - p.NS];
        const float lam = S.lam(m), mu = S.mu(m);
        const float z = (re * xo[m] + lam + rd * dd - mu) * ired;
        if (LAST) {
          dz[m] = z - S.z(m);
          sv[m] += re * dz[m];
          acc_sq_diff(rp, xo[m], z);
          acc_sq_diff(rp, z, dd);
        }
        const float mun = mu + rd * (z - dd);
        S.set_dyn(m, z, lam + re * (xo[m] - z), mun);
        tp[R::Ex2 + 4 * m] = mun + rd * z;
        if constexpr (CL && !LAST)
          if (p.first) st_async(p.halo1 + R::Ex2 + 4 * m, p.rank - 1, mun + rd * z, &p.hb->bar[1]);
      }
  }
  if constexpr (GROUP) {
    if (threadIdx.x < 32) {
      const double sum = group_collect(P, G, X);
      if (p.i == 0 && p.active) {
        const double v = group_mean(G, sum, q);
        G->u0[q] = v;
        const float uh = (float)(v - G->ub[q]);
        const float nu = S.nu(3);
        if (LAST) { sv[3] += rg * (uh - S.hat(3)); acc_sq_diff(rp, xo[3], uh); }
        S.set_box(3, uh, nu + rg * (xo[3] - uh), true);
      }
    }
    group_advance(P, X);
  }
  if constexpr (LAST) {
    // dual residual needs rho_dyn (z_{i+1,new} - z_{i+1,old}) from the right neighbour
    if constexpr (CL) cluster_sync();
    else __syncthreads();
    if (p.later) {
#pragma unroll
      for (int m = 0; m < RX; ++m)
        if (rows_is_x<M>(m, q)) {
          tp[R::Ex1 + 4 * m] = rd * dz[m];
          if constexpr (CL)
            if (p.first) st_cluster(p.halo1 + R::Ex1 + 4 * m, p.rank - 1, rd * dz[m]);
        }
    }
    if constexpr (CL) cluster_sync();
    else __syncthreads();
    float e[RX], ge[RE];
#pragma unroll
    for (int m = 0; m < RX; ++m) e[m] = p.hasU && rows_is_x<M>(m, q) ? tp[p.NS + R::Ex1 + 4 * m] : 0.0f;
    rows_GT<M>(A, e, ge);
    if (p.active) {
#pragma unroll
      for (int m = 0; m < RE; ++m)
        if (m < 4 || q == 0) {
          if (rows_is_x<M>(m, q) || p.hasU) acc_sq(rdl, sv[m] + ge[m]);
        }
    }
  }
  __syncthreads();
}

// `iters` iterations; the squared residual norms of the last one (this CTA's
// nodes) in res[0..1].
template <class M, bool GROUP, bool CL, bool REG>
__device__ __forceinline__ void rows_admm(const RowPos& p, const RowMats<M>& A, const RowConst<M>& K, const Layout& L,
                                          const Inst<float>& I, float mg, float re, float rd, float rg, int iters,
                                          InstShared& sh, double* res, GroupShared* G, GroupX& X, const ProblemDev& P,
                                          RowHaloPhase& hp) {
  const float irg = 1.0f / rg, ired = 1.0f / (re + rd);
  DF rp, rdl;
  RowState<M, REG> S;
  S.load(p);
  for (int it = 0; it + 1 < iters; ++it)
    rows_iteration<M, false, GROUP, CL>(p, A, K, S, L, I, mg, re, rd, rg, irg, ired, it == 0, hp, rp, rdl, G, X, P);
  rows_iteration<M, true, GROUP, CL>(p, A, K, S, L, I, mg, re, rd, rg, irg, ired, iters == 1, hp, rp, rdl, G, X, P);
  S.store(p);
  reduce_residuals(sh, rp, rdl, res);
}

// ------------------------------------------------------------------ per-SCP-iteration set-up
// The lane's rows of G = [A B] by forward-mode differentiation of the RK4 map
// (Eq. (2b)): the lane pushes the directions of its own rows and the lanes
// exchange the columns.
template <class M>
__device__ __forceinline__ void rows_put_column(RowMats<M>& A, const float* col, int k, int q, bool on) {
  constexpr int NX = M::NX, RX = RowMats<M>::RX;
#pragma unroll
  for (int m = 0; m < RX; ++m) {
    float own[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) own[j] = 4 * m + j < NX ? col[4 * m + j] : 0.0f;
    float got[4];
#pragma unroll
    for (int s = 0; s < 4; ++s) got[s] = rows_xor(sel4(own[0], own[1], own[2], own[3], q ^ s), s);
    A.g[m][k][0] = on ? float2{got[0], got[1]} : float2{0.0f, 0.0f};
    A.g[m][k][1] = on ? float2{got[2], got[3]} : float2{0.0f, 0.0f};
  }
}
template <class M, int K>
__device__ __forceinline__ void rows_jacobians(const RowPos& p, const Node<float, 2>& nd, RowMats<M>& A,
                                               const float* prm, const Step3<float>& hs) {
  constexpr int NX = M::NX, NU = M::NU, RX = RowMats<M>::RX;
  float xt[NX], ut[NU];
#pragma unroll
  for (int j = 0; j < NX; ++j) xt[j] = df_to_float(nd.dat(Rec<M>::Xbar, j));
#pragma unroll
  for (int j = 0; j < NU; ++j) ut[j] = p.hasU ? df_to_float(nd.dat(Rec<M>::Ubar, j)) : 1.0f;
  // one pass of code for all columns (what the set-up phases wait for is
  // instruction fetch): the columns move up a group per pass, so that the
  // register indexes stay fixed
#pragma unroll 1
  for (int k = 0; k < 4; k += K) {
    float cols[K][NX];
    if constexpr (K == 2) rk4_jvpn<M, float, 2>(prm, hs, xt, ut, p.q + 4 * k, 4, cols);
    else rk4_jvp<M, float>(prm, hs, xt, ut, p.q + 4 * k, cols[0]);
#pragma unroll
    for (int m = 0; m < RX; ++m)
#pragma unroll
      for (int c = 0; c + K < 4; ++c) { A.g[m][c][0] = A.g[m][c + K][0]; A.g[m][c][1] = A.g[m][c + K][1]; }
#pragma unroll
    for (int c = 0; c < K; ++c) rows_put_column<M>(A, cols[c], 4 - K + c, p.q, p.hasU);
  }
  if constexpr (RowMats<M>::EX) {   // column 16: the same pass in all four lanes
    float col[NX];
    rk4_jvp<M, float>(prm, hs, xt, ut, 16, col);
#pragma unroll
    for (int m = 0; m < RX; ++m) {
      float own[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) own[j] = 4 * m + j < NX ? col[4 * m + j] : 0.0f;
      A.gx[m] = p.hasU ? sel4(own[0], own[1], own[2], own[3], p.q) : 0.0f;
    }
  }
}

// Packed columns of a caller's A, B (ucn_admm_solve): the lane's rows of G.
template <class M>
__device__ __forceinline__ void rows_load_G(const RowPos& p, RowMats<M>& A, const double* Ag, const double* Bg, long long g) {
  constexpr int NX = M::NX, NU = M::NU, RX = RowMats<M>::RX;
#pragma unroll
  for (int m = 0; m < RX; ++m) {
    const int r = 4 * m + p.q;
    const bool on = p.hasU && rows_is_x<M>(m, p.q);
    const double* a = Ag + (g * NX + r) * NX;
    const double* b = Bg + (g * NX + r) * NU;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      float v[4];
#pragma unroll
      for (int s = 0; s < 4; ++s) {
        const int c = 4 * k + (s ^ p.q);
        v[s] = on ? (float)(c < NX ? a[c] : b[c - NX]) : 0.0f;
      }
      A.g[m][k][0] = {v[0], v[1]};
      A.g[m][k][1] = {v[2], v[3]};
    }
    if constexpr (RowMats<M>::EX) A.gx[m] = on ? (float)b[16 - NX] : 0.0f;
  }
}

// The lane's cost gradient, diagonal of H and boxes (Eq. (2c)), as node_setup.
template <class M>
__device__ __forceinline__ void rows_setup(const RowPos& p, const Node<float, 2>& nd,
                                           const Inst<float>& I, float rad, unsigned tmask, float re, float rg,
                                           RowConst<M>& K) {
  typedef CB<M> C;
  typedef Rec<M, 2> R;
  constexpr int NX = M::NX, RE = RowConst<M>::R;
  const DF* cb = nd.c;
  const bool term = p.i == p.N;
#pragma unroll
  for (int m = 0; m < RE; ++m) {
    const int e = m < 4 ? 4 * m + p.q : 16;
    float kq = 0.0f, khd = 1.0f, lo = 0.0f, hi = 0.0f;
    if (m < 4 && rows_is_x<M>(m, p.q)) {
      const DF xb = nd.dat(Rec<M>::Xbar, e), w = cb[(term ? C::QNd : C::Qd) + e];
      if (term || I.run_cost) {
        DF gq = df_mul(df_sub(xb, cb[C::Xref + e]), w);
        if (term) gq = df_add(gq, cb[C::QN + e]);
        kq = df_to_float(gq);
      }
      khd = df_to_float(w) + rg + (p.i > 0 ? re : 0.0f);
      lo = fmaxf(wide_diff<float>(cb[C::Xlo + e], xb), -rad);
      hi = fminf(wide_diff<float>(cb[C::Xhi + e], xb), rad);
      if (p.i == 0) lo = hi = wide_diff<float>(cb[C::Xinit + e], xb);
      else if (term && (tmask >> e & 1u)) lo = hi = wide_diff<float>(cb[C::Xtgt + e], xb);
    } else if (p.hasU) {   // node N's control rows: an identity block of H, a box at 0
      const int j = e - NX;
      const DF ub = nd.dat(Rec<M>::Ubar, j), w = cb[C::Rd + j];
      if (I.run_cost) kq = df_to_float(df_mul(df_sub(ub, cb[C::Uref + j]), w));
      khd = df_to_float(w) + rg;
      lo = fmaxf(wide_diff<float>(cb[C::Ulo + j], ub), -rad);
      hi = fminf(wide_diff<float>(cb[C::Uhi + j], ub), rad);
    }
    K.kq[m] = p.active ? kq : 0.0f;
    K.khd[m] = p.active ? khd : 0.0f;
    if (p.active) {
      p.tp[R::Xlo + (m < 4 ? 4 * m : 16 - p.q)] = lo;
      p.tp[R::Xhi + (m < 4 ? 4 * m : 16 - p.q)] = hi;
      p.tp[R::Kq + (m < 4 ? 4 * m : 16 - p.q)] = kq;
      p.tp[R::Khd + (m < 4 ? 4 * m : 16 - p.q)] = khd;
    }
  }
}

// The lane's linearised obstacles (normals, bounds), the re-seeded mirrors, the
// Gram row of the lane's position row (slot order, times rho_geo) and the first
// right-hand-side sum; as node_mirror_data and node_reseed.
template <class M>
__device__ __forceinline__ float rows_obstacle_setup(const RowPos& p, const Node<float, 2>& nd, const Layout& L,
                                                     const ProblemDev& P, int b, int nobs, float rg, bool kept,
                                                     RowConst<M>& K) {
  typedef Rec<M, 2> R;
  float G[6] = {0, 0, 0, 0, 0, 0}, a0 = 0.0f, a1 = 0.0f, a2 = 0.0f;
  if (p.active) {
    const float x0 = df_to_float(nd.dat(Rec<M>::Xbar, 0)), x1 = df_to_float(nd.dat(Rec<M>::Xbar, 1)),
                x2 = df_to_float(nd.dat(Rec<M>::Xbar, 2));
    const float* hat = p.tp - p.q + R::Xh;
    float* md = p.tp + L.oMd;
    float* ms = p.tp + L.oS;
    const float* mn = p.tp + L.oNus;
    for (int o = p.q; o < nobs; o += 4, md += 16, ms += 4, mn += 4) {
      const double* c = &P.obs_c[((long long)b * P.max_obs + o) * 3];
      const float d0 = x0 - (float)c[0], d1 = x1 - (float)c[1], d2 = x2 - (float)c[2];
      float v0 = d0, v1 = d1, v2 = d2, nn = sqrtf(d0 * d0 + d1 * d1 + d2 * d2);
      if (nn < 1e-12f) { v0 = 0.0f; v1 = 0.0f; v2 = 1.0f; nn = 1.0f; }
      const float inn = 1.0f / nn;
      const float n0 = v0 * inn, n1 = v1 * inn, n2 = v2 * inn;
      const float bd = -(n0 * d0 + n1 * d1 + n2 * d2) + (float)P.obs_r[(long long)b * P.max_obs + o];
      md[0] = n0; md[4] = n1; md[8] = n2; md[12] = bd;
      const float s = kept ? ms[0] : fmaxf(bd, n0 * hat[0] + n1 * hat[1] + n2 * hat[2]);
      ms[0] = s;
      const float a = rg * s - mn[0];
      a0 += n0 * a; a1 += n1 * a; a2 += n2 * a;
      G[0] += n0 * n0; G[1] += n0 * n1; G[2] += n0 * n2; G[3] += n1 * n1; G[4] += n1 * n2; G[5] += n2 * n2;
    }
  }
#pragma unroll
  for (int k = 0; k < 6; ++k) G[k] = rg * rows_sum(G[k]);
  a0 = rows_sum(a0); a1 = rows_sum(a1); a2 = rows_sum(a2);
  // row q of the Gram matrix, slot s holding column q ^ s
  const float r0 = sel4(G[0], G[1], G[2], 0.0f, p.q), r1 = sel4(G[1], G[3], G[4], 0.0f, p.q),
              r2 = sel4(G[2], G[4], G[5], 0.0f, p.q);
#pragma unroll
  for (int s = 0; s < 4; ++s) {
    K.gram[s] = sel4(r0, r1, r2, 0.0f, p.q ^ s);
    if (p.active) p.tp[R::Gr + 4 * s] = K.gram[s];
  }
  return sel4(a0, a1, a2, 0.0f, p.q);
}

// H_i of Eq. (4) with the mirror Gram terms, assembled by rows over the lanes,
// and its inverse by Gauss-Jordan elimination in place (H is symmetric positive
// definite: no pivoting; its pivots are those of the Cholesky factorisation).
// Returns false on a non-positive pivot (replaced by 1).
template <class M>
__device__ __forceinline__ bool rows_factor(const RowPos& p, RowMats<M>& A, const RowConst<M>& K, const Inst<float>& I,
                                            float rd, float rg) {
  constexpr int RX = RowMats<M>::RX;
  constexpr bool EX = RowMats<M>::EX;
  const int q = p.q;
  float h[4][16], hx[4], rx[17];   // own rows, their column 16, row 16
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    hx[m] = 0.0f;
#pragma unroll
    for (int c = 0; c < 16; ++c) h[m][c] = 0.0f;
  }
#pragma unroll
  for (int c = 0; c < 17; ++c) rx[c] = 0.0f;
  // sum over the rows of G of their outer products: a group of four rows (one
  // per lane) per pass, the groups moving up in between
#pragma unroll 1
  for (int k0 = 0; k0 < RX; ++k0) {
#pragma unroll
    for (int o = 0; o < 4; ++o) {
      float row[17];
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        row[4 * c + (0 ^ o)] = rows_from(A.g[0][c][0].x, o);
        row[4 * c + (1 ^ o)] = rows_from(A.g[0][c][0].y, o);
        row[4 * c + (2 ^ o)] = rows_from(A.g[0][c][1].x, o);
        row[4 * c + (3 ^ o)] = rows_from(A.g[0][c][1].y, o);
      }
      if constexpr (EX) row[16] = rows_from(A.gx[0], o);
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        const float f = sel4(row[4 * m], row[4 * m + 1], row[4 * m + 2], row[4 * m + 3], q);
#pragma unroll
        for (int c = 0; c < 16; ++c) h[m][c] += f * row[c];
        if constexpr (EX) hx[m] += f * row[16];
      }
      if constexpr (EX) {
#pragma unroll
        for (int c = 0; c < 17; ++c) rx[c] += row[16] * row[c];
      }
    }
    // (after RX passes the rows are back in place)
#pragma unroll
    for (int c = 0; c < 4; ++c)
#pragma unroll
      for (int s = 0; s < 2; ++s) {
        const float2 t = A.g[0][c][s];
#pragma unroll
        for (int m = 0; m + 1 < RX; ++m) A.g[m][c][s] = A.g[m + 1][c][s];
        A.g[RX - 1][c][s] = t;
      }
    if constexpr (EX) {
      const float t = A.gx[0];
#pragma unroll
      for (int m = 0; m + 1 < RX; ++m) A.gx[m] = A.gx[m + 1];
      A.gx[RX - 1] = t;
    }
  }
#pragma unroll
  for (int m = 0; m < 4; ++m) {
#pragma unroll
    for (int c = 0; c < 16; ++c) h[m][c] *= rd;
    hx[m] *= rd;
    // the diagonal and the Gram row
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (j == q) h[m][4 * m + j] += p.active ? K.khd[m] : 1.0f;
  }
  if constexpr (EX) {
#pragma unroll
    for (int c = 0; c < 17; ++c) rx[c] *= rd;
    rx[16] += p.active ? K.khd[4] : 1.0f;
  }
#pragma unroll
  for (int c = 0; c < 3; ++c) h[0][c] += sel4(K.gram[0], K.gram[1], K.gram[2], K.gram[3], q ^ c);
  // Gauss-Jordan, four pivots (one per lane) per pass; rows and columns rotate by
  // four in between, back in place after the fourth pass
  bool ok = true;
#pragma unroll 1
  for (int k0 = 0; k0 < 4; ++k0) {
#pragma unroll
    for (int o = 0; o < 4; ++o) {
      float row[17];
#pragma unroll
      for (int c = 0; c < 16; ++c) row[c] = rows_from(h[0][c], o);
      if constexpr (EX) row[16] = rows_from(hx[0], o);
      if (!(row[o] > 0.0f)) { ok = false; row[o] = 1.0f; }
      const float d = __frcp_rn(row[o]);
#pragma unroll
      for (int c = 0; c < (EX ? 17 : 16); ++c) row[c] *= d;
      row[o] = d;
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        const float f = h[m][o];
        const bool mine = m == 0 && q == o;
#pragma unroll
        for (int c = 0; c < 16; ++c) h[m][c] = mine ? row[c] : (c == o ? -f * d : h[m][c] - f * row[c]);
        if constexpr (EX) hx[m] = mine ? row[16] : hx[m] - f * row[16];
      }
      if constexpr (EX) {
        const float f = rx[o];
#pragma unroll
        for (int c = 0; c < 17; ++c) rx[c] = c == o ? -f * d : rx[c] - f * row[c];
      }
    }
    float h0[16];
#pragma unroll
    for (int c = 0; c < 16; ++c) h0[c] = h[0][(c + 4) & 15];
#pragma unroll
    for (int m = 0; m < 3; ++m) {
      float t[16];
#pragma unroll
      for (int c = 0; c < 16; ++c) t[c] = h[m + 1][(c + 4) & 15];
#pragma unroll
      for (int c = 0; c < 16; ++c) h[m][c] = t[c];
    }
#pragma unroll
    for (int c = 0; c < 16; ++c) h[3][c] = h0[c];
    if constexpr (EX) {
      const float x0 = hx[0];
      hx[0] = hx[1]; hx[1] = hx[2]; hx[2] = hx[3]; hx[3] = x0;
      float t[16];
#pragma unroll
      for (int c = 0; c < 16; ++c) t[c] = rx[(c + 4) & 15];
#pragma unroll
      for (int c = 0; c < 16; ++c) rx[c] = t[c];
    }
  }
  if constexpr (EX) {   // the last pivot, row 16
    if (!(rx[16] > 0.0f)) { ok = false; rx[16] = 1.0f; }
    const float d = __frcp_rn(rx[16]);
#pragma unroll
    for (int c = 0; c < 16; ++c) rx[c] *= d;
    rx[16] = d;
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      const float f = hx[m];
#pragma unroll
      for (int c = 0; c < 16; ++c) h[m][c] -= f * rx[c];
      hx[m] = -f * d;
    }
  }
  // columns into slot order (exchange by the bits of q); threads without a node: zero
#pragma unroll
  for (int m = 0; m < 4; ++m) {
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const float a0 = h[m][4 * c], a1 = h[m][4 * c + 1], a2 = h[m][4 * c + 2], a3 = h[m][4 * c + 3];
      const float b0 = (q & 1) ? a1 : a0, b1 = (q & 1) ? a0 : a1, b2 = (q & 1) ? a3 : a2, b3 = (q & 1) ? a2 : a3;
      A.h[m][c][0] = p.active ? ((q & 2) ? float2{b2, b3} : float2{b0, b1}) : float2{0.0f, 0.0f};
      A.h[m][c][1] = p.active ? ((q & 2) ? float2{b0, b1} : float2{b2, b3}) : float2{0.0f, 0.0f};
    }
    if constexpr (EX) A.hx[m] = p.active ? hx[m] : 0.0f;
  }
  if constexpr (EX) A.hxx = p.active ? rx[16] : 0.0f;
  return ok;
}

// Everything an ADMM call needs at the nominal, G given: constants, boxes,
// mirror sets, H^-1 and the published mu + rho_dyn z.  Ends with a barrier.
// The mirrors are re-projected from (x-hat, u-hat), or kept as imported.
template <class M, bool CL>
__device__ __forceinline__ float rows_prepare(const RowPos& p, const Node<float, 2>& nd, const Layout& L,
                                              const ProblemDev& P, const Inst<float>& I, int b, float rad, float re,
                                              float rd, float rg, RowMats<M>& A, RowConst<M>& K, InstShared& sh,
                                              bool kept = false) {
  typedef Rec<M, 2> R;
  constexpr int RX = RowMats<M>::RX;
  rows_setup<M>(p, nd, I, rad, sh.tmask, re, rg, K);
  const float mg = rows_obstacle_setup<M>(p, nd, L, P, b, I.nobs, rg, kept, K);
  if (!rows_factor<M>(p, A, K, I, rd, rg)) atomicOr(&sh.fail, 1);
  if (p.later) {
#pragma unroll
    for (int m = 0; m < RX; ++m)
      if (rows_is_x<M>(m, p.q)) {
        const float v = p.tp[R::Mu + 4 * m] + rd * p.tp[R::Z + 4 * m];
        p.tp[R::Ex2 + 4 * m] = v;
        if constexpr (CL)
          if (p.first) st_cluster(p.halo1 + R::Ex2 + 4 * m, p.rank - 1, v);
      }
  }
  __syncthreads();
  return mg;
}

// ------------------------------------------------------------------ the fused solve
struct RowCluster {
  RowHalo halo;
  double x[2][16][6];   // totals of the CTAs of an instance (double-buffered)
  unsigned par;
};

// The totals v[0, nsum) summed and v[nsum, nval) maxed over the cluster's CTAs,
// in rank order in every CTA (the same bits).  Every thread holds v of its CTA.
__device__ __forceinline__ void rows_combine(RowCluster& c, unsigned& par, unsigned rank, unsigned n, double* v, int nsum,
                                             int nval) {
  if (threadIdx.x < n)
    for (int k = 0; k < nval; ++k) st_cluster(&c.x[par][rank][k], threadIdx.x, v[k]);
  cluster_sync();
  for (int k = 0; k < nval; ++k) {
    double a = c.x[par][0][k];
    for (unsigned r = 1; r < n; ++r) a = k < nsum ? a + c.x[par][r][k] : fmax(a, c.x[par][r][k]);
    v[k] = a;
  }
  par ^= 1u;
}

// The thread's place in the instance and the node views of the two mappings:
// nd (four lanes per node) and ndd (one thread per node).
template <class M, bool CL>
__device__ __forceinline__ RowPos rows_place(const ProblemDev& P, const Layout& L, unsigned char* smem, int b,
                                             Node<float, 2>& nd, Node<float, 2>& ndd, bool& dact) {
  RowPos p;
  p.rank = CL ? cluster_rank() : 0u;
  const int base = CL ? (int)p.rank * L.chunk : 0, halo = CL ? 1 : 0;
  const int il = (int)threadIdx.x / 4;
  p.N = P.N[b];
  p.q = (int)threadIdx.x & 3;
  p.i = base + il;
  p.active = il < L.chunk && p.i <= p.N;
  p.hasU = p.active && p.i < p.N;
  p.later = p.active && p.i >= 1;
  p.NS = L.NS;
  float* t = (float*)smem;
  p.tp = t + ((p.active ? il : 0) + halo) * L.NS + p.q;
  p.first = CL && p.active && il == 0 && p.rank > 0;
  p.last = CL && p.hasU && il == L.chunk - 1;
  p.halo0 = t + p.q;
  p.halo1 = t + (L.chunk + 1) * L.NS + p.q;
  nd.t = t + (halo - base) * L.NS;
  nd.d = (DF*)(smem + L.tbytes) + (halo - base) * L.DS;
  nd.c = (DF*)(smem + L.oC);
  nd.S = L.S; nd.NS = L.NS; nd.DS = L.DS; nd.N = p.N;
  ndd = nd;
  nd.i = p.active ? p.i : base;   // (a thread without a node reads the CTA's first record)
  ndd.i = base + (int)threadIdx.x;
  dact = (int)threadIdx.x < L.chunk && ndd.i <= p.N;
  return p;
}

// The candidate's linear-model defect (l1) and largest step over the lane's rows.
template <class M>
__device__ __forceinline__ void rows_linear_model(const RowPos& p, const RowMats<M>& A, float& lin1, float& st) {
  typedef Rec<M, 2> R;
  constexpr int RX = RowMats<M>::RX, RE = RowConst<M>::R;
  float xh[RE];
#pragma unroll
  for (int m = 0; m < RE; ++m) {
    xh[m] = p.active ? p.tp[R::Xh + (m < 4 ? 4 * m : 16 - p.q)] : 0.0f;
    st = fmaxf(st, fabsf(xh[m]));
  }
  float2 v[4][2];
  rows_gather<4>(xh, v);
  float t[RX];
  rows_G<M>(A, v, xh[RE - 1], t);
  if (p.hasU) {
#pragma unroll
    for (int m = 0; m < RX; ++m)
      if (rows_is_x<M>(m, p.q)) lin1 += fabsf(p.tp[R::C + 4 * m] - p.tp[p.NS + R::Xh + 4 * m] + t[m]);
  }
}

// scp_candidate with several lanes per node: the rollout one thread per node, the
// linear model by rows.
template <class E>
__device__ __forceinline__ void split_candidate(const typename E::Pos& p, const Node<typename E::T, 2>& nd, bool dact,
                                                const typename E::Mats& A, const Layout& L, const ProblemDev& P,
                                                const Inst<typename E::T>& I, int b, const GroupShared* G,
                                                InstShared& sh, typename WideOf<typename E::T>::type* xc,
                                                typename WideOf<typename E::T>::type* uc,
                                                typename WideOf<typename E::T>::type* fc, double* v) {
  typedef typename E::M M;
  typedef typename E::T T;
  typedef typename WideOf<T>::type W;
  typedef Rec<M, 2> R;
  constexpr int NX = M::NX, NU = M::NU;
  const int i = nd.i, N = nd.N;
  if (dact) {
    for (int j = 0; j < NX; ++j) {
      xc[j] = wide_add(nd.dat(R::Xbar, j), nd.at(R::Xh, j));
      nd.dat(R::Xc, j) = xc[j];
      if constexpr (E::CL)
        if (threadIdx.x == 0 && p.rank > 0) st_cluster(nd.d + (i + L.chunk) * L.DS + R::Xc + j, p.rank - 1, xc[j]);
    }
    for (int j = 0; j < NU; ++j) uc[j] = i < N ? wide_add(nd.dat(R::Ubar, j), nd.at(R::Uh, j)) : W();
    if constexpr (E::GROUP) {
      if (i == 0)
        for (int j = 0; j < NU; ++j) uc[j] = wide_from_double<W>(G->u0[j]);
    }
  }
  if constexpr (E::CL) {
    E::push_hat(p);
    cluster_sync();
  } else {
    __syncthreads();
  }
  T lin1 = T(0), st = T(0);
  E::linear_model(p, A, L, lin1, st);
  W vs[3] = {W(), W(), W()};
  decltype(wide_abs_round(W())) dinf = 0;
  if (dact) {
    vs[0] = node_cost<M, T, 2>(nd, P, I, b, i, N, xc, uc);
    if (i < N) {
      rk4_wide<M, T, 2>(nd, P, b, xc, uc, fc);
#pragma unroll
      for (int r = 0; r < NX; ++r) {
        fc[r] = fc[r] - nd.dnb(R::Xc, r, i + 1);
        vs[1] = vs[1] + wide_abs(fc[r]);
        dinf = maxv(dinf, wide_abs_round(fc[r]));
      }
    }
  }
  if constexpr (IsDF<T>::value) {
    vs[2] = df_from(lin1);
    float mx[2] = {dinf, st};
    block_reduce_df(sh, vs, 3, mx, 2, v);
  } else {
    v[0] = vs[0]; v[1] = vs[1]; v[2] = lin1; v[3] = dinf; v[4] = st;
    block_reduce(sh, v, 3, 5);
  }
}

// The row kernel as an engine of the split solve.
template <class M_, bool GROUP_, bool CL_, bool REG>
struct RowEngine {
  typedef M_ M;
  typedef float T;
  static constexpr bool GROUP = GROUP_, CL = CL_;
  typedef RowPos Pos;
  typedef RowMats<M> Mats;
  typedef RowConst<M> Const;
  __device__ static __forceinline__ Pos place(const ProblemDev& P, const Layout& L, unsigned char* smem, int b,
                                              Node<float, 2>& nd, Node<float, 2>& ndd, bool& dact) {
    return rows_place<M, CL>(P, L, smem, b, nd, ndd, dact);
  }
  __device__ static __forceinline__ void jacobians(const Pos& p, const Node<float, 2>& nd, Mats& A, const float* prm,
                                                   const Step3<float>& hs, const Layout&) {
    rows_jacobians<M, REG ? 2 : 1>(p, nd, A, prm, hs);
  }
  __device__ static __forceinline__ float prepare(const Pos& p, const Node<float, 2>& nd, const Layout& L,
                                                  const ProblemDev& P, const Inst<float>& I, int b, float rad, float re,
                                                  float rd, float rg, Mats& A, Const& K, InstShared& sh) {
    return rows_prepare<M, CL>(p, nd, L, P, I, b, rad, re, rd, rg, A, K, sh);
  }
  __device__ static __forceinline__ void admm(const Pos& p, const Mats& A, const Const& K, const Layout& L,
                                              const Inst<float>& I, float mg, float re, float rd, float rg, int iters,
                                              InstShared& sh, double* res, GroupShared* G, GroupX& X,
                                              const ProblemDev& P, RowHaloPhase& hp) {
    rows_admm<M, GROUP, CL, REG>(p, A, K, L, I, mg, re, rd, rg, iters, sh, res, G, X, P, hp);
  }
  // the first node's candidate, for the linear model of the previous CTA's last node
  __device__ static __forceinline__ void push_hat(const Pos& p) {
    typedef Rec<M, 2> R;
    if (p.first) {
#pragma unroll
      for (int m = 0; m < RowMats<M>::RX; ++m)
        if (rows_is_x<M>(m, p.q)) st_cluster(p.halo1 + R::Xh + 4 * m, p.rank - 1, p.tp[R::Xh + 4 * m]);
    }
  }
  __device__ static __forceinline__ void linear_model(const Pos& p, const Mats& A, const Layout&, float& lin1, float& st) {
    rows_linear_model<M>(p, A, lin1, st);
  }
};

// The fused solve (scp_body) by an engine E that puts several lanes on a node.
template <class E>
__device__ __forceinline__ void scp_split_body(const ProblemDev& P, const Layout& L, const double* x0, const double* u0,
                                              double* xout, double* uout, ucn_scp_stats* stats, int* status_out,
                                              const int b) {
  typedef typename E::M M;
  typedef typename E::T T;
  typedef typename WideOf<T>::type W;
  constexpr bool GROUP = E::GROUP, CL = E::CL;
  static_assert(!(GROUP && CL), "a scenario group's cluster holds one CTA per scenario");
  constexpr int NX = M::NX, NU = M::NU;
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ InstShared sh;
  GroupShared* G = group_slot<GROUP>();
  RowCluster* cl = nullptr;
  if constexpr (CL) {
    __shared__ RowCluster rc;
    cl = &rc;
    if (threadIdx.x == 0) halo_init<(unsigned)(sizeof(T) * M::NX)>(&rc.halo);
  }
  RowHaloPhase hp{{0u, 0u}};
  unsigned par = 0;
  const unsigned ncta = CL ? (unsigned)L.csize : 1u;
  GroupX X{0u, 0, 0};
  if constexpr (GROUP) {
    X.g = (int)blockIdx.x / P.group;
    X.k = (int)blockIdx.x % P.group;
    if (threadIdx.x == 0) group_init(P, G);
  }
  Node<T, 2> nd, ndd;
  bool dact;
  typename E::Pos pos = E::place(P, L, smem, b, nd, ndd, dact);
  if constexpr (CL) pos.hb = &cl->halo;
  const typename E::Pos& p = pos;
  const bool lead = p.rank == 0;
  typename E::Mats A;
  typename E::Const K;
  const long long xo = P.xoff[b], uo = P.uoff[b];
  const Step3<T> hs = step_of<T>(P.dt[b]);
  const unsigned long long t0 = globaltimer_ns();
  const Inst<T> I = make_inst<M, T>(P, b);
  if (threadIdx.x == 0) {
    sh.fail = 0; sh.status = ST_OK; sh.radius = P.tr_init; sh.stop = 0;
    split_barrier_init(sh.xbar, blockDim.x);
  }
  X.bar = sh.xbar;
  X.in = &sh.red[0][0];
  // the records start at zero: rows beyond a model's are read, never set
  for (int e = threadIdx.x; e < (L.chunk + (CL ? 2 : 0)) * L.NS; e += blockDim.x) ((T*)smem)[e] = T(0);
  nd.prm = ndd.prm = sh.prm;
  stage_params<M>(sh, P, b);
  stage_consts<M, T, 2>(ndd, P, b);
  if (dact) load_nominal<M, T, 2>(ndd, L, x0, u0, xo, uo);
  if constexpr (CL) {   // the halo's nominal: the next CTA's first node
    const int ih = ndd.i;
    if ((int)threadIdx.x == L.chunk && ih <= p.N)
      for (int j = 0; j < NX; ++j) ndd.dat(Rec<M, 2>::Xbar, j) = wide_from_double<W>(x0[(xo + ih) * NX + j]);
    cluster_sync();
  } else {
    __syncthreads();
  }
  flag_bad_inputs<M>(P, b, x0, u0, xo, uo, sh);
  scp_start<M, T, 2>(ndd, P, I, b, dact, sh);
  if (dact) node_start<M, T, 2>(ndd, L, P, b);
  __syncthreads();
  double Jn0[1];
  if constexpr (CL) {   // J(nominal) over the instance (scp_start left this CTA's share)
    Jn0[0] = sh.Jn;
    rows_combine(*cl, par, p.rank, ncta, Jn0, 1, 1);
    __syncthreads();
    if (threadIdx.x == 0) sh.Jn = Jn0[0];
  }
  int accepted = 0, iters_run = 0;
  unsigned long long mask = 0ull;
  double res[2] = {0, 0}, last_step = 0.0;
  const int Kscp = P.scp_iters;
  for (int k = 0; k < Kscp; ++k) {
    if (threadIdx.x == 0) {
      double f = 1.0;
      // the schedule tabulated at create; a warm start continues at its final penalty,
      // the one its kept ADMM state was computed at
      const int ks = (P.warm && P.warm[b]) ? Kscp - 1 : k;
      if (P.rho_fac) f = P.rho_fac[ks];
      else if (P.rho_final > 0.0 && Kscp > 1) f = pow(P.rho_final / P.rho_geo, (double)ks / (double)(Kscp - 1));
      sh.rho[0] = P.rho_eq * f; sh.rho[1] = P.rho_dyn * f; sh.rho[2] = P.rho_geo * f;
      for (int r = 0; r < 3; ++r) sh.rhof[r] = (float)sh.rho[r];
      sh.rhof[3] = (float)sh.radius;
    }
    __syncthreads();
    const T re = rho_of<T>(sh, 0), rd = rho_of<T>(sh, 1), rg = rho_of<T>(sh, 2);
    E::jacobians(p, nd, A, prm_of<T>(sh), hs, L);
    const T mg = E::prepare(p, nd, L, P, I, b, radius_of<T>(sh), re, rd, rg, A, K, sh);
    if constexpr (CL) {   // a failed factorisation anywhere stops the instance
      if (sh.fail && threadIdx.x < ncta) st_cluster(&sh.fail, threadIdx.x, 1);
      cluster_sync();
    }
    if constexpr (GROUP) {
      if (p.i == 0 && p.active) {
        group_box_put(G, X, p.q, wide_to_double(nd.dat(Rec<M, 2>::Ubar, p.q)), p.tp[Rec<M, 2>::Xlo + 12],
                      p.tp[Rec<M, 2>::Xhi + 12]);
      }
      group_begin(P, G, X, sh);
    }
    if (sh.fail) { if (threadIdx.x == 0) sh.status = ST_NUMERIC; iters_run++; break; }
    E::admm(p, A, K, L, I, mg, re, rd, rg, P.admm_iters, sh, res, G, X, P, hp);
    ++iters_run;
    W xc[NX], uc[NU], fc[NX];
    double v[6] = {0, 0, 0, 0, 0, 0};
    split_candidate<E>(p, ndd, dact, A, L, P, I, b, G, sh, xc, uc, fc, v);
    bool timed_out = false;
    if (threadIdx.x == 0) timed_out = globaltimer_ns() - t0 > P.timeout_ns;
    if constexpr (CL) {   // rank 0's clock decides (thread 0 of each CTA writes all the shares)
      if (threadIdx.x == 0 && lead && timed_out) sh.out[5] = 1.0;
      else if (threadIdx.x == 0) sh.out[5] = 0.0;
      __syncthreads();
      v[5] = sh.out[5];
      rows_combine(*cl, par, p.rank, ncta, v, 3, 6);
      timed_out = v[5] != 0.0;
    }
    double Jn = sh.Jn, Jc = v[0] + P.w_d * v[1], Lc = v[0] + P.w_d * v[2];
    const double Jc_own = Jc;
    if constexpr (GROUP) {
      if (threadIdx.x == 0) {
        double* m = G->mine[X.epoch & 1];
        m[0] = Jn; m[1] = Jc; m[2] = Lc; m[3] = v[3]; m[4] = v[4]; m[5] = timed_out ? 1.0 : 0.0;
      }
      double a[6];
      group_allreduce<6>(P, G, X, 3, a);
      if (threadIdx.x == 0) {
        Jn = a[0]; Jc = a[1]; Lc = a[2]; v[3] = a[3]; v[4] = a[4]; timed_out = a[5] != 0.0;
      }
    }
    if (threadIdx.x == 0) scp_decide(sh, P, Jn, Jc, Lc, Jc_own, v[3], v[4], timed_out, k, Kscp);
    __syncthreads();
    last_step = v[4];
    if (sh.accept) {
      ++accepted;
      if (k < 64) mask |= (1ull << k);
      if (dact) scp_move_nominal<M, T, 2>(ndd, L, P, b, xc, uc, fc);
      if constexpr (CL) {
        if ((int)threadIdx.x == L.chunk && ndd.i <= p.N)
          for (int j = 0; j < NX; ++j) ndd.dat(Rec<M, 2>::Xbar, j) = ndd.dat(Rec<M, 2>::Xc, j);
      }
    }
    __syncthreads();
    if (sh.stop) break;
  }
  double w[6] = {0, 0, 0, 0, 0, 0};
  scp_finish<M, T, 2>(ndd, L, P, I, b, dact, xo, uo, xout, uout, sh, w);
  if constexpr (CL) {
    // cost, l1 defect, the two residual norms | max defect
    double t[6] = {w[0], w[1], res[0], res[1], w[2], sh.xbar[1] || cl->halo.fail ? 1.0 : 0.0};
    __threadfence();
    rows_combine(*cl, par, p.rank, ncta, t, 4, 6);
    w[0] = t[0]; w[1] = t[1]; res[0] = t[2]; res[1] = t[3]; w[2] = t[4];
    if (threadIdx.x == 0 && t[5] != 0.0) sh.xbar[1] = 1ull;   // (reported as a numerical failure)
  }
  if (threadIdx.x == 0 && lead) {
    bool gfail = false;
    if constexpr (GROUP) gfail = G->gfail;   // the group lost its consensus partner
    scp_report(sh, P, b, w, res, last_step, iters_run, accepted, mask, t0, gfail, stats, status_out);
  }
  __syncthreads();
  if (lead) deliver_result(P, b, xout, uout, stats);
  if constexpr (CL) cluster_sync();   // no CTA leaves while another may write to it
  if constexpr (GROUP) group_finish(P);
}

// One instance per cluster of L.csize CTAs (CL) or per CTA.
template <class M, bool GROUP, bool CL, int MAXT, bool REG>
__global__ void __launch_bounds__(MAXT, 1) scp_rows_kernel(ProblemDev P, Layout L, const double* x0, const double* u0,
                                                           double* xout, double* uout, ucn_scp_stats* stats,
                                                           int* status_out) {
  const int k = CL ? (int)blockIdx.x / L.csize : (int)blockIdx.x;
  const int b = (GROUP || !P.order) ? k : P.order[k];
  scp_split_body<RowEngine<M, GROUP, CL, REG>>(P, L, x0, u0, xout, uout, stats, status_out, b);
}

// The stand-alone ADMM call (admm_kernel) on the row mapping: the caller's A, B
// go straight into the lanes' registers.
template <class M, bool CL, int MAXT, bool REG>
__global__ void __launch_bounds__(MAXT, 1) admm_rows_kernel(ProblemDev P, Layout L, const double* xbar,
                                                            const double* ubar, const double* Ag, const double* Bg,
                                                            const double* dg, const double* radius, int iters, int warm,
                                                            double* xhat, double* uhat, double* res, int* status) {
  typedef Rec<M, 2> R;
  constexpr int NX = M::NX, NU = M::NU, RX = RowMats<M>::RX;
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ InstShared sh;
  RowCluster* cl = nullptr;
  if constexpr (CL) {
    __shared__ RowCluster rc;
    cl = &rc;
    if (threadIdx.x == 0) halo_init<4 * M::NX>(&rc.halo);
  }
  RowHaloPhase hp{{0u, 0u}};
  unsigned par = 0;
  const unsigned ncta = CL ? (unsigned)L.csize : 1u;
  // the longest instances first, as the fused solve takes them
  const int b = P.order[CL ? (int)blockIdx.x / L.csize : (int)blockIdx.x];
  Node<float, 2> nd, ndd;
  bool dact;
  RowPos p = rows_place<M, CL>(P, L, smem, b, nd, ndd, dact);
  if constexpr (CL) p.hb = &cl->halo;
  RowMats<M> A;
  RowConst<M> K;
  const long long xo = P.xoff[b], uo = P.uoff[b];
  const Inst<float> I = make_inst<M, float>(P, b);
  if (threadIdx.x == 0) { sh.fail = 0; split_barrier_init(sh.xbar, blockDim.x); }
  for (int e = threadIdx.x; e < (L.chunk + (CL ? 2 : 0)) * L.NS; e += blockDim.x) ((float*)smem)[e] = 0.0f;
  nd.prm = ndd.prm = sh.prm;
  stage_params<M>(sh, P, b);
  stage_consts<M, float, 2>(ndd, P, b);
  if (dact) load_nominal<M, float, 2>(ndd, L, xbar, ubar, xo, uo);
  // a cluster's CTAs have all started and cleared their records before the first
  // store into one of them (rows_prepare's halo)
  if constexpr (CL) cluster_sync();
  else __syncthreads();
  rows_load_G<M>(p, A, Ag, Bg, uo + p.i);
  if (p.hasU) {
    // deviation affine term c_i = A xbar_i + B ubar_i + d_i - xbar_{i+1} in FP64 (once per call)
    const long long g = uo + p.i;
#pragma unroll
    for (int m = 0; m < RX; ++m)
      if (rows_is_x<M>(m, p.q)) {
        const int r = 4 * m + p.q;
        double acc = dg[g * NX + r];
        for (int c = 0; c < NX; ++c) acc += Ag[(g * NX + r) * NX + c] * df_to_double(nd.dat(R::Xbar, c));
        for (int c = 0; c < NU; ++c) acc += Bg[(g * NX + r) * NU + c] * df_to_double(nd.dat(R::Ubar, c));
        p.tp[R::C + 4 * m] = (float)(acc - df_to_double(df_from(xbar[(xo + p.i + 1) * NX + r])));
      }
  }
  if (dact) {
    if (warm) {
      DF xb[NX], ub[NU];
      read_nominal<M, float, 2>(ndd, ndd.i < ndd.N, xb, ub);
      node_mirror_data<M, float, 2>(ndd, L, P, b, xb, ub);   // the import takes the mirrors relative to it
      node_import<M, float, 2>(ndd, L, P, b, P.state_abs + P.soff[b]);
    } else {
      node_cold_start<M, float, 2>(ndd, L);
    }
  }
  __syncthreads();
  const float re = (float)P.rho_eq, rd = (float)P.rho_dyn, rg = (float)P.rho_geo;
  const float mg = rows_prepare<M, CL>(p, nd, L, P, I, b, (float)radius[b], re, rd, rg, A, K, sh, warm != 0);
  if constexpr (CL) {
    if (sh.fail && threadIdx.x < ncta) st_cluster(&sh.fail, threadIdx.x, 1);
    cluster_sync();
  }
  double r2[2] = {0.0, 0.0};
  GroupX X{0u, 0, 0, 0u, nullptr, sh.xbar, 0u};
  if (!sh.fail) rows_admm<M, false, CL, REG>(p, A, K, L, I, mg, re, rd, rg, iters, sh, r2, nullptr, X, P, hp);
  __syncthreads();
  if (dact) {
    const int i = ndd.i;
    node_export<M, float, 2>(ndd, L, P, b, P.state_abs + P.soff[b]);
    for (int j = 0; j < NX; ++j) xhat[(xo + i) * NX + j] = df_to_double(ndd.dat(R::Xbar, j)) + (double)ndd.at(R::Xh, j);
    if (i < p.N)
      for (int j = 0; j < NU; ++j) uhat[(uo + i) * NU + j] = df_to_double(ndd.dat(R::Ubar, j)) + (double)ndd.at(R::Uh, j);
  }
  if constexpr (CL) {
    double t[3] = {r2[0], r2[1], sh.xbar[1] || cl->halo.fail ? 1.0 : 0.0};
    rows_combine(*cl, par, p.rank, ncta, t, 2, 3);
    r2[0] = t[0]; r2[1] = t[1];
    if (threadIdx.x == 0 && t[2] != 0.0) sh.xbar[1] = 1ull;
  }
  if (threadIdx.x == 0 && p.rank == 0) {
    res[2 * b] = sqrt(r2[0]);
    res[2 * b + 1] = sqrt(r2[1]);
    status[b] = (sh.fail || sh.xbar[1]) ? ST_NUMERIC : ST_OK;
  }
  if constexpr (CL) cluster_sync();
}

}  // namespace ucn
