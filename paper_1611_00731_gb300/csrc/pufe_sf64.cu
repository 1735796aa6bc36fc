// FP64 assembly of H and S by sum factorization (rules of >= 4 points per axis on
// every (sub)cell).
//
// What bounds it: GB300 issues two FP64 multiply-adds per clock and SM (1/64
// of the FP32 rate), so a kernel of this kind is as fast as the number of FP64
// operations it can avoid; shared-memory traffic, integer work and the FP64
// atomics of the scatter hide behind them.  The direct element contraction
// (k_assemble_fp64) takes 5 n_e (n_e + 1) / 2 multiply-adds per point, about
// 19,000 on the 12^3 rocksalt cell's elements of 104 functions; the forms below
// take about 2,000.
//
// On a p^3 (sub)cell every integral is a projection of a few per-point fields
// onto products of 1D polynomials, contracted one axis at a time (z, y, x):
//
//  * FE x FE: w V onto the 10 products L_a L_b per axis (1,000 values; the
//    kinetic and overlap parts are constants of the mesh).
//  * FE x enrichment: with b_r = phi_v Psi, phi_v = 1/8 prod_d (1 + s_d x_d),
//      8 H_ir = <w V Psi, M M M> + sum_d [ 1/2 (2/h_d) <w d_d Psi, D on d, M else>
//                                       + 1/2 (2/h_d)^2 s_d <w Psi, L' on d, M else> ],
//      8 S_ir = <w Psi, M M M>,   M = L_a (1 + s x), D = L'_a (1 + s x).
//    (x - x_a) L_a = kappa_a omega with the nodal quartic omega, so the eight M
//    of an axis lie in the span of L_0..L_3 and omega, and D, L' in that of
//    L_0..L_3 (their nodal values are the coefficients).  A slot's five fields
//    therefore need 125 + 125 + 3 * 100 moments in all, 30 p^3 + 115 p^2 + 550 p
//    operations; the 512 entries of its eight vertex columns follow from the
//    moments axis by axis, two operations per M (fxe_expand, 11,500 per slot).
//    Projecting onto the eight M directly, as the mixed path does, takes
//    48 p^3 + 320 p^2 + 2,048 p: 34,000 against 25,000 operations at p = 6,
//    100,000 against 58,000 at p = 10.
//  * enrichment x enrichment, per slot pair (alpha, beta): the products of two
//    trilinear PU factors are quadratics u_0, u_1, u_2 = (1-x)^2, 1-x^2, (1+x)^2
//    per axis, those of a PU slope and a PU factor linears l_0, l_1 = 1 -+ x:
//      64 H_rs = <E, u u u> + 1/2 sum_d (2/h_d)^2 s_d s'_d <A, u u, 1 on d>
//             + 1/2 sum_d (2/h_d) (s_d <C_d, u u, l_b'd on d> + s'_d <B_d, u u, l_bd on d>),
//      64 S_rs = <A, u u u>,
//      A = w Psi_a Psi_b, E = w (V Psi_a Psi_b + 1/2 grad Psi_a . grad Psi_b),
//      B_d = w Psi_b d_d Psi_a, C_d = w Psi_a d_d Psi_b,
//    with <., 1> = (u_0 + 2 u_1 + u_2) / 4 of the A moments: 162 moments,
//    36 p^3 + 60 p^2 + 162 p operations for the pair's 64 vertex pairs.
//    Elements whose slots hold few vertex columns take the direct products of
//    their columns where those are fewer operations (sf64_work_list).
//
// General (triclinic) cells: the fields are (J^-1 grad Psi)_d and the metric
// G = J^-1 J^-T replaces (2/h_d)^2; its off-diagonal terms pair a slope on one axis
// with a slope on another, projections of w Psi (of A) that the same moments hold.
// The serendipity functions are sums of tricubic ones (their nodal values, R), so
// their rows are R^T times the tricubic rows.
//
// One launch over a work list of (element, kind, range) items, largest first:
// FE x FE blocks, slot ranges, pair ranges and the direct blocks' point ranges,
// cut so that the items of small meshes still fill the chip.  All blocks meet in
// FP64 atomics.
//
// Measured (kernel time, direct kernel before): 12^3 rocksalt cell 18.8 -> 1.31 ms,
// CsCl-like 16^3 cell 23.7 -> 2.62 ms, two-atom 4^3 cell 1.72 -> 0.094 ms, eight
// elements of 6^3 points 377 -> 35 us; triclinic serendipity 6^3 at a wavevector 1.15
// -> 0.21 ms.
#include <algorithm>

#include "pufe_internal.h"

namespace pufe {
namespace {

constexpr int A64_NT = 128;

struct Asm64 {
  const int32_t *items;   // six per item: element, kind, range, (sub)cell range
  const int64_t *qoff;
  const double *w, *xi;
  const int32_t *partoff, *part_p, *part_q;
  const int64_t *doff;
  const int32_t *ecol, *aoff;
  const int64_t *toff;
  const double *psi;
  const int64_t *soff;
  const int32_t *smap;
  const double *V, *Tfe, *Sfe;
  double *H, *Hi, *S, *Si;
  const uint8_t *eshift;
  PhaseTab ph;
  // first and second order factors of the fields: orthorhombic cells 2 / h_d with
  // the physical gradients; general cells (GEN) jit = J^-T, the fields
  // (J^-1 grad Psi)_d and the metric G = J^-1 J^-T
  double sc[3], jit[9], G[9];
  // serendipity space (nfe = 32): the tricubic nodes where function c is not zero
  // and its values there, rl per function (padded with zeros)
  const int32_t *ri;
  const double *rv;
  int rl, nfe;
  int want, work;   // PUFE_WANT_* mask; doubles of the shared work area
  unsigned *err;
};

// value hv, sv of the local pair (i, j) into H and S; Bloch: with the phase
// conj(exp(i k.R_i)) exp(i k.R_j) (a zero imaginary part is not added, unless
// the value is not finite)
template <bool BLOCH>
__device__ __forceinline__ void add_entry(const Asm64 &P, int64_t slot, double hv, double sv,
                                          bool h, bool s, int ci, int cj) {
  if (!BLOCH) {
    if (h) atomicAdd(P.H + slot, hv);
    if (s) atomicAdd(P.S + slot, sv);
    return;
  }
  double pr = 1.0, pi = 0.0;
  if (ci != cj) {
    pr = P.ph.re[ci] * P.ph.re[cj] + P.ph.im[ci] * P.ph.im[cj];
    pi = P.ph.re[ci] * P.ph.im[cj] - P.ph.im[ci] * P.ph.re[cj];
  }
  if (h) {
    atomicAdd(P.H + slot, hv * pr);
    if (pi != 0.0 || !isfinite(hv)) atomicAdd(P.Hi + slot, hv * pi);
  }
  if (s) {
    atomicAdd(P.S + slot, sv * pr);
    if (pi != 0.0) atomicAdd(P.Si + slot, sv * pi);
  }
}

__device__ __forceinline__ int pidx64(int a, int b) {   // unordered pair -> 0..9
  const int lo = a < b ? a : b, hi = a < b ? b : a;
  return lo * 4 - (lo * (lo - 1)) / 2 + (hi - lo);
}

// coordinate of point t of axis d of the (sub)cell starting at point qs
__device__ __forceinline__ double axis_xi(const Asm64 &P, int64_t qs, int p, int d, int t) {
  const int64_t stride = d == 0 ? 1 : (d == 1 ? p : (int64_t)p * p);
  return P.xi[3 * (qs + t * stride) + d];
}

// ---- FE x FE block -----------------------------------------------------------
template <bool BLOCH>
__device__ void fefe_item(const Asm64 &P, int e, int cb, int ce, double *sm) {
  const int tid = threadIdx.x;
  double *M = sm;   // 1000 moments
  for (int o = tid; o < 1000; o += A64_NT) M[o] = 0.0;
  const bool h = (P.want & PUFE_WANT_H) != 0;
  if (!h && P.V && cb == 0) {   // an S-only call still reports a V that is not finite
    bool bad = false;
    for (int64_t q = P.qoff[e] + tid; q < P.qoff[e + 1]; q += A64_NT) bad |= !isfinite(P.V[q]);
    if (bad) atomicOr(P.err, DEVERR_NONFINITE);
  }
  for (int k = P.partoff[e] + cb; h && k < P.partoff[e] + ce; ++k) {
    const int p = P.part_p[k], p2 = p * p;
    double *F = M + 1000;           // [axis][10][p]
    double *G1 = F + 30 * p;        // [10][p^2]
    double *G2 = G1 + 10 * p2;      // [100][p]
    const int64_t qs = P.qoff[e] + P.part_q[k];
    __syncthreads();
    for (int o = tid; o < 3 * p; o += A64_NT) {
      const int d = o / p, t = o - d * p;
      double L[4], dL[4];
      lagrange3(axis_xi(P, qs, p, d, t), L, dL);
      int c = 0;
      for (int a = 0; a < 4; ++a)
        for (int b = a; b < 4; ++b) F[(d * 10 + c++) * p + t] = L[a] * L[b];
    }
    __syncthreads();
    bool bad = false;
    for (int o = tid; o < 2 * p2; o += A64_NT) {   // z: five of the ten products each
      const int half = o / p2, qxy = o - half * p2;
      const double *f = F + (20 + 5 * half) * p;
      double s[5] = {0, 0, 0, 0, 0};
      for (int qz = 0; qz < p; ++qz) {
        const int64_t q = qs + qxy + p2 * qz;
        const double v = P.V[q];
        bad |= !isfinite(v);
        const double wv = P.w[q] * v;
#pragma unroll
        for (int u = 0; u < 5; ++u) s[u] = fma(wv, f[u * p + qz], s[u]);
      }
#pragma unroll
      for (int u = 0; u < 5; ++u) G1[(5 * half + u) * p2 + qxy] = s[u];
    }
    if (bad) atomicOr(P.err, DEVERR_NONFINITE);
    __syncthreads();
    for (int o = tid; o < 20 * p; o += A64_NT) {   // y: (z product, half of the y products, qx)
      const int r = o / p, qx = o - r * p, cc = r >> 1, half = r & 1;
      const double *f = F + (10 + 5 * half) * p, *g = G1 + cc * p2 + qx;
      double s[5] = {0, 0, 0, 0, 0};
      for (int qy = 0; qy < p; ++qy) {
        const double t = g[p * qy];
#pragma unroll
        for (int u = 0; u < 5; ++u) s[u] = fma(t, f[u * p + qy], s[u]);
      }
#pragma unroll
      for (int u = 0; u < 5; ++u) G2[((5 * half + u) * 10 + cc) * p + qx] = s[u];
    }
    __syncthreads();
    for (int o = tid; o < 200; o += A64_NT) {      // x
      const int r = o >> 1, half = o & 1;
      const double *f = F + 5 * half * p, *g = G2 + r * p;
      double s[5] = {0, 0, 0, 0, 0};
      for (int qx = 0; qx < p; ++qx) {
        const double t = g[qx];
#pragma unroll
        for (int u = 0; u < 5; ++u) s[u] = fma(t, f[u * p + qx], s[u]);
      }
#pragma unroll
      for (int u = 0; u < 5; ++u) M[(5 * half + u) * 100 + r] += s[u];
    }
  }
  __syncthreads();
  const int n = (int)(P.doff[e + 1] - P.doff[e]);
  const int32_t *m = P.smap + P.soff[e];
  const uint8_t *es = P.eshift + P.doff[e];
  auto tri = [&](int i, int j) -> double {   // tricubic entry
    return M[pidx64(i & 3, j & 3) * 100 + pidx64((i >> 2) & 3, (j >> 2) & 3) * 10 +
             pidx64(i >> 4, j >> 4)];
  };
  // serendipity: R^T M, R the nodal values of its functions, transposed [64][32];
  // a warp works on one function's nodes, so that its list is uniform
  double *Y = M + 1000;
  if (P.nfe == 32 && h) {
    for (int o = tid; o < 2048; o += A64_NT) {
      const int c = o >> 6, k = o & 63;
      double s = 0.0;
      for (int u = 0; u < P.rl; ++u) s = fma(P.rv[c * P.rl + u], tri(P.ri[c * P.rl + u], k), s);
      Y[k * 32 + c] = s;
    }
    __syncthreads();
  }
  // the constants come with the element's first (sub)cell range; S starts as their
  // sum at the Gamma point, so a wavevector adds only what the phases change
  const bool s = BLOCH && (P.want & PUFE_WANT_S) && cb == 0;
  const int nf = P.nfe;
  for (int o = tid; o < nf * nf; o += A64_NT) {
    const int i = o / nf, j = o - i * nf;
    double v = 0.0;
    if (nf == 64) {
      v = tri(i, j);
    } else if (h) {   // (symmetric: row i from function i's list, column j from Y)
      for (int u = 0; u < P.rl; ++u)
        v = fma(P.rv[i * P.rl + u], Y[P.ri[i * P.rl + u] * 32 + j], v);
    }
    const int ci = BLOCH ? es[i] : 0, cj = BLOCH ? es[j] : 0;
    add_entry<BLOCH>(P, m[i * n + j], h && cb == 0 ? P.Tfe[o] + v : v, 0.0, h, false, ci, cj);
    if (s && ci != cj) {
      const double pr = P.ph.re[ci] * P.ph.re[cj] + P.ph.im[ci] * P.ph.im[cj];
      const double pi = P.ph.re[ci] * P.ph.im[cj] - P.ph.im[ci] * P.ph.re[cj];
      atomicAdd(P.S + m[i * n + j], P.Sfe[o] * (pr - 1.0));
      atomicAdd(P.Si + m[i * n + j], P.Sfe[o] * pi);
    }
  }
}

// ---- FE x enrichment blocks of the slots [s0, s1) ------------------------------
// 1D constants.  With s = -1, +1 for t = 0, 1: M_a,t = L_a (1 + s x) =
// alpha_a,t L_a + s kappa_a omega, alpha_a,t = 1 + s x_a = 0, 2/3, 4/3 or 2.  Both
// values of each constant are known at compile time and picked by t, so that no
// FP64 operation is spent on them.
__device__ __forceinline__ double alpha1(int a, bool t) {
  return t ? (a == 0 ? 0.0 : (a == 1 ? 2.0 / 3.0 : (a == 2 ? 4.0 / 3.0 : 2.0)))
           : (a == 3 ? 0.0 : (a == 2 ? 2.0 / 3.0 : (a == 1 ? 4.0 / 3.0 : 2.0)));
}
__device__ __forceinline__ double kappa1(int a, bool t) {   // s kappa_a
  const double k = (a & 1 ? 1.0 : -1.0) * (a == 0 || a == 3 ? 0.5625 : 1.6875);
  return t ? k : -k;
}
// L'_a(x_j), row a
__constant__ double c_d1[16] = {-2.75, -0.5, 0.25, -0.5, 4.5,  -0.75, -1.5, 2.25,
                                -2.25, 1.5,  0.75, -4.5, 0.5,  -0.25, 0.5,  2.75};

// the four M_a,t of an axis from the five moments at stride `st`
__device__ __forceinline__ void expand_m(const double *m, int st, bool t, double o[4]) {
  const double om = m[4 * st];
#pragma unroll
  for (int a = 0; a < 4; ++a) o[a] = fma(kappa1(a, t), om, alpha1(a, t) * m[a * st]);
}
// adds sum_j L'_a(x_j) ((1 + s x_j) F_j + ss S_j) to o[a] (ss: the second order
// factor times s); general cells: with x1, x2 their cross terms' moments,
// (1 + s x_j) (c1 x1_j + c2 x2_j) too
template <bool GEN = false>
__device__ __forceinline__ void expand_d(const double *F, int fst, const double *S, int sst,
                                         bool t, double ss, double o[4],
                                         const double *x1 = nullptr, int st1 = 0, double c1 = 0.0,
                                         const double *x2 = nullptr, int st2 = 0, double c2 = 0.0) {
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    double f = F[j * fst];
    if (GEN) f = fma(c1, x1[j * st1], f);
    if (GEN && x2) f = fma(c2, x2[j * st2], f);
    const double g = fma(alpha1(j, t), f, ss * S[j * sst]);
#pragma unroll
    for (int a = 0; a < 4; ++a) o[a] = fma(c_d1[a * 4 + j], g, o[a]);
  }
}
// sum_j L'_a(x_j) (1 + s x_j) S_j
__device__ __forceinline__ void slope_m(const double *S, int st, bool t, double o[4]) {
#pragma unroll
  for (int a = 0; a < 4; ++a) o[a] = 0.0;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const double g = alpha1(j, t) * S[j * st];
#pragma unroll
    for (int a = 0; a < 4; ++a) o[a] = fma(c_d1[a * 4 + j], g, o[a]);
  }
}

// doubles of the expansion's intermediates: orthorhombic, general cells' cross
// terms, the serendipity space's tricubic rows of H and S
constexpr int FXE_EXP = 1616, FXE_EXP_GEN = 1160, FXE_EXP_SER = 1024;
constexpr int FXE_MOM = 550;    // moments of a slot: S 125, V 125, Fx, Fy, Fz 100 each
constexpr int EXE_MOM = 162;    // moments of a slot pair

template <bool BLOCH, bool GEN>
__device__ void fxe_item(const Asm64 &P, int e, int s0, int s1, int cb, int ce, double *sm) {
  const int tid = threadIdx.x, G = s1 - s0;
  const bool h = (P.want & PUFE_WANT_H) != 0, ws = (P.want & PUFE_WANT_S) != 0;
  const int n = (int)(P.doff[e + 1] - P.doff[e]), nE = n - P.nfe;
  const int64_t q0 = P.qoff[e];
  const int Q = (int)(P.qoff[e + 1] - q0);
  const double *pe = P.psi + 4 * P.toff[e];
  const int32_t *ec = P.ecol + (P.doff[e] - (int64_t)P.nfe * e);
  double *mom = sm;                                        // [G][550]
  int *scol = reinterpret_cast<int *>(mom + FXE_MOM * G);  // [G][8]
  double *base = mom + FXE_MOM * G + 4 * G;
  for (int o = tid; o < FXE_MOM * G; o += A64_NT) mom[o] = 0.0;
  for (int o = tid; o < 8 * G; o += A64_NT) scol[o] = -1;
  __syncthreads();
  for (int o = tid; o < nE; o += A64_NT) {
    const int c = ec[o] - 8 * s0;
    if (c >= 0 && c < 8 * G) scol[c] = o;
  }
  const int nr1 = h ? 24 : 5, nr2 = h ? 115 : 25;   // rows of the z and y stages
  for (int k = P.partoff[e] + cb; k < P.partoff[e] + ce; ++k) {
    const int p = P.part_p[k], p2 = p * p, GP2 = G * p2, GP = G * p, pq = P.part_q[k];
    const int64_t qs = q0 + pq;
    double *F = base;              // [axis][5][p]: L_0..L_3, omega
    double *T1 = F + 15 * p;       // [24][G p^2]: S, V, Fx, Fy (5 each), Fz (4)
    double *T2 = T1 + 24 * GP2;    // [115][G p]
    __syncthreads();
    for (int o = tid; o < 3 * p; o += A64_NT) {
      const int d = o / p, t = o - d * p;
      const double x = axis_xi(P, qs, p, d, t);
      double L[4], dL[4];
      lagrange3(x, L, dL);
      double *f = F + d * 5 * p + t;
      const double c8 = d == 2 ? 0.125 : 1.0;   // the 1/8 of phi_v, once
      for (int a = 0; a < 4; ++a) f[a * p] = c8 * L[a];
      f[4 * p] = c8 * ((x + 1.0) * (x + 1.0 / 3.0) * (x - 1.0 / 3.0) * (x - 1.0));
    }
    __syncthreads();
    for (int it = tid; it < GP2; it += A64_NT) {   // z: one thread per (slot, qx, qy)
      const int g = it / p2, qxy = it - g * p2;
      const double *ps = pe + (int64_t)(s0 + g) * 4 * Q + pq + qxy;
      const double *f = F + 10 * p;
      double a[24];
#pragma unroll
      for (int u = 0; u < 24; ++u) a[u] = 0.0;
      for (int qz = 0; qz < p; ++qz) {
        const int64_t q = qs + qxy + p2 * qz;
        const double w = P.w[q], fS = w * ps[p2 * qz];
        double fk[5];
#pragma unroll
        for (int u = 0; u < 5; ++u) fk[u] = f[u * p + qz];
#pragma unroll
        for (int u = 0; u < 5; ++u) a[u] = fma(fS, fk[u], a[u]);
        if (h) {
          const double fV = fS * P.V[q];
          double fx = ps[Q + p2 * qz], fy = ps[2 * Q + p2 * qz], fz = ps[3 * Q + p2 * qz];
          if (GEN) {   // J^-1 grad
            const double gx = fx, gy = fy, gz = fz;
            fx = P.jit[0] * gx + P.jit[3] * gy + P.jit[6] * gz;
            fy = P.jit[1] * gx + P.jit[4] * gy + P.jit[7] * gz;
            fz = P.jit[2] * gx + P.jit[5] * gy + P.jit[8] * gz;
          }
          fx *= w;
          fy *= w;
          fz *= w;
#pragma unroll
          for (int u = 0; u < 5; ++u) {
            a[5 + u] = fma(fV, fk[u], a[5 + u]);
            a[10 + u] = fma(fx, fk[u], a[10 + u]);
            a[15 + u] = fma(fy, fk[u], a[15 + u]);
          }
#pragma unroll
          for (int u = 0; u < 4; ++u) a[20 + u] = fma(fz, fk[u], a[20 + u]);
        }
      }
#pragma unroll
      for (int u = 0; u < 24; ++u)
        if (u < nr1) T1[u * GP2 + it] = a[u];
    }
    __syncthreads();
    for (int it = tid; it < nr1 * GP; it += A64_NT) {   // y: one thread per (z row, slot, qx)
      const int r = it / GP, gq = it - r * GP, g = gq / p, qx = gq - g * p;
      const double *t1 = T1 + r * GP2 + g * p2 + qx, *f = F + 5 * p;
      double a[5] = {0, 0, 0, 0, 0};
      for (int qy = 0; qy < p; ++qy) {
        const double t = t1[p * qy];
#pragma unroll
        for (int u = 0; u < 4; ++u) a[u] = fma(t, f[u * p + qy], a[u]);
        if (r < 15 || r >= 20) a[4] = fma(t, f[4 * p + qy], a[4]);
      }
      // rows 0-14 and 20-23 keep five y moments, Fy (15-19) four
      const int o = r < 15 ? 5 * r : (r < 20 ? 75 + 4 * (r - 15) : 95 + 5 * (r - 20));
#pragma unroll
      for (int u = 0; u < 4; ++u) T2[(o + u) * GP + gq] = a[u];
      if (r < 15 || r >= 20) T2[(o + 4) * GP + gq] = a[4];
    }
    __syncthreads();
    for (int it = tid; it < nr2 * G; it += A64_NT) {   // x: one thread per (y row, slot)
      const int r = it / G, g = it - r * G;
      const double *t2 = T2 + r * GP + g * p, *f = F;
      double a[5] = {0, 0, 0, 0, 0};
      for (int qx = 0; qx < p; ++qx) {
        const double t = t2[qx];
#pragma unroll
        for (int u = 0; u < 4; ++u) a[u] = fma(t, f[u * p + qx], a[u]);
        if (r < 50 || r >= 75) a[4] = fma(t, f[4 * p + qx], a[4]);
      }
      // rows 50-74 (Fx) keep four x moments, the others five
      double *mo = mom + g * FXE_MOM + (r < 50 ? 5 * r : (r < 75 ? 250 + 4 * (r - 50) : 350 + 5 * (r - 75)));
#pragma unroll
      for (int u = 0; u < 4; ++u) mo[u] += a[u];
      if (r < 50 || r >= 75) mo[4] += a[4];
    }
  }
  // the entries from the moments, axis by axis, one slot at a time
  const int32_t *m = P.smap + P.soff[e];
  const uint8_t *es = P.eshift + P.doff[e];
  double *XS = base, *XFy = XS + 200, *XFz = XFy + 160, *R1 = XFz + 160;   // [z][y][x 8]
  double *YS = R1 + 200, *YFz = YS + 320, *R2 = YFz + 256;                 // [z][y 8][x 8]
  // general cells: D on x; its M on y; D on y of M on x; M on y of s_x L on x
  double *XD = R2 + 320, *YXD = XD + 200, *YD = YXD + 320, *YXL = YD + 320;
  double *HS = base + FXE_EXP + (GEN ? FXE_EXP_GEN : 0);   // serendipity: [64][H, S][vertex]
  // 1/2 of the first order factor goes into the moments of Fx, Fy, Fz, 1/2 of the
  // second into cc
  const double cc[3] = {0.5 * (GEN ? P.G[0] : P.sc[0] * P.sc[0]),
                        0.5 * (GEN ? P.G[4] : P.sc[1] * P.sc[1]),
                        0.5 * (GEN ? P.G[8] : P.sc[2] * P.sc[2])};
  if (h) {
    __syncthreads();
    for (int o = tid; o < 300 * G; o += A64_NT) {
      const int g = o / 300, i = o - 300 * g;
      mom[g * FXE_MOM + 250 + i] *= GEN ? 0.5 : 0.5 * P.sc[i / 100];
    }
  }
  const double gxy = 0.5 * P.G[1], gxz = 0.5 * P.G[2], gyz = 0.5 * P.G[5];
  const bool ser = P.nfe == 32;
  for (int g = 0; g < G; ++g) {
    const double *S = mom + g * FXE_MOM, *Vm = S + 125, *Fx = S + 250, *Fy = S + 350, *Fz = S + 450;
    const int *sc8 = scol + 8 * g;
    int vm = 0;   // vertices that hold a column
#pragma unroll
    for (int v = 0; v < 8; ++v) vm |= (sc8[v] >= 0) << v;
    // vertex codes with t = 0 / t = 1 on each axis
    const int xm = ((vm & 0x55) != 0) | ((vm & 0xAA) != 0) << 1;
    const int ym = ((vm & 0x33) != 0) | ((vm & 0xCC) != 0) << 1;
    __syncthreads();
    for (int it = tid; it < 130; it += A64_NT) {   // x
      const int t = it & 1, r = it >> 1;
      if (!(xm >> t & 1)) continue;
      double o[4];
      if (r < 25) {
        expand_m(S + 5 * r, 1, t, o);
        for (int a = 0; a < 4; ++a) XS[r * 8 + 4 * t + a] = o[a];
        if (h) {
          expand_m(Vm + 5 * r, 1, t, o);
          expand_d(Fx + 4 * r, 1, S + 5 * r, 1, t, t ? cc[0] : -cc[0], o);
          for (int a = 0; a < 4; ++a) R1[r * 8 + 4 * t + a] = o[a];
          if (GEN) {
            slope_m(S + 5 * r, 1, t, o);
            for (int a = 0; a < 4; ++a) XD[r * 8 + 4 * t + a] = o[a];
          }
        }
      } else if (h) {
        const bool y = r < 45;
        const int rr = y ? r - 25 : r - 45;
        expand_m((y ? Fy : Fz) + 5 * rr, 1, t, o);
        for (int a = 0; a < 4; ++a) (y ? XFy : XFz)[rr * 8 + 4 * t + a] = o[a];
      }
    }
    __syncthreads();
    for (int it = tid; it < 144; it += A64_NT) {   // y: (z row, t, x)
      const int x = it & 7, t = (it >> 3) & 1, z = it >> 4;
      if (!(ym >> t & 1) || !(xm >> (x >> 2) & 1)) continue;
      const double s = t ? 1.0 : -1.0;
      double o[4];
      if (z < 5) {
        expand_m(XS + z * 40 + x, 8, t, o);
        for (int b = 0; b < 4; ++b) YS[z * 64 + (4 * t + b) * 8 + x] = o[b];
        if (h) {
          expand_m(R1 + z * 40 + x, 8, t, o);
          if (GEN) {
            // s_x L_a on x: the moments of L_a themselves, signed
            const double sx = x >> 2 ? 1.0 : -1.0, *xl = S + z * 25 + (x & 3);
            expand_d<true>(XFy + z * 32 + x, 8, XS + z * 40 + x, 8, t, s * cc[1], o, xl, 5,
                           gxy * sx);
            for (int b = 0; b < 4; ++b) {
              o[b] = fma(gxy * s, XD[z * 40 + b * 8 + x], o[b]);
              R2[z * 64 + (4 * t + b) * 8 + x] = o[b];
            }
            expand_m(XD + z * 40 + x, 8, t, o);
            for (int b = 0; b < 4; ++b) YXD[z * 64 + (4 * t + b) * 8 + x] = o[b];
            slope_m(XS + z * 40 + x, 8, t, o);
            for (int b = 0; b < 4; ++b) YD[z * 64 + (4 * t + b) * 8 + x] = o[b];
            expand_m(xl, 5, t, o);
            for (int b = 0; b < 4; ++b) YXL[z * 64 + (4 * t + b) * 8 + x] = sx * o[b];
          } else {
            expand_d(XFy + z * 32 + x, 8, XS + z * 40 + x, 8, t, t ? cc[1] : -cc[1], o);
            for (int b = 0; b < 4; ++b) R2[z * 64 + (4 * t + b) * 8 + x] = o[b];
          }
        }
      } else if (h) {
        expand_m(XFz + (z - 5) * 40 + x, 8, t, o);
        for (int b = 0; b < 4; ++b) YFz[(z - 5) * 64 + (4 * t + b) * 8 + x] = o[b];
      }
    }
    __syncthreads();
    for (int it = tid; it < 128; it += A64_NT) {   // z and the scatter: (t_z, y 8, x 8)
      const int xy = it & 63, t = it >> 6, x = xy & 7, y = xy >> 3;
      const int v = (x >> 2) | ((y >> 2) << 1) | (t << 2), r = sc8[v];
      if (r < 0) continue;
      const double s = t ? 1.0 : -1.0;
      double so[4], ho[4] = {0, 0, 0, 0};
      expand_m(YS + xy, 64, t, so);
      if (h) {
        expand_m(R2 + xy, 64, t, ho);
        if (GEN) {
          const double sy = y >> 2 ? 1.0 : -1.0;
          expand_d<true>(YFz + xy, 64, YS + xy, 64, t, s * cc[2], ho, YXL + xy, 64, gxz,
                         XS + (y & 3) * 8 + x, 40, gyz * sy);
          for (int c = 0; c < 4; ++c)
            ho[c] = fma(s, fma(gxz, YXD[c * 64 + xy], gyz * YD[c * 64 + xy]), ho[c]);
        } else {
          expand_d(YFz + xy, 64, YS + xy, 64, t, t ? cc[2] : -cc[2], ho);
        }
      }
      for (int c = 0; c < 4; ++c) {
        const int i = (x & 3) + 4 * (y & 3) + 16 * c;
        if (ser) {
          HS[i * 16 + v] = ho[c];
          HS[i * 16 + 8 + v] = so[c];
          continue;
        }
        const int j = 64 + r;
        const int ci = BLOCH ? es[i] : 0, cj = BLOCH ? es[j] : 0;
        add_entry<BLOCH>(P, m[i * n + j], ho[c], so[c], h, ws, ci, cj);
        add_entry<BLOCH>(P, m[j * n + i], ho[c], so[c], h, ws, cj, ci);
      }
    }
    if (!ser) continue;
    __syncthreads();
    // rows of the serendipity functions: half a warp per function (its H and S of
    // the eight vertices), whose list is uniform there
    for (int it = tid; it < 512; it += A64_NT) {
      const int i = it >> 4, hsv = it & 15, r = sc8[hsv & 7];
      if (r < 0 || !(hsv < 8 ? h : ws)) continue;
      double t = 0.0;
      for (int u = 0; u < P.rl; ++u)
        t = fma(P.rv[i * P.rl + u], HS[P.ri[i * P.rl + u] * 16 + hsv], t);
      const int j = 32 + r;
      const int ci = BLOCH ? es[i] : 0, cj = BLOCH ? es[j] : 0;
      add_entry<BLOCH>(P, m[i * n + j], t, t, hsv < 8, hsv >= 8, ci, cj);
      add_entry<BLOCH>(P, m[j * n + i], t, t, hsv < 8, hsv >= 8, cj, ci);
    }
  }
}

// ---- enrichment x enrichment block of the slot pairs [k0, k1) ------------------
// z rows: A u (3), E u (3), B_x u, C_x u, B_y u, C_y u (3 each), B_z l, C_z l (2 each)
template <bool BLOCH, bool GEN>
__device__ void exe_item(const Asm64 &P, int e, int k0, int k1, int cb, int ce, double *sm) {
  const int tid = threadIdx.x;
  const bool h = (P.want & PUFE_WANT_H) != 0, ws = (P.want & PUFE_WANT_S) != 0;
  const int n = (int)(P.doff[e + 1] - P.doff[e]), nE = n - P.nfe;
  const int64_t q0 = P.qoff[e];
  const int Q = (int)(P.qoff[e + 1] - q0), A = P.aoff[e + 1] - P.aoff[e];
  const double *pe = P.psi + 4 * P.toff[e];
  const int32_t *ec = P.ecol + (P.doff[e] - (int64_t)P.nfe * e);
  const int32_t *m = P.smap + P.soff[e];
  const uint8_t *es = P.eshift + P.doff[e];
  int *scol = reinterpret_cast<int *>(sm);   // [A][8]
  double *base = sm + 4 * A;
  for (int o = tid; o < 8 * A; o += A64_NT) scol[o] = -1;
  __syncthreads();
  for (int o = tid; o < nE; o += A64_NT) scol[ec[o]] = o;
  int pmax = 1;
  for (int k = P.partoff[e]; k < P.partoff[e + 1]; ++k) pmax = max(pmax, P.part_p[k]);
  const int avail = P.work - 4 * A - 18 * pmax;
  const int fit = max(1, avail / (22 * pmax * pmax + 60 * pmax + EXE_MOM + 1));
  const int nch = (k1 - k0 + fit - 1) / fit, npc = (k1 - k0 + nch - 1) / nch;
  const int nr1 = h ? 22 : 3, nr2 = h ? 60 : 9;
  // factors of the entries' terms with the scaled 1D functions: 1/4 (2/h_d) (first
  // order; general cells: 1/4) and 1/8 (2/h_d)^2 (G_dd / 8)
  const double c1[3] = {GEN ? 0.25 : 0.25 * P.sc[0], GEN ? 0.25 : 0.25 * P.sc[1],
                        GEN ? 0.25 : 0.25 * P.sc[2]};
  const double cq[3] = {0.125 * (GEN ? P.G[0] : P.sc[0] * P.sc[0]),
                        0.125 * (GEN ? P.G[4] : P.sc[1] * P.sc[1]),
                        0.125 * (GEN ? P.G[8] : P.sc[2] * P.sc[2])};
  for (int c0 = k0; c0 < k1; c0 += npc) {
    const int nc = min(npc, k1 - c0);
    double *mom = base;                                         // [nc][162]
    int *pr = reinterpret_cast<int *>(mom + EXE_MOM * nc);      // [nc][2]: alpha, beta
    double *F = mom + EXE_MOM * nc + nc;                        // [axis][u_0, u_1, u_2, 1, l_0, l_1][p]
    __syncthreads();
    for (int o = tid; o < EXE_MOM * nc; o += A64_NT) mom[o] = 0.0;
    for (int o = tid; o < nc; o += A64_NT) {   // pair c0 + o of the alpha-major list, alpha <= beta
      int a = 0, t = c0 + o;
      while (t >= A - a) t -= A - a++;
      pr[2 * o] = a;
      pr[2 * o + 1] = a + t;
    }
    for (int k = P.partoff[e] + cb; k < P.partoff[e] + ce; ++k) {
      const int p = P.part_p[k], p2 = p * p, NP2 = nc * p2, NP = nc * p, pq = P.part_q[k];
      const int64_t qs = q0 + pq;
      double *T1 = F + 18 * p;      // [22][nc p^2]
      double *T2 = T1 + 22 * NP2;   // [60][nc p]
      __syncthreads();
      for (int o = tid; o < 3 * p; o += A64_NT) {
        const int d = o / p, t = o - d * p;
        // (halved linears: u_k / 4 and l_t / 2, so the 1/64 of phi_v phi_v' is in them)
        const double x = axis_xi(P, qs, p, d, t), l0 = 0.5 - 0.5 * x, l1 = 0.5 + 0.5 * x;
        double *f = F + d * 6 * p + t;
        f[0] = l0 * l0;
        f[p] = l0 * l1;
        f[2 * p] = l1 * l1;
        f[3 * p] = 0.0;
        f[4 * p] = l0;
        f[5 * p] = l1;
      }
      __syncthreads();
      for (int it = tid; it < NP2; it += A64_NT) {   // z: one thread per (pair, qx, qy)
        const int g = it / p2, qxy = it - g * p2;
        const double *pa = pe + (int64_t)pr[2 * g] * 4 * Q + pq + qxy;
        const double *pb = pe + (int64_t)pr[2 * g + 1] * 4 * Q + pq + qxy;
        const bool diag = pa == pb;
        const double *f = F + 12 * p;
        double a[22];
#pragma unroll
        for (int u = 0; u < 22; ++u) a[u] = 0.0;
        for (int qz = 0; qz < p; ++qz) {
          const int64_t q = qs + qxy + p2 * qz;
          const int z = p2 * qz;
          const double w = P.w[q], a0 = pa[z], b0 = pb[z], wb = w * b0, fA = a0 * wb;
          const double u0 = f[qz], u1 = f[p + qz], u2 = f[2 * p + qz];
          a[0] = fma(fA, u0, a[0]);
          a[1] = fma(fA, u1, a[1]);
          a[2] = fma(fA, u2, a[2]);
          if (h) {
            double a1 = pa[Q + z], a2 = pa[2 * Q + z], a3 = pa[3 * Q + z];
            double b1 = pb[Q + z], b2 = pb[2 * Q + z], b3 = pb[3 * Q + z];
            const double l0 = f[4 * p + qz], l1 = f[5 * p + qz];
            const double fE = fma(P.V[q], fA, 0.5 * w * fma(a1, b1, fma(a2, b2, a3 * b3)));
            a[3] = fma(fE, u0, a[3]);
            a[4] = fma(fE, u1, a[4]);
            a[5] = fma(fE, u2, a[5]);
            if (GEN) {   // J^-1 grad
              const double ax = a1, ay = a2, az = a3, bx = b1, by = b2, bz = b3;
              a1 = P.jit[0] * ax + P.jit[3] * ay + P.jit[6] * az;
              a2 = P.jit[1] * ax + P.jit[4] * ay + P.jit[7] * az;
              a3 = P.jit[2] * ax + P.jit[5] * ay + P.jit[8] * az;
              b1 = P.jit[0] * bx + P.jit[3] * by + P.jit[6] * bz;
              b2 = P.jit[1] * bx + P.jit[4] * by + P.jit[7] * bz;
              b3 = P.jit[2] * bx + P.jit[5] * by + P.jit[8] * bz;
            }
            const double Bx = wb * a1, By = wb * a2, Bz = wb * a3;
            a[6] = fma(Bx, u0, a[6]);
            a[7] = fma(Bx, u1, a[7]);
            a[8] = fma(Bx, u2, a[8]);
            a[12] = fma(By, u0, a[12]);
            a[13] = fma(By, u1, a[13]);
            a[14] = fma(By, u2, a[14]);
            a[18] = fma(Bz, l0, a[18]);
            a[19] = fma(Bz, l1, a[19]);
            if (!diag) {   // C of a pair alpha = beta is its B
              const double wa = w * a0, Cx = wa * b1, Cy = wa * b2, Cz = wa * b3;
              a[9] = fma(Cx, u0, a[9]);
              a[10] = fma(Cx, u1, a[10]);
              a[11] = fma(Cx, u2, a[11]);
              a[15] = fma(Cy, u0, a[15]);
              a[16] = fma(Cy, u1, a[16]);
              a[17] = fma(Cy, u2, a[17]);
              a[20] = fma(Cz, l0, a[20]);
              a[21] = fma(Cz, l1, a[21]);
            }
          }
        }
        if (diag) {
#pragma unroll
          for (int u = 0; u < 3; ++u) {
            a[9 + u] = a[6 + u];
            a[15 + u] = a[12 + u];
          }
          a[20] = a[18];
          a[21] = a[19];
        }
#pragma unroll
        for (int u = 0; u < 22; ++u)
          if (u < nr1) T1[u * NP2 + it] = a[u];
      }
      __syncthreads();
      for (int it = tid; it < nr1 * NP; it += A64_NT) {   // y: one thread per (z row, pair, qx)
        const int r = it / NP, gq = it - r * NP, g = gq / p, qx = gq - g * p;
        const double *t1 = T1 + r * NP2 + g * p2 + qx;
        // B_y, C_y (rows 12-17) on the two linears, the others on the quadratics
        const bool lin = r >= 12 && r < 18;
        const double *f = F + (6 + (lin ? 4 : 0)) * p;
        double x0 = 0.0, x1 = 0.0, x2 = 0.0;
        for (int qy = 0; qy < p; ++qy) {
          const double t = t1[p * qy];
          x0 = fma(t, f[qy], x0);
          x1 = fma(t, f[p + qy], x1);
          if (!lin) x2 = fma(t, f[2 * p + qy], x2);
        }
        const int o = r < 12 ? 3 * r : (lin ? 36 + 2 * (r - 12) : 48 + 3 * (r - 18));
        T2[o * NP + gq] = x0;
        T2[(o + 1) * NP + gq] = x1;
        if (!lin) T2[(o + 2) * NP + gq] = x2;
      }
      __syncthreads();
      for (int it = tid; it < nr2 * nc; it += A64_NT) {   // x: one thread per (y row, pair)
        const int r = it / nc, g = it - r * nc;
        const double *t2 = T2 + r * NP + g * p;
        const bool lin = r >= 18 && r < 36;   // B_x, C_x
        const double *f = F + (lin ? 4 : 0) * p;
        double x0 = 0.0, x1 = 0.0, x2 = 0.0;
        for (int qx = 0; qx < p; ++qx) {
          const double t = t2[qx];
          x0 = fma(t, f[qx], x0);
          x1 = fma(t, f[p + qx], x1);
          if (!lin) x2 = fma(t, f[2 * p + qx], x2);
        }
        double *mo = mom + g * EXE_MOM + (r < 18 ? 3 * r : (lin ? 54 + 2 * (r - 18) : 90 + 3 * (r - 36)));
        mo[0] += x0;
        mo[1] += x1;
        if (!lin) mo[2] += x2;
      }
    }
    __syncthreads();
    // <A, 1 on d> = A_0 + 2 A_1 + A_2 along d (scaled u), for the other two indices
    double *ones = F;   // [nc][3][9]; the 1D factors and stages are done with
    if (h) {
      for (int o = tid; o < 27 * nc; o += A64_NT) {
        const int g = o / 27, r = o - 27 * g, d = r / 9, u = (r % 9) / 3, w = r % 3;
        const double *a = mom + g * EXE_MOM + (d == 0 ? u * 9 + w * 3 : (d == 1 ? u * 9 + w : u * 3 + w));
        const int st = d == 0 ? 1 : (d == 1 ? 3 : 9);
        ones[o] = fma(2.0, a[st], a[0] + a[2 * st]);
      }
      __syncthreads();
    }
    // entries (v, alpha) x (v', beta) and, for alpha != beta, their transposes
    for (int it = tid; it < nc * 64; it += A64_NT) {
      const int g = it >> 6, v = (it >> 3) & 7, vp = it & 7;
      const int al = pr[2 * g], be = pr[2 * g + 1];
      const int r = scol[al * 8 + v], c = scol[be * 8 + vp];
      if (r < 0 || c < 0) continue;
      const double *M = mom + g * EXE_MOM, *A1 = ones + 27 * g;
      const int bx = v & 1, by = (v >> 1) & 1, bz = v >> 2, cx = vp & 1, cy = (vp >> 1) & 1, cz = vp >> 2;
      const int kx = bx + cx, ky = by + cy, kz = bz + cz, kzy = (kz * 3 + ky);
      const double sv = M[kzy * 3 + kx];
      double hv = 0.0;
      if (h) {   // (signs picked, not multiplied: no FP64 operation goes into them)
        hv = M[27 + kzy * 3 + kx];
        hv = fma(bx == cx ? cq[0] : -cq[0], A1[kzy], hv);
        hv = fma(by == cy ? cq[1] : -cq[1], A1[9 + kz * 3 + kx], hv);
        hv = fma(bz == cz ? cq[2] : -cq[2], A1[18 + ky * 3 + kx], hv);
        hv = fma(bx ? c1[0] : -c1[0], M[72 + kzy * 2 + cx], hv);
        hv = fma(cx ? c1[0] : -c1[0], M[54 + kzy * 2 + bx], hv);
        hv = fma(by ? c1[1] : -c1[1], M[108 + (kz * 2 + cy) * 3 + kx], hv);
        hv = fma(cy ? c1[1] : -c1[1], M[90 + (kz * 2 + by) * 3 + kx], hv);
        hv = fma(bz ? c1[2] : -c1[2], M[144 + (cz * 3 + ky) * 3 + kx], hv);
        hv = fma(cz ? c1[2] : -c1[2], M[126 + (bz * 3 + ky) * 3 + kx], hv);
        if (GEN) {
          // 1/2 G_de s_d s'_e <A, l_b'd on d, l_be on e> for d != e, with
          // l_t = (u_t + u_(t+1)) / 2
          const int b3[3] = {bx, by, bz}, c3[3] = {cx, cy, cz}, k3[3] = {kx, ky, kz},
                    st[3] = {1, 3, 9};
#pragma unroll
          for (int d = 0; d < 3; ++d)
#pragma unroll
            for (int f = 0; f < 3; ++f) {
              if (d == f) continue;
              const int o = 3 - d - f;
              const double *q = M + k3[o] * st[o] + c3[d] * st[d] + b3[f] * st[f];
              const double gdf = 0.125 * P.G[3 * d + f];
              hv = fma(b3[d] == c3[f] ? gdf : -gdf,
                       q[0] + q[st[d]] + q[st[f]] + q[st[d] + st[f]], hv);
            }
        }
      }
      const int i = P.nfe + r, j = P.nfe + c;
      const int ci = BLOCH ? es[i] : 0, cj = BLOCH ? es[j] : 0;
      add_entry<BLOCH>(P, m[i * n + j], hv, sv, h, ws, ci, cj);
      if (al != be) add_entry<BLOCH>(P, m[j * n + i], hv, sv, h, ws, cj, ci);
    }
  }
}

// ---- enrichment x enrichment block, direct products over the points [qa, qb) ----
// Per chunk of points the columns' sqrt(w/2) grad b_r, sqrt(w) b_r and V sqrt(w) b_r
// go to shared memory; a thread owns up to EED_PER entries (r, c), c <= r, and the
// PG groups of threads that an element of few entries leaves split the points.
// One entry per thread instead of a register tile: an FP64 multiply-add takes
// the SM 16 cycles per warp against 2 for a shared-memory read of 8 bytes, so
// reads are not what bounds it, and no lane works on a tile's padding.
constexpr int EED_PER = 4;

template <bool BLOCH, bool GEN>
__device__ void eed_item(const Asm64 &P, int e, int qa, int qb, double *sm) {
  const int tid = threadIdx.x;
  const bool h = (P.want & PUFE_WANT_H) != 0, ws = (P.want & PUFE_WANT_S) != 0;
  const int n = (int)(P.doff[e + 1] - P.doff[e]), nE = n - P.nfe, nent = nE * (nE + 1) / 2;
  const int64_t q0 = P.qoff[e];
  const int Q = (int)(P.qoff[e + 1] - q0);
  const double *pe = P.psi + 4 * P.toff[e];
  const int32_t *ec = P.ecol + (P.doff[e] - (int64_t)P.nfe * e);
  const int32_t *m = P.smap + P.soff[e];
  const uint8_t *es = P.eshift + P.doff[e];
  const int QC = max(1, min((P.work - 2 * A64_NT) / (5 * nE), qb - qa));
  double *X = sm;                   // [QC][5][nE]: three gradients, b, V b
  double *red = sm + 5 * nE * QC;   // [2][A64_NT]
  const int PG = max(1, A64_NT / nent);
  const int grp = nent < A64_NT ? tid / nent : 0, e0 = nent < A64_NT ? tid % nent : tid;
  for (int base = 0; base < nent; base += EED_PER * A64_NT) {
    int r[EED_PER], c[EED_PER];
    double hs[EED_PER], ss[EED_PER];
#pragma unroll
    for (int u = 0; u < EED_PER; ++u) {
      const int t = base + e0 + u * A64_NT;
      r[u] = c[u] = -1;
      hs[u] = ss[u] = 0.0;
      if (t < nent && grp < PG) {
        int i = (int)((sqrtf(8.0f * t + 1.0f) - 1.0f) * 0.5f);
        while ((i + 1) * (i + 2) / 2 <= t) ++i;
        while (i * (i + 1) / 2 > t) --i;
        r[u] = i;
        c[u] = t - i * (i + 1) / 2;
      }
    }
    for (int qc = qa; qc < qb; qc += QC) {
      const int nq = min(QC, qb - qc);
      __syncthreads();
      for (int it = tid; it < nq * nE; it += A64_NT) {
        const int qq = it / nE, j = it - qq * nE, q = qc + qq;
        const int code = ec[j], lv = code & 7;
        const double *ps = pe + (int64_t)(code >> 3) * 4 * Q + q, *x = P.xi + 3 * (q0 + q);
        const double sx = lv & 1 ? 1.0 : -1.0, sy = lv & 2 ? 1.0 : -1.0, sz = lv & 4 ? 1.0 : -1.0;
        const double lx = fma(sx, x[0], 1.0), ly = fma(sy, x[1], 1.0), lz = fma(sz, x[2], 1.0);
        const double w1 = 0.125 * sqrt(P.w[q0 + q]), w2 = w1 * 0.70710678118654752440;
        const double yz = ly * lz, phi = lx * yz, v = ps[0], b = w1 * phi * v;
        double *o = X + qq * 5 * nE + j;
        if (h) {
          double dx = sx * yz, dy = sy * lx * lz, dz = sz * lx * ly;   // 8 grad_xi phi
          if (GEN) {
            const double gx = dx, gy = dy, gz = dz;
            dx = P.jit[0] * gx + P.jit[1] * gy + P.jit[2] * gz;
            dy = P.jit[3] * gx + P.jit[4] * gy + P.jit[5] * gz;
            dz = P.jit[6] * gx + P.jit[7] * gy + P.jit[8] * gz;
          } else {
            dx *= P.sc[0];
            dy *= P.sc[1];
            dz *= P.sc[2];
          }
          o[0] = w2 * fma(phi, ps[Q], dx * v);
          o[nE] = w2 * fma(phi, ps[2 * Q], dy * v);
          o[2 * nE] = w2 * fma(phi, ps[3 * Q], dz * v);
          o[4 * nE] = P.V[q0 + q] * b;
        }
        o[3 * nE] = b;
      }
      __syncthreads();
#pragma unroll
      for (int u = 0; u < EED_PER; ++u) {
        if (r[u] < 0) continue;
        const double *xr = X + r[u], *xc = X + c[u];
        double a = hs[u], b = ss[u];
        for (int qq = grp; qq < nq; qq += PG) {
          const double *yr = xr + qq * 5 * nE, *yc = xc + qq * 5 * nE;
          const double z = yc[3 * nE];
          b = fma(yr[3 * nE], z, b);
          if (h) {
            a = fma(yr[0], yc[0], a);
            a = fma(yr[nE], yc[nE], a);
            a = fma(yr[2 * nE], yc[2 * nE], a);
            a = fma(yr[4 * nE], z, a);
          }
        }
        hs[u] = a;
        ss[u] = b;
      }
    }
    if (PG > 1) {   // the point groups of one entry meet in shared memory
      __syncthreads();
      for (int o = tid; o < 2 * A64_NT; o += A64_NT) red[o] = 0.0;
      __syncthreads();
      if (r[0] >= 0) {
        atomicAdd(red + e0, hs[0]);
        atomicAdd(red + A64_NT + e0, ss[0]);
      }
      __syncthreads();
      if (grp > 0) r[0] = -1;
      hs[0] = red[e0];
      ss[0] = red[A64_NT + e0];
    }
#pragma unroll
    for (int u = 0; u < EED_PER; ++u) {
      if (r[u] < 0) continue;
      const int i = P.nfe + r[u], j = P.nfe + c[u];
      const int ci = BLOCH ? es[i] : 0, cj = BLOCH ? es[j] : 0;
      add_entry<BLOCH>(P, m[i * n + j], hs[u], ss[u], h, ws, ci, cj);
      if (i != j) add_entry<BLOCH>(P, m[j * n + i], hs[u], ss[u], h, ws, cj, ci);
    }
  }
}

template <bool BLOCH, bool GEN>
__global__ void __launch_bounds__(A64_NT) k_assemble_sf64(Asm64 P) {
  extern __shared__ __align__(16) double sm64[];
  const int32_t *it = P.items + 6ll * blockIdx.x;
  const int e = it[0], kind = it[1], a = it[2], b = it[3], cb = it[4], ce = it[5];
  if (kind == 0)
    fefe_item<BLOCH>(P, e, cb, ce, sm64);
  else if (kind == 1)
    fxe_item<BLOCH, GEN>(P, e, a, b, cb, ce, sm64);
  else if (kind == 2)
    exe_item<BLOCH, GEN>(P, e, a, b, cb, ce, sm64);
  else
    eed_item<BLOCH, GEN>(P, e, a, b, sm64);
}

// shared doubles of one item
int fefe_doubles(int p, bool ser) {
  return 1000 + std::max(30 * p + 10 * p * p + 100 * p, ser ? 2048 : 0);
}
int fxe_doubles(int G, int p, bool gen, bool ser) {
  return (FXE_MOM + 4) * G +
         std::max(FXE_EXP + (gen ? FXE_EXP_GEN : 0) + (ser ? FXE_EXP_SER : 0),
                  15 * p + G * (24 * p * p + 115 * p));
}
int exe_doubles(int A, int nc, int p) {
  return 4 * A + 18 * p + nc * (22 * p * p + 60 * p + EXE_MOM + 1);
}

// work area of a CTA: 56 KB, so that four CTAs share an SM (FP64 issue needs
// few warps; more shared memory would only serve more slots or pairs between
// barriers)
constexpr int A64_WORK = 7000;

}  // namespace

// Operations of an element's enrichment-enrichment block: the direct products of
// its nE columns (5 multiply-adds per point and entry of the lower triangle, 20
// operations per point and column to form the columns) and the pair form of its
// A slots (`cells`: its (sub)cells' points per axis)
static double ee_direct_ops(int nE, double points) {
  return points * (2.5 * nE * (nE + 1.0) + 20.0 * nE);
}
static double ee_pair_ops(const std::vector<int32_t> &cells) {
  double c = 64.0 * 12.0;
  for (double p : cells) c += 36 * p * p * p + 60 * p * p + 162 * p;
  return c;
}

// Work list of the sum-factorized FP64 assembly (host): items (element, kind 0
// FE x FE / 1 slot range / 2 pair range / 3 point range of the direct E x E
// products, begin, end, (sub)cell range), largest first.  Items are cut to the
// mean cost of a CTA slot (four per SM) as far as slots, pairs and points allow,
// then by (sub)cells where the cells' work is several times what a range adds
// (the expansion of its moments and the scatter); slot ranges also to what the
// shared work area holds.  The E x E block takes the form of
// fewer operations: slots of one vertex column each (64 + 30 functions, 30 slots,
// 4,096 points: 12 M direct against 88 M) fall on the direct side, slots of eight
// (64 + 40, 5 slots, 216 points: 1.06 M against 0.18 M) on the other.
void sf64_work_list(const pufe_ctx *ctx, std::vector<int32_t> &items, int &work) {
  const int nsm = ctx->nsm;
  items.clear();
  work = 0;
  if (!ctx->fe_exact || ctx->max_part_p > 16) return;
  const int64_t ne = (int64_t)ctx->n_e.size();
  struct Item {
    int32_t e, kind, a, b, cb, ce;
    double c;
  };
  double total = 0.0;
  std::vector<double> cf(ne), cs(ne), cp(ne), cd(ne);
  std::vector<int> pm(ne);
  for (int64_t e = 0; e < ne; ++e) {
    cf[e] = 4096;
    cs[e] = 11500;
    for (int p : ctx->part_p_host[e]) {
      const double d = p;
      pm[e] = std::max(pm[e], p);
      cf[e] += 10 * d * d * d + 100 * d * d + 1000 * d;
      cs[e] += 30 * d * d * d + 115 * d * d + 550 * d;
    }
    const double A = ctx->n_slot[e], np = 0.5 * A * (A + 1);
    cp[e] = ee_pair_ops(ctx->part_p_host[e]);
    cd[e] = ee_direct_ops(ctx->n_e[e] - ctx->nfe_e, ctx->q_e[e]);
    total += cf[e] + A * cs[e] + std::min(np * cp[e], cd[e]);
  }
  const double target = std::max(1.0, total / (4.0 * nsm));
  std::vector<Item> L;
  // one range over (sub)cell ranges of at least `least` operations
  auto cells = [&](int64_t e, int kind, int a, int b, double c, double least) {
    const int nc = (int)ctx->part_p_host[e].size();
    const double m = std::min(std::min(std::ceil(c / target), c / least), (double)nc);
    const int cuts = std::max(1, (int)m);
    for (int j = 0; j < cuts; ++j)
      L.push_back(Item{(int32_t)e, kind, a, b, (int)((int64_t)j * nc / cuts),
                       (int)((int64_t)(j + 1) * nc / cuts), c / cuts});
  };
  for (int64_t e = 0; e < ne; ++e) {
    const int A = ctx->n_slot[e], np = A * (A + 1) / 2, p = pm[e], nE = ctx->n_e[e] - ctx->nfe_e;
    cells(e, 0, 0, 0, cf[e], 40000.0);
    work = std::max(work, fefe_doubles(p, ctx->ser));
    if (A == 0) continue;
    int G = std::max(1, std::min(A, (int)std::min(1e6, target / cs[e])));
    while (G > 1 && fxe_doubles(G, p, ctx->general, ctx->ser) > A64_WORK) --G;
    work = std::max(work, fxe_doubles(G, p, ctx->general, ctx->ser));
    for (int a = 0; a < A; a += G)
      cells(e, 1, a, std::min(A, a + G), cs[e] * std::min(G, A - a), 40000.0 * G);
    if (cd[e] < np * cp[e]) {
      const int Q = ctx->q_e[e];
      const int cuts = std::max(1, std::min(Q / 32, (int)std::min(1e6, std::ceil(cd[e] / target))));
      work = std::max(work, 5 * nE + 2 * A64_NT);
      work = std::max(work, std::min(A64_WORK, 5 * nE * ((Q + cuts - 1) / cuts) + 2 * A64_NT));
      for (int j = 0; j < cuts; ++j) {
        const int a = (int)((int64_t)j * Q / cuts), b = (int)((int64_t)(j + 1) * Q / cuts);
        L.push_back(Item{(int32_t)e, 3, a, b, 0, 0, cd[e] * (b - a) / Q});
      }
      continue;
    }
    work = std::max(work, exe_doubles(A, 1, p));
    const int M = std::max(1, std::min(np, (int)std::min(1e6, target / cp[e])));
    const int cuts = (np + M - 1) / M;
    for (int j = 0; j < cuts; ++j) {
      const int a = (int)((int64_t)j * np / cuts), b = (int)((int64_t)(j + 1) * np / cuts);
      cells(e, 2, a, b, cp[e] * (b - a), 8000.0 * (b - a));
      for (int c = b - a; c > 1; --c)   // pairs that fit the work area together
        if (exe_doubles(A, c, p) <= A64_WORK) {
          work = std::max(work, exe_doubles(A, c, p));
          break;
        }
    }
  }
  std::stable_sort(L.begin(), L.end(), [](const Item &x, const Item &y) { return x.c > y.c; });
  for (const Item &i : L) items.insert(items.end(), {i.e, i.kind, i.a, i.b, i.cb, i.ce});
}

// H (and Hi, Si at a wavevector: ph != nullptr) must hold zeros, S the summed
// FE-FE overlap constants
pufe_status launch_assemble_sf64(pufe_ctx *ctx, const PhaseTab *ph, const double *V, int what,
                                 double *H, double *Hi, double *S, double *Si, cudaStream_t st) {
  auto &D = ctx->d;
  Asm64 P{};
  P.items = D.aitems;
  P.qoff = D.qoff;
  P.w = D.w;
  P.xi = D.xi;
  P.partoff = D.partoff;
  P.part_p = D.part_p;
  P.part_q = D.part_q;
  P.doff = D.doff;
  P.ecol = D.ecol;
  P.aoff = D.aoff;
  P.toff = D.toff;
  P.psi = D.psi;
  P.soff = D.soff;
  P.smap = D.smap;
  P.V = V;
  P.Tfe = D.Tfe;
  P.Sfe = D.Sfe;
  P.H = H;
  P.Hi = Hi;
  P.S = S;
  P.Si = Si;
  P.eshift = D.eshift;
  if (ph) P.ph = *ph;
  for (int d = 0; d < 3 && !ctx->general; ++d) P.sc[d] = 2.0 / ctx->h[d];
  if (ctx->general)
    for (int d = 0; d < 3; ++d)
      for (int c = 0; c < 3; ++c) {
        P.jit[3 * d + c] = ctx->Jit[3 * d + c];
        for (int r = 0; r < 3; ++r) P.G[3 * d + c] += ctx->Jit[3 * r + d] * ctx->Jit[3 * r + c];
      }
  P.ri = D.rser_i;
  P.rv = D.rser_v;
  P.rl = ctx->rser_len;
  P.nfe = ctx->nfe_e;
  P.want = what;
  P.work = ctx->asm64_work;
  P.err = D.err;
  const size_t sm = (size_t)ctx->asm64_work * sizeof(double);
  if (sm > 227 * 1024) return fail(PUFE_EINVAL, "element too large for the FP64 assembly");
  auto kern = ph ? (ctx->general ? k_assemble_sf64<true, true> : k_assemble_sf64<true, false>)
                 : (ctx->general ? k_assemble_sf64<false, true> : k_assemble_sf64<false, false>);
  PUFE_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
  kern<<<(unsigned)ctx->n_aitems, A64_NT, sm, st>>>(P);
  PUFE_CUDA_TRY(cudaGetLastError());
  return PUFE_OK;
}

}  // namespace pufe
