// FP64 quantities at the quadrature points by sum factorization on the p^3
// (sub)cells: the adjoint of V -> H and the density.
//
// As in the FP64 assembly (pufe_sf64.cu) the two FP64 multiply-adds per clock
// and SM are what binds, so the forms are those of fewest FP64 operations and
// shared-memory reads, gathers and the atomics on the outputs hide behind them.
//
// Adjoint, Vbar_q = w_q b_q^T Hbar_e b_q, as polynomials in the 1D factors of the
// element, evaluated axis by axis (x, y, z):
//  * FE x FE: Hbar_e enters only through its sums over the index swaps of each
//    axis, 1,000 coefficients on the products L_a L_b: 4,096 additions, then
//    1,000 p + 100 p^2 + 10 p^3 operations per cell against the 4,096 p +
//    256 p^2 + 16 p^3 of the unsymmetrised contraction.
//  * FE x enrichment, per slot: sum_v phi_v sum_j (Hbar_rj + Hbar_jr) phi_j is a
//    polynomial of degree 4 per axis (M_a,t = (1 + s x_a) L_a + s kappa_a omega):
//    its 512 coefficients are collapsed to 125 on {L_0..L_3, omega}
//    (2 operations per entry), evaluated in 125 p + 25 p^2 + 5 p^3 and
//    multiplied by Psi.
//  * enrichment x enrichment, per slot pair: 27 coefficients on the quadratics,
//    27 p + 9 p^2 + 3 p^3, times Psi_a Psi_b; or the direct products of the
//    columns where the slots hold few vertices.
// 97,000 operations for an element of 104 functions and 6^3 points against the
// 2,360,000 of contracting the element's whole block at every point.  The parts add into Vbar (zeroed
// first) with one atomic per point, so that an element's parts can run on
// different SMs.
//
// Density, n_q = sum_k f_k (sum_j B_qj C_jk)^2: the 64 tricubic functions by
// sum factorization per state (64 p + 16 p^2 + 4 p^3 against 64 p^3), the
// enrichment columns directly, each point's b_r formed once for the group of up to 16
// columns that its thread carries.
//
// Measured, direct kernels before: adjoint 12^3 rocksalt 9.34 -> 0.35 ms, CsCl-like
// 16^3 19.4 -> 0.60 ms, two-atom 4^3 1.06 -> 0.031 ms; density 0.80 -> 0.23 ms (8
// states), 17.5 -> 0.99 ms (35 states), 0.21 -> 0.025 ms (2 states).
#include <cooperative_groups.h>

#include <algorithm>

#include "pufe_internal.h"

namespace pufe {
namespace {

constexpr int P64_NT = 128;
constexpr int P64_WORK = 7000;   // shared doubles of an adjoint CTA: 56 KB, four CTAs per SM
// Direct enrichment blocks of the adjoint.  A triangle goes through shared memory whole,
// beside 64 points, up to P64_WHOLE doubles (163 columns); larger ones in ranges of
// rows of P64_ROWS doubles (112 KB, two CTAs per SM), with room for P64_QC_MIN points.
// Eight elements of one-vertex slots and 4^3 points: 150 columns 217 us whole, 225 us in
// ranges; 185 columns 331 and 262 us.
constexpr int P64_WHOLE = 24000, P64_ROWS = 14000, P64_QC_MIN = 16, P64_MAX = 227 * 1024 / 8;

struct Adj64 {
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
  const double *Hr, *Hi;
  const uint8_t *eshift;
  PhaseTab ph;
  double *out;
  const double *Rser;   // serendipity space: nodal values 64 x 32 (nfe = 32)
  int nfe, work;
};

// the element's cotangent entries (the phased real part at a wavevector)
template <bool BLOCH>
struct CotElem {
  const double *Hr, *Hi;
  const int32_t *m;
  const uint8_t *es;
  const PhaseTab *ph;
  int n;
  __device__ __forceinline__ double operator()(int i, int j) const {
    const int32_t sl = m[(int64_t)i * n + j];
    return BLOCH ? cot_entry(Hr[sl], Hi[sl], es[i], es[j], *ph) : Hr[sl];
  }
};

template <bool BLOCH>
__device__ __forceinline__ CotElem<BLOCH> cot_elem(const Adj64 &P, int e) {
  return CotElem<BLOCH>{P.Hr, P.Hi, P.smap + P.soff[e], P.eshift + P.doff[e], &P.ph,
                        (int)(P.doff[e + 1] - P.doff[e])};
}

__device__ __forceinline__ double pt_axis_xi(const double *xi, int64_t qs, int p, int d, int t) {
  const int64_t stride = d == 0 ? 1 : (d == 1 ? p : (int64_t)p * p);
  return xi[3 * (qs + t * stride) + d];
}
__device__ __forceinline__ double pt_node(int a) { return -1.0 + a * (2.0 / 3.0); }
__device__ __forceinline__ double pt_kappa(int a) {
  return (a & 1 ? 1.0 : -1.0) * (a == 0 || a == 3 ? 0.5625 : 1.6875);
}
// unordered pairs 0..9 of four indices
__device__ __forceinline__ int pair_lo(int c) { return c < 4 ? 0 : (c < 7 ? 1 : (c < 9 ? 2 : 3)); }
__device__ __forceinline__ int pair_hi(int c) {
  return c < 4 ? c : (c < 7 ? c - 3 : (c < 9 ? c - 5 : 3));
}

template <bool BLOCH>
__device__ void adj_fefe(const Adj64 &P, int e, int cb, int ce, double *sm) {
  const int tid = threadIdx.x;
  const CotElem<BLOCH> H = cot_elem<BLOCH>(P, e);
  double *C = sm, *X = sm + 1000;   // coefficients [z][y][x]; the gathered block, then the stages
  if (P.nfe == 64) {
#pragma unroll 4
    for (int o = tid; o < 4096; o += P64_NT) X[o] = H(o >> 6, o & 63);
  } else {   // serendipity: R Hbar R^T, R the nodal values of its functions
    double *Y = X + 4096;
    for (int o = tid; o < 1024; o += P64_NT) X[o] = H(o >> 5, o & 31);
    __syncthreads();
    // (a warp works on one node, whose zeros it skips as a whole; R Hbar is kept
    // transposed, [32][64], and the result too: the sums below take both halves)
    for (int o = tid; o < 2048; o += P64_NT) {
      const int j = o >> 5, d = o & 31;
      double s = 0.0;
      for (int c = 0; c < 32; ++c) {
        const double r = P.Rser[j * 32 + c];
        if (r != 0.0) s = fma(r, X[c * 32 + d], s);
      }
      Y[d * 64 + j] = s;
    }
    __syncthreads();
    for (int o = tid; o < 4096; o += P64_NT) {
      const int j = o >> 6, i = o & 63;
      double s = 0.0;
      for (int c = 0; c < 32; ++c) {
        const double r = P.Rser[j * 32 + c];
        if (r != 0.0) s = fma(r, Y[c * 64 + i], s);
      }
      X[o] = s;
    }
  }
  __syncthreads();
  for (int o = tid; o < 1000; o += P64_NT) {
    const int x = o % 10, y = (o / 10) % 10, z = o / 100;
    const int a[2] = {pair_lo(x), pair_hi(x)}, b[2] = {pair_lo(y), pair_hi(y)},
              c[2] = {pair_lo(z), pair_hi(z)};
    double s = 0.0;
    for (int u = 0; u < 8; ++u) {   // the swaps of each axis pair (equal indices: one)
      const int ux = u & 1, uy = (u >> 1) & 1, uz = u >> 2;
      if ((ux && a[0] == a[1]) || (uy && b[0] == b[1]) || (uz && c[0] == c[1])) continue;
      s += X[(a[ux] + 4 * b[uy] + 16 * c[uz]) * 64 + a[1 - ux] + 4 * b[1 - uy] + 16 * c[1 - uz]];
    }
    C[o] = s;
  }
  for (int k = P.partoff[e] + cb; k < P.partoff[e] + ce; ++k) {
    const int p = P.part_p[k], p2 = p * p, p3 = p2 * p;
    const int64_t qs = P.qoff[e] + P.part_q[k];
    double *F = X, *T1 = F + 30 * p, *T2 = T1 + 100 * p;   // [axis][10][p], [z y][p], [z][p^2]
    __syncthreads();
    for (int o = tid; o < 3 * p; o += P64_NT) {
      const int d = o / p, t = o - d * p;
      double L[4], dL[4];
      lagrange3(pt_axis_xi(P.xi, qs, p, d, t), L, dL);
      int c = 0;
      for (int a = 0; a < 4; ++a)
        for (int b = a; b < 4; ++b) F[(d * 10 + c++) * p + t] = L[a] * L[b];
    }
    __syncthreads();
    for (int o = tid; o < 100 * p; o += P64_NT) {
      const int r = o / p, qx = o - r * p;
      double s = 0.0;
#pragma unroll
      for (int c = 0; c < 10; ++c) s = fma(C[r * 10 + c], F[c * p + qx], s);
      T1[o] = s;
    }
    __syncthreads();
    for (int o = tid; o < 10 * p2; o += P64_NT) {
      const int z = o / p2, r = o - z * p2, qy = r / p, qx = r - qy * p;
      double s = 0.0;
#pragma unroll
      for (int c = 0; c < 10; ++c) s = fma(T1[(z * 10 + c) * p + qx], F[(10 + c) * p + qy], s);
      T2[o] = s;
    }
    __syncthreads();
    for (int q = tid; q < p3; q += P64_NT) {
      const int qz = q / p2, r = q - qz * p2;
      double s = 0.0;
#pragma unroll
      for (int c = 0; c < 10; ++c) s = fma(T2[c * p2 + r], F[(20 + c) * p + qz], s);
      atomicAdd(P.out + qs + q, P.w[qs + q] * s);
    }
  }
}

// shared doubles of the FE x FE part and, per slot and per pair, of the others
int adj_fefe_doubles(int p, bool ser) {
  return 1000 + std::max(ser ? 6144 : 4096, 130 * p + 10 * p * p);
}
__host__ __device__ inline int adj_slot_doubles(int p) {
  const int ev = 25 * p + 5 * p * p;
  return 125 + (ev > 832 ? ev : 832);
}
__host__ __device__ inline int adj_pair_doubles(int p) { return 28 + 9 * p + 3 * p * p; }

template <bool BLOCH>
__device__ void adj_slots(const Adj64 &P, int e, int s0, int s1, int cb, int ce, double *sm) {
  const int tid = threadIdx.x, G = s1 - s0;
  const CotElem<BLOCH> H = cot_elem<BLOCH>(P, e);
  const int nE = H.n - P.nfe;
  const int64_t q0 = P.qoff[e];
  const int Q = (int)(P.qoff[e + 1] - q0);
  const double *pe = P.psi + 4 * P.toff[e];
  const int32_t *ec = P.ecol + (P.doff[e] - (int64_t)P.nfe * e);
  int *scol = reinterpret_cast<int *>(sm);   // [G][8]
  double *K = sm + 4 * G, *base = K + 125 * G;
  double *R = base, *X = R + 512 * G, *Y = R;   // [g][z 8][y 8][x 8] -> [g][zy][5] -> [g][z 8][25]
  for (int o = tid; o < 8 * G; o += P64_NT) scol[o] = -1;
  __syncthreads();
  for (int o = tid; o < nE; o += P64_NT) {
    const int c = ec[o] - 8 * s0;
    if (c >= 0 && c < 8 * G) scol[c] = o;
  }
  __syncthreads();
  if (P.nfe == 32) {   // serendipity: its 32 coefficients per vertex first
    for (int o = tid; o < 256 * G; o += P64_NT) {   // [function][slot, vertex]
      const int j = o & 31, gv = o >> 5, r = scol[gv];
      X[j * 8 * G + gv] = r < 0 ? 0.0 : H(32 + r, j) + H(j, 32 + r);
    }
    __syncthreads();
  }
#pragma unroll 4
  for (int o = tid; o < 512 * G; o += P64_NT) {   // (vertex, tricubic function) coefficients
    // lanes along the functions of one vertex, or (serendipity) along the vertices
    // of one node, whose nonzeros they share
    const int j = P.nfe == 64 ? o & 63 : o / (8 * G), gv = P.nfe == 64 ? o >> 6 : o % (8 * G);
    const int v = gv & 7, r = scol[gv];
    double c = 0.0;
    if (P.nfe == 64) {
      if (r >= 0) c = H(64 + r, j) + H(j, 64 + r);
    } else {
      for (int k = 0; k < 32; ++k) {
        const double w = P.Rser[j * 32 + k];
        if (w != 0.0) c = fma(w, X[k * 8 * G + gv], c);
      }
    }
    const int x = (j & 3) + 4 * (v & 1), y = ((j >> 2) & 3) + 4 * ((v >> 1) & 1),
              z = (j >> 4) + 4 * (v >> 2);
    R[(gv >> 3) * 512 + (z * 8 + y) * 8 + x] = c;
  }
  // eight coefficients on M_a,t at stride `st` -> five on {L_0..L_3, omega}
  auto collapse = [](const double *h, int st, double o[5]) {
    o[4] = 0.0;
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      const double h0 = h[a * st], h1 = h[(4 + a) * st];
      o[a] = fma(1.0 - pt_node(a), h0, (1.0 + pt_node(a)) * h1);
      o[4] = fma(pt_kappa(a), h1 - h0, o[4]);
    }
  };
  __syncthreads();
  for (int o = tid; o < 64 * G; o += P64_NT) {
    double c[5];
    collapse(R + 8 * o, 1, c);
    for (int u = 0; u < 5; ++u) X[5 * o + u] = c[u];
  }
  __syncthreads();
  for (int o = tid; o < 40 * G; o += P64_NT) {   // (g z, x 5)
    const int gz = o / 5, x = o - 5 * gz;
    double c[5];
    collapse(X + gz * 40 + x, 5, c);
    for (int u = 0; u < 5; ++u) Y[gz * 25 + 5 * u + x] = c[u];
  }
  __syncthreads();
  for (int o = tid; o < 25 * G; o += P64_NT) {   // (g, yx 25)
    const int g = o / 25, yx = o - 25 * g;
    double c[5];
    collapse(Y + g * 200 + yx, 25, c);
    for (int u = 0; u < 5; ++u) K[g * 125 + 25 * u + yx] = 0.125 * c[u];
  }
  for (int k = P.partoff[e] + cb; k < P.partoff[e] + ce; ++k) {
    const int p = P.part_p[k], p2 = p * p, p3 = p2 * p, pq = P.part_q[k];
    const int64_t qs = q0 + pq;
    double *T1 = base, *T2 = T1 + 25 * G * p, *F = sm + P.work - 15 * p;
    __syncthreads();
    for (int o = tid; o < 3 * p; o += P64_NT) {
      const int d = o / p, t = o - d * p;
      const double x = pt_axis_xi(P.xi, qs, p, d, t);
      double L[4], dL[4];
      lagrange3(x, L, dL);
      double *f = F + d * 5 * p + t;
      for (int a = 0; a < 4; ++a) f[a * p] = L[a];
      f[4 * p] = (x + 1.0) * (x + 1.0 / 3.0) * (x - 1.0 / 3.0) * (x - 1.0);
    }
    __syncthreads();
    for (int o = tid; o < 25 * G * p; o += P64_NT) {   // (g z y, qx)
      const int r = o / p, qx = o - r * p;
      double s = 0.0;
#pragma unroll
      for (int u = 0; u < 5; ++u) s = fma(K[r * 5 + u], F[u * p + qx], s);
      T1[o] = s;
    }
    __syncthreads();
    for (int o = tid; o < 5 * G * p2; o += P64_NT) {   // (g z, qx qy)
      const int r = o / p2, xy = o - r * p2, qy = xy / p, qx = xy - qy * p;
      double s = 0.0;
#pragma unroll
      for (int u = 0; u < 5; ++u) s = fma(T1[(r * 5 + u) * p + qx], F[(5 + u) * p + qy], s);
      T2[o] = s;
    }
    __syncthreads();
    for (int q = tid; q < p3; q += P64_NT) {
      const int qz = q / p2, xy = q - qz * p2;
      double fz[5], s = 0.0;
#pragma unroll
      for (int u = 0; u < 5; ++u) fz[u] = F[(10 + u) * p + qz];
      for (int g = 0; g < G; ++g) {
        double t = 0.0;
#pragma unroll
        for (int u = 0; u < 5; ++u) t = fma(T2[(g * 5 + u) * p2 + xy], fz[u], t);
        s = fma(pe[(int64_t)(s0 + g) * 4 * Q + pq + q], t, s);
      }
      atomicAdd(P.out + qs + q, P.w[qs + q] * s);
    }
  }
}

template <bool BLOCH>
__device__ void adj_pairs(const Adj64 &P, int e, int k0, int k1, int cb, int ce, double *sm) {
  const int tid = threadIdx.x;
  const CotElem<BLOCH> H = cot_elem<BLOCH>(P, e);
  const int nE = H.n - P.nfe, A = P.aoff[e + 1] - P.aoff[e];
  const int64_t q0 = P.qoff[e];
  const int Q = (int)(P.qoff[e + 1] - q0);
  const double *pe = P.psi + 4 * P.toff[e];
  const int32_t *ec = P.ecol + (P.doff[e] - (int64_t)P.nfe * e);
  int *scol = reinterpret_cast<int *>(sm);   // [A][8]
  for (int o = tid; o < 8 * A; o += P64_NT) scol[o] = -1;
  __syncthreads();
  for (int o = tid; o < nE; o += P64_NT) scol[ec[o]] = o;
  int pmax = 1;
  for (int k = P.partoff[e]; k < P.partoff[e + 1]; ++k) pmax = max(pmax, P.part_p[k]);
  const int fit = max(1, (P.work - 4 * A - 9 * pmax) / adj_pair_doubles(pmax));
  const int nch = (k1 - k0 + fit - 1) / fit, npc = (k1 - k0 + nch - 1) / nch;
  for (int c0 = k0; c0 < k1; c0 += npc) {
    const int nc = min(npc, k1 - c0);
    double *F0 = sm + 4 * A, *K = F0 + 9 * pmax;             // factors [axis][3][p]; [nc][27]
    int *pr = reinterpret_cast<int *>(K + 27 * nc);          // [nc][2]
    double *T1 = K + 28 * nc;
    __syncthreads();
    for (int o = tid; o < nc; o += P64_NT) {   // pair c0 + o of the alpha-major list
      int a = 0, t = c0 + o;
      while (t >= A - a) t -= A - a++;
      pr[2 * o] = a;
      pr[2 * o + 1] = a + t;
    }
    __syncthreads();
    for (int o = tid; o < 27 * nc; o += P64_NT) {   // sums over the vertex pairs of each product
      const int g = o / 27, k = o - 27 * g, kx = k % 3, ky = (k / 3) % 3, kz = k / 9;
      const int al = pr[2 * g], be = pr[2 * g + 1];
      double s = 0.0;
      for (int u = 0; u < 8; ++u) {   // bits of the first vertex; the second's follow
        const int bx = u & 1, by = (u >> 1) & 1, bz = u >> 2;
        const int cx = kx - bx, cy = ky - by, cz = kz - bz;
        if ((unsigned)cx > 1u || (unsigned)cy > 1u || (unsigned)cz > 1u) continue;
        const int r = scol[al * 8 + u], c = scol[be * 8 + (cx | (cy << 1) | (cz << 2))];
        if (r < 0 || c < 0) continue;
        s += H(P.nfe + r, P.nfe + c);
        if (al != be) s += H(P.nfe + c, P.nfe + r);
      }
      K[o] = s * (1.0 / 64.0);
    }
    for (int k = P.partoff[e] + cb; k < P.partoff[e] + ce; ++k) {
      const int p = P.part_p[k], p2 = p * p, p3 = p2 * p, pq = P.part_q[k];
      const int64_t qs = q0 + pq;
      double *T2 = T1 + 9 * nc * p, *F = F0;
      __syncthreads();
      for (int o = tid; o < 3 * p; o += P64_NT) {
        const int d = o / p, t = o - d * p;
        const double x = pt_axis_xi(P.xi, qs, p, d, t), l0 = 1.0 - x, l1 = 1.0 + x;
        double *f = F + d * 3 * p + t;
        f[0] = l0 * l0;
        f[p] = l0 * l1;
        f[2 * p] = l1 * l1;
      }
      __syncthreads();
      for (int o = tid; o < 9 * nc * p; o += P64_NT) {   // (g z y, qx)
        const int r = o / p, qx = o - r * p;
        T1[o] = fma(K[r * 3], F[qx], fma(K[r * 3 + 1], F[p + qx], K[r * 3 + 2] * F[2 * p + qx]));
      }
      __syncthreads();
      for (int o = tid; o < 3 * nc * p2; o += P64_NT) {   // (g z, qx qy)
        const int r = o / p2, xy = o - r * p2, qy = xy / p, qx = xy - qy * p;
        const double *t = T1 + r * 3 * p + qx, *f = F + 3 * p + qy;
        T2[o] = fma(t[0], f[0], fma(t[p], f[p], t[2 * p] * f[2 * p]));
      }
      __syncthreads();
      for (int q = tid; q < p3; q += P64_NT) {
        const int qz = q / p2, xy = q - qz * p2;
        const double f0 = F[6 * p + qz], f1 = F[7 * p + qz], f2 = F[8 * p + qz];
        double s = 0.0;
        for (int g = 0; g < nc; ++g) {
          const double *t = T2 + g * 3 * p2 + xy;
          const double v = fma(t[0], f0, fma(t[p2], f1, t[2 * p2] * f2));
          s = fma(pe[(int64_t)pr[2 * g] * 4 * Q + pq + q] * pe[(int64_t)pr[2 * g + 1] * 4 * Q + pq + q],
                  v, s);
        }
        atomicAdd(P.out + qs + q, P.w[qs + q] * s);
      }
    }
  }
}

// direct E x E products of the block's rows [ra, rb) over the points [qa, qb): those
// rows of the symmetrised block and the columns' values of a chunk of points in shared
// memory, threads over points and row groups
template <bool BLOCH>
__device__ void adj_direct(const Adj64 &P, int e, int qa, int qb, int ra, int rb, double *sm) {
  const int tid = threadIdx.x;
  const CotElem<BLOCH> H = cot_elem<BLOCH>(P, e);
  const int h0 = ra * (ra + 1) / 2, nent = rb * (rb + 1) / 2 - h0;   // packed rows ra .. rb - 1
  const int64_t q0 = P.qoff[e];
  const int Q = (int)(P.qoff[e + 1] - q0);
  const double *pe = P.psi + 4 * P.toff[e];
  const int32_t *ec = P.ecol + (P.doff[e] - (int64_t)P.nfe * e);
  double *Hs = sm, *B = sm + nent;
  for (int o = tid; o < (rb - ra) * rb; o += P64_NT) {
    const int r = ra + o / rb, c = o % rb;
    if (c > r) continue;
    Hs[r * (r + 1) / 2 - h0 + c] =
        r == c ? H(P.nfe + r, P.nfe + r) : H(P.nfe + r, P.nfe + c) + H(P.nfe + c, P.nfe + r);
  }
  const int QC = max(1, min(min((P.work - nent) / rb, P64_NT), qb - qa)), PG = P64_NT / QC;
  const int qq = tid % QC, grp = tid / QC;
  for (int qc = qa; qc < qb; qc += QC) {
    const int nq = min(QC, qb - qc);
    __syncthreads();
    for (int o = tid; o < rb * nq; o += P64_NT) {
      const int j = o / nq, t = o - j * nq, q = qc + t, code = ec[j];
      const double *x = P.xi + 3 * (q0 + q);
      const double lx = code & 1 ? 1.0 + x[0] : 1.0 - x[0], ly = code & 2 ? 1.0 + x[1] : 1.0 - x[1],
                   lz = code & 4 ? 1.0 + x[2] : 1.0 - x[2];
      B[j * QC + t] = 0.125 * lx * (ly * lz) * pe[(int64_t)(code >> 3) * 4 * Q + q];
    }
    __syncthreads();
    if (qq < nq && grp < PG) {
      double s = 0.0;
      for (int r = ra + grp; r < rb; r += PG) {
        const double *h = Hs + r * (r + 1) / 2 - h0;
        double g = 0.0;
        for (int c = 0; c <= r; ++c) g = fma(h[c], B[c * QC + qq], g);
        s = fma(B[r * QC + qq], g, s);
      }
      atomicAdd(P.out + q0 + qc + qq, P.w[q0 + qc + qq] * s);
    }
  }
}

template <bool BLOCH>
__global__ void __launch_bounds__(P64_NT) k_adjoint_sf64(Adj64 P) {
  extern __shared__ __align__(16) double sma64[];
  const int32_t *it = P.items + 6ll * blockIdx.x;
  const int e = it[0], kind = it[1], a = it[2], b = it[3], cb = it[4], ce = it[5];
  if (kind == 0)
    adj_fefe<BLOCH>(P, e, cb, ce, sma64);
  else if (kind == 1)
    adj_slots<BLOCH>(P, e, a, b, cb, ce, sma64);
  else if (kind == 2)
    adj_pairs<BLOCH>(P, e, a, b, cb, ce, sma64);
  else
    adj_direct<BLOCH>(P, e, a, b, cb, ce, sma64);
}

// ---- density ------------------------------------------------------------------
// One CTA per (unit, group of KC real columns): a unit is a (sub)cell of an element
// and a range of its z planes, a column a state (Gamma) or the real or imaginary
// part of one (Bloch).
//
// The groups of a unit meet in an order that the launch fixes, so that the density
// repeats bit for bit (one atomic per group does not, from three groups on):
//  * two halves of the groups on two CTAs, which keep their sum in shared memory and add
//    it into the zeroed density with one atomic per point (two terms commute);
//  * from three groups on, on a mesh too small to fill the chip with that (all units and
//    groups fit four CTAs per SM), a CTA per group: up to five as one cluster, more as two
//    of them, whose CTAs read one another's sums through distributed shared memory, in
//    rank order.
// 64 complex states, against one CTA and atomic per group: eight elements of 6^3 points
// 38 -> 40 us (halves alone 85 us), 6^3 rocksalt 1,073 -> 1,140 us (clusters 1,169 us),
// 12^3 rocksalt 3,495 -> 3,447 us; 35 real states on the CsCl-like 16^3 cell 975 -> 967
// us (clusters 1,045 us); one group, which needs neither, two-atom 4^3 40 -> 35 us.
constexpr int DEN_CLUSTER = 8;   // largest portable cluster

struct Den64 {
  const int4 *units;   // element, (sub)cell, first plane, end plane
  const int64_t *qoff;
  const double *xi;
  const int32_t *part_p, *part_q;
  const int64_t *doff;
  const int32_t *dofs, *ecol;
  const int64_t *toff;
  const double *psi, *C, *Ci, *f, *Rser;
  int64_t ldc;
  int ncol, groups, nfe;
  int halves, cs;   // halves of the groups (or 1: all together), CTAs in the cluster of one
  const uint8_t *eshift;
  PhaseTab ph;
  double *rho;
};

// doubles of one column: its coefficients (64 FE functions whatever the space) and, for
// the serendipity space, its own; x and y stages
int den_column(int n, int p) { return n + 32 + 16 * p + 4 * p * p; }
// kc columns and their occupations; 1D factors; phi_v of each thread
int den_doubles(int column, int p, int kc) { return kc * (column + 1) + 12 * p + 8 * P64_NT; }

template <bool BLOCH, int KC>
__global__ void __launch_bounds__(P64_NT) k_density_sf64(Den64 P) {
  extern __shared__ __align__(16) double smd64[];
  const int4 u = P.units[blockIdx.x];
  const int tid = threadIdx.x, e = u.x;
  const int n = (int)(P.doff[e + 1] - P.doff[e]), nE = n - P.nfe;
  const int p = P.part_p[u.y], p2 = p * p, pq = P.part_q[u.y];
  const int64_t q0 = P.qoff[e], qs = q0 + pq;
  const int Q = (int)(P.qoff[e + 1] - q0);
  const double *pe = P.psi + 4 * P.toff[e];
  const int32_t *ec = P.ecol + (P.doff[e] - (int64_t)P.nfe * e), *dl = P.dofs + P.doff[e];
  const uint8_t *es = P.eshift + P.doff[e];
  double *fs = smd64, *Cs = fs + KC;            // [64 + nE][KC]
  double *L = Cs + (64 + nE) * KC;              // [axis][4][p]
  double *T1 = L + 12 * p, *T2 = T1 + 16 * p * KC;   // [bc][k][qx], [c][k][qx qy]
  double *ph8 = T2 + 4 * p2 * KC;               // [vertex][thread]
  double *acc = ph8 + 8 * P64_NT;               // [point]: sum over this CTA's groups
  double *raw = P.nfe == 64 ? Cs : T1;          // serendipity coefficients before the lift
  for (int o = tid; o < 3 * p; o += P64_NT) {
    const int d = o / p, t = o - d * p;
    double l[4], dl4[4];
    lagrange3(pt_axis_xi(P.xi, qs, p, d, t), l, dl4);
    for (int a = 0; a < 4; ++a) L[(d * 4 + a) * p + t] = l[a];
  }
  const int first = u.z * p2, np = (u.w - u.z) * p2;   // the unit's points
  // this CTA's groups: its share of all of them or of one half
  const int half = blockIdx.y / P.cs, rank = blockIdx.y - half * P.cs;
  const int cut = P.halves == 1 ? P.groups : (P.groups + 1) / 2;
  const int h0 = half ? cut : 0, hn = half ? P.groups - cut : cut;
  const int g0 = h0 + rank * hn / P.cs, g1 = h0 + (rank + 1) * hn / P.cs;
  const bool direct = P.groups <= 2;   // one group to a CTA, which needs no sum
  if (g0 == g1)
    for (int q = tid; q < np; q += P64_NT) acc[q] = 0.0;
  for (int grp = g0; grp < g1; ++grp) {
    const int k0 = grp * KC;
    __syncthreads();
    for (int o = tid; o < KC; o += P64_NT) {
      const int k = k0 + o;
      fs[o] = k < P.ncol ? P.f[BLOCH ? k >> 1 : k] : 0.0;
    }
    for (int o = tid; o < n * KC; o += P64_NT) {
      const int j = o / KC, kk = o - j * KC, k = k0 + kk;
      double c = 0.0;
      if (k < P.ncol) {
        const int64_t g = (int64_t)dl[j] * P.ldc;
        if (!BLOCH) {
          c = P.C[g + k];
        } else {   // real (even k) or imaginary part of the phased coefficient
          const double ar = P.C[g + (k >> 1)], ai = P.Ci[g + (k >> 1)];
          const int s = es[j];
          c = k & 1 ? P.ph.re[s] * ai + P.ph.im[s] * ar : P.ph.re[s] * ar - P.ph.im[s] * ai;
        }
      }
      if (j < P.nfe)
        raw[o] = c;
      else
        Cs[(64 + j - P.nfe) * KC + kk] = c;
    }
    __syncthreads();
    if (P.nfe != 64) {   // the serendipity functions in the tricubic ones: their nodal values
      for (int o = tid; o < 64 * KC; o += P64_NT) {
        const int j = o / KC, kk = o - j * KC;
        double s = 0.0;
        for (int c = 0; c < 32; ++c) {
          const double r = P.Rser[j * 32 + c];
          if (r != 0.0) s = fma(r, raw[c * KC + kk], s);
        }
        Cs[o] = s;
      }
      __syncthreads();
    }
    for (int o = tid; o < 16 * p * KC; o += P64_NT) {   // x: (b c, k, qx)
      const int r = o / p, qx = o - r * p, bc = r / KC, kk = r - bc * KC;
      const double *c = Cs + 4 * bc * KC + kk;
      T1[o] = fma(c[0], L[qx], fma(c[KC], L[p + qx], fma(c[2 * KC], L[2 * p + qx], c[3 * KC] * L[3 * p + qx])));
    }
    __syncthreads();
    for (int o = tid; o < 4 * p2 * KC; o += P64_NT) {   // y: (c, k, qx qy)
      const int r = o / p2, xy = o - r * p2, qy = xy / p, qx = xy - qy * p, c = r / KC, kk = r - c * KC;
      const double *t = T1 + (4 * c * KC + kk) * p + qx, *l = L + 4 * p + qy;
      const int st = KC * p;
      T2[o] = fma(t[0], l[0], fma(t[st], l[p], fma(t[2 * st], l[2 * p], t[3 * st] * l[3 * p])));
    }
    __syncthreads();
    double *ph = ph8 + tid;
    auto point = [&](int q) -> double {   // this group's part of the density at point q
      const int qz = q / p2, xy = q - qz * p2;
      double a[KC];
      {
        const double l0 = L[8 * p + qz], l1 = L[9 * p + qz], l2 = L[10 * p + qz], l3 = L[11 * p + qz];
#pragma unroll
        for (int k = 0; k < KC; ++k) {
          const double *t = T2 + k * p2 + xy;
          a[k] = fma(t[0], l0, fma(t[KC * p2], l1, fma(t[2 * KC * p2], l2, t[3 * KC * p2] * l3)));
        }
      }
      if (nE > 0) {
        const double *x = P.xi + 3 * (qs + q);
        const double lx[2] = {0.125 * (1.0 - x[0]), 0.125 * (1.0 + x[0])},
                     ly[2] = {1.0 - x[1], 1.0 + x[1]}, lz[2] = {1.0 - x[2], 1.0 + x[2]};
#pragma unroll
        for (int v = 0; v < 8; ++v)
          ph[v * P64_NT] = lx[v & 1] * ly[(v >> 1) & 1] * lz[v >> 2];
        for (int j = 0; j < nE; ++j) {
          const int code = ec[j];
          const double b = ph[(code & 7) * P64_NT] * pe[(int64_t)(code >> 3) * 4 * Q + pq + q];
          const double *c = Cs + (64 + j) * KC;
#pragma unroll
          for (int k = 0; k < KC; ++k) a[k] = fma(b, c[k], a[k]);
        }
      }
      double r = 0.0;
#pragma unroll
      for (int k = 0; k < KC; ++k) r = fma(fs[k] * a[k], a[k], r);
      return r;
    };
    // (a thread meets its own points again in the next group)
    double *o = direct ? P.rho + qs + first : acc;
    for (int q = tid; q < np; q += P64_NT) {
      const double r = point(first + q);
      if (direct && P.halves == 2)
        atomicAdd(o + q, r);
      else
        o[q] = grp > g0 ? o[q] + r : r;
    }
  }
  if (direct) return;
  const auto cluster = cooperative_groups::this_cluster();
  if (P.cs > 1) cluster.sync();
  for (int q = rank * P64_NT + tid; q < np; q += P.cs * P64_NT) {
    double r = 0.0;
    for (int y = 0; y < P.cs; ++y) r += *cluster.map_shared_rank(acc + q, y);
    if (P.halves == 2)
      atomicAdd(P.rho + qs + first + q, r);
    else
      P.rho[qs + first + q] = r;
  }
  if (P.cs > 1) cluster.sync();   // no CTA leaves while its part is read
}

}  // namespace

// Work lists (host).  Adjoint: items (element, kind 0 FE x FE / 1 slot range /
// 2 pair range / 3 point range of the direct E x E products, begin, end, (sub)cell
// range, or for kind 3 the range of the block's rows) cut to the mean cost of a CTA
// slot (four per SM), by (sub)cells where their work outweighs the coefficients that
// every range forms, and to the shared work area, largest first.  The E x E block takes
// the form of fewer operations, but the pair form, which any work area holds, where
// one row of the triangle and its columns' points are beyond half an SM's shared
// memory (over 907 columns; eight such elements of 912 columns 5.5 ms, of 800 in the
// direct form 1.0 ms).  Density: int4 units (element, (sub)cell, first z plane, end z plane),
// cut to the mean cost of a CTA slot; the doubles that one column takes and the points
// that one unit has at most.
void pt64_work_lists(const pufe_ctx *ctx, std::vector<int32_t> &adj, int &adj_work,
                     std::vector<int32_t> &den, int &den_col, int &den_pts) {
  const int nsm = ctx->nsm;
  adj.clear();
  den.clear();
  adj_work = den_col = den_pts = 0;
  const int64_t ne = (int64_t)ctx->n_e.size();
  struct Item {
    int32_t v[6];
    double c;
  };
  std::vector<Item> L;
  auto emit = [&](std::vector<int32_t> &out, int width) {
    std::stable_sort(L.begin(), L.end(), [](const Item &x, const Item &y) { return x.c > y.c; });
    for (const Item &i : L) out.insert(out.end(), i.v, i.v + width);
  };
  {
    std::vector<double> cf(ne), cs(ne), cp(ne), cd(ne);
    double total = 0.0;
    for (int64_t e = 0; e < ne; ++e) {
      cf[e] = 4096;
      cs[e] = 2100;
      cp[e] = 128;
      for (double d : ctx->part_p_host[e]) {
        cf[e] += 1000 * d + 100 * d * d + 10 * d * d * d;
        cs[e] += 125 * d + 25 * d * d + 6 * d * d * d;
        cp[e] += 27 * d + 9 * d * d + 5 * d * d * d;
      }
      const double nE = ctx->n_e[e] - ctx->nfe_e, A = ctx->n_slot[e];
      cd[e] = (double)ctx->q_e[e] * (0.5 * nE * (nE + 1) + 5 * nE);
      total += cf[e] + A * cs[e] + std::min(0.5 * A * (A + 1) * cp[e], cd[e]);
    }
    const double target = std::max(1.0, total / (4.0 * nsm));
    // one range over (sub)cell ranges of at least `least` operations
    auto cells = [&](int64_t e, int kind, int a, int b, double c, double least) {
      const int nc = (int)ctx->part_p_host[e].size();
      const double m = std::min(std::min(std::ceil(c / target), c / least), (double)nc);
      const int cuts = std::max(1, (int)m);
      for (int j = 0; j < cuts; ++j)
        L.push_back(Item{{(int32_t)e, kind, a, b, (int)((int64_t)j * nc / cuts),
                          (int)((int64_t)(j + 1) * nc / cuts)},
                         c / cuts});
    };
    for (int64_t e = 0; e < ne; ++e) {
      int p = 1;
      for (int d : ctx->part_p_host[e]) p = std::max(p, d);
      const int A = ctx->n_slot[e], np = A * (A + 1) / 2, nE = ctx->n_e[e] - ctx->nfe_e;
      adj_work = std::max(adj_work, adj_fefe_doubles(p, ctx->ser));
      cells(e, 0, 0, 0, cf[e], 30000.0);
      if (A == 0) continue;
      int G = std::max(1, std::min(A, (int)std::min(1e6, target / cs[e])));
      G = std::max(1, std::min(G, (P64_WORK - 15 * p) / (adj_slot_doubles(p) + 4)));
      adj_work = std::max(adj_work, G * (adj_slot_doubles(p) + 4) + 15 * p);
      for (int a = 0; a < A; a += G)
        cells(e, 1, a, std::min(A, a + G), cs[e] * std::min(G, A - a), 8000.0 * G);
      if (cd[e] < np * cp[e] && (nE + 1) * P64_QC_MIN <= P64_MAX / 2) {
        const int Q = ctx->q_e[e];
        const int cuts = std::max(1, std::min(Q / 32, (int)std::min(1e6, std::ceil(cd[e] / target))));
        // the whole triangle where it fits beside up to 64 points, else ranges of rows
        // beside P64_QC_MIN of them
        const int whole = nE * (nE + 1) / 2 + nE * std::min(64, Q);
        const int qc = std::min(P64_QC_MIN, Q);
        const int area = std::max(P64_ROWS, 2 * nE * qc);
        for (int ra = 0, rb; ra < nE; ra = rb) {
          rb = whole <= P64_WHOLE ? nE : ra + 1;
          int ent = rb * (rb + 1) / 2 - ra * (ra + 1) / 2;
          while (rb < nE && ent + rb + 1 + nE * qc <= area) ent += ++rb;
          adj_work = std::max(adj_work, whole <= P64_WHOLE ? whole : ent + nE * qc);
          const double c = cd[e] * ent / (0.5 * nE * (nE + 1));
          for (int j = 0; j < cuts; ++j) {
            const int a = (int)((int64_t)j * Q / cuts), b = (int)((int64_t)(j + 1) * Q / cuts);
            L.push_back(Item{{(int32_t)e, 3, a, b, ra, rb}, c * (b - a) / Q});
          }
        }
        continue;
      }
      const int M = std::max(1, std::min(np, (int)std::min(1e6, target / cp[e])));
      const int cuts = (np + M - 1) / M;
      adj_work = std::max(adj_work, 4 * A + 9 * p + adj_pair_doubles(p));
      for (int j = 0; j < cuts; ++j) {
        const int a = (int)((int64_t)j * np / cuts), b = (int)((int64_t)(j + 1) * np / cuts);
        cells(e, 2, a, b, cp[e] * (b - a), 1000.0 * (b - a));
        for (int c = b - a; c > 1; --c)
          if (4 * A + 9 * p + c * adj_pair_doubles(p) <= P64_WORK) {
            adj_work = std::max(adj_work, 4 * A + 9 * p + c * adj_pair_doubles(p));
            break;
          }
      }
    }
    emit(adj, 6);
  }
  // density units, in operations per state
  L.clear();
  auto plane = [&](int64_t e, double p) {
    return p * p * (6.0 + 1.4 * (ctx->n_e[e] - ctx->nfe_e));
  };
  double total = 0.0;
  for (int64_t e = 0; e < ne; ++e)
    for (double p : ctx->part_p_host[e]) total += 64 * p + 16 * p * p + p * plane(e, p);
  const double target = std::max(1.0, total / (4.0 * nsm));
  int32_t cell = 0;
  for (int64_t e = 0; e < ne; ++e)
    for (int p : ctx->part_p_host[e]) {
      den_col = std::max(den_col, den_column(ctx->n_e[e], p));
      const double fix = 64.0 * p + 16.0 * p * p, pl = plane(e, p);
      const int cuts = std::max(1, std::min(p, (int)std::min(64.0, std::ceil(p * pl / target))));
      den_pts = std::max(den_pts, (p + cuts - 1) / cuts * p * p);
      for (int j = 0; j < cuts; ++j)
        L.push_back(Item{{(int32_t)e, cell, j * p / cuts, (j + 1) * p / cuts},
                         fix + pl * ((j + 1) * p / cuts - j * p / cuts)});
      ++cell;
    }
  emit(den, 4);
}

pufe_status launch_adjoint_sf64(pufe_ctx *ctx, const PhaseTab *ph, const double *Hr,
                                const double *Hi, double *Vbar, cudaStream_t st) {
  auto &D = ctx->d;
  Adj64 P{};
  P.items = D.jitems;
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
  P.Hr = Hr;
  P.Hi = Hi;
  P.eshift = D.eshift;
  if (ph) P.ph = *ph;
  P.out = Vbar;
  P.Rser = D.Rser;
  P.nfe = ctx->nfe_e;
  P.work = ctx->adj64_work;
  const size_t sm = (size_t)ctx->adj64_work * sizeof(double);
  if (sm > 227 * 1024) return fail(PUFE_EINVAL, "element too large for the FP64 adjoint");
  PUFE_CUDA_TRY(cudaMemsetAsync(Vbar, 0, (size_t)ctx->nq * sizeof(double), st));
  auto kern = ph ? k_adjoint_sf64<true> : k_adjoint_sf64<false>;
  PUFE_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
  kern<<<(unsigned)ctx->n_jitems, P64_NT, sm, st>>>(P);
  PUFE_CUDA_TRY(cudaGetLastError());
  return PUFE_OK;
}

// ph == nullptr: Gamma point, real C; else C + i Ci at the wavevector of ph
pufe_status launch_density_sf64(pufe_ctx *ctx, const PhaseTab *ph, const double *C,
                                const double *Ci, int64_t ldc, const double *f, int nocc,
                                double *rho, cudaStream_t st) {
  auto &D = ctx->d;
  Den64 P{};
  P.units = reinterpret_cast<const int4 *>(D.dunits);
  P.qoff = D.qoff;
  P.xi = D.xi;
  P.part_p = D.part_p;
  P.part_q = D.part_q;
  P.doff = D.doff;
  P.dofs = D.dofs;
  P.ecol = D.ecol;
  P.toff = D.toff;
  P.psi = D.psi;
  P.C = C;
  P.Ci = Ci;
  P.f = f;
  P.Rser = D.Rser;
  P.ldc = ldc;
  P.ncol = ph ? 2 * nocc : nocc;
  P.nfe = ctx->nfe_e;
  P.eshift = D.eshift;
  if (ph) P.ph = *ph;
  P.rho = rho;
  // columns per CTA: the width (a multiple of 4, up to 16) that pads the fewest; less
  // where the work area of the largest (sub)cell does not fit an SM
  const int most = (P.ncol + 15) / 16;
  int kc = ((P.ncol + most - 1) / most + 3) & ~3;
  auto bytes = [&] {   // (the sums of a unit's points from three groups on)
    const int sums = P.ncol > 2 * kc ? ctx->den64_points : 0;
    return (size_t)(den_doubles(ctx->den64_column, ctx->max_part_p, kc) + sums) * sizeof(double);
  };
  while (kc > 4 && bytes() > 227 * 1024) kc -= 4;
  const int groups = P.groups = (P.ncol + kc - 1) / kc;
  P.cs = 1;
  P.halves = std::min(groups, 2);
  if (groups > 2 && (int64_t)ctx->n_dunits * groups <= 4 * ctx->nsm) {
    P.halves = groups > 5 ? 2 : 1;
    P.cs = std::min(DEN_CLUSTER, (groups + P.halves - 1) / P.halves);
  }
  const int ny = P.halves * P.cs;
  const size_t sm = bytes();
  if (sm > 227 * 1024) return fail(PUFE_EINVAL, "n_e too large for the density kernel");
  if (P.halves == 2) PUFE_CUDA_TRY(cudaMemsetAsync(rho, 0, (size_t)ctx->nq * sizeof(double), st));
  auto run = [&](auto kern) -> pufe_status {
    PUFE_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = at[0].val.clusterDim.z = 1;
    at[0].val.clusterDim.y = (unsigned)P.cs;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)ctx->n_dunits, (unsigned)ny);
    cfg.blockDim = dim3(P64_NT);
    cfg.dynamicSmemBytes = sm;
    cfg.stream = st;
    cfg.attrs = at;
    cfg.numAttrs = P.cs > 1 ? 1 : 0;
    PUFE_CUDA_TRY(cudaLaunchKernelEx(&cfg, kern, P));
    return PUFE_OK;
  };
  if (ph) {
    if (kc == 4) return run(k_density_sf64<true, 4>);
    if (kc == 8) return run(k_density_sf64<true, 8>);
    if (kc == 12) return run(k_density_sf64<true, 12>);
    return run(k_density_sf64<true, 16>);
  }
  if (kc == 4) return run(k_density_sf64<false, 4>);
  if (kc == 8) return run(k_density_sf64<false, 8>);
  if (kc == 12) return run(k_density_sf64<false, 12>);
  return run(k_density_sf64<false, 16>);
}

}  // namespace pufe
