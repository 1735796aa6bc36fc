// FP64 CUDA-core kernels of the PUFE hot path:
//   K0  enrichment tabulation (Sec. 5.1, eqs. Psitilde/Psi)
//   K1+K2+K3  element basis tile, contraction and scatter (Sec. 4, eq. disceig3d)
//
// The element basis (the FE columns -- 64 tricubic or 32 cubic serendipity
// functions -- then phi_v^PU Psi_alpha columns) is rebuilt on chip from the reference coordinates of each quadrature point
// and the tabulated Psi / grad Psi; it is never stored in HBM.
//
// The contraction here is the direct one, for rules of fewer than 4 points per axis; the
// others, the density and the adjoint are sum factorized (pufe_sf64.cu, pufe_pt64.cu).
#include <math.h>

#include "pufe_internal.h"

namespace pufe {

namespace {

constexpr int QC = 8;         // quadrature points per chunk
constexpr int ASM_NT = 256;   // threads of the assembly kernel

__device__ __forceinline__ void set_err(unsigned *err, unsigned bit) { atomicOr(err, bit); }

// ---------------------------------------------------------------------------
// K0: Psi and grad Psi for every (enrichment slot, quadrature point) of an element.
// Layout per element: psi[4*toff[e] + (slot*4 + comp)*Q + q].
//
// One CTA per work item, a run of slots of one element that share an atom and
// TAB64_NT of its points; one thread per point.  FP64 operations bind it (two
// multiply-adds per clock and SM), so what the orbitals of an atom share is
// formed once per point: the displacement, its length, the cutoff and its slope;
// the exponential and the radial function carry over while consecutive slots have
// the same exponent and the same (n, l).  Only the images that can lie within r_c
// are visited: those with |s_d + i| <= r_c b_d on every lattice direction (s_d the
// displacement in lattice coordinates, 1/b_d the distance of the lattice planes),
// one or two per axis instead of 27 in all.  On the 12^3 rocksalt cell that is
// about 40 operations per value in place of 400, and the elements of 30 slots and
// 4,096 points of the CsCl-like cell spread over 32 CTAs each instead of one.
// Measured: 12^3 rocksalt 2.19 -> 0.19 ms, CsCl-like 16^3 30.3 -> 0.26 ms, two-atom
// 4^3 377 -> 28 us.
// ---------------------------------------------------------------------------
constexpr int TAB64_NT = 128;

// (general cells: `gen`, Sec. 6.2)
__global__ void __launch_bounds__(TAB64_NT) k_tabulate(
    const int4 *__restrict__ items, const int64_t *__restrict__ qoff,
    const double *__restrict__ x, const int32_t *__restrict__ aoff,
    const int32_t *__restrict__ alist, const int64_t *__restrict__ toff,
    const Orbital *__restrict__ orb, LatticeDev lat, float b0, float b1, float b2, int gen,
    double *__restrict__ psi) {
  const int4 it = items[blockIdx.x];   // element, first slot, slots, first point
  const int64_t e = it.x, q0 = qoff[e];
  const int Q = (int)(qoff[e + 1] - q0);
  const int32_t *al = alist + aoff[e] + it.y;
  double *out = psi + 4 * toff[e] + (int64_t)it.y * 4 * Q;
  for (int q = it.w + threadIdx.x; q < min(it.w + TAB64_CHUNK, Q); q += TAB64_NT) {
    const Orbital &o0 = orb[al[0]];   // the atom and the cutoff of the run
    const double rc = o0.rc, irc = o0.inv_rc, rc2 = rc * rc;
    const float bn[3] = {b0, b1, b2};
    double d[3], s[3];
    int lo[3], hi[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) d[k] = x[3 * (q0 + q) + k] - o0.tau[k];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      s[k] = gen ? lat.Lit[3 * k] * d[0] + lat.Lit[3 * k + 1] * d[1] + lat.Lit[3 * k + 2] * d[2]
                 : d[k] * lat.Lit[4 * k];
      // (in FP32; r < r_c decides below.  The margin covers the rounding, since |s| stays
      // small: the setup looks for an atom's images at most two cells from its given
      // position, on general cells as many as r_c spans, and an element has no slot of
      // an atom further off)
      const float reach = (float)rc * bn[k] * 1.0001f + 1e-4f, sf = (float)s[k];
      lo[k] = (int)ceilf(-reach - sf);
      hi[k] = (int)floorf(reach - sf);
    }
    bool first = true;
    for (int i = lo[0]; i <= hi[0]; ++i)
      for (int j = lo[1]; j <= hi[1]; ++j)
        for (int k = lo[2]; k <= hi[2]; ++k) {
          double v[3];
          if (gen) {
#pragma unroll
            for (int m = 0; m < 3; ++m)
              v[m] = d[m] + (i * lat.L[m] + j * lat.L[3 + m] + k * lat.L[6 + m]);
          } else {
            v[0] = d[0] + i * lat.L[0];
            v[1] = d[1] + j * lat.L[4];
            v[2] = d[2] + k * lat.L[8];
          }
          const double r2 = v[0] * v[0] + v[1] * v[1] + v[2] * v[2];
          if (r2 >= rc2) continue;
          // one reciprocal square root for r and 1 / r (0 at the nucleus); r is corrected
          // by its residual to the rounded root, since the exponential of a sharp orbital
          // shows its last place (CsCl-like density: error against 64 bits 4.2e-16
          // without, 1.9e-16 with; no difference in time)
          const double ir = r2 > 1e-28 ? rsqrt(r2) : 0.0;
          const double r0 = r2 * ir;
          const double r = r2 > 1e-28 ? fma(fma(-r0, r0, r2), 0.5 * ir, r0) : sqrt(r2);
          const double t = r * irc, t3 = t * t * t, om = 1.0 - t;
          const double hc = 1.0 + t3 * t * (-35.0 + t * (84.0 + t * (-70.0 + 20.0 * t)));
          const double dh = -140.0 * irc * t3 * om * om * om;
          double zeta = -1.0, ex = 0.0, f = 0.0, df = 0.0;
          int pn = -1, pl = -1;
          for (int c = 0; c < it.z; ++c) {
            const Orbital &o = orb[al[c]];
            if (o.zeta != zeta || o.n != pn || o.l != pl) {   // the radial function of (n, l, zeta)
              if (o.zeta != zeta) ex = exp(-o.zeta * r);
              zeta = o.zeta;
              pn = o.n;
              pl = o.l;
              const int kk = pn - 1 - pl;
              double rk = 1.0, rkm = 0.0;
              for (int u = 0; u < kk; ++u) {
                rkm = rk;
                rk *= r;
              }
              const double ez = o.norm * ex, rh = rk * hc;
              f = ez * rh;
              df = ez * fma(rk, dh, fma((double)kk * rkm, hc, -zeta * rh)) * ir;
            }
            double gs[3];
            const double S = solid_harmonic<double>(o.l, o.m, v[0], v[1], v[2], gs);
            const double ds = df * S;
            double *dst = out + (int64_t)c * 4 * Q + q;
            double w0 = f * S, w1 = fma(ds, v[0], f * gs[0]), w2 = fma(ds, v[1], f * gs[1]),
                   w3 = fma(ds, v[2], f * gs[2]);
            if (!first) {   // a second image within r_c adds to the first's
              w0 += dst[0];
              w1 += dst[Q];
              w2 += dst[2 * Q];
              w3 += dst[3 * Q];
            }
            dst[0] = w0;
            dst[Q] = w1;
            dst[2 * Q] = w2;
            dst[3 * Q] = w3;
          }
          first = false;
        }
    if (first)
      for (int c = 0; c < 4 * it.z; ++c) out[(int64_t)c * Q + q] = 0.0;
  }
}

// Basis values and physical gradients of column c at reference point xi.
// FE column c: node (c&3, (c>>2)&3, c>>4) from the 1D tables L, dL.
// Enrichment column: PU vertex lv times Psi (value/gradient g4).
struct Tab1D {
  double L[3][4], dL[3][4];
};

__device__ __forceinline__ void fe_column(const Tab1D &t, int c, const double s[3], double &b,
                                          double &gx, double &gy, double &gz) {
  const int ia = c & 3, ib = (c >> 2) & 3, ic = c >> 4;
  const double lx = t.L[0][ia], ly = t.L[1][ib], lz = t.L[2][ic];
  b = lx * ly * lz;
  gx = t.dL[0][ia] * ly * lz * s[0];
  gy = lx * t.dL[1][ib] * lz * s[1];
  gz = lx * ly * t.dL[2][ic] * s[2];
}

__device__ __forceinline__ void pu_column(const double xi[3], int lv, const double s[3],
                                          const double ps[4], double &b, double &gx, double &gy,
                                          double &gz) {
  double h[3], dh[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const int bit = (lv >> d) & 1;
    h[d] = bit ? 0.5 * (1.0 + xi[d]) : 0.5 * (1.0 - xi[d]);
    dh[d] = (bit ? 0.5 : -0.5) * s[d];
  }
  const double phi = h[0] * h[1] * h[2];
  b = phi * ps[0];
  gx = dh[0] * h[1] * h[2] * ps[0] + phi * ps[1];
  gy = h[0] * dh[1] * h[2] * ps[0] + phi * ps[2];
  gz = h[0] * h[1] * dh[2] * ps[0] + phi * ps[3];
}

// ---------------------------------------------------------------------------
// K1+K2+K3 (FP64): one CTA per work item -- an element, or with the setup's
// point-range list (`wsplit`) the points [qa, qb) of one.  Per chunk of QC
// points the CTA builds y_d = sqrt(w/2) G_d, z = sqrt(w) B and zv = V z in
// shared memory; each thread owns 4x4 blocks of the lower triangle and
// accumulates
//   H += sum_d y_d y_d^T + zv z^T,   S += z z^T,
// over the item's points, then adds its entries into the CSR values through
// the scatter map (the ranges of one element meet in these atomics).
// ---------------------------------------------------------------------------
// BLOCH: the scatter carries the phase exp(i k.(R_j - R_i)) of the column
// pair (lattice shifts from `eshift`, phases of the 8 shift codes in `ph`)
// into separate real and imaginary outputs (Sec. 4, eq. bloch).  GEN: a
// general cell, physical gradients J^-T grad_xi with jit = J^-T (row-major).
struct Mat3 {
  double m[9];
};

template <bool BLOCH, bool GEN>
__global__ void __launch_bounds__(ASM_NT) k_assemble_fp64(
    const int32_t *__restrict__ order, const int64_t *__restrict__ qoff,
    const double *__restrict__ w, const double *__restrict__ xi_all,
    const int64_t *__restrict__ doff, const int32_t *__restrict__ ecol,
    const int64_t *__restrict__ toff, const double *__restrict__ psi,
    const int64_t *__restrict__ soff, const int32_t *__restrict__ smap,
    const double *__restrict__ V, double sx, double sy, double sz, int npad_max, int want,
    double *__restrict__ H, double *__restrict__ S, unsigned *err,
    const uint8_t *__restrict__ eshift, PhaseTab ph, double *__restrict__ Hi,
    double *__restrict__ Si, const int32_t *__restrict__ wsplit, Mat3 jit, int nfe) {
  extern __shared__ __align__(16) double smem[];
  // work item: a whole element, or the point range [qa, qb) of one
  const int e = wsplit ? wsplit[3 * blockIdx.x] : order[blockIdx.x];
  const int64_t q0 = qoff[e];
  const int Q = (int)(qoff[e + 1] - q0);
  const int qa = wsplit ? max(wsplit[3 * blockIdx.x + 1], 0) : 0;
  const int qb = wsplit ? min(wsplit[3 * blockIdx.x + 2], Q) : Q;
  const int n = (int)(doff[e + 1] - doff[e]);
  const int npad = (n + 3) & ~3;
  if (npad > npad_max) {
    if (threadIdx.x == 0) set_err(err, DEVERR_SHAPE);
    return;
  }
  const int32_t *ec = ecol + (doff[e] - (int64_t)nfe * e);
  const double *pe = psi + 4 * toff[e];
  // shared layout: 5 arrays [QC][npad] then 1D tables
  double *Y0 = smem, *Y1 = Y0 + QC * npad, *Y2 = Y1 + QC * npad, *Z = Y2 + QC * npad,
         *ZV = Z + QC * npad;
  Tab1D *tab = reinterpret_cast<Tab1D *>(ZV + QC * npad);
  const double s[3] = {sx, sy, sz};

  const int nb = npad / 4;
  const int nblk = nb * (nb + 1) / 2;
  for (int base = 0; base < nblk; base += ASM_NT) {
    const int t = base + threadIdx.x;
    const bool active = t < nblk;
    int I = 0, J = 0;
    if (active) {
      I = (int)((sqrt(8.0 * t + 1.0) - 1.0) * 0.5);
      while ((I + 1) * (I + 2) / 2 <= t) ++I;
      while (I * (I + 1) / 2 > t) --I;
      J = t - I * (I + 1) / 2;
    }
    const int i0 = 4 * I, j0 = 4 * J;
    double h[4][4], sv[4][4];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int b = 0; b < 4; ++b) h[a][b] = sv[a][b] = 0.0;

    for (int qc = qa; qc < qb; qc += QC) {
      __syncthreads();
      // 1D Lagrange tables of the chunk's points
      for (int k = threadIdx.x; k < QC * 3; k += ASM_NT) {
        const int qq = k / 3, d = k - 3 * qq;
        const int q = qc + qq;
        const double xv = (q < qb) ? xi_all[3 * (q0 + q) + d] : 0.0;
        double L[4], dL[4];
        lagrange3(xv, L, dL);
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          tab[qq].L[d][c] = L[c];
          tab[qq].dL[d][c] = dL[c];
        }
      }
      __syncthreads();
      for (int k = threadIdx.x; k < QC * npad; k += ASM_NT) {
        const int qq = k / npad, c = k - qq * npad;
        const int q = qc + qq;
        double b = 0, gx = 0, gy = 0, gz = 0, sw = 0, vv = 0;
        if (q < qb && c < n) {
          // GEN: reference gradients (unit scales) mapped by J^-T
          const double one[3] = {1.0, 1.0, 1.0};
          auto tomap = [&](double &x, double &y, double &z) {
            const double rx = x, ry = y, rz = z;
            x = jit.m[0] * rx + jit.m[1] * ry + jit.m[2] * rz;
            y = jit.m[3] * rx + jit.m[4] * ry + jit.m[5] * rz;
            z = jit.m[6] * rx + jit.m[7] * ry + jit.m[8] * rz;
          };
          if (c < nfe) {   // FE column: tricubic (64) or serendipity (32)
            if (nfe == 64) {
              fe_column(tab[qq], c, GEN ? one : s, b, gx, gy, gz);
            } else {
              const double xq[3] = {xi_all[3 * (q0 + q)], xi_all[3 * (q0 + q) + 1],
                                    xi_all[3 * (q0 + q) + 2]};
              const double *sc = GEN ? one : s;
              double g3[3];
              serendipity32(c, xq, b, g3);
              gx = g3[0] * sc[0];
              gy = g3[1] * sc[1];
              gz = g3[2] * sc[2];
            }
            if (GEN) tomap(gx, gy, gz);
          } else {
            const int code = ec[c - nfe];
            const int slot = code >> 3, lv = code & 7;
            const double *pp = pe + (int64_t)slot * 4 * Q + q;
            const double ps[4] = {pp[0], pp[Q], pp[2 * Q], pp[3 * Q]};
            const double xq[3] = {xi_all[3 * (q0 + q)], xi_all[3 * (q0 + q) + 1],
                                  xi_all[3 * (q0 + q) + 2]};
            if (GEN) {   // phi_v and its mapped gradient, then the product rule
              const double unit[4] = {1.0, 0.0, 0.0, 0.0};
              double phi;
              pu_column(xq, lv, one, unit, phi, gx, gy, gz);
              tomap(gx, gy, gz);
              b = phi * ps[0];
              gx = gx * ps[0] + phi * ps[1];
              gy = gy * ps[0] + phi * ps[2];
              gz = gz * ps[0] + phi * ps[3];
            } else {
              pu_column(xq, lv, s, ps, b, gx, gy, gz);
            }
          }
          sw = w[q0 + q];
          vv = V ? V[q0 + q] : 0.0;
          if (!isfinite(vv)) atomicOr(err, DEVERR_NONFINITE);
        }
        const double r2 = sqrt(0.5 * sw), r1 = sqrt(sw);
        Y0[k] = r2 * gx;
        Y1[k] = r2 * gy;
        Y2[k] = r2 * gz;
        Z[k] = r1 * b;
        ZV[k] = vv * r1 * b;
      }
      __syncthreads();
      if (active) {
        const int qn = min(QC, qb - qc);
        for (int qq = 0; qq < qn; ++qq) {
          const int ro = qq * npad;
          double ai[5][4], bj[4][4];
#pragma unroll
          for (int a = 0; a < 4; ++a) {
            ai[0][a] = Y0[ro + i0 + a];
            ai[1][a] = Y1[ro + i0 + a];
            ai[2][a] = Y2[ro + i0 + a];
            ai[3][a] = ZV[ro + i0 + a];
            ai[4][a] = Z[ro + i0 + a];
            bj[0][a] = Y0[ro + j0 + a];
            bj[1][a] = Y1[ro + j0 + a];
            bj[2][a] = Y2[ro + j0 + a];
            bj[3][a] = Z[ro + j0 + a];
          }
#pragma unroll
          for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b) {
              double acc = h[a][b];
              acc = fma(ai[0][a], bj[0][b], acc);
              acc = fma(ai[1][a], bj[1][b], acc);
              acc = fma(ai[2][a], bj[2][b], acc);
              acc = fma(ai[3][a], bj[3][b], acc);
              h[a][b] = acc;
              sv[a][b] = fma(ai[4][a], bj[3][b], sv[a][b]);
            }
        }
      }
    }
    // scatter the owned lower-triangle entries (both (i,j) and (j,i))
    if (active) {
      const int32_t *m = smap + soff[e];
#pragma unroll
      for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) {
          const int i = i0 + a, j = j0 + b;
          if (i >= n || j >= n || j > i) continue;
          const int32_t sij = m[(int64_t)i * n + j];
          const int32_t sji = m[(int64_t)j * n + i];
          if (BLOCH) {
            // (i, j) gets conj(ph_i) ph_j, (j, i) its conjugate
            const int ci = eshift[doff[e] + i], cj = eshift[doff[e] + j];
            double pr = 1.0, pim = 0.0;
            if (ci != cj) {
              pr = ph.re[ci] * ph.re[cj] + ph.im[ci] * ph.im[cj];
              pim = ph.re[ci] * ph.im[cj] - ph.im[ci] * ph.re[cj];
            }
            if (want & PUFE_WANT_H) {
              atomicAdd(H + sij, h[a][b] * pr);
              atomicAdd(Hi + sij, h[a][b] * pim);
              if (i != j) {
                atomicAdd(H + sji, h[a][b] * pr);
                atomicAdd(Hi + sji, -h[a][b] * pim);
              }
            }
            if (want & PUFE_WANT_S) {
              atomicAdd(S + sij, sv[a][b] * pr);
              atomicAdd(Si + sij, sv[a][b] * pim);
              if (i != j) {
                atomicAdd(S + sji, sv[a][b] * pr);
                atomicAdd(Si + sji, -sv[a][b] * pim);
              }
            }
            continue;
          }
          if (want & PUFE_WANT_H) {
            atomicAdd(H + sij, h[a][b]);
            if (i != j) atomicAdd(H + sji, h[a][b]);
          }
          if (want & PUFE_WANT_S) {
            atomicAdd(S + sij, sv[a][b]);
            if (i != j) atomicAdd(S + sji, sv[a][b]);
          }
        }
    }
  }
}

}  // namespace

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
// the lattice of a general cell for the image sums
static LatticeDev lattice_of(const pufe_ctx *ctx) {
  LatticeDev l{};
  if (!ctx->general) return l;
  const double *L = ctx->lat;
  for (int k = 0; k < 9; ++k) l.L[k] = L[k];
  const double det = L[0] * (L[4] * L[8] - L[5] * L[7]) - L[1] * (L[3] * L[8] - L[5] * L[6]) +
                     L[2] * (L[3] * L[7] - L[4] * L[6]);
  const double C[9] = {L[4] * L[8] - L[5] * L[7], L[5] * L[6] - L[3] * L[8],
                       L[3] * L[7] - L[4] * L[6], L[2] * L[7] - L[1] * L[8],
                       L[0] * L[8] - L[2] * L[6], L[1] * L[6] - L[0] * L[7],
                       L[1] * L[5] - L[2] * L[4], L[2] * L[3] - L[0] * L[5],
                       L[0] * L[4] - L[1] * L[3]};
  for (int k = 0; k < 9; ++k) l.Lit[k] = C[k] / det;
  for (int k = 0; k < 3; ++k) l.img[k] = ctx->images[k];
  return l;
}

static Mat3 jit_of(const pufe_ctx *ctx) {
  Mat3 m{};
  for (int k = 0; k < 9; ++k) m.m[k] = ctx->Jit[k];
  return m;
}

pufe_status launch_tabulate(pufe_ctx *ctx, cudaStream_t st) {
  if (ctx->n_kitems == 0) return PUFE_OK;
  auto &D = ctx->d;
  LatticeDev lat = lattice_of(ctx);
  double bn[3];   // inverse distances of the lattice planes
  for (int k = 0; k < 3; ++k) {
    if (!ctx->general) {
      lat.L[4 * k] = ctx->a[k];
      lat.Lit[4 * k] = 1.0 / ctx->a[k];
    }
    bn[k] = sqrt(lat.Lit[3 * k] * lat.Lit[3 * k] + lat.Lit[3 * k + 1] * lat.Lit[3 * k + 1] +
                 lat.Lit[3 * k + 2] * lat.Lit[3 * k + 2]);
  }
  k_tabulate<<<(unsigned)ctx->n_kitems, TAB64_NT, 0, st>>>(
      reinterpret_cast<const int4 *>(D.kitems), D.qoff, D.x, D.aoff, D.alist, D.toff, D.orb, lat,
      (float)bn[0], (float)bn[1], (float)bn[2], ctx->general ? 1 : 0, D.psi);
  PUFE_CUDA_TRY(cudaGetLastError());
  return PUFE_OK;
}

// CTAs of the FP64 assembly and adjoint: one per work item of the point-range
// list when the setup made one, else one per element
static unsigned fp64_items(const pufe_ctx *ctx) {
  return ctx->d.wsplit ? (unsigned)ctx->n_wsplit : (unsigned)ctx->nelem;
}

// FP64 assembly into caller arrays: H (and Hi, Si at a wavevector, ph != nullptr)
// zeroed here, S too -- or, on the sum-factorized path, set to the constant FE-FE
// overlap that path does not add
pufe_status launch_assemble_fp64(pufe_ctx *ctx, const PhaseTab *ph, const double *V, int what,
                                 double *H, double *Hi, double *S, double *Si, cudaStream_t st) {
  auto &D = ctx->d;
  const int npad = (ctx->max_basis + 3) & ~3;
  const size_t sm = (size_t)5 * QC * npad * sizeof(double) + QC * sizeof(Tab1D);
  if (sm > 227 * 1024) return fail(PUFE_EINVAL, "element basis too large for the FP64 kernel");
  const size_t bytes = (size_t)ctx->nnz * sizeof(double);
  if (what & PUFE_WANT_H) {
    PUFE_CUDA_TRY(cudaMemsetAsync(H, 0, bytes, st));
    if (ph) PUFE_CUDA_TRY(cudaMemsetAsync(Hi, 0, bytes, st));
  }
  if (what & PUFE_WANT_S) {
    if (ctx->n_aitems > 0)
      PUFE_CUDA_TRY(cudaMemcpyAsync(S, D.S0, bytes, cudaMemcpyDeviceToDevice, st));
    else
      PUFE_CUDA_TRY(cudaMemsetAsync(S, 0, bytes, st));
    if (ph) PUFE_CUDA_TRY(cudaMemsetAsync(Si, 0, bytes, st));
  }
  if (ctx->n_aitems > 0) return launch_assemble_sf64(ctx, ph, V, what, H, Hi, S, Si, st);
  auto kern = ph ? (ctx->general ? k_assemble_fp64<true, true> : k_assemble_fp64<true, false>)
                 : (ctx->general ? k_assemble_fp64<false, true> : k_assemble_fp64<false, false>);
  PUFE_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
  kern<<<fp64_items(ctx), ASM_NT, sm, st>>>(
      D.order, D.qoff, D.w, D.xi, D.doff, D.ecol, D.toff, D.psi, D.soff, D.smap, V,
      2.0 / ctx->h[0], 2.0 / ctx->h[1], 2.0 / ctx->h[2], npad, what, H, S, D.err, D.eshift,
      ph ? *ph : PhaseTab{}, Hi, Si, D.wsplit, jit_of(ctx), ctx->nfe_e);
  PUFE_CUDA_TRY(cudaGetLastError());
  return PUFE_OK;
}

pufe_status launch_density_fp64(pufe_ctx *ctx, const double *C, int64_t ldc, const double *f,
                                int nocc, double *rho, cudaStream_t st) {
  auto &D = ctx->d;
  const int noccp = (nocc + 7) & ~7;
  // (the call's limit of basis x states; the kernel's own need is less)
  const size_t sm = ((size_t)ctx->max_basis * noccp + noccp) * sizeof(double);
  if (sm > 227 * 1024) return fail(PUFE_EINVAL, "n_e * nocc too large for the density kernel");
  return launch_density_sf64(ctx, nullptr, C, nullptr, ldc, f, nocc, rho, st);
}

pufe_status launch_adjoint_fp64(pufe_ctx *ctx, const double *Hbar, double *Vbar, cudaStream_t st) {
  return launch_adjoint_sf64(ctx, nullptr, Hbar, nullptr, Vbar, st);
}

// ---------------------------------------------------------------------------
// Bloch (k != 0) launchers
// ---------------------------------------------------------------------------
PhaseTab phase_table(const pufe_ctx *ctx, const double k[3]) {
  PhaseTab t;
  for (int c = 0; c < 8; ++c) {
    double th = 0.0;
    for (int d = 0; d < 3; ++d)
      if ((c >> d) & 1) {
        if (ctx->general)   // the lattice vector a_d
          th += k[0] * ctx->lat[3 * d] + k[1] * ctx->lat[3 * d + 1] + k[2] * ctx->lat[3 * d + 2];
        else
          th += k[d] * ctx->a[d];
      }
    t.re[c] = cos(th);
    t.im[c] = sin(th);
  }
  return t;
}

pufe_status launch_density_fp64_bloch(pufe_ctx *ctx, const PhaseTab &ph, const double *Cr,
                                      const double *Ci, int64_t ldc, const double *f, int nocc,
                                      double *rho, cudaStream_t st) {
  auto &D = ctx->d;
  const int noccp = (nocc + 7) & ~7;
  const size_t sm = ((size_t)2 * ctx->max_basis * noccp + noccp) * sizeof(double);
  if (sm > 227 * 1024) return fail(PUFE_EINVAL, "n_e * nocc too large for the density kernel");
  return launch_density_sf64(ctx, &ph, Cr, Ci, ldc, f, nocc, rho, st);
}

pufe_status launch_adjoint_fp64_bloch(pufe_ctx *ctx, const PhaseTab &ph, const double *Hr,
                                      const double *Hi, double *Vbar, cudaStream_t st) {
  return launch_adjoint_sf64(ctx, &ph, Hr, Hi, Vbar, st);
}

}  // namespace pufe
