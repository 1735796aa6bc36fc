// Projections of the basis onto separable nonlocal projectors (Sec. 4),
//   F[g_i, p] = sum_e sum_q w_q b_i(x_q) v_p(x_q),
//   v_p = N r^l exp(-r^2 / (2 r_p^2)) Y_lm summed over the periodic images,
// in FP64 by sum factorization on the p^3 (sub)cells.
//
// GB300's two FP64 multiply-adds per clock and SM bind it, so:
//  * a Gaussian times a solid harmonic is a sum of at most three products of
//    functions of one coordinate, and the images of an orthorhombic cell are a
//    product of three sums, so the projector's values come from the tables
//      X_a(x) = sum_i (x + i a_x)^a exp(-(x + i a_x)^2 / (2 r_p^2)),  a = 0..3,
//    of each axis (images within the radius where the Gaussian falls below
//    1e-20) -- 3 p exponentials per image instead of p^3;
//  * the 64 FE functions take 4 p^3 + 16 p^2 + 64 p operations per projector
//    instead of 64 p^3, the vertex columns of a slot 2 p^3 + 4 p^2 + 8 p.
// At a wavevector (Sec. 4, eqs. bloch, strong) the image at lattice vector a_n
// carries exp(i k.a_n), a factor per axis of the same tables, and element column
// i the factor exp(-i k.R_i) of its lattice shift: the real and imaginary parts
// go through the contractions as two fields.
//
// One CTA per element and group of `pc` projectors, chosen so that the work area
// leaves four CTAs per SM and small meshes still fill the chip.
//
// Measured: 32 s and p projectors on the 12^3 rocksalt cell 13.9 -> 1.07 ms at the
// Gamma point (before: every projector's images and exponential per point).
#include <algorithm>

#include "pufe_internal.h"

namespace pufe {
namespace {

constexpr int PJ_NT = 128;
constexpr int PJ_WORK = 7000;   // shared doubles aimed at: 56 KB

struct ProjArgs {
  const int64_t *qoff;
  const double *w, *xi, *x;
  const int32_t *partoff, *part_p, *part_q;
  const int64_t *doff;
  const int32_t *dofs, *ecol, *aoff;
  const int64_t *toff;
  const double *psi;
  const ProjDev *pj;
  int P, pc, sc;   // projectors, per CTA, slots per pass
  double a[3], k[3];
  const uint8_t *eshift;
  PhaseTab ph;
  double *F, *Fi;
};

// doubles of a CTA: fields, tables, 1D factors, accumulators and the larger of the
// FE pass's and a slot pass's stages
__host__ __device__ inline int proj_doubles(int nf, int pc, int sc, int A, int p, int parts) {
  const int p2 = p * p, fe = nf * (4 * p2 + 16 * p), sl = nf * sc * (2 * p2 + 4 * p);
  return nf * p2 * p + pc * 12 * p * parts + 18 * p + nf * (64 + 8 * A) + (fe > sl ? fe : sl);
}

template <bool BLOCH>
__global__ void __launch_bounds__(PJ_NT) k_projections_sf(ProjArgs P) {
  extern __shared__ __align__(16) double smpj[];
  constexpr int NC = BLOCH ? 2 : 1;
  const int tid = threadIdx.x, e = blockIdx.x, j0 = blockIdx.y * P.pc, pc = min(P.pc, P.P - j0),
            nf = NC * pc;
  const int64_t q0 = P.qoff[e];
  const int Q = (int)(P.qoff[e + 1] - q0), A = P.aoff[e + 1] - P.aoff[e], na = 64 + 8 * A;
  const double *pe = P.psi + 4 * P.toff[e];
  double *acc = smpj, *base = acc + nf * na;   // [field][64 + 8 slot + vertex]
  for (int o = tid; o < nf * na; o += PJ_NT) acc[o] = 0.0;
  for (int k = P.partoff[e]; k < P.partoff[e + 1]; ++k) {
    const int p = P.part_p[k], p2 = p * p, p3 = p2 * p, pq = P.part_q[k];
    const int64_t qs = q0 + pq;
    double *f = base;                    // [field][p^3]: w v_p
    double *T = f + nf * p3;             // [projector][axis][power][p] (x NC: re, im)
    double *L = T + 12 * NC * pc * p;    // [axis][4][p], then [axis][l_0, l_1][p]
    double *l = L + 12 * p, *W = l + 6 * p;
    __syncthreads();
    for (int o = tid; o < 3 * p; o += PJ_NT) {
      const int d = o / p, t = o - d * p;
      const int64_t at = qs + (int64_t)t * (d == 0 ? 1 : (d == 1 ? p : p2));
      const double x = P.xi[3 * at + d];
      double L4[4], dL4[4];
      lagrange3(x, L4, dL4);
      for (int a = 0; a < 4; ++a) L[(d * 4 + a) * p + t] = L4[a];
      l[(2 * d) * p + t] = 0.5 * (1.0 - x);
      l[(2 * d + 1) * p + t] = 0.5 * (1.0 + x);
    }
    for (int o = tid; o < 3 * p * pc; o += PJ_NT) {   // the projectors' 1D tables
      const int g = o / (3 * p), r = o - g * 3 * p, d = r / p, t = r - d * p;
      const ProjDev &pr = P.pj[j0 + g];
      const int64_t at = qs + (int64_t)t * (d == 0 ? 1 : (d == 1 ? p : p2));
      const double a = P.a[d], x = P.x[3 * at + d] - pr.tau[d], i2 = 1.0 / (2.0 * pr.rp * pr.rp);
      double s[4] = {0, 0, 0, 0}, si[4] = {0, 0, 0, 0};
      const int lo = (int)ceil((-pr.rcut - x) / a), hi = (int)floor((pr.rcut - x) / a);
      for (int i = lo; i <= hi; ++i) {
        const double y = x + i * a;
        double v = exp(-y * y * i2), vi = 0.0;
        if (BLOCH) {   // exp(i k.a_n): this term is v(x - tau - a_n), a_n = -i a
          double sn, cs;
          sincos(-P.k[d] * (i * a), &sn, &cs);
          vi = v * sn;
          v *= cs;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          s[u] += v;
          v *= y;
          if (BLOCH) {
            si[u] += vi;
            vi *= y;
          }
        }
      }
      double *o4 = T + (g * 3 + d) * 4 * NC * p + t;
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        o4[u * p] = s[u];
        if (BLOCH) o4[(4 + u) * p] = si[u];
      }
    }
    __syncthreads();
    for (int o = tid; o < pc * p3; o += PJ_NT) {   // w v_p at the points
      const int g = o / p3, q = o - g * p3, qz = q / p2, r = q - qz * p2, qy = r / p, qx = r - qy * p;
      const ProjDev &pr = P.pj[j0 + g];
      const double *tx = T + g * 12 * NC * p + qx, *ty = T + (g * 3 + 1) * 4 * NC * p + qy,
                   *tz = T + (g * 3 + 2) * 4 * NC * p + qz;
      double v = 0.0, vi = 0.0;
      for (int u = 0; u < pr.nterm; ++u) {
        const int ax = pr.pw[u][0] * p, ay = pr.pw[u][1] * p, az = pr.pw[u][2] * p;
        if (BLOCH) {
          const double xr = tx[ax], xm = tx[4 * p + ax], yr = ty[ay], ym = ty[4 * p + ay];
          const double zr = pr.coef[u] * tz[az], zm = pr.coef[u] * tz[4 * p + az];
          const double rr = xr * yr - xm * ym, ri = xr * ym + xm * yr;
          v += rr * zr - ri * zm;
          vi += rr * zm + ri * zr;
        } else {
          v = fma(pr.coef[u] * tz[az], tx[ax] * ty[ay], v);
        }
      }
      const double w = P.w[qs + q];
      f[NC * g * p3 + q] = w * v;
      if (BLOCH) f[(NC * g + 1) * p3 + q] = w * vi;
    }
    __syncthreads();
    {   // FE functions: z, y, x
      double *T1 = W, *T2 = W + 4 * nf * p2;   // [c][field][p^2], [b c][field][p]
      for (int o = tid; o < nf * p2; o += PJ_NT) {
        const int g = o / p2, xy = o - g * p2;
        double s[4] = {0, 0, 0, 0};
        for (int qz = 0; qz < p; ++qz) {
          const double v = f[g * p3 + p2 * qz + xy];
#pragma unroll
          for (int c = 0; c < 4; ++c) s[c] = fma(v, L[(8 + c) * p + qz], s[c]);
        }
#pragma unroll
        for (int c = 0; c < 4; ++c) T1[c * nf * p2 + o] = s[c];
      }
      __syncthreads();
      for (int o = tid; o < 4 * nf * p; o += PJ_NT) {
        const int cg = o / p, qx = o - cg * p;   // (c, field)
        double s[4] = {0, 0, 0, 0};
        for (int qy = 0; qy < p; ++qy) {
          const double v = T1[cg * p2 + p * qy + qx];
#pragma unroll
          for (int b = 0; b < 4; ++b) s[b] = fma(v, L[(4 + b) * p + qy], s[b]);
        }
        const int c = cg / nf, g = cg - c * nf;
#pragma unroll
        for (int b = 0; b < 4; ++b) T2[((c * 4 + b) * nf + g) * p + qx] = s[b];
      }
      __syncthreads();
      for (int o = tid; o < 16 * nf; o += PJ_NT) {
        const int cb = o / nf, g = o - cb * nf;
        double s[4] = {0, 0, 0, 0};
        for (int qx = 0; qx < p; ++qx) {
          const double v = T2[o * p + qx];
#pragma unroll
          for (int a = 0; a < 4; ++a) s[a] = fma(v, L[a * p + qx], s[a]);
        }
#pragma unroll
        for (int a = 0; a < 4; ++a) acc[g * na + 4 * cb + a] += s[a];
      }
    }
    for (int s0 = 0; s0 < A; s0 += P.sc) {   // slots: z, y, x on the two linears
      const int ns = min(P.sc, A - s0), np = ns * nf;
      double *T1 = W, *T2 = W + 2 * np * p2;   // [t_z][slot field][p^2], [t_y t_z][slot field][p]
      __syncthreads();
      for (int o = tid; o < np * p2; o += PJ_NT) {
        const int sg = o / p2, xy = o - sg * p2, sl = sg / nf, g = sg - sl * nf;
        const double *ps = pe + (int64_t)(s0 + sl) * 4 * Q + pq + xy;
        double a = 0.0, b = 0.0;
        for (int qz = 0; qz < p; ++qz) {
          const double v = f[g * p3 + p2 * qz + xy] * ps[p2 * qz];
          a = fma(v, l[4 * p + qz], a);
          b = fma(v, l[5 * p + qz], b);
        }
        T1[o] = a;
        T1[np * p2 + o] = b;
      }
      __syncthreads();
      for (int o = tid; o < 2 * np * p; o += PJ_NT) {
        const int zs = o / p, qx = o - zs * p;   // (t_z, slot field)
        double a = 0.0, b = 0.0;
        for (int qy = 0; qy < p; ++qy) {
          const double v = T1[zs * p2 + p * qy + qx];
          a = fma(v, l[2 * p + qy], a);
          b = fma(v, l[3 * p + qy], b);
        }
        const int tz = zs / np, sg = zs - tz * np;
        T2[((2 * tz) * np + sg) * p + qx] = a;
        T2[((2 * tz + 1) * np + sg) * p + qx] = b;
      }
      __syncthreads();
      for (int o = tid; o < 4 * np; o += PJ_NT) {
        const int zy = o / np, sg = o - zy * np, sl = sg / nf, g = sg - sl * nf;
        double a = 0.0, b = 0.0;
        for (int qx = 0; qx < p; ++qx) {
          const double v = T2[o * p + qx];
          a = fma(v, l[qx], a);
          b = fma(v, l[p + qx], b);
        }
        double *t = acc + g * na + 64 + 8 * (s0 + sl) + 2 * zy;   // vertex code t_x + 2 t_y + 4 t_z
        t[0] += a;
        t[1] += b;
      }
    }
  }
  __syncthreads();
  const int n = (int)(P.doff[e + 1] - P.doff[e]);
  const int32_t *ec = P.ecol + (P.doff[e] - 64ll * e);
  for (int o = tid; o < n * pc; o += PJ_NT) {
    const int i = o / pc, g = o - i * pc;
    const double *t = acc + NC * g * na + (i < 64 ? i : 64 + ec[i - 64]);
    const int64_t to = (int64_t)P.dofs[P.doff[e] + i] * P.P + j0 + g;
    if (BLOCH) {   // times conj(exp(i k.R_i))
      const int c = P.eshift[P.doff[e] + i];
      const double cr = P.ph.re[c], ci = -P.ph.im[c], ar = t[0], ai = t[na];
      atomicAdd(P.F + to, cr * ar - ci * ai);
      atomicAdd(P.Fi + to, cr * ai + ci * ar);
    } else {
      atomicAdd(P.F + to, t[0]);
    }
  }
}

}  // namespace

pufe_status launch_projections(pufe_ctx *ctx, const ProjDev *pj, int P, const double *k,
                               double *F, double *Fi, cudaStream_t st) {
  auto &D = ctx->d;
  const int n = ctx->max_basis, nc = k ? 2 : 1;
  // (the element blocks that the call takes: n_e x nproj values per part)
  if (((size_t)8 * n + (size_t)nc * (8 + n) * P) * sizeof(double) + 8 * 24 * sizeof(double) >
      227 * 1024)
    return fail(PUFE_EINVAL, "n_e * nproj too large for the projection kernel");
  ProjArgs A{};
  A.qoff = D.qoff;
  A.w = D.w;
  A.xi = D.xi;
  A.x = D.x;
  A.partoff = D.partoff;
  A.part_p = D.part_p;
  A.part_q = D.part_q;
  A.doff = D.doff;
  A.dofs = D.dofs;
  A.ecol = D.ecol;
  A.aoff = D.aoff;
  A.toff = D.toff;
  A.psi = D.psi;
  A.pj = pj;
  A.P = P;
  for (int d = 0; d < 3; ++d) A.a[d] = ctx->a[d];
  A.eshift = D.eshift;
  A.F = F;
  A.Fi = Fi;
  if (k) {
    A.ph = phase_table(ctx, k);
    for (int d = 0; d < 3; ++d) A.k[d] = k[d];
  }
  // projectors per CTA: as many (up to 8) as the work area holds with one slot per
  // pass and as leave two CTAs per SM; then the slots per pass that still fit
  const int amax = std::max(1, ctx->max_alpha), pm = ctx->max_part_p;
  A.pc = std::min(8, P);
  while (A.pc > 1 && (proj_doubles(nc * A.pc, A.pc, 1, amax, pm, nc) > PJ_WORK ||
                      ctx->nelem * ((P + A.pc - 1) / A.pc) < 2 * ctx->nsm))
    A.pc = (A.pc + 1) / 2;
  A.sc = 1;
  while (A.sc < amax && proj_doubles(nc * A.pc, A.pc, A.sc + 1, amax, pm, nc) <= PJ_WORK) ++A.sc;
  const size_t sm = (size_t)proj_doubles(nc * A.pc, A.pc, A.sc, amax, pm, nc) * sizeof(double);
  if (sm > 227 * 1024) return fail(PUFE_EINVAL, "n_e * nproj too large for the projection kernel");
  auto kern = k ? k_projections_sf<true> : k_projections_sf<false>;
  PUFE_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
  const dim3 grid((unsigned)ctx->nelem, (unsigned)((P + A.pc - 1) / A.pc));
  kern<<<grid, PJ_NT, sm, st>>>(A);
  PUFE_CUDA_TRY(cudaGetLastError());
  return PUFE_OK;
}

}  // namespace pufe
