// Self-consistent-field step (Sec. 3): ionic charge, total Coulomb potential,
// LDA exchange-correlation, occupations, density mixing and total energy.
//
// Coulomb potential.  Sec. 3 (eq. poisson) obtains V_C = V_I + V_H from one
// Poisson equation for the total charge rho = rho_I - n (Gaussian ionic
// charges, electrons with density n).  It is solved in the tricubic FE space
// of the mesh:  -K v = 4 pi b,  K_ij = int grad phi_i . grad phi_j,
// b_i = int phi_i rho (shared element rule), zero cell average.  The mesh is
// a periodic tensor grid, so K = K1 (x) M1 (x) M1 + M1 (x) K1 (x) M1 +
// M1 (x) M1 (x) K1 with the 1D periodic cubic stiffness K1 and mass M1 of each
// axis.  With the 1D generalized eigenvectors X (K1 X = M1 X Lambda,
// X^T M1 X = I), K^+ = (X (x) X (x) X) D^+ (X (x) X (x) X)^T with
// D = Lambda_x + Lambda_y + Lambda_z: the solve is three small dense
// transforms along the axes, a diagonal scaling with the constant mode set to
// zero (which is exactly the zero-average solution), and three transforms
// back (the fast diagonalization method of Lynch, Rice and Thomas, 1964).
//
// LDA: Dirac exchange plus the Perdew-Zunger 1981 fit of the Ceperley-Alder
// correlation, unpolarised (the paper names the LDA without its fit).
// Everything here is FP64.
#include <algorithm>
#include <cmath>
#include <vector>

#include "pufe_internal.h"

namespace pufe {

// per-context work arrays of the SCF calls (allocated on first use)
constexpr int SCF_SUMS = 4, SCF_SLOTS = 32;   // reductions, partial sums of each
struct ScfState {
  int n1[3] = {0, 0, 0};
  double *X[3] = {nullptr, nullptr, nullptr};     // n1 x n1, row-major X[node][mode]
  double *lam[3] = {nullptr, nullptr, nullptr};   // n1, ascending
  bool b_dirty = false;     // a solve that failed left the load vector b as it was
  double *b = nullptr, *t0 = nullptr, *t1 = nullptr;   // n_fe each
  double *n_out = nullptr;  // n_q: output density of a step
  double *sums = nullptr;   // SCF_SUMS x SCF_SLOTS partial sums of the energies
  double *h_sums = nullptr; // pinned host copy
  double *f = nullptr;      // occupations: 64 states x up to 64 k-points (k-major)
  double *nk = nullptr;     // n_q: one k-point's density (k-point steps)
  double *atoms = nullptr;  // 5 per atom: tau (3), Z, sigma
  int atoms_cap = 0;
  double e_self = 0.0;      // self-energy of the last ionic charge set
  // Pulay history: ring of PULAY_MAX (input density, residual) pairs
  double *hist_n = nullptr, *hist_R = nullptr, *dots = nullptr;
  std::vector<int> slots;   // active slots, oldest first
  double gram[8][8] = {{0}};
  int next_slot = 0;
};

namespace {

constexpr double PI = 3.14159265358979323846;

// ---------------------------------------------------------------------------
// host: 1D periodic cubic FE matrices and their generalized eigenvectors
// ---------------------------------------------------------------------------

// cyclic Jacobi rotations: A (n x n, symmetric, row-major) -> Q Lambda Q^T
static void jacobi_eigen(int n, std::vector<double> &A, std::vector<double> &Q,
                         std::vector<double> &lam) {
  Q.assign((size_t)n * n, 0.0);
  for (int i = 0; i < n; ++i) Q[(size_t)i * n + i] = 1.0;
  double norm = 0.0;
  for (double v : A) norm += v * v;
  for (int sweep = 0; sweep < 100; ++sweep) {
    double off = 0.0;
    for (int i = 0; i < n; ++i)
      for (int j = i + 1; j < n; ++j) off += A[(size_t)i * n + j] * A[(size_t)i * n + j];
    if (off <= 1e-32 * norm) break;
    for (int p = 0; p < n; ++p)
      for (int q = p + 1; q < n; ++q) {
        const double apq = A[(size_t)p * n + q];
        if (std::fabs(apq) < 1e-300) continue;
        const double app = A[(size_t)p * n + p], aqq = A[(size_t)q * n + q];
        const double theta = (aqq - app) / (2.0 * apq);
        const double t = (theta >= 0 ? 1.0 : -1.0) / (std::fabs(theta) + std::sqrt(theta * theta + 1.0));
        const double c = 1.0 / std::sqrt(t * t + 1.0), s = t * c;
        for (int k = 0; k < n; ++k) {   // A <- J^T A J, columns p and q
          const double akp = A[(size_t)k * n + p], akq = A[(size_t)k * n + q];
          A[(size_t)k * n + p] = c * akp - s * akq;
          A[(size_t)k * n + q] = s * akp + c * akq;
        }
        for (int k = 0; k < n; ++k) {   // rows p and q
          const double apk = A[(size_t)p * n + k], aqk = A[(size_t)q * n + k];
          A[(size_t)p * n + k] = c * apk - s * aqk;
          A[(size_t)q * n + k] = s * apk + c * aqk;
        }
        for (int k = 0; k < n; ++k) {
          const double qkp = Q[(size_t)k * n + p], qkq = Q[(size_t)k * n + q];
          Q[(size_t)k * n + p] = c * qkp - s * qkq;
          Q[(size_t)k * n + q] = s * qkp + c * qkq;
        }
      }
  }
  lam.resize(n);
  for (int i = 0; i < n; ++i) lam[i] = A[(size_t)i * n + i];
}

// K1 X = M1 X Lambda, X^T M1 X = I for the periodic 1D cubic space of nel
// elements of length h (3 nel nodes); modes sorted by ascending Lambda
static void axis_modes(int nel, double h, std::vector<double> &X, std::vector<double> &lam) {
  const int n = 3 * nel;
  // 4-point Gauss-Legendre (exact for the degree-6 mass integrand)
  const double a = std::sqrt(3.0 / 7.0 - 2.0 / 7.0 * std::sqrt(6.0 / 5.0));
  const double b = std::sqrt(3.0 / 7.0 + 2.0 / 7.0 * std::sqrt(6.0 / 5.0));
  const double wa = (18.0 + std::sqrt(30.0)) / 36.0, wb = (18.0 - std::sqrt(30.0)) / 36.0;
  const double gx[4] = {-b, -a, a, b}, gw[4] = {wb, wa, wa, wb};
  double Ke[4][4] = {{0}}, Me[4][4] = {{0}};
  for (int g = 0; g < 4; ++g) {
    double L[4], dL[4];
    lagrange3(gx[g], L, dL);
    for (int i = 0; i < 4; ++i)
      for (int j = 0; j < 4; ++j) {
        Me[i][j] += gw[g] * L[i] * L[j] * (h / 2.0);
        Ke[i][j] += gw[g] * dL[i] * dL[j] * (2.0 / h);
      }
  }
  std::vector<double> K((size_t)n * n, 0.0), M((size_t)n * n, 0.0);
  for (int e = 0; e < nel; ++e)
    for (int i = 0; i < 4; ++i)
      for (int j = 0; j < 4; ++j) {
        const int gi = (3 * e + i) % n, gj = (3 * e + j) % n;
        K[(size_t)gi * n + gj] += Ke[i][j];
        M[(size_t)gi * n + gj] += Me[i][j];
      }
  // M = L L^T
  std::vector<double> Lc((size_t)n * n, 0.0);
  for (int i = 0; i < n; ++i)
    for (int j = 0; j <= i; ++j) {
      double s = M[(size_t)i * n + j];
      for (int k = 0; k < j; ++k) s -= Lc[(size_t)i * n + k] * Lc[(size_t)j * n + k];
      Lc[(size_t)i * n + j] = (i == j) ? std::sqrt(s) : s / Lc[(size_t)j * n + j];
    }
  // Li = L^{-1} (lower triangular)
  std::vector<double> Li((size_t)n * n, 0.0);
  for (int j = 0; j < n; ++j) {
    Li[(size_t)j * n + j] = 1.0 / Lc[(size_t)j * n + j];
    for (int i = j + 1; i < n; ++i) {
      double s = 0.0;
      for (int k = j; k < i; ++k) s -= Lc[(size_t)i * n + k] * Li[(size_t)k * n + j];
      Li[(size_t)i * n + j] = s / Lc[(size_t)i * n + i];
    }
  }
  // A = L^{-1} K L^{-T}
  std::vector<double> T((size_t)n * n, 0.0), A((size_t)n * n, 0.0);
  for (int i = 0; i < n; ++i)
    for (int j = 0; j < n; ++j) {
      double s = 0.0;
      for (int k = 0; k <= i; ++k) s += Li[(size_t)i * n + k] * K[(size_t)k * n + j];
      T[(size_t)i * n + j] = s;
    }
  for (int i = 0; i < n; ++i)
    for (int j = 0; j < n; ++j) {
      double s = 0.0;
      for (int k = 0; k <= j; ++k) s += T[(size_t)i * n + k] * Li[(size_t)j * n + k];
      A[(size_t)i * n + j] = s;
    }
  for (int i = 0; i < n; ++i)   // exact symmetry before the rotations
    for (int j = i + 1; j < n; ++j) {
      const double s = 0.5 * (A[(size_t)i * n + j] + A[(size_t)j * n + i]);
      A[(size_t)i * n + j] = A[(size_t)j * n + i] = s;
    }
  std::vector<double> Q, l;
  jacobi_eigen(n, A, Q, l);
  std::vector<int> idx(n);
  for (int i = 0; i < n; ++i) idx[i] = i;
  std::sort(idx.begin(), idx.end(), [&](int p, int q) { return l[p] < l[q]; });
  // X = L^{-T} Q, columns in ascending Lambda
  X.assign((size_t)n * n, 0.0);
  lam.resize(n);
  for (int m = 0; m < n; ++m) {
    const int src = idx[m];
    lam[m] = l[src];
    for (int i = 0; i < n; ++i) {
      double s = 0.0;
      for (int k = i; k < n; ++k) s += Li[(size_t)k * n + i] * Q[(size_t)k * n + src];
      X[(size_t)i * n + m] = s;
    }
  }
  lam[0] = 0.0;   // the constant mode (zero up to rounding)
}

// ---------------------------------------------------------------------------
// kernels (FP64)
// ---------------------------------------------------------------------------

// rho_I(x_q) = sum_a Z_a e^{-r^2/s_a^2} / (pi^{3/2} s_a^3) over every periodic
// image within 6.8 s_a (where the Gaussian is below 1e-20)
__global__ void k_ion_density(int64_t nq, const double *__restrict__ x, int natoms,
                              const double *__restrict__ atoms, double ax, double ay, double az,
                              double *__restrict__ rho) {
  const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= nq) return;
  const double av[3] = {ax, ay, az};
  double s = 0.0;
  for (int ia = 0; ia < natoms; ++ia) {
    const double *at = atoms + 5 * ia;
    const double sig = at[4], rc = 6.8 * sig;
    double d[3];
    int lo[3], hi[3];
    for (int k = 0; k < 3; ++k) {
      d[k] = x[3 * q + k] - at[k];
      lo[k] = (int)ceil((-rc - d[k]) / av[k]);
      hi[k] = (int)floor((rc - d[k]) / av[k]);
    }
    const double amp = at[3] / (PI * sqrt(PI) * sig * sig * sig), is2 = 1.0 / (sig * sig);
    for (int i = lo[0]; i <= hi[0]; ++i)
      for (int j = lo[1]; j <= hi[1]; ++j)
        for (int k = lo[2]; k <= hi[2]; ++k) {
          const double dx = d[0] + i * ax, dy = d[1] + j * ay, dz = d[2] + k * az;
          s += amp * exp(-(dx * dx + dy * dy + dz * dz) * is2);
        }
  }
  rho[q] = s;
}

constexpr int SCF_PMAX = 16;   // largest points per axis of a (sub)cell
constexpr int SCF_NT = 128;

// 1D Lagrange factors of one p^3 (sub)cell along its three axes:
// L1[(d * 4 + a) * p + t] for axis d, function a, axis point t
__device__ __forceinline__ void cell_tables(const double *__restrict__ xi, int64_t qs, int p,
                                            double *L1) {
  for (int o = threadIdx.x; o < 3 * p; o += SCF_NT) {
    const int d = o / p, t = o - d * p;
    const int64_t stride = d == 0 ? 1 : (d == 1 ? p : (int64_t)p * p);
    double L[4], dL[4];
    lagrange3(xi[3 * (qs + t * stride) + d], L, dL);
    for (int a = 0; a < 4; ++a) L1[(d * 4 + a) * p + t] = L[a];
  }
}

// b_i += scale sum_q w_q phi_i(x_q) (n_q - rho_I,q) over the 64 FE functions of
// every element, by sum factorization over each p^3 (sub)cell (contract z, then y,
// then x: 5 p^3 + 16 p^2 + 64 p FP64 operations per cell, which bind it; a column
// of points is read once for its four z functions).  Also clears the energy sums
// of the step.
__global__ void __launch_bounds__(SCF_NT) k_fe_load(
    const int64_t *__restrict__ qoff, const double *__restrict__ w, const double *__restrict__ xi,
    const int32_t *__restrict__ partoff, const int32_t *__restrict__ part_p,
    const int32_t *__restrict__ part_q, const int64_t *__restrict__ doff,
    const int32_t *__restrict__ dofs, const double *__restrict__ n,
    const double *__restrict__ rho_I, double scale, int pm, double *__restrict__ b,
    double *__restrict__ sums) {
  extern __shared__ __align__(16) double sml[];
  double *L1 = sml, *T1 = L1 + 12 * pm, *T2 = T1 + 4 * pm * pm, *bl = T2 + 16 * pm;
  const int e = blockIdx.x, tid = threadIdx.x;
  if (e == 0)
    for (int o = tid; o < SCF_SUMS * SCF_SLOTS; o += SCF_NT) sums[o] = 0.0;
  for (int o = tid; o < 64; o += SCF_NT) bl[o] = 0.0;
  for (int k = partoff[e]; k < partoff[e + 1]; ++k) {
    const int p = part_p[k], p2 = p * p;
    const int64_t qs = qoff[e] + part_q[k];
    __syncthreads();
    cell_tables(xi, qs, p, L1);
    __syncthreads();
    for (int it = tid; it < p2; it += SCF_NT) {   // z: [c][qx + p qy]
      double s[4] = {0, 0, 0, 0};
#pragma unroll 4
      for (int qz = 0; qz < p; ++qz) {
        const int64_t q = qs + it + (int64_t)p2 * qz;
        const double v = w[q] * (n[q] - rho_I[q]);
#pragma unroll
        for (int c = 0; c < 4; ++c) s[c] = fma(v, L1[(8 + c) * p + qz], s[c]);
      }
#pragma unroll
      for (int c = 0; c < 4; ++c) T1[c * p2 + it] = s[c];
    }
    __syncthreads();
    for (int it = tid; it < p * 16; it += SCF_NT) {   // y: [b + 4 c][qx]
      const int bc = it / p, qx = it - bc * p, bb = bc & 3, c = bc >> 2;
      double s = 0.0;
      for (int qy = 0; qy < p; ++qy) s = fma(T1[c * p2 + p * qy + qx], L1[(4 + bb) * p + qy], s);
      T2[it] = s;
    }
    __syncthreads();
    for (int it = tid; it < 64; it += SCF_NT) {       // x
      const int a = it & 3, bc = it >> 2;
      double s = 0.0;
      for (int qx = 0; qx < p; ++qx) s = fma(T2[bc * p + qx], L1[a * p + qx], s);
      bl[it] += s;
    }
  }
  __syncthreads();
  for (int o = tid; o < 64; o += SCF_NT) atomicAdd(b + dofs[doff[e] + o], scale * bl[o]);
}

// One axis of the (n0, n1, n2) node array (x fastest): out[.., j, ..] =
// sum_k M[k][j] in[.., k, ..] with M = X (fwd) or X^T (back), X row-major
// [node][mode].  A CTA takes `nb` lines (8; fewer on very long axes).  n FP64
// multiply-adds per node bind it (2.7 us for 36^3 nodes) as long as nothing waits:
// M is staged in shared memory by one round of independent loads (reading it from
// L2 inside the sums, a few values ahead, took 13-25 us), and a sum runs in four
// chains.  M of more than AX_STAGE nodes per axis is read in place: its stage leaves two
// CTAs per SM, then one (whole potential at 96 nodes per axis 1,556 us staged, 1,582 us in
// place; at 102 2,085 and 1,838 us, at 111 2,724 and 2,483 us).
// `clear` (may be null): an array of the same size set to zero.
constexpr int AX_NT = 256;
constexpr int AX_STAGE = 96;

__device__ __forceinline__ int64_t line_base(int n0, int n1, int axis, int64_t line) {
  if (axis == 0) return line * n0;
  if (axis == 1) return (line % n0) + (line / n0) * ((int64_t)n0 * n1);
  return line;
}

// M into shared memory as [k][j] (staged) or left in place; entry (k, j) then is at
// k sk + j sj of the returned pointer
__device__ __forceinline__ const double *axis_matrix(const double *__restrict__ X, bool fwd, int n,
                                                     bool staged, double *M, int &sk, int &sj) {
  if (!staged) {
    sk = fwd ? n : 1;
    sj = fwd ? 1 : n;
    return X;
  }
  if (fwd)
    for (int o = threadIdx.x; o < n * n; o += AX_NT) M[o] = X[o];
  else
    for (int o = threadIdx.x; o < n * n; o += AX_NT) {
      const int j = o / n, k = o - j * n;
      M[k * n + j] = X[o];
    }
  sk = n;
  sj = 1;
  return M;
}

__device__ __forceinline__ double line_sum(const double *m, int sk, int n, const double *in,
                                           int nb) {
  double s[4] = {0, 0, 0, 0};
  int k = 0;
  for (; k + 4 <= n; k += 4) {
#pragma unroll
    for (int u = 0; u < 4; ++u) s[u] = fma(m[(int64_t)(k + u) * sk], in[(k + u) * nb], s[u]);
  }
  for (; k < n; ++k) s[0] = fma(m[(int64_t)k * sk], in[k * nb], s[0]);
  return (s[0] + s[1]) + (s[2] + s[3]);
}

__global__ void __launch_bounds__(AX_NT) k_axis(int n0, int n1, int n2, int axis, int nb,
                                                bool staged, const double *__restrict__ X,
                                                bool fwd, const double *__restrict__ in,
                                                double *__restrict__ out,
                                                double *__restrict__ clear) {
  extern __shared__ __align__(16) double smx[];   // [k][line], then M
  const int n = axis == 0 ? n0 : (axis == 1 ? n1 : n2);
  const int64_t lines = (int64_t)n0 * n1 * n2 / n, l0 = (int64_t)blockIdx.x * nb;
  const int nl = (int)min((int64_t)nb, lines - l0);
  const int64_t stride = axis == 0 ? 1 : (axis == 1 ? n0 : (int64_t)n0 * n1);
  int sk, sj;
  const double *M = axis_matrix(X, fwd, n, staged, smx + n * nb, sk, sj);
  for (int o = threadIdx.x; o < nl * n; o += AX_NT) {
    const int l = axis == 0 ? o / n : o % nl, k = axis == 0 ? o - l * n : o / nl;
    smx[k * nb + l] = in[line_base(n0, n1, axis, l0 + l) + k * stride];
  }
  __syncthreads();
  for (int o = threadIdx.x; o < nl * n; o += AX_NT) {
    const int l = axis == 0 ? o / n : o % nl, j = axis == 0 ? o - l * n : o / nl;
    const int64_t at = line_base(n0, n1, axis, l0 + l) + j * stride;
    out[at] = line_sum(M + (int64_t)j * sj, sk, n, smx + l, nb);
    if (clear) clear[at] = 0.0;
  }
}

// The z axis both ways around the modal scaling: forward, c_abc / (lx_a + ly_b +
// lz_c) with the constant mode (0, 0, 0) set to zero, and back, on the same lines
// (back reads the same staged matrix by rows).
__global__ void __launch_bounds__(AX_NT) k_axis_z(int n0, int n1, int n2, int nb, bool staged,
                                                  const double *__restrict__ X,
                                                  const double *__restrict__ lx,
                                                  const double *__restrict__ ly,
                                                  const double *__restrict__ lz,
                                                  const double *__restrict__ in,
                                                  double *__restrict__ out) {
  extern __shared__ __align__(16) double smx[];   // [k][line], twice, then X
  double *c = smx + n2 * nb;
  const int64_t plane = (int64_t)n0 * n1, l0 = (int64_t)blockIdx.x * nb;
  const int nl = (int)min((int64_t)nb, plane - l0);
  int sk, sj;
  const double *M = axis_matrix(X, true, n2, staged, c + n2 * nb, sk, sj);
  for (int o = threadIdx.x; o < nl * n2; o += AX_NT) {
    const int l = o % nl, k = o / nl;
    smx[k * nb + l] = in[l0 + l + k * plane];
  }
  __syncthreads();
  for (int o = threadIdx.x; o < nl * n2; o += AX_NT) {
    const int l = o % nl, j = o / nl;
    const int64_t xy = l0 + l;
    const double s = line_sum(M + (int64_t)j * sj, sk, n2, smx + l, nb);
    c[j * nb + l] = (xy == 0 && j == 0) ? 0.0 : s / (lx[xy % n0] + ly[xy / n0] + lz[j]);
  }
  __syncthreads();
  for (int o = threadIdx.x; o < nl * n2; o += AX_NT) {
    const int l = o % nl, j = o / nl;
    out[l0 + l + j * plane] = line_sum(M + (int64_t)j * sk, sj, n2, c + l, nb);
  }
}

// Powers for the LDA from their FP32 values, each refined once by Householder's
// iteration of third order (the residual r of an FP32 start is about 2^-22, so the
// terms left out are below 2^-62): a handful of FP64 operations each, where the
// library's cbrt, square root and division take tens -- and FP64 operations are what
// binds a pass over the points.
// n^(-1/3), 1e-30 < n: y <- y (1 + r / 3 + 2 r^2 / 9), r = 1 - n y^3 (values beyond
// the FP32 range take cbrt)
__device__ __forceinline__ double inv_cbrt(double n) {
  if (!(n < 1e37)) return 1.0 / cbrt(n);
  const double y = (double)rcbrtf((float)n);
  const double r = fma(-n * y, y * y, 1.0);
  return fma(y * r, fma(r, 2.0 / 9.0, 1.0 / 3.0), y);
}
// x^(-1/2), 1 <= x < 1e30: y <- y (1 + r / 2 + 3 r^2 / 8), r = 1 - x y^2
__device__ __forceinline__ double inv_sqrt(double x) {
  const double y = (double)rsqrtf((float)x);
  const double r = fma(-x * y, y, 1.0);
  return fma(y * r, fma(r, 0.375, 0.5), y);
}
// 1 / x, 1 <= x < 1e30: y <- y (1 + r + r^2), r = 1 - x y
__device__ __forceinline__ double inverse(double x) {
  const double y = (double)(1.0f / (float)x);
  const double r = fma(-x, y, 1.0);
  return fma(y * r, r + 1.0, y);
}

// Dirac exchange + Perdew-Zunger 1981 correlation (unpolarised); 0 for n <= 1e-30.
// The energy per electron (v false) or the potential (v true).
__device__ __forceinline__ double lda_pz81(double n, bool v) {
  if (!(n > 1e-30)) return 0.0;
  const double y = inv_cbrt(n);
  const double rs = 0.62035049089940009 * y;           // (3 / (4 pi))^(1/3) n^(-1/3)
  const double ex = -0.73855876638202240 * (n * y * y);   // -3/4 (3 / pi)^(1/3) n^(1/3)
  if (rs >= 1.0) {
    const double sq = rs * inv_sqrt(rs);
    const double inv = inverse(fma(1.0529, sq, fma(0.3334, rs, 1.0)));
    if (!v) return fma(-0.1423, inv, ex);
    return fma(4.0 / 3.0, ex,
               -0.1423 * fma(7.0 / 6.0 * 1.0529, sq, fma(4.0 / 3.0 * 0.3334, rs, 1.0)) * inv * inv);
  }
  const double lr = log(rs);
  if (!v) return ex + (0.0311 * lr - 0.048 + 0.0020 * rs * lr - 0.0116 * rs);
  return fma(4.0 / 3.0, ex,
             0.0311 * lr + (-0.048 - 0.0311 / 3.0) + 2.0 / 3.0 * 0.0020 * rs * lr +
                 (2.0 * -0.0116 - 0.0020) / 3.0 * rs);
}

// V_C(x_q) = sum_i v_i phi_i(x_q) over the 64 FE functions, by sum factorization
// over each p^3 (sub)cell (x, then y, then z), and what the caller makes of it at
// the point while it is in a register:
//  * V_eff != nullptr: V_eff = V_C + v_xc(n), and V_C, eps_xc where wanted;
//  * else the energies of n (an output density) and its mixing: partial sums
//    [0] += w n V_in, [1] += w (rho_I - n) V_C, [2] += w n eps_xc, [3] += w |n - n_in|
//    (32 partial sums each: thousands of atomics on one address would take longer
//    than the sums themselves), then n_in <- n_in + alpha (n - n_in).
struct InterpOut {
  const double *n;
  double *V_eff, *V_C, *eps_xc;
  const double *w, *V_in, *rho_I;
  double alpha;
  double *n_in, *sums;
};

__global__ void __launch_bounds__(SCF_NT) k_fe_interp(
    const int64_t *__restrict__ qoff, const double *__restrict__ xi,
    const int32_t *__restrict__ partoff, const int32_t *__restrict__ part_p,
    const int32_t *__restrict__ part_q, const int64_t *__restrict__ doff,
    const int32_t *__restrict__ dofs, const double *__restrict__ v, int pm, InterpOut O) {
  extern __shared__ __align__(16) double smi[];
  double *L1 = smi, *ve = L1 + 12 * pm, *T1 = ve + 64, *T2 = T1 + 16 * pm;   // T2: [c][qx + p qy]
  double *red = T2 + 4 * pm * pm;                                            // [4][warps]
  const int e = blockIdx.x, tid = threadIdx.x;
  for (int o = tid; o < 64; o += SCF_NT) ve[o] = v[dofs[doff[e] + o]];
  double s4[SCF_SUMS] = {0.0, 0.0, 0.0, 0.0};
  for (int k = partoff[e]; k < partoff[e + 1]; ++k) {
    const int p = part_p[k], p2 = p * p;
    const int64_t qs = qoff[e] + part_q[k];
    __syncthreads();
    cell_tables(xi, qs, p, L1);
    __syncthreads();
    for (int it = tid; it < 16 * p; it += SCF_NT) {   // x
      const int bc = it / p, qx = it - bc * p;
      double s = 0.0;
#pragma unroll
      for (int a = 0; a < 4; ++a) s = fma(ve[a + 4 * bc], L1[a * p + qx], s);
      T1[it] = s;
    }
    __syncthreads();
    for (int it = tid; it < 4 * p2; it += SCF_NT) {   // y
      const int c = it / p2, qxy = it - c * p2, qy = qxy / p, qx = qxy - qy * p;
      double s = 0.0;
#pragma unroll
      for (int bb = 0; bb < 4; ++bb) s = fma(T1[(bb + 4 * c) * p + qx], L1[(4 + bb) * p + qy], s);
      T2[it] = s;
    }
    __syncthreads();
    for (int it = tid; it < p2 * p; it += SCF_NT) {   // z
      const int qz = it / p2, qxy = it - qz * p2;
      const int64_t q = qs + it;
      double vc = 0.0;
#pragma unroll
      for (int c = 0; c < 4; ++c) vc = fma(T2[c * p2 + qxy], L1[(8 + c) * p + qz], vc);
      const double n = O.n[q];
      if (O.V_eff) {
        if (O.V_C) O.V_C[q] = vc;
        if (O.eps_xc) O.eps_xc[q] = lda_pz81(n, false);
        O.V_eff[q] = vc + lda_pz81(n, true);
      } else {
        const double w = O.w[q], wn = w * n, ni = O.n_in[q];
        s4[0] = fma(wn, O.V_in[q], s4[0]);
        s4[1] = fma(w * (O.rho_I[q] - n), vc, s4[1]);
        s4[2] = fma(wn, lda_pz81(n, false), s4[2]);
        s4[3] = fma(w, fabs(n - ni), s4[3]);
        O.n_in[q] = ni + O.alpha * (n - ni);
      }
    }
  }
  if (O.V_eff) return;
  const int lane = tid & 31, warp = tid >> 5, nw = (SCF_NT + 31) / 32;
  for (int k = 0; k < SCF_SUMS; ++k) {
    double t = s4[k];
    for (int off = 16; off > 0; off >>= 1) t += __shfl_xor_sync(0xffffffffu, t, off);
    if (lane == 0) red[k * nw + warp] = t;
  }
  __syncthreads();
  for (int k = tid; k < SCF_SUMS; k += SCF_NT) {
    double t = 0.0;
    for (int i = 0; i < nw; ++i) t += red[k * nw + i];
    atomicAdd(O.sums + k * SCF_SLOTS + (e & (SCF_SLOTS - 1)), t);
  }
}

__global__ void k_add(int64_t nq, const double *__restrict__ a, const double *__restrict__ b,
                      double *__restrict__ out) {    // out = a + b
  const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (q < nq) out[q] = a[q] + b[q];
}

constexpr int PULAY_MAX = 8;
struct SlotList {
  int m;
  int s[PULAY_MAX];
  double c[PULAY_MAX];
};

// store (n_in, n_out - n_in) in slot `slot` of the history and accumulate
// dots[j] += sum_q w_q R_new R_j for the active slots
__global__ void k_pulay_store(int64_t nq, const double *__restrict__ w,
                              const double *__restrict__ n_in, const double *__restrict__ n_out,
                              int slot, SlotList L, double *__restrict__ hn, double *__restrict__ hR,
                              double *__restrict__ dots) {
  __shared__ double red[PULAY_MAX][8];
  const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  double r = 0.0, wq = 0.0;
  if (q < nq) {
    r = n_out[q] - n_in[q];
    wq = w[q];
    hn[(int64_t)slot * nq + q] = n_in[q];
    hR[(int64_t)slot * nq + q] = r;
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int j = 0; j < L.m; ++j) {
    double t = 0.0;
    if (q < nq) t = wq * r * (L.s[j] == slot ? r : hR[(int64_t)L.s[j] * nq + q]);
    for (int off = 16; off > 0; off >>= 1) t += __shfl_xor_sync(0xffffffffu, t, off);
    if (lane == 0) red[j][warp] = t;
  }
  __syncthreads();
  if (threadIdx.x < L.m) {
    double t = 0.0;
    for (int i = 0; i < (int)(blockDim.x >> 5); ++i) t += red[threadIdx.x][i];
    atomicAdd(dots + threadIdx.x, t);
  }
}

// n = sum_i c_i (n_i + alpha R_i) over the active slots
__global__ void k_pulay_mix(int64_t nq, SlotList L, double alpha, const double *__restrict__ hn,
                            const double *__restrict__ hR, double *__restrict__ n) {
  const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= nq) return;
  double s = 0.0;
  for (int i = 0; i < L.m; ++i)
    s += L.c[i] * (hn[(int64_t)L.s[i] * nq + q] + alpha * hR[(int64_t)L.s[i] * nq + q]);
  n[q] = s;
}

// solve the (m + 1) bordered system [A 1; 1^T 0] [c; l] = [0; 1] by Gaussian
// elimination with partial pivoting (m <= 8)
static bool pulay_coefficients(int m, const double A[8][8], double *c) {
  double M[9][10] = {{0}};
  double tr = 0.0;
  for (int i = 0; i < m; ++i) tr += A[i][i];
  const double ridge = 1e-12 * tr / m;
  for (int i = 0; i < m; ++i) {
    for (int j = 0; j < m; ++j) M[i][j] = A[i][j] + (i == j ? ridge : 0.0);
    M[i][m] = 1.0;
    M[m][i] = 1.0;
  }
  M[m][m + 1] = 1.0;
  const int n = m + 1;
  for (int k = 0; k < n; ++k) {
    int piv = k;
    for (int i = k + 1; i < n; ++i)
      if (std::fabs(M[i][k]) > std::fabs(M[piv][k])) piv = i;
    if (std::fabs(M[piv][k]) < 1e-300) return false;
    for (int j = 0; j <= n; ++j) std::swap(M[k][j], M[piv][j]);
    for (int i = k + 1; i < n; ++i) {
      const double f = M[i][k] / M[k][k];
      for (int j = k; j <= n; ++j) M[i][j] -= f * M[k][j];
    }
  }
  double x[9];
  for (int i = n - 1; i >= 0; --i) {
    double t = M[i][n];
    for (int j = i + 1; j < n; ++j) t -= M[i][j] * x[j];
    x[i] = t / M[i][i];
  }
  for (int i = 0; i < m; ++i) c[i] = x[i];
  return true;
}

inline unsigned blocks(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }

}  // namespace

pufe_status scf_prepare(pufe_ctx *ctx) {
  if (ctx->scf) return PUFE_OK;
  if (ctx->max_part_p > SCF_PMAX) return fail(PUFE_EINVAL, "rule with more than 16 points per axis");
  auto *S = new ScfState();
  ctx->scf = S;
  auto &D = ctx->d;
  (void)D;
  for (int d = 0; d < 3; ++d) {
    std::vector<double> X, lam;
    axis_modes(ctx->nel[d], ctx->h[d], X, lam);
    S->n1[d] = 3 * ctx->nel[d];
    PUFE_CUDA_TRY(cudaMalloc((void **)&S->X[d], X.size() * sizeof(double)));
    PUFE_CUDA_TRY(cudaMalloc((void **)&S->lam[d], lam.size() * sizeof(double)));
    PUFE_CUDA_TRY(cudaMemcpy(S->X[d], X.data(), X.size() * sizeof(double), cudaMemcpyHostToDevice));
    PUFE_CUDA_TRY(
        cudaMemcpy(S->lam[d], lam.data(), lam.size() * sizeof(double), cudaMemcpyHostToDevice));
  }
  const size_t nfe = (size_t)ctx->n_fe * sizeof(double), nq = (size_t)ctx->nq * sizeof(double);
  PUFE_CUDA_TRY(cudaMalloc((void **)&S->b, nfe));
  PUFE_CUDA_TRY(cudaMemset(S->b, 0, nfe));
  PUFE_CUDA_TRY(cudaMalloc((void **)&S->t0, nfe));
  PUFE_CUDA_TRY(cudaMalloc((void **)&S->t1, nfe));
  PUFE_CUDA_TRY(cudaMalloc((void **)&S->n_out, nq));
  PUFE_CUDA_TRY(cudaMalloc((void **)&S->sums, SCF_SUMS * SCF_SLOTS * sizeof(double)));
  PUFE_CUDA_TRY(cudaMallocHost((void **)&S->h_sums, SCF_SUMS * SCF_SLOTS * sizeof(double)));
  PUFE_CUDA_TRY(cudaMalloc((void **)&S->f, 64 * 64 * sizeof(double)));
  // the copies and the clearing above are done before a solve on a caller's stream,
  // which need not wait for the default one
  PUFE_CUDA_TRY(cudaStreamSynchronize(0));
  return PUFE_OK;
}

void scf_free(pufe_ctx *ctx) {
  ScfState *S = ctx->scf;
  if (!S) return;
  void *ptrs[] = {S->X[0], S->X[1], S->X[2], S->lam[0], S->lam[1], S->lam[2], S->b, S->t0,
                  S->t1, S->n_out, S->sums, S->f, S->nk, S->atoms,
                  S->hist_n, S->hist_R, S->dots};
  for (void *p : ptrs)
    if (p) cudaFree(p);
  if (S->h_sums) cudaFreeHost(S->h_sums);
  delete S;
  ctx->scf = nullptr;
}

pufe_status launch_ion_density(pufe_ctx *ctx, int natoms, const double *tau, const double *Z,
                               const double *sigma, double *rho, cudaStream_t st) {
  if (pufe_status e0 = scf_prepare(ctx)) return e0;
  ScfState *S = ctx->scf;
  if (natoms > S->atoms_cap) {
    if (S->atoms) PUFE_CUDA_TRY(cudaFree(S->atoms));
    S->atoms = nullptr;
    PUFE_CUDA_TRY(cudaMalloc((void **)&S->atoms, (size_t)5 * std::max(1, natoms) * sizeof(double)));
    S->atoms_cap = natoms;
  }
  std::vector<double> at((size_t)5 * std::max(1, natoms), 0.0);
  double es = 0.0;
  for (int a = 0; a < natoms; ++a) {
    for (int k = 0; k < 3; ++k) at[5 * a + k] = tau[3 * a + k];
    at[5 * a + 3] = Z[a];
    at[5 * a + 4] = sigma[a];
    es += Z[a] * Z[a] / (sigma[a] * std::sqrt(2.0 * PI));
  }
  S->e_self = es;
  // synchronous copy: the host vector is a temporary
  PUFE_CUDA_TRY(cudaMemcpy(S->atoms, at.data(), at.size() * sizeof(double), cudaMemcpyHostToDevice));
  k_ion_density<<<blocks(ctx->nq, 256), 256, 0, st>>>(ctx->nq, ctx->d.x, natoms, S->atoms,
                                                      ctx->a[0], ctx->a[1], ctx->a[2], rho);
  PUFE_CUDA_TRY(cudaGetLastError());
  return PUFE_OK;
}

// V_C with del^2 V_C = 4 pi (rho_I - n), zero cell average, and at every point what
// `O` asks for (its n is this n)
static pufe_status coulomb(pufe_ctx *ctx, const double *rho_I, const InterpOut &O,
                           cudaStream_t st) {
  ScfState *S = ctx->scf;
  auto &D = ctx->d;
  const int n0 = S->n1[0], n1 = S->n1[1], n2 = S->n1[2], pm = std::max(1, ctx->max_part_p);
  const int64_t nfe = ctx->n_fe;
  const size_t sm_load = (size_t)(12 * pm + 4 * pm * pm + 16 * pm + 64) * sizeof(double);
  const size_t sm_out = (size_t)(12 * pm + 64 + 16 * pm + 4 * pm * pm + 16) * sizeof(double);
  int nb = 8;   // lines per CTA: what two copies of the longest axis' lines leave
  const int nmax = std::max(n0, std::max(n1, n2));
  while (nb > 1 && (size_t)2 * nmax * nb * sizeof(double) > 96 * 1024) nb /= 2;
  const bool staged = nmax <= AX_STAGE;   // the matrix beside the lines
  const size_t sm_ax = ((size_t)2 * nmax * nb + (staged ? (size_t)nmax * nmax : 0)) * sizeof(double);
  if (sm_ax > 227 * 1024)
    return fail(PUFE_EINVAL, "more nodes per axis than the Poisson solve takes");
  auto lines = [&](int n) { return (unsigned)((nfe / n + nb - 1) / nb); };
  PUFE_CUDA_TRY(cudaFuncSetAttribute(k_axis, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm_ax));
  PUFE_CUDA_TRY(cudaFuncSetAttribute(k_axis_z, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm_ax));
  // the load vector is zero here unless a launch of an earlier solve failed between
  // the kernel that adds into it and the one that clears it
  if (S->b_dirty) PUFE_CUDA_TRY(cudaMemsetAsync(S->b, 0, nfe * sizeof(double), st));
  S->b_dirty = true;
  // -K v = 4 pi int phi (rho_I - n)  <=>  K v = 4 pi int phi (n - rho_I)
  k_fe_load<<<(unsigned)ctx->nelem, SCF_NT, sm_load, st>>>(
      D.qoff, D.w, D.xi, D.partoff, D.part_p, D.part_q, D.doff, D.dofs, O.n, rho_I, 4.0 * PI, pm,
      S->b, S->sums);
  k_axis<<<lines(n0), AX_NT, sm_ax, st>>>(n0, n1, n2, 0, nb, staged, S->X[0], true, S->b, S->t0,
                                                    nullptr);
  k_axis<<<lines(n1), AX_NT, sm_ax, st>>>(n0, n1, n2, 1, nb, staged, S->X[1], true, S->t0, S->t1,
                                                    S->b);
  PUFE_CUDA_TRY(cudaGetLastError());
  S->b_dirty = false;
  k_axis_z<<<lines(n2), AX_NT, sm_ax, st>>>(n0, n1, n2, nb, staged, S->X[2], S->lam[0], S->lam[1],
                                                      S->lam[2], S->t1, S->t0);
  k_axis<<<lines(n1), AX_NT, sm_ax, st>>>(n0, n1, n2, 1, nb, staged, S->X[1], false, S->t0, S->t1,
                                                    nullptr);
  k_axis<<<lines(n0), AX_NT, sm_ax, st>>>(n0, n1, n2, 0, nb, staged, S->X[0], false, S->t1, S->t0,
                                                    nullptr);
  k_fe_interp<<<(unsigned)ctx->nelem, SCF_NT, sm_out, st>>>(
      D.qoff, D.xi, D.partoff, D.part_p, D.part_q, D.doff, D.dofs, S->t0, pm, O);
  PUFE_CUDA_TRY(cudaGetLastError());
  return PUFE_OK;
}

pufe_status launch_effective_potential(pufe_ctx *ctx, const double *n, const double *rho_I,
                                       double *V_eff, double *V_C, double *eps_xc,
                                       cudaStream_t st) {
  if (pufe_status e0 = scf_prepare(ctx)) return e0;
  InterpOut O{};
  O.n = n;
  O.V_eff = V_eff;
  O.V_C = V_C;
  O.eps_xc = eps_xc;
  return coulomb(ctx, rho_I, O, st);
}

void scf_reset(pufe_ctx *ctx) {
  if (!ctx->scf) return;
  ctx->scf->slots.clear();
  ctx->scf->next_slot = 0;
}

// Fermi-Dirac occupations of nk k-points x nstates states (eps and f
// k-major) with weights wk (nullptr: one k-point of weight 1): mu by bisection
// on sum_k w_k sum_n f_nk = nelec; the band energy and the entropy sum
// sum_k w_k sum_n [g ln g + (1 - g) ln(1 - g)] (g = f / 2) weighted alike.
static double occupations(int nk, const double *wk, int nstates, const double *eps, double nelec,
                          double kT, std::vector<double> &f, double &e_band, double &ts) {
  const int nt = nk * nstates;
  double lo = eps[0], hi = eps[0];
  for (int k = 1; k < nt; ++k) {
    lo = std::min(lo, eps[k]);
    hi = std::max(hi, eps[k]);
  }
  lo -= 50.0 * kT + 1.0;
  hi += 50.0 * kT + 1.0;
  f.assign(nt, 0.0);
  auto occ = [&](double mu) {
    double s = 0.0;
    for (int k = 0; k < nt; ++k) {
      const double x = std::min(700.0, std::max(-700.0, (eps[k] - mu) / kT));
      f[k] = 2.0 / (1.0 + std::exp(x));
      s += (wk ? wk[k / nstates] : 1.0) * f[k];
    }
    return s;
  };
  for (int it = 0; it < 200; ++it) {
    const double mid = 0.5 * (lo + hi);
    if (occ(mid) < nelec)
      lo = mid;
    else
      hi = mid;
  }
  const double mu = 0.5 * (lo + hi);
  occ(mu);
  e_band = 0.0;
  ts = 0.0;
  for (int k = 0; k < nt; ++k) {
    const double w = wk ? wk[k / nstates] : 1.0;
    e_band += w * f[k] * eps[k];
    const double g = f[k] / 2.0;
    if (g > 1e-300 && g < 1.0 - 1e-16) ts += w * (g * std::log(g) + (1.0 - g) * std::log1p(-g));
  }
  ts *= -2.0;
  return mu;
}

static pufe_status scf_finish(pufe_ctx *ctx, double mu, double e_band, double ts, double kT,
                              double alpha, int pulay, const double *rho_I,
                              const double *V_eff_in, double *n, double *V_eff_out,
                              pufe_scf_info *info, cudaStream_t st);

pufe_status launch_scf_step(pufe_ctx *ctx, int nstates, const double *eps, const double *C,
                            int64_t ldc, double nelec, double kT, double alpha, int pulay, int prec,
                            const double *rho_I, const double *V_eff_in, double *n, double *V_eff_out,
                            double *f_out, pufe_scf_info *info, cudaStream_t st) {
  if (pufe_status e0 = scf_prepare(ctx)) return e0;
  ScfState *S = ctx->scf;
  std::vector<double> f;
  double e_band = 0.0, ts = 0.0;
  const double mu = occupations(1, nullptr, nstates, eps, nelec, kT, f, e_band, ts);
  if (f_out) std::copy(f.begin(), f.end(), f_out);
  PUFE_CUDA_TRY(cudaMemcpyAsync(S->f, f.data(), nstates * sizeof(double), cudaMemcpyHostToDevice, st));
  pufe_status e1 = (prec == PUFE_FP64)
                       ? launch_density_fp64(ctx, C, ldc, S->f, nstates, S->n_out, st)
                       : launch_density_tc(ctx, C, ldc, S->f, nstates, S->n_out, st);
  if (e1 != PUFE_OK) return e1;
  return scf_finish(ctx, mu, e_band, ts, kT, alpha, pulay, rho_I, V_eff_in, n, V_eff_out, info, st);
}

pufe_status launch_scf_step_bloch(pufe_ctx *ctx, int nk, const double *kpts, const double *wk,
                                  int nstates, const double *eps, const double *const *C_re,
                                  const double *const *C_im, int64_t ldc, double nelec, double kT,
                                  double alpha, int pulay, int prec, const double *rho_I,
                                  const double *V_eff_in, double *n, double *V_eff_out,
                                  double *f_out, pufe_scf_info *info, cudaStream_t st) {
  if (pufe_status e0 = scf_prepare(ctx)) return e0;
  ScfState *S = ctx->scf;
  if (!S->nk) PUFE_CUDA_TRY(cudaMalloc((void **)&S->nk, (size_t)ctx->nq * sizeof(double)));
  std::vector<double> f;
  double e_band = 0.0, ts = 0.0;
  const double mu = occupations(nk, wk, nstates, eps, nelec, kT, f, e_band, ts);
  if (f_out) std::copy(f.begin(), f.end(), f_out);
  // n_out = sum_k w_k sum_n f_nk |psi_nk|^2: each k's density with the
  // occupations w_k f_nk, added into n_out
  std::vector<double> fw(f.size());
  for (size_t i = 0; i < f.size(); ++i) fw[i] = wk[i / nstates] * f[i];
  PUFE_CUDA_TRY(cudaMemcpyAsync(S->f, fw.data(), fw.size() * sizeof(double), cudaMemcpyHostToDevice,
                                st));
  for (int i = 0; i < nk; ++i) {
    const PhaseTab ph = phase_table(ctx, kpts + 3 * i);
    double *out = i == 0 ? S->n_out : S->nk;
    const double *fk = S->f + (size_t)i * nstates;
    pufe_status e1 = (prec == PUFE_FP64)
                         ? launch_density_fp64_bloch(ctx, ph, C_re[i], C_im[i], ldc, fk, nstates,
                                                     out, st)
                         : launch_density_tc(ctx, C_re[i], ldc, fk, nstates, out, st, C_im[i], &ph);
    if (e1 != PUFE_OK) return e1;
    if (i > 0) {
      k_add<<<blocks(ctx->nq, 256), 256, 0, st>>>(ctx->nq, S->n_out, S->nk, S->n_out);
      PUFE_CUDA_TRY(cudaGetLastError());
    }
  }
  return scf_finish(ctx, mu, e_band, ts, kT, alpha, pulay, rho_I, V_eff_in, n, V_eff_out, info, st);
}

// the part of an SCF step after the output density S->n_out: V_C[n_out] and
// eps_xc(n_out), the energies, mixing into n and the new potential
static pufe_status scf_finish(pufe_ctx *ctx, double mu, double e_band, double ts, double kT,
                              double alpha, int pulay, const double *rho_I,
                              const double *V_eff_in, double *n, double *V_eff_out,
                              pufe_scf_info *info, cudaStream_t st) {
  ScfState *S = ctx->scf;
  const bool use_pulay = pulay > 1;
  InterpOut O{};
  O.n = S->n_out;
  O.w = ctx->d.w;
  O.V_in = V_eff_in;
  O.rho_I = rho_I;
  O.alpha = use_pulay ? 0.0 : alpha;
  O.n_in = n;
  O.sums = S->sums;
  if (pufe_status e2 = coulomb(ctx, rho_I, O, st)) return e2;
  // (before the second solve, which clears the sums)
  PUFE_CUDA_TRY(cudaMemcpyAsync(S->h_sums, S->sums, SCF_SUMS * SCF_SLOTS * sizeof(double),
                                cudaMemcpyDeviceToHost, st));
  if (use_pulay) {
    const int depth = std::min(pulay, PULAY_MAX);
    if (!S->hist_n) {
      PUFE_CUDA_TRY(cudaMalloc((void **)&S->hist_n, (size_t)PULAY_MAX * ctx->nq * sizeof(double)));
      PUFE_CUDA_TRY(cudaMalloc((void **)&S->hist_R, (size_t)PULAY_MAX * ctx->nq * sizeof(double)));
      PUFE_CUDA_TRY(cudaMalloc((void **)&S->dots, PULAY_MAX * sizeof(double)));
    }
    // drop the oldest entries beyond depth - 1, then add this one
    while ((int)S->slots.size() > depth - 1) S->slots.erase(S->slots.begin());
    int slot = 0;
    while (std::find(S->slots.begin(), S->slots.end(), slot) != S->slots.end()) ++slot;
    S->slots.push_back(slot);
    SlotList L;
    L.m = (int)S->slots.size();
    for (int i = 0; i < L.m; ++i) L.s[i] = S->slots[i];
    PUFE_CUDA_TRY(cudaMemsetAsync(S->dots, 0, PULAY_MAX * sizeof(double), st));
    k_pulay_store<<<blocks(ctx->nq, 256), 256, 0, st>>>(ctx->nq, ctx->d.w, n, S->n_out, slot, L,
                                                        S->hist_n, S->hist_R, S->dots);
    PUFE_CUDA_TRY(cudaGetLastError());
    double dots[PULAY_MAX];
    PUFE_CUDA_TRY(cudaMemcpyAsync(dots, S->dots, L.m * sizeof(double), cudaMemcpyDeviceToHost, st));
    PUFE_CUDA_TRY(cudaStreamSynchronize(st));
    for (int j = 0; j < L.m; ++j) S->gram[slot][L.s[j]] = S->gram[L.s[j]][slot] = dots[j];
    double A[8][8];
    for (int i = 0; i < L.m; ++i)
      for (int j = 0; j < L.m; ++j) A[i][j] = S->gram[L.s[i]][L.s[j]];
    if (!pulay_coefficients(L.m, A, L.c)) return fail(PUFE_EINVAL, "Pulay system is singular");
    k_pulay_mix<<<blocks(ctx->nq, 256), 256, 0, st>>>(ctx->nq, L, alpha, S->hist_n, S->hist_R, n);
    PUFE_CUDA_TRY(cudaGetLastError());
  }
  // the new effective potential of the mixed density
  if (pufe_status e3 = launch_effective_potential(ctx, n, rho_I, V_eff_out, nullptr, nullptr, st))
    return e3;
  PUFE_CUDA_TRY(cudaStreamSynchronize(st));
  double sums[SCF_SUMS];
  for (int k = 0; k < SCF_SUMS; ++k) {
    sums[k] = 0.0;
    for (int i = 0; i < SCF_SLOTS; ++i) sums[k] += S->h_sums[k * SCF_SLOTS + i];
  }
  if (info) {
    info->mu = mu;
    info->e_band = e_band;
    info->e_dc = -sums[0];
    info->e_es = -0.5 * sums[1];
    info->e_self = S->e_self;
    info->e_xc = sums[2];
    info->e_ts = -kT * ts;
    info->e_total = info->e_band + info->e_dc + info->e_es - info->e_self + info->e_xc + info->e_ts;
    info->residual = sums[3];
  }
  return PUFE_OK;
}

}  // namespace pufe
