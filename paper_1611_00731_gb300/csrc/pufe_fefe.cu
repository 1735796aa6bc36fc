// FE-FE block of H_V = int phi_i V phi_j by sum factorization (mixed path).
//
// On a tensor-product (sub)cell rule with points q = (qx, qy, qz), the 64
// tricubic functions are products L_a(x) L_b(y) L_c(z), so
//   M[(a,b,c),(a',b',c')] = sum_q w_q V_q L_a L_a' L_b L_b' L_c L_c'
// contracts one axis at a time: first z for every (qx, qy), then y, then x.
// The integrand is symmetric in each axis pair separately, so M has only
// 10 x 10 x 10 distinct values (unordered pairs per axis).  Cost per p^3 cell:
// 10 p^3 + 100 p^2 + 1000 p multiply-adds, against 2080 p^3 for the direct
// element contraction.  (Sec. 4 eq. disceig3d, local potential term; the rule
// is the element's shared rule of Sec. 5.2.)
//
// H starts at zero; each element adds the constant 64 x 64 kinetic block of
// the tricubic functions (the same on every element of the cubic mesh, exact
// for rules with >= 4 points per axis, precomputed in FP64) plus its block of
// M through the scatter map.  The enrichment strip kernel adds the rest.
#include <algorithm>

#include "pufe_internal.h"

namespace pufe {
namespace {

constexpr int SF_NT = 128;
constexpr int SF_PMAX = 16;

__device__ __forceinline__ int pidx(int a, int b) {  // unordered pair -> 0..9
  const int lo = a < b ? a : b, hi = a < b ? b : a;
  return lo * 4 - (lo * (lo - 1)) / 2 + (hi - lo);
}

__device__ __forceinline__ void lag3(float t, float L[4]) {
  const float a = t + 1.0f, b = t + (1.0f / 3.0f), c = t - (1.0f / 3.0f), d = t - 1.0f;
  L[0] = -0.5625f * b * c * d;
  L[1] = 1.6875f * a * c * d;
  L[2] = -1.6875f * a * b * d;
  L[3] = 0.5625f * a * b * c;
}

// BLOCH (Sec. 4, eqs. bloch, strong): entry (i, j) goes into H(k) and S(k)
// with the phase conj(exp(i k.R_i)) exp(i k.R_j) of the columns' lattice
// shifts; S holds the constant overlap of the Gamma point on entry and gets the
// difference that the phases make.
//
// What bounded it before: shared memory sized for 16 points per axis (39 KB, five
// 128-thread CTAs per SM), one output per loop turn (three instructions per
// multiply-add) and the widening of each entry on the FP64 pipe (two per clock and SM).
// Now a thread owns a line of each stage with five or ten outputs, shared memory
// follows the largest rule (15 KB at 10 points: 48 registers bind, 10 CTAs per SM) and
// entries are widened on the integer pipe; what is left is the 7 M atomics.
// 12^3 rocksalt (ncu) 59 -> 33 us; at a wavevector, where elements away from the upper
// faces skip phases that are 1, 64-atom cell 2.41 -> 1.26 ms.
template <bool BLOCH>
__global__ void __launch_bounds__(SF_NT) k_fefe_sumfac(
    const int64_t *__restrict__ qoff, const double *__restrict__ w, const double *__restrict__ V,
    const double *__restrict__ xi_all, const int32_t *__restrict__ partoff,
    const int32_t *__restrict__ part_p, const int32_t *__restrict__ part_q,
    const int64_t *__restrict__ doff, const int64_t *__restrict__ soff,
    const int32_t *__restrict__ smap, const double *__restrict__ Tfe, double *__restrict__ H,
    unsigned *err, const double *__restrict__ Sfe, const uint8_t *__restrict__ eshift,
    PhaseTab ph, int what, double *__restrict__ Hi, double *__restrict__ S,
    double *__restrict__ Si, int pm) {
  // dynamic shared memory, sized for the largest per-axis count pm: P[3][pm][16], the 10
  // pair products of each axis and point as two halves of five (pitch 8); Wq[pm^3];
  // G1[qx + p qy][cc]; G2[qx][bb][cc]; M[aa][bb][cc]
  extern __shared__ __align__(16) float sm_ff[];
  float *P = sm_ff, *G2 = P + 48 * pm, *M = G2 + 100 * pm, *G1 = M + 1000, *Wq = G1 + 10 * pm * pm;
  const int e = blockIdx.x, tid = threadIdx.x;
  float m10[10];   // this thread's (bb, cc) at every aa
#pragma unroll
  for (int a = 0; a < 10; ++a) m10[a] = 0.0f;
  // acc[u] += f v over the five products of one half at one point
  auto five = [](const float *f, float v, float *acc) {
    const float4 f4 = *reinterpret_cast<const float4 *>(f);
    acc[0] = fmaf(v, f4.x, acc[0]);
    acc[1] = fmaf(v, f4.y, acc[1]);
    acc[2] = fmaf(v, f4.z, acc[2]);
    acc[3] = fmaf(v, f4.w, acc[3]);
    acc[4] = fmaf(v, f[4], acc[4]);
  };
  for (int k = partoff[e]; V != nullptr && k < partoff[e + 1]; ++k) {
    const int p = part_p[k];
    if (p > pm) {
      if (tid == 0) atomicOr(err, DEVERR_SHAPE);
      return;
    }
    const int64_t qs = qoff[e] + part_q[k];
    const int p2 = p * p, p3 = p2 * p;
    __syncthreads();
    bool bad = false;
    for (int q = tid; q < p3; q += SF_NT) {
      const double v = V[qs + q];
      bad |= !isfinite(v);
      Wq[q] = f64_to_f32(w[qs + q] * v);
    }
    if (bad) atomicOr(err, DEVERR_NONFINITE);
    for (int o = tid; o < 3 * p; o += SF_NT) {
      const int d = o / p, t = o - d * p;
      const int stride = d == 0 ? 1 : (d == 1 ? p : p2);
      float L[4];
      lag3((float)xi_all[3 * (qs + (int64_t)t * stride) + d], L);
      float *f = P + (d * pm + t) * 16;
      int c = 0;
#pragma unroll
      for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = a; b < 4; ++b, ++c) f[c < 5 ? c : c + 3] = L[a] * L[b];
    }
    __syncthreads();
    for (int o = tid; o < 2 * p2; o += SF_NT) {   // contract z: (half of cc, qx + p qy)
      const int h = o >= p2, qxy = o - h * p2;
      const float *f = P + 2 * pm * 16 + 8 * h;
      float s[5] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
      for (int qz = 0; qz < p; ++qz) five(f + 16 * qz, Wq[qxy + p2 * qz], s);
#pragma unroll
      for (int u = 0; u < 5; ++u) G1[qxy * 10 + 5 * h + u] = s[u];
    }
    __syncthreads();
    for (int o = tid; o < 20 * p; o += SF_NT) {   // contract y: (half of bb, qx, cc)
      const int h = o >= 10 * p, r = o - h * 10 * p, qx = r / 10, cc = r - qx * 10;
      const float *f = P + pm * 16 + 8 * h;
      float s[5] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
      for (int qy = 0; qy < p; ++qy) five(f + 16 * qy, G1[qy * p * 10 + r], s);
#pragma unroll
      for (int u = 0; u < 5; ++u) G2[qx * 100 + (5 * h + u) * 10 + cc] = s[u];
    }
    __syncthreads();
    if (tid < 100) {   // contract x: (bb, cc)
      float s[10];
#pragma unroll
      for (int a = 0; a < 10; ++a) s[a] = 0.0f;
      for (int qx = 0; qx < p; ++qx) {
        const float g = G2[qx * 100 + tid];
        five(P + 16 * qx, g, s);
        five(P + 16 * qx + 8, g, s + 5);
      }
#pragma unroll
      for (int a = 0; a < 10; ++a) m10[a] += s[a];
    }
  }
  if (tid < 100) {
#pragma unroll
    for (int a = 0; a < 10; ++a) M[a * 100 + tid] = m10[a];
  }
  __syncthreads();
  // add the 64 x 64 block into H through the scatter map: consecutive lanes run along
  // j and hit neighbouring CSR columns; a thread keeps its j, so its M offsets are one
  // per node of each axis
  const int n = (int)(doff[e + 1] - doff[e]);
  const int32_t *m = smap + soff[e];
  const int j = tid & 63, ih = tid >> 6;
  // most elements touch no upper face of the cell: every phase is 1.  The others read
  // the phase of a pair of shift codes, and what it adds to S, from a table (P and G2
  // are done with): formed per entry its FP64 operations bound meshes of a few hundred
  // elements, many of them at a face (7^3 rocksalt 48 us when every entry of every element
  // had them, 57 us for the faces alone with the tests on top, 44 us from the table).
  const uint8_t *es = BLOCH ? eshift + doff[e] : nullptr;
  const bool phased = BLOCH && __syncthreads_or(tid < 64 ? es[tid] : 0) != 0;
  double *tab = reinterpret_cast<double *>(sm_ff);   // [re, im, re - 1][ci][cj]
  if (phased) {
    if (tid < 64) {
      const int ci = tid >> 3, cj = tid & 7;
      const double pr = ph.re[ci] * ph.re[cj] + ph.im[ci] * ph.im[cj];
      tab[tid] = pr;
      tab[64 + tid] = ph.re[ci] * ph.im[cj] - ph.im[ci] * ph.re[cj];
      tab[128 + tid] = pr - 1.0;
    }
    __syncthreads();
  }
  const int cj = phased ? es[j] : 0;
  int pa[2], pb[4];
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    if (u < 2) pa[u] = pidx(ih + 2 * u, j & 3) * 100;
    pb[u] = pidx(u, (j >> 2) & 3) * 10;
  }
#pragma unroll 1
  for (int c = 0; c < 4; ++c) {
    const int pc = pidx(c, j >> 4);
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int i = 16 * c + 2 * u + ih, o = i * 64 + j;
      const double v = f32_to_f64(M[pa[u & 1] + pb[u >> 1] + pc]);
      const int slot = m[i * n + j];
      if (!BLOCH) {
        atomicAdd(H + slot, __ldg(Tfe + o) + v);
      } else {
        // S starts as the summed constants, so only pairs whose phase is not 1 (the
        // elements on the cell's upper faces) correct it; a zero imaginary part is
        // not added (unless the value is not finite)
        const int ci = phased ? es[i] : 0, cc = 8 * ci + cj;
        const double pr = ci != cj ? tab[cc] : 1.0, pi = ci != cj ? tab[64 + cc] : 0.0;
        if (what & PUFE_WANT_H) {
          const double hv = __ldg(Tfe + o) + v;
          atomicAdd(H + slot, ci != cj ? hv * pr : hv);
          if (pi != 0.0 || !isfinite(hv)) atomicAdd(Hi + slot, hv * pi);
        }
        if ((what & PUFE_WANT_S) && ci != cj) {
          const double sv = __ldg(Sfe + o);
          atomicAdd(S + slot, sv * tab[128 + cc]);
          atomicAdd(Si + slot, sv * pi);
        }
      }
    }
  }
}

// FE-FE part of the adjoint of V -> H on a tensor-product (sub)cell:
//   f(q) = sum_{(abc),(a'b'c')} L_a L_a' L_b L_b' L_c L_c' Hbar[(abc),(a'b'c')]
// (Hbar restricted to the element's 64 FE columns, general, not symmetric),
// contracted axis by axis: 4096 p + 256 p^2 + 16 p^3 multiply-adds per cell,
// then Vbar_q = w_q f(q) is stored (the strip kernel adds the enrichment part).
//
// What bounded a form with one output per loop turn was its instructions: two products
// and three shared-memory reads per multiply-add, beside the gather.  Here a thread
// owns a row of each stage and runs over the points: its 16 inputs stay in registers
// (for z, the 16 gathered entries themselves, through all (sub)cells), and the 16
// factors L_i L_i' of a point, formed once per cell, are four 16-byte reads that all
// lanes share.  The 16 terms keep their order.  12^3 rocksalt (ncu) 40 -> 30 us.
constexpr int AF_NT = 256;     // one thread per ((a, b), (a', b')) row
constexpr int AF_ROW = 20;     // pitches of G1 (of a row of 16, and of a qz) that keep the
constexpr int AF_QZ = 336;     // y stage's reads on different banks

__device__ __forceinline__ float af_sum(const float (&v)[16], const float4 *l) {
  float s = 0.0f;
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    const float4 f = l[c];
    s = fmaf(f.x, v[4 * c], s);
    s = fmaf(f.y, v[4 * c + 1], s);
    s = fmaf(f.z, v[4 * c + 2], s);
    s = fmaf(f.w, v[4 * c + 3], s);
  }
  return s;
}

template <bool BLOCH>
__global__ void __launch_bounds__(AF_NT, 4) k_adjoint_fefe(
    const int32_t *__restrict__ order, const int64_t *__restrict__ qoff,
    const double *__restrict__ w, const double *__restrict__ xi_all,
    const int32_t *__restrict__ partoff, const int32_t *__restrict__ part_p,
    const int32_t *__restrict__ part_q, const int64_t *__restrict__ doff,
    const int64_t *__restrict__ soff, const int32_t *__restrict__ smap,
    const double *__restrict__ Hbar, int pm, double *__restrict__ Vbar, unsigned *err,
    BlochCot bc) {
  // dynamic shared memory, sized for the largest per-axis count pm:
  // LL[3][pm][16] = L_i L_i', G1[qz][(a,b)][(a',b')], G2[(a,a')][qy + p qz]
  extern __shared__ __align__(16) float sm_adj[];
  float4 *LL = reinterpret_cast<float4 *>(sm_adj);
  float *G1 = sm_adj + 48 * pm, *G2 = G1 + AF_QZ * pm;
  const int e = order[blockIdx.x], tid = threadIdx.x;
  const int n = (int)(doff[e + 1] - doff[e]);
  const int32_t *m = smap + soff[e];
  const int ab = tid >> 4, apbp = tid & 15;
  // this row's entries, (c, c') = 0..15: eight independent (map, value) load chains
  // in flight
  float hz[16];
#pragma unroll
  for (int g = 0; g < 2; ++g) {
    int s1[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int c = 2 * g + (u >> 2), cp = u & 3;
      s1[u] = m[(ab + 16 * c) * n + apbp + 16 * cp];
    }
    double h[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) h[u] = Hbar[s1[u]];
    if (BLOCH) {   // at a wavevector: the phased real part (columns' shift codes)
      double hi[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) hi[u] = bc.Hi[s1[u]];
      const uint8_t *esh = bc.eshift + doff[e];
#pragma unroll
      for (int u = 0; u < 8; ++u)
        h[u] = cot_entry(h[u], hi[u], esh[ab + 16 * (2 * g + (u >> 2))],
                         esh[apbp + 16 * (u & 3)], bc.ph);
    }
#pragma unroll
    for (int u = 0; u < 8; ++u) hz[8 * g + u] = f64_to_f32(h[u]);
  }
  for (int k = partoff[e]; k < partoff[e + 1]; ++k) {
    const int p = part_p[k];
    if (p > pm) {
      if (tid == 0) atomicOr(err, DEVERR_SHAPE);
      return;
    }
    const int64_t qs = qoff[e] + part_q[k];
    const int p2 = p * p;
    __syncthreads();
    for (int o = tid; o < 3 * p; o += AF_NT) {
      const int d = o / p, t = o - d * p;
      const int stride = d == 0 ? 1 : (d == 1 ? p : p2);
      float L[4];
      lag3((float)xi_all[3 * (qs + (int64_t)t * stride) + d], L);
#pragma unroll
      for (int a = 0; a < 4; ++a)
        LL[(d * pm + t) * 4 + a] = make_float4(L[a] * L[0], L[a] * L[1], L[a] * L[2], L[a] * L[3]);
    }
    __syncthreads();
    // contract (c, c'): a thread's row at every qz
    for (int qz = 0; qz < p; ++qz)
      G1[qz * AF_QZ + ab * AF_ROW + apbp] = af_sum(hz, LL + (2 * pm + qz) * 4);
    __syncthreads();
    // contract (b, b'): rows (a, a', qz), their qy spread over ny threads
    const int ny = max(1, AF_NT / (16 * p));
    if (tid < 16 * p * ny) {
      const int aa = tid & 15, sq = tid >> 4, sp = sq / p, qz = sq - sp * p;
      const float *g = G1 + qz * AF_QZ + (aa >> 2) * AF_ROW + (aa & 3);
      float v[16];
#pragma unroll
      for (int b = 0; b < 4; ++b)
#pragma unroll
        for (int bp = 0; bp < 4; ++bp) v[4 * b + bp] = g[4 * b * AF_ROW + 4 * bp];
      for (int qy = sp; qy < p; qy += ny)
        G2[aa * p2 + qy + p * qz] = af_sum(v, LL + (pm + qy) * 4);
    }
    __syncthreads();
    // contract (a, a'): lines (qy, qz), their qx spread over nx threads; w_q f(q)
    const int nx = min(p, AF_NT / p2);
    if (tid < p2 * nx) {
      const int sp = tid / p2, r = tid - sp * p2;
      float v[16];
#pragma unroll
      for (int a = 0; a < 16; ++a) v[a] = G2[a * p2 + r];
      for (int qx = sp; qx < p; qx += nx) {
        const int64_t q = qs + qx + p * r;
        Vbar[q] = w[q] * f32_to_f64(af_sum(v, LL + qx * 4));
      }
    }
  }
}

// shared bytes of k_fefe_sumfac (40 KB at the 16 points per axis that the callers allow)
size_t fefe_bytes(int pm) {
  return (size_t)(148 * pm + 1000 + 10 * pm * pm + pm * pm * pm) * sizeof(float);
}

}  // namespace

// Every element adds its kinetic FE-FE block and the FE-FE block of H_V into
// H (which the caller has zeroed); V == NULL means V = 0.
pufe_status launch_fefe(pufe_ctx *ctx, const double *V, double *H, cudaStream_t st) {
  auto &D = ctx->d;
  if (ctx->max_part_p > SF_PMAX) return fail(PUFE_EINVAL, "rule with more than 16 points per axis");
  if (!D.Tfe) return fail(PUFE_ESTATE, "no exact FE-FE blocks (a rule has < 4 points per axis)");
  const int pm = std::max(1, ctx->max_part_p);
  k_fefe_sumfac<false><<<(unsigned)ctx->nelem, SF_NT, fefe_bytes(pm), st>>>(
      D.qoff, D.w, V, D.xi, D.partoff, D.part_p, D.part_q, D.doff, D.soff, D.smap, D.Tfe, H, D.err,
      nullptr, nullptr, PhaseTab{}, PUFE_WANT_H, nullptr, nullptr, nullptr, pm);
  PUFE_CUDA_TRY(cudaGetLastError());
  return PUFE_OK;
}

// Bloch form: the FE-FE blocks of H(k) (if wanted; V == NULL means V = 0) and
// S(k) (if wanted) with the column phases, into zeroed H, Hi and Si and S = S0
pufe_status launch_fefe_bloch(pufe_ctx *ctx, const PhaseTab &ph, const double *V, int what,
                              double *H, double *Hi, double *S, double *Si, cudaStream_t st) {
  auto &D = ctx->d;
  if (ctx->max_part_p > SF_PMAX) return fail(PUFE_EINVAL, "rule with more than 16 points per axis");
  if (!D.Tfe || !D.Sfe) return fail(PUFE_ESTATE, "no exact FE-FE blocks (a rule has < 4 points per axis)");
  const int pm = std::max(1, ctx->max_part_p);
  k_fefe_sumfac<true><<<(unsigned)ctx->nelem, SF_NT, fefe_bytes(pm), st>>>(
      D.qoff, D.w, (what & PUFE_WANT_H) ? V : nullptr, D.xi, D.partoff, D.part_p, D.part_q,
      D.doff, D.soff, D.smap, D.Tfe, H, D.err, D.Sfe, D.eshift, ph, what, Hi, S, Si, pm);
  PUFE_CUDA_TRY(cudaGetLastError());
  return PUFE_OK;
}

}  // namespace pufe

namespace pufe {
// Vbar = w_q (FE part of b^T Hbar b) for elements order[first .. first+count)
pufe_status launch_adjoint_fefe(pufe_ctx *ctx, const double *Hbar, double *Vbar, int first,
                                int count, cudaStream_t st, const BlochCot &bc) {
  auto &D = ctx->d;
  if (ctx->max_part_p > SF_PMAX) return fail(PUFE_EINVAL, "rule with more than 16 points per axis");
  if (count <= 0) return PUFE_OK;
  const int pm = std::max(1, ctx->max_part_p);
  const size_t sm = (size_t)((48 + AF_QZ) * pm + 16 * pm * pm) * sizeof(float);
  auto kern = bc.Hi ? k_adjoint_fefe<true> : k_adjoint_fefe<false>;
  PUFE_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
  kern<<<(unsigned)count, AF_NT, sm, st>>>(D.order + first, D.qoff, D.w, D.xi, D.partoff, D.part_p,
                                           D.part_q, D.doff, D.soff, D.smap, Hbar, pm, Vbar, D.err,
                                           bc);
  PUFE_CUDA_TRY(cudaGetLastError());
  return PUFE_OK;
}
}  // namespace pufe
