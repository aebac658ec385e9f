// SVD of the small square factor R through bidiagonalisation.
//
// The truncation at a bond needs every singular value of the triangular
// factor R (the discarded tail) and the left singular vectors of the kept
// ones (App. A, the QR-then-SVD structure of Alg. 4).  Instead of Jacobi
// rotations (O(n^3) flops per sweep, a dozen sweeps), R is reduced once:
//
//  1. Householder bidiagonalisation R = Q B P^H (Golub & Kahan 1965), B real
//     upper bidiagonal, with the reflector conventions of LAPACK's zgebrd.
//     One cooperative launch; CTA g keeps the rows r = g (mod G) of R in
//     shared memory and the CTAs meet once per column (see gebrd_kernel).
//  2. Singular values of B: eigenvalues sigma^2 of B B^T by counting with the
//     differential qd transform of B B^T - x^2 I (Fernando & Parlett 1994),
//     one CTA of 32 W threads per value and 32 W points per round of
//     multisection.  Counts are taken in double-float arithmetic (hi + lo FP32
//     pair, ~2^-45 relative): a count is exact for a bidiagonal whose entries
//     are perturbed by a few units of the working precision, and the singular
//     values of a bidiagonal move by a relative amount of the same order under
//     such perturbations (Demmel & Kahan 1990), so every value above 2^-50 of
//     the largest entry is found to a relative accuracy of ~1e-13; the ones
//     below (FP64 rounding of the bidiagonalisation) to 2^-8 by Sturm counts
//     of the Golub-Kahan tridiagonal T_GK (order 2n, zero diagonal,
//     off-diagonals d_1, e_1, d_2, ..., d_n), whose pivots stay in FP32 range.
//  3. Left singular vectors of B for the kept values: eigenvectors of B B^T
//     by twisted factorisation (Dhillon & Parlett 2004): the stationary and
//     the progressive differential qd transforms of B B^T - lambda I meet at
//     the index where the residual is smallest, one Rayleigh-quotient
//     correction of lambda, then again, FP64.  Every vector is computed by
//     itself, all of them at once; their orthogonality error is the rounding
//     over the relative gap of the values and is removed by two Newton-Schulz
//     steps of the polar factor.  Only if values agree to ~1e-11 (repeated
//     singular values) are all vectors computed again one cluster after
//     another, by inverse iteration on T_GK with modified Gram-Schmidt inside
//     clusters (as in LAPACK's dstein).  Kept values at the rounding-noise
//     level of R get an orthonormal completion (their vectors are not
//     determined by R).
//  4. U = Q [u_1 .. u_rho] by applying the left reflectors.
#include <algorithm>
#include <cfloat>

#include "kernels.h"

namespace hk {

constexpr int kBdThreads = 256;

// Values other CTAs published are read kBdBatch at a time per lane: the
// loads of a batch are independent and in flight together, one L2 round
// trip per batch on a path every column waits for; sums keep their order.
constexpr int kBdBatch = 8;
DV double sum_published(const double* p, int G) {  // lane-strided partial sum
  const int lane = threadIdx.x & 31;
  double s = 0.0;
  for (int g0 = lane; g0 < G; g0 += 32 * kBdBatch) {
    double v[kBdBatch];
#pragma unroll
    for (int u = 0; u < kBdBatch; ++u) v[u] = (g0 + 32 * u < G) ? __ldcg(p + g0 + 32 * u) : 0.0;
#pragma unroll
    for (int u = 0; u < kBdBatch; ++u)
      if (g0 + 32 * u < G) s += v[u];
  }
  return s;
}
DV cplx sum_published(const cplx* p, size_t stride, int G) {
  const int lane = threadIdx.x & 31;
  cplx s = mk(0, 0);
  for (int g0 = lane; g0 < G; g0 += 32 * kBdBatch) {
    cplx v[kBdBatch];
#pragma unroll
    for (int u = 0; u < kBdBatch; ++u) v[u] = (g0 + 32 * u < G) ? __ldcg(p + (size_t)(g0 + 32 * u) * stride) : mk(0, 0);
#pragma unroll
    for (int u = 0; u < kBdBatch; ++u)
      if (g0 + 32 * u < G) s = cadd(s, v[u]);
  }
  return s;
}
// Sum over the block delivered to lanes 0 to 7 of warp 0 only (the other warps'
// FP64 work in a block-wide reduction costs more, on this GPU's narrow FP64
// pipe, than the column's arithmetic).  Warps whose `has` is false contribute
// zero without reducing.  Its __syncthreads also publishes the block's
// shared-memory writes made before it; the next use of red has to lie behind
// another one.
DV double sum_to_warp0(double v, bool has, double* red) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  constexpr int nw = kBdThreads / 32;
  if (has) v = warp_sum(v);
  if (lane == 0) red[w] = has ? v : 0.0;
  __syncthreads();
  double s = 0.0;
  if (w == 0) {
    s = (lane < nw) ? red[lane] : 0.0;
    for (int o = nw / 2; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  }
  return s;
}

// ---- 1. bidiagonalisation -------------------------------------------------------
// Column i, with H = I - tau v v^H the left reflector (v_i = 1,
// v_r = A[r,i] * scale for r > i) and w_c = sum_r conj(v_r) A[r,c]:
//   w_c = A[i,c] + conj(scale) * sum_{r>i} conj(A[r,i]) A[r,c].
// Each CTA writes its partial sums over its own rows (and the owner of row
// i publishes that row); after a grid barrier, CTA g reduces the columns
// c = i+1+g (mod G) and publishes conj(tau) w_c and the updated row i,
// A[i,c] - conj(tau) w_c; after a second barrier every CTA forms the right
// reflector G = I - taup u u^H of that row itself and applies both
// reflectors to its own rows.  (Reducing every column in every CTA would
// save the second barrier but costs G times the FP64 additions, which on
// this GPU's narrow FP64 pipe outweigh the barrier.)  The exchange buffers
// alternate between two halves by column parity: a CTA writing column
// i+2's data has passed both barriers of column i+1, so every reader of
// column i's half is done.
// FAST: reflector scalars from the reciprocal root and reciprocal of
// common.cuh, about 800 cycles less on each of a column's two scalar chains.
// Without it the IEEE forms (bd_serial_kernel says where the factors are kept
// to the last bit).
template <bool FAST>
__global__ void __launch_bounds__(kBdThreads, 1)
gebrd_kernel(cplx* A, int lda, int n, int nloc, double* dg, double* eg, cplx* tauq, cplx* taup,
             CoopWs ws, cplx* rows_global) {
  extern __shared__ __align__(16) unsigned char bd_smem[];
  // own rows (nloc x n, row-major) in shared memory, or, for a factor too
  // large for it, in this CTA's slice of a global workspace (L2-resident)
  cplx* rows = rows_global ? rows_global + (size_t)blockIdx.x * nloc * n : reinterpret_cast<cplx*>(bd_smem);
  cplx* fv = rows_global ? reinterpret_cast<cplx*>(bd_smem) : rows + (size_t)nloc * n;  // conj(tau) w_c
  cplx* nrow = fv + n;                           // updated row i
  cplx* uv = nrow + n;                           // right reflector u
  cplx* vloc = uv + n;                           // v_r of own rows (nloc)
  __shared__ double dred[32];
  __shared__ cplx bc[4];
  __shared__ cplx bcr[4];
  const int G = gridDim.x, g = blockIdx.x, tid = threadIdx.x;
  const int lane = tid & 31, wid = tid >> 5, nw = blockDim.x >> 5;
  const size_t pstride = (size_t)n + 1;
  GridSync gs{ws.bar, 0u};
  auto grow = [&](int lr) { return g + lr * G; };
  auto R = [&](int lr, int c) -> cplx& { return rows[(size_t)lr * n + c]; };
  const int nact = min(nloc, (n - g + G - 1) / G);  // local rows that exist

  for (int lr = 0; lr < nloc; ++lr) {
    const int r = grow(lr);
    for (int c = tid; c < n; c += blockDim.x) R(lr, c) = (r < n) ? A[r + (size_t)lda * c] : mk(0, 0);
  }
  __syncthreads();

  for (int i = 0; i < n; ++i) {
    const int buf = i & 1;
    cplx* pc = ws.pc + (size_t)buf * G * pstride;
    double* pr = ws.pr + buf * G;
    cplx* rowb = ws.wfin + (size_t)buf * 3 * n;  // row i as published by its owner
    cplx* fvg = rowb + n;                        // conj(tau) w_c
    cplx* nrg = fvg + n;                         // updated row i
    const int C = n - i - 1;
    // first own local row strictly below i (rows of this CTA: g + lr G)
    const int lr0 = (i + 1 > g) ? (i + 1 - g + G - 1) / G : 0;
    const bool owner = (i % G == g);
    // (a) partial sums over own rows r > i.  Up to eight rows (three at full
    // grid size) are summed by one thread, in the order of a warp's exchange
    // (the same bits): a block-wide sum held every column up by two exchanges
    // and two barriers, 0.2 of 6.4 us.
    if (nact - lr0 <= 8) {
      if (tid == kBdThreads - 1) {
        double v[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) v[q] = lr0 + q < nact ? cabs2(R(lr0 + q, i)) : 0.0;
#pragma unroll
        for (int o = 4; o > 0; o >>= 1)
#pragma unroll
          for (int q = 0; q < o; ++q) v[q] += v[q + o];
        pr[g] = v[0];
      }
    } else {
      double sq = 0.0;
      for (int lr = lr0 + tid; lr < nact; lr += blockDim.x) sq += cabs2(R(lr, i));
      sq = sum_to_warp0(sq, lr0 + 32 * wid < nact, dred);
      if (tid == 0) pr[g] = sq;
    }
    for (int c = i + 1 + tid; c < n; c += blockDim.x) {
      cplx acc = mk(0, 0);
      for (int lr = lr0; lr < nact; ++lr) acc = cfmac(R(lr, i), R(lr, c), acc);
      pc[(size_t)g * pstride + c] = acc;
    }
    if (owner)
      for (int c = i + tid; c < n; c += blockDim.x) rowb[c] = R(i / G, c);
    if (grid_sync(gs)) return;
    // (b1) left reflector of column i (every CTA, warp 0) while the other
    // warps sum this CTA's columns; a second round only where a CTA has more
    // columns than warps
    cplx acc = mk(0, 0), a_ic = mk(0, 0);
    int cc = g + (wid - 1) * G;
    if (wid == 0) {
      const cplx al = __ldcg(rowb + i);
      const double s2 = warp_sum(sum_published(pr, G));
      if constexpr (FAST) {
        house_fast(al, s2, bc);
      } else {
        cplx tq, sc;
        double beta;
        house_warp(al, s2, &tq, &sc, &beta);
        if (lane == 0) {
          bc[0] = tq;
          bc[1] = sc;
          bc[2] = mk(beta, 0.0);
        }
      }
    } else if (cc < C) {
      a_ic = __ldcg(rowb + i + 1 + cc);
      acc = warp_sum(sum_published(pc + i + 1 + cc, pstride, G));
    }
    __syncthreads();
    const cplx tq = bc[0], scq = bc[1];
    const cplx ctq = cconj(tq), cscq = cconj(scq);
    if (wid > 0)
      while (cc < C) {
        const int c = i + 1 + cc;
        if (lane == 0) {
          // (the compiler may fuse a product's rounding into the sum around it)
          const cplx f = FAST ? cmul(ctq, cadd(a_ic, cmul(cscq, acc)))
                              : cmul_rounded(ctq, cadd(a_ic, cmul_rounded(cscq, acc)));
          fvg[c] = f;
          nrg[c] = csub(a_ic, f);
        }
        cc += (nw - 1) * G;
        if (cc < C) {
          a_ic = __ldcg(rowb + i + 1 + cc);
          acc = warp_sum(sum_published(pc + i + 1 + cc, pstride, G));
        }
      }
    if (grid_sync(gs)) return;
    // (b2) left update of own rows r > i: A[r,c] -= v_r conj(tau) w_c;
    // column i keeps v_r
    for (int lr = lr0 + tid; lr < nact; lr += blockDim.x) vloc[lr] = cmul(R(lr, i), scq);
    double sqp = 0.0;
    for (int c = i + 1 + tid; c < n; c += blockDim.x) {
      fv[c] = __ldcg(fvg + c);
      const cplx nr = __ldcg(nrg + c);
      nrow[c] = nr;
      if (c >= i + 2) sqp += cabs2(nr);
    }
    sqp = sum_to_warp0(sqp, i + 1 + 32 * wid < n, dred);  // its barrier also publishes fv / nrow / vloc
    if (owner && tid == 0) {
      R(i / G, i) = bc[2];
      dg[i] = bc[2].x;
      tauq[i] = tq;
    }
    // warp 0 forms the right reflector of the updated row i (every CTA
    // does; it zeroes the row beyond i+1) while warps 1.. apply the left
    // reflector to the own rows: A[r,c] -= v_r conj(tau) w_c, column i
    // keeps v_r
    if (wid == 0) {
      if (FAST && i + 1 < n) {
        house_fast(cconj(nrow[i + 1]), sqp, bcr);
      } else if (i + 1 < n) {
        cplx tp, sp;
        double beta;
        house_warp(cconj(nrow[i + 1]), sqp, &tp, &sp, &beta);
        if (lane == 0) {
          bcr[0] = tp;
          bcr[1] = sp;
          bcr[2] = mk(beta, 0.0);
        }
      }
    } else {
      const int t1 = tid - 32, nt1 = blockDim.x - 32;
      for (int c = i + 1 + t1; c < n; c += nt1) {
        const cplx f = fv[c];
        const cplx nf = mk(-f.x, -f.y);
        for (int lr = lr0; lr < nact; ++lr) R(lr, c) = cfma(vloc[lr], nf, R(lr, c));
      }
      for (int lr = lr0 + t1; lr < nact; lr += nt1) R(lr, i) = vloc[lr];
    }
    if (i + 1 >= n) break;
    __syncthreads();
    const cplx tp = bcr[0], scp = bcr[1];
    for (int c = i + 1 + tid; c < n; c += blockDim.x) {
      const cplx u = (c == i + 1) ? mk(1, 0) : cmul(cconj(nrow[c]), scp);
      uv[c] = u;
      if (owner) R(i / G, c) = (c == i + 1) ? bcr[2] : cconj(u);
    }
    if (owner && tid == 0) {
      eg[i] = bcr[2].x;
      taup[i] = tp;
    }
    __syncthreads();
    // right update of own rows r > i: A[r,:] -= taup (A[r,:] . u) u^H
    for (int lr = lr0 + wid; lr < nact; lr += nw) {
      cplx dot = mk(0, 0);
      if constexpr (FAST) {
        // a warp's FP64 instructions follow one another at the pace of a
        // dependent chain: one sum (four cost six more additions)
#pragma unroll 4
        for (int c = i + 1 + lane; c < n; c += 32) dot = cfma(R(lr, c), uv[c], dot);
        dot = warp_sum(dot);
      } else {
        cplx d0 = mk(0, 0), d1 = mk(0, 0), d2 = mk(0, 0), d3 = mk(0, 0);
        int c = i + 1 + lane;
        for (; c + 96 < n; c += 128) {
          d0 = cfma(R(lr, c), uv[c], d0);
          d1 = cfma(R(lr, c + 32), uv[c + 32], d1);
          d2 = cfma(R(lr, c + 64), uv[c + 64], d2);
          d3 = cfma(R(lr, c + 96), uv[c + 96], d3);
        }
        for (; c < n; c += 32) d0 = cfma(R(lr, c), uv[c], d0);
        dot = warp_sum(cadd(cadd(d0, d1), cadd(d2, d3)));
      }
      const cplx f = cmul(tp, dot);
      const cplx nf = mk(-f.x, -f.y);
      for (int c = i + 1 + lane; c < n; c += 32) R(lr, c) = cfma(nf, cconj(uv[c]), R(lr, c));
    }
    __syncthreads();
  }
  __syncthreads();
  for (int lr = 0; lr < nact; ++lr) {
    const int r = grow(lr);
    for (int c = tid; c < n; c += blockDim.x) A[r + (size_t)lda * c] = R(lr, c);
  }
}

// Grid of the bidiagonalisation: rows resident in shared memory when they
// fit (*global_rows = false), else all SMs with the rows in a global
// workspace of gebrd_rows_elems(n) elements (when allowed).
int gebrd_grid(int n, int sms, int* nloc_out, size_t* smem_out, bool allow_global, bool* global_rows) {
  const DevInfo& di = dev_info();
  int G = std::max(1, std::min(sms, (n + 2) / 3));
  *global_rows = false;
  for (;;) {
    const int nloc = (n + G - 1) / G;
    const size_t smem = ((size_t)nloc * n + 3 * (size_t)n + nloc) * sizeof(cplx);
    if (smem + 8192 <= (size_t)di.max_smem_optin) {
      *nloc_out = nloc;
      *smem_out = smem;
      return G;
    }
    if (G >= sms) break;
    G = std::min(sms, G + 8);
  }
  const int nloc = (n + G - 1) / G;
  const size_t smem = (3 * (size_t)n + nloc) * sizeof(cplx);
  if (!allow_global || smem + 8192 > (size_t)di.max_smem_optin) return 0;
  *global_rows = true;
  *nloc_out = nloc;
  *smem_out = smem;
  return G;
}

size_t gebrd_rows_elems(int n, int sms) {
  const int G = std::max(1, std::min(sms, (n + 2) / 3));
  return (size_t)(n + G) * (size_t)n;
}

size_t bd_vectors_smem(int n);

bool gebrd_fits(int n, const CoopWs& ws, bool have_rows_ws) {
  int nloc;
  size_t smem;
  bool glob;
  return n >= 1 && gebrd_grid(n, coop_sms(ws), &nloc, &smem, have_rows_ws, &glob) > 0 &&
         bd_vectors_smem(n) <= (size_t)dev_info().max_smem_optin;
}

cudaError_t gebrd(cplx* A, int lda, int n, double* d, double* e, cplx* tauq, cplx* taup,
                  const CoopWs& ws, cudaStream_t s, cplx* rows_ws, int kept) {
  if (n <= 0) return cudaSuccess;
  int nloc;
  size_t smem;
  bool glob = false;
  const int G = gebrd_grid(n, coop_sms(ws), &nloc, &smem, rows_ws != nullptr, &glob);
  if (G <= 0) return cudaErrorInvalidValue;
  cplx* rows_global = glob ? rows_ws : nullptr;
  if ((size_t)2 * G * (n + 1) > ws.pc_elems || (size_t)6 * n > ws.wfin_elems || 2 * G > 1024)
    return cudaErrorInvalidValue;
  void* fn = kept ? (void*)gebrd_kernel<false> : (void*)gebrd_kernel<true>;
  cudaError_t err = allow_smem(fn, smem);
  if (err != cudaSuccess) return err;
  err = cudaMemsetAsync(&ws.bar->count, 0, sizeof(unsigned int), s);
  if (err != cudaSuccess) return err;
  CoopWs w = ws;
  void* args[] = {&A, &lda, &n, &nloc, &d, &e, &tauq, &taup, &w, &rows_global};
  return cudaLaunchCooperativeKernel(fn, dim3(G), dim3(kBdThreads), args, smem, s);
}

// ---- 2. singular values ------------------------------------------------------------
// Double-float reals: value = h + l, |l| <= ulp(h)/2.
struct dfr {
  float h, l;
};
DV dfr df_quick(float a, float b) {  // |a| >= |b|
  const float s = a + b;
  return dfr{s, b - (s - a)};
}
DV dfr df_add(dfr a, dfr b) {
  const float s = a.h + b.h;
  const float bb = s - a.h;
  const float e = (a.h - (s - bb)) + (b.h - bb) + a.l + b.l;
  return df_quick(s, e);
}
DV dfr df_div(dfr a, dfr b) {
  // long division: q1 = a/b to FP32, exact remainder a - q1 b, q2 = rem/b
  const float r = __frcp_rn(b.h);
  const float q1 = a.h * r;
  const float p = q1 * b.h;
  const float pe = fmaf(q1, b.h, -p);
  const float rem = (((a.h - p) - pe) + a.l) - q1 * b.l;
  return df_quick(q1, rem * r);
}
DV dfr df_of(double x) {
  const float h = (float)x;
  return dfr{h, (float)(x - (double)h)};
}

// Prepare the scaled squares a2[2i] = (d_i / amax)^2, a2[2i+1] = (e_i / amax)^2
// (the squared off-diagonals of T_GK in order) as double-float; info[0] = amax,
// info[1] = Gershgorin bound of T_GK / amax (2n entries, the last one zero).
__global__ void bd_prep_kernel(const double* __restrict__ d, const double* __restrict__ e, int n,
                               float2* __restrict__ a2, double* __restrict__ info) {
  __shared__ double red[32];
  const int N = 2 * n;
  auto off = [&](int k) { return (k & 1) ? e[k >> 1] : d[k >> 1]; };
  const int nw = blockDim.x >> 5;
  double m = 0.0;
  for (int k = threadIdx.x; k < N - 1; k += blockDim.x) m = fmax(m, fabs(off(k)));
  for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
  __syncthreads();
  double amax = 0.0;
  for (int w = 0; w < nw; ++w) amax = fmax(amax, red[w]);
  __syncthreads();
  const double inv = amax > 0.0 ? 1.0 / amax : 0.0;
  double bnd = 0.0;
  for (int k = threadIdx.x; k < N - 1; k += blockDim.x) {
    const double a = fabs(off(k)) * inv;
    const double a_sq = a * a;
    float2 v = make_float2(0.f, 0.f);
    if (a_sq >= 1e-36) {
      v.x = (float)a_sq;
      v.y = (float)(a_sq - (double)v.x);
    }
    a2[k] = v;
    // row k+1 of T_GK holds a_k and a_{k+1}
    const double nb = (k + 1 < N - 1) ? fabs(off(k + 1)) * inv : 0.0;
    bnd = fmax(bnd, a + nb);
  }
  for (int o = 16; o > 0; o >>= 1) bnd = fmax(bnd, __shfl_xor_sync(0xffffffffu, bnd, o));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = bnd;
  __syncthreads();
  if (threadIdx.x == 0) {
    double b = 0.0;
    for (int w = 0; w < nw; ++w) b = fmax(b, red[w]);
    info[0] = amax;
    info[1] = b * (1.0 + 1e-6) + 1e-30;
    info[2] = 0.0;  // set when the vectors of nearly equal values need the clustered path
    a2[N - 1] = make_float2(0.f, 0.f);
  }
}

// Number of eigenvalues of the scaled T_GK below x: negative pivots of the
// LDL^T factorisation of T_GK - x I (pivots clamped away from zero).
__device__ __forceinline__ int sturm_count_df(const float2* __restrict__ a2, int N, double x) {
  const float pivmin = 1e-30f;
  const dfr xd = df_of(x);
  dfr q{-xd.h, -xd.l};
  if (fabsf(q.h) < pivmin) q = dfr{-pivmin, 0.f};
  int cnt = (q.h < 0.f);
  for (int k = 1; k < N; ++k) {
    const float2 a = __ldg(a2 + k - 1);
    const dfr t = df_div(dfr{a.x, a.y}, q);
    const dfr s = df_add(xd, t);
    q = dfr{-s.h, -s.l};
    if (fabsf(q.h) < pivmin) q = dfr{-pivmin, 0.f};
    cnt += (q.h < 0.f);
  }
  return cnt;
}

// a + b with an error of a few 2^-48 of the *result* (both parts summed
// without error first), so that it also holds when the operands cancel: the
// relative accuracy of the qd recurrence rests on it.
DV dfr df_add_rel(dfr a, dfr b) {
  const float s = a.h + b.h, sb = s - a.h;
  const float se = (a.h - (s - sb)) + (b.h - sb);
  const float t = a.l + b.l, tb = t - a.l;
  const float te = (a.l - (t - tb)) + (b.l - tb);
  const dfr v = df_quick(s, se + t);
  return df_quick(v.h, te + v.l);
}
DV dfr df_mul(dfr a, dfr b) {
  const float p = a.h * b.h;
  return df_quick(p, fmaf(a.h, b.h, -p) + fmaf(a.h, b.l, a.l * b.h));
}

// Number of singular values below x (x >= 2^-50: x^2 and the pivots stay far
// inside the FP32 range): negative pivots p_i of B B^T - x^2 I = L D L^T from
// the top, in differential form: with q_i = d_i^2 and eps_i = e_i^2,
//   s_1 = q_1 - x^2,  p_i = s_i + eps_i,  s_{i+1} = q_{i+1} (s_i / p_i) - x^2
// (the quotient first: s_i q_{i+1} would leave the FP32 range).  Per row one
// division, one product and two additions, against two divisions and two
// additions in the two T_GK rows it replaces.
__device__ __forceinline__ int qd_count_df(const float4* __restrict__ qe, int n, double x) {
  const float pivmin = 1e-36f;
  const dfr lam = df_of(x * x);
  const dfr ml{-lam.h, -lam.l};
  float4 cur = __ldg(qe);
  dfr s = df_add_rel(dfr{cur.x, cur.y}, ml);
  int cnt = 0;
  for (int i = 0; i < n; ++i) {
    const float4 nxt = __ldg(qe + (i + 1 < n ? i + 1 : i));
    const dfr ep{cur.z, cur.w};
    dfr p = df_add_rel(s, ep);
    if (fabsf(p.h) < pivmin) {
      p = dfr{p.h < 0.f ? -pivmin : pivmin, 0.f};
      s = df_add_rel(p, dfr{-ep.h, -ep.l});
    }
    cnt += (p.h < 0.f);
    s = df_add_rel(df_mul(df_div(s, p), dfr{nxt.x, nxt.y}), ml);
    cur = nxt;
  }
  return cnt;
}

// One CTA of 32 W threads per value: sig[k] = k-th largest singular value of
// B.  The bracket [lo, hi) keeps #{sigma < lo} < target <= #{sigma < hi} with
// target = n - k; each round the threads count at 32 W interior points, the
// first round's spaced geometrically from 2^-50, so that small values cost no
// more rounds than large ones.  Bound: the latency of the count's dependent
// chain (n rows of ~50 FP32 operations), times the rounds.  32 W points per
// round cut the rounds to 7 (W = 4); W = 1 once n values of 4 warps would
// queue for the issue slots instead of waiting for latency.  A value below
// 2^-50 amax is rounding noise of the FP64 bidiagonalisation and is found to
// 2^-8 relative by two rounds of T_GK counts.
template <int W>
__global__ void __launch_bounds__(32 * W)
bd_sigma_kernel(const float2* __restrict__ a2, const double* __restrict__ info, int n, double* __restrict__ sig) {
  const int P = 32 * W, t = threadIdx.x, k = blockIdx.x;
  const double amax = info[0];
  if (amax == 0.0) {
    if (t == 0) sig[k] = 0.0;
    return;
  }
  const int target = n - k;
  const float4* qe = reinterpret_cast<const float4*>(a2);
  const double bound = info[1], floor_hi = 0x1p-50;
  double lo = floor_hi, hi = bound;
  bool tiny = false;
  {
    // point 0 is the floor itself
    const double step = log2(bound / floor_hi) / P;
    auto at = [&](int j) { return floor_hi * exp2(step * j); };
    const int first = __syncthreads_count(qd_count_df(qe, n, at(t)) < target);
    if (first == 0) tiny = true;
    else {
      lo = at(first - 1);
      if (first < P) hi = at(first);
    }
  }
  if (tiny) {
    const double base = 0x1p-106;
    lo = 0.0;
    hi = floor_hi;
    for (int it = 0; it < 2; ++it) {
      const double l0 = lo, h0 = hi;
      auto at = [&](int j) {
        return it == 0 ? base * exp2(56.0 / P * j) : l0 + (h0 - l0) * (double)(j + 1) * (1.0 / (P + 1));
      };
      const int first = __syncthreads_count(sturm_count_df(a2, 2 * n, at(t)) - n < target);
      if (first > 0) lo = at(first - 1);
      if (first < P) hi = at(first);
      if (lo == 0.0) break;  // below 2^-106
    }
  } else {
    for (int it = 0; it < 24; ++it) {
      if (hi - lo <= 0x1p-42 * hi) break;
      const double l0 = lo, h0 = hi;
      auto at = [&](int j) { return l0 + (h0 - l0) * (double)(j + 1) * (1.0 / (P + 1)); };
      const int first = __syncthreads_count(qd_count_df(qe, n, at(t)) < target);
      if (first > 0) lo = at(first - 1);
      if (first < P) hi = at(first);
    }
  }
  if (t == 0) sig[k] = 0.5 * (lo + hi) * amax;
}

// The kept form of the values (see bd_serial_kernel): one warp per value on T_GK,
// sig[k] = k-th largest singular value of B.  The
// bracket [lo, hi) keeps #{sigma < lo} < target <= #{sigma < hi} with
// target = n - k; each round the lanes count at 32 interior points.
__global__ void bd_sigma_gk_kernel(const float2* __restrict__ a2, const double* __restrict__ info, int n,
                                double* __restrict__ sig) {
  const int lane = threadIdx.x & 31;
  const int k = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (k >= n) return;
  const double amax = info[0];
  if (amax == 0.0) {
    if (lane == 0) sig[k] = 0.0;
    return;
  }
  const int N = 2 * n, target = n - k;
  double lo = 0.0, hi = info[1];
  for (int it = 0; it < 24; ++it) {
    if (hi - lo <= 0x1p-42 * hi || hi - lo <= 1e-32) break;
    const double x = lo + (hi - lo) * (double)(lane + 1) * (1.0 / 33.0);
    const int below = sturm_count_df(a2, N, x) - n;
    const unsigned ok = __ballot_sync(0xffffffffu, below >= target);
    const int first = ok ? (__ffs(ok) - 1) : 32;
    const double xl = __shfl_sync(0xffffffffu, x, first == 0 ? 0 : first - 1);
    const double xh = __shfl_sync(0xffffffffu, x, first == 32 ? 31 : first);
    if (first > 0) lo = xl;
    if (first < 32) hi = xh;
  }
  if (lane == 0) sig[k] = 0.5 * (lo + hi) * amax;
}

cudaError_t bd_sigma(const double* d, const double* e, int n, float2* a2, double* info, double* sig,
                     int kept, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  bd_prep_kernel<<<1, 256, 0, s>>>(d, e, n, a2, info);
  cudaError_t err = cudaGetLastError();
  if (err != cudaSuccess) return err;
  if (kept) bd_sigma_gk_kernel<<<(n + 3) / 4, 128, 0, s>>>(a2, info, n, sig);
  else if (n <= 512) bd_sigma_kernel<4><<<n, 128, 0, s>>>(a2, info, n, sig);
  else bd_sigma_kernel<1><<<n, 32, 0, s>>>(a2, info, n, sig);
  return cudaGetLastError();
}
// Rank rule on the sorted values (the same rule as rank_select), one CTA:
// suffix sums of sigma^2 by a block scan, the rank as the smallest index
// that passes the test.
constexpr int kRankThreads = 256;
__global__ void __launch_bounds__(kRankThreads)
bd_rank_kernel(const double* __restrict__ sig, int n, const double* __restrict__ eps_hat, int cap,
               int forced, int* __restrict__ out_int, double* __restrict__ out_dbl,
               double* __restrict__ tail2) {
  __shared__ double wtot[kRankThreads / 32];
  __shared__ int rmin[2];
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int per = (n + kRankThreads - 1) / kRankThreads;
  const int a = min(n, tid * per), b = min(n, a + per);
  double own = 0.0;
  for (int r = a; r < b; ++r) own += sig[r] * sig[r];
  // suffix sum over threads: inclusive from the right within the warp
  double suf = own;
  for (int o = 1; o < 32; o <<= 1) {
    const double v = __shfl_down_sync(0xffffffffu, suf, o);
    if (lane + o < 32) suf += v;
  }
  if (lane == 0) wtot[wid] = suf;
  if (tid == 0) {
    rmin[0] = n;
    rmin[1] = n;
  }
  __syncthreads();
  double after = 0.0;  // sum over later warps
  for (int w = wid + 1; w < kRankThreads / 32; ++w) after += wtot[w];
  // tail2[r] = sum_{q >= r} sig_q^2 for this thread's chunk
  double run = suf - own + after;  // everything after this chunk
  for (int r = b - 1; r >= a; --r) {
    run += sig[r] * sig[r];
    tail2[r] = run;
  }
  if (tid == 0) tail2[n] = 0.0;
  __syncthreads();
  const double eh = *eps_hat;
  const double fro = sqrt(tail2[0]);
  const double thr = 2.0 * n * DBL_EPSILON * fro;
  for (int r = 1 + tid; r <= n; r += kRankThreads)
    if (sqrt(tail2[r]) <= eh) atomicMin(&rmin[0], r);
  for (int k = tid; k < n; k += kRankThreads)
    if (!(sig[k] > thr)) atomicMin(&rmin[1], k);
  __syncthreads();
  if (tid == 0) {
    const int rho_tol = rmin[0];
    int rho = forced > 0 ? forced : (rho_tol < cap ? rho_tol : cap);
    rho = rho < 1 ? 1 : (rho > n ? n : rho);
    // kept values at the noise level of a factorisation of B (their vectors
    // are not determined by B and are completed instead)
    const int kt = min(rmin[1], rho);
    out_int[0] = rho;
    out_int[1] = rho_tol;
    out_int[2] = kt;
    out_dbl[0] = sqrt(tail2[rho]);
    out_dbl[1] = sig[rho - 1];
    out_dbl[2] = tail2[0];
  }
}

cudaError_t bd_rank(const double* sig, int n, const double* eps_hat, int cap, int forced, int* out_int,
                    double* out_dbl, double* tail2, cudaStream_t s) {
  bd_rank_kernel<<<1, kRankThreads, 0, s>>>(sig, n, eps_hat, cap, forced, out_int, out_dbl, tail2);
  return cudaGetLastError();
}

// ---- 3. singular vectors of B -------------------------------------------------------------
DV double hash_unit(unsigned a, unsigned b) {
  unsigned h = a * 0x9E3779B1u ^ (b + 0x7F4A7C15u) * 0x85EBCA77u;
  h ^= h >> 15;
  h *= 0x2C1B3C6Du;
  h ^= h >> 12;
  h *= 0x297A2D39u;
  h ^= h >> 15;
  return (double)(h & 0xFFFFFFu) * (1.0 / 16777216.0) - 0.5;
}

// Entry i of the start vector of inverse iteration for value k.
DV double start_value(int i, int k) { return 1.0 + 0.25 * hash_unit((unsigned)i, (unsigned)k); }

// Solver arrays of T_GK - lam I (length N each) in shared memory, and the
// scaled off-diagonals (staged once per launch).
enum { L_DINV = 0, L_C1 = 1, L_C2 = 2, L_DL = 3, L_PV = 4, L_B = 5, L_OFF = 6 };
constexpr int kSolveArrays = 7;
size_t bd_vectors_smem(int n) { return sizeof(double) * kSolveArrays * 2 * (size_t)n; }

// LU with partial pivoting of T_GK - lam I (off-diagonals at L_OFF, scaled
// by 1 / amax); one thread.  Row i of U is stored as (1 / pivot, super /
// pivot, second super / pivot), so that the back substitution has one
// dependent multiply-add per row, and the multiplier uses the reciprocal of
// the pivot: one reciprocal and one multiply-add on the serial chain.
DV void gk_factor(int N, double lam, double* w) {
  double* Dinv = w + L_DINV * N;
  double* C1 = w + L_C1 * N;
  double* C2 = w + L_C2 * N;
  double* DL = w + L_DL * N;
  double* PV = w + L_PV * N;
  const double* off = w + L_OFF * N;
  const double tiny = 4.0 * DBL_EPSILON;
  auto guard = [&](double p) { return d_mag_less(p, tiny) ? (d_neg(p) ? -tiny : tiny) : p; };
  double di = -lam, dui = (N > 1) ? off[0] : 0.0;
  double sub = dui;
  for (int i = 0; i < N - 1; ++i) {
    const double un = (i + 1 < N - 1) ? off[i + 1] : 0.0;
    if (!d_mag_less(di, sub)) {
      const double rp = 1.0 / guard(di);
      const double f = sub * rp;
      Dinv[i] = rp;
      C1[i] = dui * rp;
      C2[i] = 0.0;
      DL[i] = f;
      PV[i] = 0.0;
      di = fma(-f, dui, -lam);
      dui = un;
    } else {
      // rows i and i+1 swapped: new row i = (sub, -lam, un)
      const double rs = 1.0 / sub;
      const double f = di * rs;
      Dinv[i] = rs;
      C1[i] = -lam * rs;
      C2[i] = un * rs;
      DL[i] = f;
      PV[i] = 1.0;
      di = fma(f, lam, dui);
      dui = -f * un;
    }
    sub = un;  // the sub-diagonal of row i+2 equals the super-diagonal off(i+1)
  }
  Dinv[N - 1] = 1.0 / guard(di);
}

// Solve with the factors at w, in place on B, by a whole warp (its results need
// a __syncwarp).  An FP64 instruction of a warp takes 64 cycles, one lane or all: comparisons are
// on the bits, the products with the reciprocal pivots run on all lanes, and
// the chains of lane 0 have one multiply-add per row (two where rows were
// swapped).
DV void gk_solve(int N, const double* w, double* B) {
  const double* Dinv = w + L_DINV * N;
  const double* C1 = w + L_C1 * N;
  const double* C2 = w + L_C2 * N;
  const double* DL = w + L_DL * N;
  const double* PV = w + L_PV * N;
  const int lane = threadIdx.x & 31;
  double cur = B[0];
  if (lane == 0) {
    double bn = B[min(1, N - 1)], f = DL[0];
    bool swap = !d_zero(PV[0]);
    for (int i = 0; i < N - 1; ++i) {
      // the next row's inputs are loaded ahead of the chain
      const int in = min(i + 1, N - 2);
      const double bnn = B[in + 1], fn = DL[in], pn = PV[in];
      const double row = swap ? bn : cur;
      B[i] = row;
      cur = fma(-f, row, swap ? cur : bn);
      bn = bnn;
      f = fn;
      swap = !d_zero(pn);
    }
  }
  __syncwarp();
  for (int i = lane; i < N - 1; i += 32) B[i] *= Dinv[i];
  __syncwarp();
  if (lane == 0) {
    double x2 = 0.0, x1 = cur * Dinv[N - 1];
    B[N - 1] = x1;
    int i = N - 2;
    double t = B[max(i, 0)], c1 = C1[max(i, 0)], c2 = C2[max(i, 0)];
    for (; i >= 0; --i) {
      const int in = max(i - 1, 0);
      const double tn = B[in], c1n = C1[in], c2n = C2[in];
      if (!d_zero(c2)) t = fma(-c2, x2, t);  // swapped rows only
      const double x = fma(-c1, x1, t);
      B[i] = x;
      x2 = x1;
      x1 = x;
      t = tn;
      c1 = c1n;
      c2 = c2n;
    }
  }
}

// One warp per kept value: left vector u_k of B as the eigenvector of B B^T
// by twisted factorisation.  With q_i = d_i^2, eps_i = e_i^2 (scaled by
// 1 / amax^2) and lambda = (sig_k / amax)^2, lane 0 runs
//   s_1 = q_1 - lambda, p_i = s_i + eps_i, s_{i+1} = q_{i+1} s_i / p_i - lambda
// from the top while lane 1 runs
//   t_n = -lambda, r_i = q_i + t_i, t_{i-1} = eps_{i-1} t_i / r_i - lambda
// from the bottom; gamma_i = s_i + t_i + lambda is the residual of the vector
// that solves every equation but row i, and the row where it is smallest
// starts the two products z_{i} = -(d_{i+1} e_i / p_i) z_{i+1} upwards and
// z_{i+1} = -(d_{i+1} e_i / r_{i+1}) z_i downwards.  lambda + gamma / |z|^2 is
// the Rayleigh quotient: one correction brings the multisection's 2^-42 to
// rounding level.  Bound by the latency of the FP64 chain, two sweeps of n
// rows of one reciprocal and three dependent operations.  The serial form it
// replaces (one warp per cluster, LU with pivoting and three solves of 2n
// rows per vector, one vector after another in a cluster) needed 14.3 ms per
// factor at n = 384 and 64 kept values when the values decay.
enum { V_Q = 0, V_EP = 1, V_OFF = 2, V_S = 3, V_T = 4, V_P = 5, V_R = 6, V_Z = 7 };
constexpr int kVecArrays = 8;

__global__ void __launch_bounds__(32)
bd_vectors_kernel(const double* __restrict__ d, const double* __restrict__ e, int n,
                  const double* __restrict__ info, const double* __restrict__ sig, double* __restrict__ X,
                  int ldx) {
  extern __shared__ __align__(16) double vsm[];
  const int k = blockIdx.x, lane = threadIdx.x;
  const double amax = info[0];
  if (amax == 0.0) return;
  const double inv = 1.0 / amax;
  double *Q = vsm + V_Q * n, *EP = vsm + V_EP * n, *OFF = vsm + V_OFF * n, *Sv = vsm + V_S * n, *Tv = vsm + V_T * n,
         *Pi = vsm + V_P * n, *Ri = vsm + V_R * n, *Z = vsm + V_Z * n;
  for (int i = lane; i < n; i += 32) {
    const double di = d[i] * inv, ei = (i + 1 < n) ? e[i] * inv : 0.0;
    Q[i] = di * di;
    EP[i] = ei * ei;
    OFF[i] = (i + 1 < n) ? d[i + 1] * inv * ei : 0.0;
  }
  __syncwarp();
  double lam = sig[k] * inv;
  lam *= lam;
  const double tiny = 1e-150;
  for (int pass = 0; pass < 2; ++pass) {
    if (lane < 2) {
      const bool up = lane == 1;  // lane 1 walks from the bottom
      double v = up ? -lam : Q[0] - lam;
      double* V = up ? Tv : Sv;
      double* C = up ? Ri : Pi;
      int i = up ? n - 1 : 0;
      const int di = up ? -1 : 1;
      double add = up ? Q[i] : EP[i];
      for (int step = 0; step < n; ++step) {
        // the next row's inputs are loaded ahead of the chain
        const int in = (step + 1 < n) ? i + di : i;
        const double mul = up ? EP[in] : Q[in];
        const double addn = up ? Q[in] : EP[in];
        double piv = v + add;
        if (d_mag_less(piv, tiny)) {
          piv = d_neg(piv) ? -tiny : tiny;
          v = piv - add;
        }
        V[i] = v;
        const double vm = v * mul;
        const double rc = rcp_fast(piv);
        C[i] = rc;
        v = fma(vm, rc, -lam);
        add = addn;
        i = in;
      }
    }
    __syncwarp();
    // twist row: smallest |gamma|
    double best = 1e300;
    int tw = 0;
    for (int i = lane; i < n; i += 32) {
      const double g = fabs(Sv[i] + Tv[i] + lam);
      if (g < best) {
        best = g;
        tw = i;
      }
    }
    for (int o = 16; o >= 1; o >>= 1) {
      const double ob = __shfl_xor_sync(0xffffffffu, best, o);
      const int ot = __shfl_xor_sync(0xffffffffu, tw, o);
      if (ob < best || (ob == best && ot < tw)) {
        best = ob;
        tw = ot;
      }
    }
    const double gam = Sv[tw] + Tv[tw] + lam;
    __syncwarp();
    for (int i = lane; i < n; i += 32) {
      Pi[i] *= -OFF[i];
      if (i > 0) Ri[i] *= -OFF[i - 1];
    }
    __syncwarp();
    if (lane < 2) {
      double v = 1.0;
      if (lane == 0) {
        Z[tw] = 1.0;
        for (int i = tw - 1; i >= 0; --i) {
          v *= Pi[i];
          Z[i] = v;
        }
      } else {
        for (int i = tw + 1; i < n; ++i) {
          v *= Ri[i];
          Z[i] = v;
        }
      }
    }
    __syncwarp();
    double nrm = 0.0;
    for (int i = lane; i < n; i += 32) nrm = fma(Z[i], Z[i], nrm);
    nrm = warp_sum(nrm);
    if (pass == 0) {
      const double corr = gam / nrm;
      if (fabs(corr) <= 1e-9 * lam) lam += corr;
    } else {
      const double s = 1.0 / sqrt(nrm);
      for (int i = lane; i < n; i += 32) X[i + (size_t)ldx * k] = Z[i] * s;
    }
  }
}

// One Newton-Schulz step towards the polar factor of X (n x k, columns of
// norm one and nearly orthogonal): X_out = X + X (I - X^T X) / 2, whose
// orthogonality error is 3/4 of the square of X's; the columns' span is
// unchanged.  One CTA per column: its k dot products, then its row of the
// update.  The first step sets info[2] when a pair of columns is not even
// orthogonal to 1e-4 (values equal to ~1e-11): the clustered path then
// computes all vectors again.
constexpr int kOrthThreads = 256;
// The clustered path's vectors take two steps of their own (only where it
// ran): orthogonal vectors of T_GK leave their left parts orthogonal to
// rounding times sigma_max / sigma only.
enum { kOrthFirst = 1, kOrthNext = 0, kOrthClustered = 2 };
__global__ void __launch_bounds__(kOrthThreads)
bd_orth_kernel(int n, int k, const double* __restrict__ X, int ldx, double* __restrict__ Xo, int ldo,
               double* __restrict__ info, int mode) {
  if (mode == kOrthClustered && info[2] == 0.0) return;
  extern __shared__ __align__(16) double osm[];  // column j [n], e_j [k]
  double* xj = osm;
  double* ej = osm + n;
  const int j = blockIdx.x, lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = kOrthThreads >> 5;
  for (int i = threadIdx.x; i < n; i += kOrthThreads) xj[i] = X[i + (size_t)ldx * j];
  __syncthreads();
  // two columns at a time per warp: independent chains
  for (int c = 2 * wid; c < k; c += 2 * nw) {
    const bool two = c + 1 < k;
    const double *a = X + (size_t)ldx * c, *b = X + (size_t)ldx * (two ? c + 1 : c);
    double s0 = 0.0, s1 = 0.0;
    for (int i = lane; i < n; i += 32) {
      s0 = fma(a[i], xj[i], s0);
      s1 = fma(b[i], xj[i], s1);
    }
    s0 = warp_sum(s0);
    s1 = warp_sum(s1);
    if (lane < 2 && c + lane < k) {
      const double g = lane ? s1 : s0;
      const double ee = (c + lane == j) ? 1.0 - g : -g;
      ej[c + lane] = 0.5 * ee;
      if (mode == kOrthFirst && !(fabs(ee) <= 1e-4)) info[2] = 1.0;  // also for NaN
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < n; i += kOrthThreads) {
    double v0 = 0.0, v1 = 0.0;
    int c = 0;
    for (; c + 1 < k; c += 2) {
      v0 = fma(X[i + (size_t)ldx * c], ej[c], v0);
      v1 = fma(X[i + (size_t)ldx * (c + 1)], ej[c + 1], v1);
    }
    if (c < k) v0 = fma(X[i + (size_t)ldx * c], ej[c], v0);
    Xo[i + (size_t)ldo * j] = xj[i] + (v0 + v1);
  }
}

// The path for repeated values (runs when bd_orth_kernel has set info[2]): one
// warp per cluster of kept values (consecutive values closer than 1e-3
// sigma_max): inverse iteration for each member, re-orthogonalised
// against the members before it.  Lane 0 runs the tridiagonal recurrences
// out of shared memory; the warp does the products and norms.  X (n x
// nvec, ldx) receives the normalised left vectors u_k.  Every k < nvec is
// above the noise level (the caller passes the count of such values).
__global__ void bd_cluster_kernel(const double* __restrict__ d, const double* __restrict__ e, int n,
                                  const double* __restrict__ info, const double* __restrict__ sig,
                                  int nvec, double* __restrict__ X, int ldx, double* __restrict__ Zs) {
  extern __shared__ __align__(16) double vsm[];  // kSolveArrays * N
  const int k0 = blockIdx.x, lane = threadIdx.x;
  const int N = 2 * n;
  if (k0 >= nvec || info[2] == 0.0) return;
  const double amax = info[0];
  if (amax == 0.0) return;
  const double gap_tol = 1e-3 * sig[0];
  if (k0 > 0 && sig[k0 - 1] - sig[k0] < gap_tol) return;  // not the first of its cluster
  int k1 = k0 + 1;
  while (k1 < nvec && sig[k1 - 1] - sig[k1] < gap_tol) ++k1;
  const double inv = 1.0 / amax;
  double* B = vsm + L_B * N;
  double* off = vsm + L_OFF * N;
  for (int i = lane; i < N - 1; i += 32) off[i] = ((i & 1) ? e[i >> 1] : d[i >> 1]) * inv;
  __syncwarp();
  for (int k = k0; k < k1; ++k) {
    if (lane == 0) gk_factor(N, sig[k] * inv, vsm);
    for (int i = lane; i < N; i += 32) B[i] = start_value(i, k);
    __syncwarp();
    for (int it = 0; it < 3; ++it) {
      gk_solve(N, vsm, B);
      __syncwarp();
      for (int j = k0; j < k; ++j) {
        const double* zj = Zs + (size_t)j * N;
        double dot = 0.0;
        for (int i = lane; i < N; i += 32) dot += zj[i] * B[i];
        dot = warp_sum(dot);
        for (int i = lane; i < N; i += 32) B[i] -= dot * zj[i];
        __syncwarp();
      }
      double nrm = 0.0;
      for (int i = lane; i < N; i += 32) nrm += B[i] * B[i];
      nrm = warp_sum(nrm);
      const double s = nrm > 0.0 ? 1.0 / sqrt(nrm) : 0.0;
      for (int i = lane; i < N; i += 32) B[i] *= s;
      __syncwarp();
    }
    double* zk = Zs + (size_t)k * N;
    double un = 0.0;
    for (int i = lane; i < N; i += 32) {
      const double z = B[i];
      zk[i] = z;
      if (i & 1) un += z * z;
    }
    un = warp_sum(un);
    const double s = un > 0.0 ? 1.0 / sqrt(un) : 0.0;
    for (int i = lane; i < n; i += 32) X[i + (size_t)ldx * k] = B[2 * i + 1] * s;
    __syncwarp();
  }
}

// ---- vectors kept to the last bit ----------------------------------------------
// In a mixed context with digit products U is cut at 2^-40 of its largest
// entry, about the 1e-12 by which a vector in a cluster of values moves with the
// rounding of its computation; the flipped digits move a covariance (a second
// difference of Phi) by 1e-10 to 2e-9.  There the vectors are those of
// bd_cluster_kernel, in its order of operations, from two kernels instead of
// one: bd_factor_kernel does for all values at once what does not wait for other
// vectors (the LU factors, a division per row on the chain, and the first
// solve), bd_serial_kernel the rest, one CTA per cluster.
//   lu: 5 N doubles per value (the factor arrays), Z: N per value.
__global__ void __launch_bounds__(32)
bd_factor_kernel(const double* __restrict__ d, const double* __restrict__ e, int n, const double* __restrict__ info,
                 const double* __restrict__ sig, double* __restrict__ lu, double* __restrict__ Z) {
  extern __shared__ __align__(16) double vsm[];  // kSolveArrays * N
  const int k = blockIdx.x, lane = threadIdx.x, N = 2 * n;
  const double amax = info[0];
  if (amax == 0.0) return;
  const double inv = 1.0 / amax;
  double *off = vsm + L_OFF * N, *B = vsm + L_B * N;
  for (int i = lane; i < N - 1; i += 32) off[i] = ((i & 1) ? e[i >> 1] : d[i >> 1]) * inv;
  __syncwarp();
  if (lane == 0) gk_factor(N, sig[k] * inv, vsm);
  for (int i = lane; i < N; i += 32) B[i] = start_value(i, k);
  __syncwarp();
  // (the last rows of C1, C2, DL, PV are never written or read)
  double* f = lu + (size_t)k * 5 * N;
  for (int i = lane; i < 5 * N; i += 32)
    if (i < N || i % N < N - 1) f[i] = vsm[i];
  gk_solve(N, vsm, B);
  __syncwarp();
  for (int i = lane; i < N; i += 32) Z[(size_t)k * N + i] = B[i];
}

// Per vector of a cluster: Gram-Schmidt against the members before it,
// normalisation, and twice solve, Gram-Schmidt, normalisation.  A dot product's
// 32 chains (one per lane) fix warp 0 to it; the other warps stage the next
// vector meanwhile and share the update, and while warp 0 solves they load the
// next value's factors (two buffers of each, where they fit).  Bound by warp 0's
// FP64 instructions: per pair N / 32 of the chain, 5 of the sum, N / 128 of the
// update.
constexpr int kSerialThreads = 128;
size_t bd_serial_smem(int n, int buffers) { return sizeof(double) * (6 * (size_t)buffers + 1) * 2 * n; }

__global__ void __launch_bounds__(kSerialThreads)
bd_serial_kernel(int n, const double* __restrict__ info, const double* __restrict__ sig, int nvec,
                 const double* __restrict__ lu, double* Z, double* __restrict__ X, int ldx, int buffers) {
  extern __shared__ __align__(16) double ssm[];
  __shared__ double bcast;
  const int N = 2 * n, k0 = blockIdx.x, tid = threadIdx.x, lane = tid & 31;
  if (info[0] == 0.0) return;
  const double gap_tol = 1e-3 * sig[0];
  if (k0 > 0 && sig[k0 - 1] - sig[k0] < gap_tol) return;  // not the first of its cluster
  int k1 = k0 + 1;
  while (k1 < nvec && sig[k1 - 1] - sig[k1] < gap_tol) ++k1;
  double* F = ssm;                                // [buffers][5 N]
  double* B = F + (size_t)buffers * 5 * N;        // [N]
  double* zb = B + N;                             // [buffers][N]
  const int odd = buffers - 1;  // with two buffers odd values and vectors use the second
  // factors of value k by the threads from t0 on
  auto load_factors = [&](int k, int t0) {
    double* dst = F + (size_t)((k & 1) & odd) * 5 * N;
    const double* src = lu + (size_t)k * 5 * N;
    for (int i = tid - t0; i < 5 * N; i += kSerialThreads - t0)
      if (i < N || i % N < N - 1) dst[i] = src[i];
  };
  auto load_vector = [&](double* dst, int j, int t0) {
    for (int i = tid - t0; i < N; i += kSerialThreads - t0) dst[i] = Z[(size_t)j * N + i];
  };
  load_factors(k0, 0);
  for (int k = k0; k < k1; ++k) {
    load_vector(B, k, 0);
    __syncthreads();
    const double* f = F + (size_t)((k & 1) & odd) * 5 * N;
    for (int it = 0; it < 3; ++it) {
      if (it > 0) {
        if (tid < 32) gk_solve(N, f, B);
        else if (it == 1 && buffers == 2 && k + 1 < k1) load_factors(k + 1, 32);
        __syncthreads();
      }
      if (k > k0) load_vector(zb, k0, 0);
      __syncthreads();
      for (int j = k0; j < k; ++j) {
        const double* zj = zb + (size_t)((j - k0) & odd) * N;
        if (tid < 32) {
          double dot = 0.0;
          for (int i = lane; i < N; i += 32) dot = fma(zj[i], B[i], dot);
          dot = warp_sum(dot);
          if (lane == 0) bcast = dot;
        } else if (buffers == 2 && j + 1 < k) {
          load_vector(zb + (size_t)((j + 1 - k0) & 1) * N, j + 1, 32);
        }
        __syncthreads();
        const double dot = bcast;
        for (int i = tid; i < N; i += kSerialThreads) B[i] = fma(-dot, zj[i], B[i]);
        if (buffers == 1 && j + 1 < k) {
          __syncthreads();
          load_vector(zb, j + 1, 0);
        }
        __syncthreads();
      }
      if (tid < 32) {
        double nrm = 0.0;
        for (int i = lane; i < N; i += 32) nrm = fma(B[i], B[i], nrm);
        nrm = warp_sum(nrm);
        if (lane == 0) bcast = nrm > 0.0 ? 1.0 / sqrt(nrm) : 0.0;
      }
      __syncthreads();
      const double s = bcast;
      for (int i = tid; i < N; i += kSerialThreads) B[i] *= s;
      __syncthreads();
    }
    for (int i = tid; i < N; i += kSerialThreads) Z[(size_t)k * N + i] = B[i];
    if (tid < 32) {
      double un = 0.0;
      for (int i = lane; i < N; i += 32)
        if (i & 1) un = fma(B[i], B[i], un);
      un = warp_sum(un);
      if (lane == 0) bcast = un > 0.0 ? 1.0 / sqrt(un) : 0.0;
    }
    if (buffers == 1 && k + 1 < k1) load_factors(k + 1, 0);
    __syncthreads();
    const double s = bcast;
    for (int i = tid; i < n; i += kSerialThreads) X[i + (size_t)ldx * k] = B[2 * i + 1] * s;
    __syncthreads();
  }
}

// Orthonormal completion for kept values at the noise level (indices
// kt..nvec-1): pseudo-random vectors, classical Gram-Schmidt twice against
// every earlier column of X.  One CTA.
__global__ void bd_complete_kernel(int n, int kt, int nvec, double* __restrict__ X, int ldx) {
  extern __shared__ __align__(16) unsigned char cs_smem[];
  double* x = reinterpret_cast<double*>(cs_smem);  // n
  double* dots = x + n;                             // nvec
  __shared__ double red[32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  for (int k = kt; k < nvec; ++k) {
    for (int i = threadIdx.x; i < n; i += blockDim.x) x[i] = hash_unit((unsigned)i + 7919u, (unsigned)k * 31u + 3u);
    __syncthreads();
    for (int pass = 0; pass < 2; ++pass) {
      for (int j = wid; j < k; j += nw) {
        double s = 0.0;
        for (int i = lane; i < n; i += 32) s += X[i + (size_t)ldx * j] * x[i];
        s = warp_sum(s);
        if (lane == 0) dots[j] = s;
      }
      __syncthreads();
      for (int i = threadIdx.x; i < n; i += blockDim.x) {
        double v = x[i];
        for (int j = 0; j < k; ++j) v -= dots[j] * X[i + (size_t)ldx * j];
        x[i] = v;
      }
      __syncthreads();
    }
    double s = 0.0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) s += x[i] * x[i];
    s = block_sum(s, red);
    const double sc = s > 0.0 ? 1.0 / sqrt(s) : 0.0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) X[i + (size_t)ldx * k] = x[i] * sc;
    __syncthreads();
  }
}


size_t bd_lu_elems(int n, int kt) { return (size_t)10 * n * kt; }

cudaError_t bd_vectors(const double* d, const double* e, int n, double* info, const double* sig,
                       int kt, int nvec, double* X, int ldx, double* Zs, double* lu, cudaStream_t s) {
  if (nvec <= 0) return cudaSuccess;
  if (kt > 0 && lu) {
    const size_t fsmem = bd_vectors_smem(n);
    const int buffers = bd_serial_smem(n, 2) <= (size_t)dev_info().max_smem_optin - 1024 ? 2 : 1;
    const size_t smem = bd_serial_smem(n, buffers);
    cudaError_t err = allow_smem((const void*)bd_factor_kernel, fsmem);
    if (err == cudaSuccess) err = allow_smem((const void*)bd_serial_kernel, smem);
    if (err != cudaSuccess) return err;
    bd_factor_kernel<<<kt, 32, fsmem, s>>>(d, e, n, info, sig, lu, Zs);
    bd_serial_kernel<<<kt, kSerialThreads, smem, s>>>(n, info, sig, kt, lu, Zs, X, ldx, buffers);
    err = cudaGetLastError();
    if (err != cudaSuccess) return err;
  } else if (kt > 0) {
    const size_t vsmem = sizeof(double) * kVecArrays * (size_t)n, csmem = bd_vectors_smem(n);
    const size_t osmem = sizeof(double) * ((size_t)n + kt);
    cudaError_t err = allow_smem((const void*)bd_orth_kernel, osmem);
    if (err == cudaSuccess) err = allow_smem((const void*)bd_cluster_kernel, csmem);
    if (err == cudaSuccess) err = allow_smem((const void*)bd_vectors_kernel, vsmem);
    if (err != cudaSuccess) return err;
    bd_vectors_kernel<<<kt, 32, vsmem, s>>>(d, e, n, info, sig, X, ldx);
    bd_orth_kernel<<<kt, kOrthThreads, osmem, s>>>(n, kt, X, ldx, Zs, n, info, kOrthFirst);
    bd_orth_kernel<<<kt, kOrthThreads, osmem, s>>>(n, kt, Zs, n, X, ldx, info, kOrthNext);
    bd_cluster_kernel<<<kt, 32, csmem, s>>>(d, e, n, info, sig, kt, X, ldx, Zs);
    bd_orth_kernel<<<kt, kOrthThreads, osmem, s>>>(n, kt, X, ldx, Zs, n, info, kOrthClustered);
    bd_orth_kernel<<<kt, kOrthThreads, osmem, s>>>(n, kt, Zs, n, X, ldx, info, kOrthClustered);
    err = cudaGetLastError();
    if (err != cudaSuccess) return err;
  }
  if (kt < nvec) {
    const size_t smem = sizeof(double) * ((size_t)n + nvec);
    bd_complete_kernel<<<1, 256, smem, s>>>(n, kt, nvec, X, ldx);
  }
  return cudaGetLastError();
}

// ---- 4. back-transformation -------------------------------------------------------------------
// u_k <- Q u_k with Q = H_0 H_1 ... H_{n-1} (reflector j: unit entry at j,
// tail A[j+1:n, j], tau[j]).  One vector per CTA, so that the FP64 work
// (about 10 n^2 / 2 operations per vector) spreads over many SMs.  A warp's
// FP64 instruction holds its quarter of the SM for 64 cycles, so one warp per
// vector ran at a quarter of the SM's rate (7400 cycles for two reflectors at
// n = 192; a factor of the C3 mixed step 520 us, 289 with four).  Four warps
// share a reflector: the real and the imaginary part of the dot product on two
// of them each, by halves of the rows (SPLIT; without it one warp's order of
// the sums and its bits, bd_serial_kernel says where), then a quarter of the
// rows' update each.
// kBackStage further warps stage the next reflectors in shared memory.
// The result goes to U (n x nvec, ldu) and to Xp (mrows x nvec, ldp, zero
// below row n).
constexpr int kBackStage = 2, kBackWarps = 4;
template <bool SPLIT>
__global__ void __launch_bounds__(32 * (kBackStage + kBackWarps))
bd_back_kernel(const cplx* __restrict__ A, int lda, const cplx* __restrict__ tauq, int n,
               const double* __restrict__ Xr, int ldx, int nvec, cplx* __restrict__ U, int ldu,
               cplx* __restrict__ Xp, int ldp, int mrows) {
  extern __shared__ __align__(16) unsigned char bk_smem[];
  constexpr int S = kBackStage;
  cplx* vb = reinterpret_cast<cplx*>(bk_smem);  // [2][S][n] staged reflectors
  cplx* x = vb + 2 * (size_t)S * n;             // [n]
  __shared__ cplx tb[2 * S];                    // their tau
  __shared__ double red[2][kBackWarps];
  const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int k = blockIdx.x;
  if (k >= nvec) return;
  // reflector j (none if negative) into slot q
  auto stage = [&](int j, int q) {
    if (j < 0) return;
    cplx* v = vb + (size_t)q * n;
    const cplx* a = A + (size_t)lda * j;
    if (lane == 0) {
      v[j] = mk(1, 0);
      tb[q] = __ldg(tauq + j);
    }
    for (int i0 = j + 1 + lane; i0 < n; i0 += 128) {
      cplx r[4];
#pragma unroll
      for (int t = 0; t < 4; ++t) r[t] = (i0 + 32 * t < n) ? __ldg(a + i0 + 32 * t) : mk(0, 0);
#pragma unroll
      for (int t = 0; t < 4; ++t)
        if (i0 + 32 * t < n) v[i0 + 32 * t] = r[t];
    }
  };
  if (wid < kBackWarps) {
    for (int i = threadIdx.x; i < n; i += 32 * kBackWarps) x[i] = mk(Xr[i + (size_t)ldx * k], 0.0);
  } else {
    stage(n - 1 - (wid - kBackWarps), wid - kBackWarps);
  }
  __syncthreads();
  for (int j0 = n - 1, h = 0; j0 >= 0; j0 -= S, h ^= 1) {
    if (wid >= kBackWarps) {
      stage(j0 - S - (wid - kBackWarps), (h ^ 1) * S + wid - kBackWarps);
    } else {
      for (int w = 0; w < S && j0 - w >= 0; ++w) {
        const int j = j0 - w;
        const cplx t = tb[h * S + w];
        if (t.x == 0.0 && t.y == 0.0) continue;  // the same for every thread
        const cplx* v = vb + (size_t)(h * S + w) * n;
        double* rd = red[w & 1];
        // part wid & 1 of v^H x
        double acc = 0.0;
        if (SPLIT || wid < 2) {
          const int step = SPLIT ? 64 : 32;
          int i = j + lane + (SPLIT ? 32 * (wid >> 1) : 0);
          if (wid & 1) {
            for (; i < n; i += step) acc = fma(v[i].x, x[i].y, fma(-v[i].y, x[i].x, acc));
          } else {
            for (; i < n; i += step) acc = fma(v[i].x, x[i].x, fma(v[i].y, x[i].y, acc));
          }
          acc = warp_sum(acc);
          if (lane == 0) rd[wid] = acc;
        }
        asm volatile("bar.sync 1, %0;" ::"n"(32 * kBackWarps) : "memory");
        const cplx dot = SPLIT ? mk(rd[0] + rd[2], rd[1] + rd[3]) : mk(rd[0], rd[1]);
        const cplx f = cmul(t, dot);
        const cplx nf = mk(-f.x, -f.y);
        for (int i = j + threadIdx.x; i < n; i += 32 * kBackWarps) x[i] = cfma(v[i], nf, x[i]);
        asm volatile("bar.sync 1, %0;" ::"n"(32 * kBackWarps) : "memory");
      }
    }
    __syncthreads();
  }
  for (int i = threadIdx.x; i < mrows; i += blockDim.x) {
    const cplx v = (i < n) ? x[i] : mk(0, 0);
    if (i < n) U[i + (size_t)ldu * k] = v;
    Xp[i + (size_t)ldp * k] = v;
  }
}

cudaError_t bd_back(const cplx* A, int lda, const cplx* tauq, int n, const double* X, int ldx, int nvec,
                    cplx* U, int ldu, cplx* Xp, int ldp, int mrows, int kept, cudaStream_t s) {
  if (nvec <= 0) return cudaSuccess;
  // 80 bytes per row: less than the vectors' own solves keep (bd_vectors_smem)
  const size_t smem = sizeof(cplx) * (size_t)n * (2 * kBackStage + 1);
  const auto fn = kept ? bd_back_kernel<false> : bd_back_kernel<true>;
  cudaError_t err = allow_smem((const void*)fn, smem);
  if (err != cudaSuccess) return err;
  fn<<<nvec, 32 * (kBackStage + kBackWarps), smem, s>>>(A, lda, tauq, n, X, ldx, nvec, U, ldu, Xp, ldp, mrows);
  return cudaGetLastError();
}

}  // namespace hk
