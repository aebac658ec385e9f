// The values of Phi that the central differences of the moments read: Phi at
// a = 0, one step along every axis, and one step along every pair of axes
// (Sec. 1: moments are functional derivatives of Phi at theta = 0).
//
// The 1 + 2d + 2d(d-1) points differ from the centre in at most two modes, so
// their products share almost everything.  With E_k^o the slice of core k at
// index n/2 + o, L_k = E_0^0 ... E_{k-1}^0 and R_k = E_k^0 ... E_{d-1}^0,
//   Phi(0) = L_d,   Phi(s e_k) = L_k (E_k^s R_{k+1}),
//   Phi(s e_j + s' e_k) = [L_j E_j^s E_{j+1}^0 ... E_{k-1}^0] (E_k^s' R_{k+1}).
// moment_chains_kernel runs the 2d row chains (the prefix L, and for every
// j < d-1 and sign the bracket, kept for every k) and the suffix chain R at
// once, d steps each; moment_pairs_kernel forms y = E_k^s' R_{k+1} per (k, s')
// and its products with the brackets.  O(d^2 r^2) multiply-adds instead of
// O(d^3 r^2) for one product per point, which was bound by the FP64 units
// (1.88 ms at d = 32, r = 64).  What bounds the chains is the latency of d
// dependent matrix-vector products, each r^2 complex FP64 multiply-adds (4 us
// on one SM at r = 64): a thread-block cluster splits every product by
// columns and exchanges the vector through distributed shared memory.
#include <cooperative_groups.h>

#include <algorithm>

#include "kernels.h"

namespace cg = cooperative_groups;

namespace hk {

namespace {

constexpr int kMomThreads = 256;

DV cplx shfl_xor_c(cplx v, int o) {
  return mk(__shfl_xor_sync(0xffffffffu, v.x, o), __shfl_xor_sync(0xffffffffu, v.y, o));
}

// Lanes that share one output of a product: few for many outputs (fewer FP64
// additions across lanes), more when the outputs do not fill the CTA.
DV int lanes_per_output(int outputs) {
  int s = 4;
  while (s < 32 && outputs * s * 2 <= kMomThreads) s *= 2;
  return s;
}

// out(j, sum_i v_i E[i + cs j]) for j in [j0, j1): S adjacent lanes per
// column take interleaved i (contiguous in memory).
template <class F>
DV void row_times(const cplx* __restrict__ E, size_t cs, int a, const cplx* v, int j0, int j1, F out) {
  const int S = lanes_per_output(j1 - j0);
  const int seg = threadIdx.x % S, per = kMomThreads / S;
  for (int jb = j0; jb < j1; jb += per) {
    const int j = jb + threadIdx.x / S;
    cplx acc = mk(0, 0), acc2 = mk(0, 0);
    if (j < j1) {
      const cplx* col = E + cs * j;
      int i = seg;
      for (; i + 3 * S < a; i += 4 * S) {
        const cplx e0 = __ldg(col + i), e1 = __ldg(col + i + S), e2 = __ldg(col + i + 2 * S), e3 = __ldg(col + i + 3 * S);
        acc = cfma(v[i], e0, acc);
        acc2 = cfma(v[i + S], e1, acc2);
        acc = cfma(v[i + 2 * S], e2, acc);
        acc2 = cfma(v[i + 3 * S], e3, acc2);
      }
      for (; i < a; i += S) acc = cfma(v[i], __ldg(col + i), acc);
    }
    acc = cadd(acc, acc2);
    for (int o = 1; o < S; o <<= 1) acc = cadd(acc, shfl_xor_c(acc, o));
    if (seg == 0 && j < j1) out(j, acc);
  }
}

// out(i, sum_j E[i + cs j] v_j) for i in [i0, i1): neighbouring lanes take
// neighbouring i, S groups of lanes interleaved j.
template <class F>
DV void times_col(const cplx* __restrict__ E, size_t cs, int c, const cplx* v, int i0, int i1, F out) {
  const int S = lanes_per_output(i1 - i0), L = 32 / S;
  const int lane = threadIdx.x & 31, seg = lane / L, per = kMomThreads / S;
  for (int ib = i0; ib < i1; ib += per) {
    const int i = ib + (threadIdx.x >> 5) * L + lane % L;
    cplx acc = mk(0, 0), acc2 = mk(0, 0);
    if (i < i1) {
      int j = seg;
      for (; j + 3 * S < c; j += 4 * S) {
        const cplx e0 = __ldg(E + i + cs * j), e1 = __ldg(E + i + cs * (j + S)), e2 = __ldg(E + i + cs * (j + 2 * S)),
                   e3 = __ldg(E + i + cs * (j + 3 * S));
        acc = cfma(v[j], e0, acc);
        acc2 = cfma(v[j + S], e1, acc2);
        acc = cfma(v[j + 2 * S], e2, acc);
        acc2 = cfma(v[j + 3 * S], e3, acc2);
      }
      for (; j < c; j += S) acc = cfma(v[j], __ldg(E + i + cs * j), acc);
    }
    acc = cadd(acc, acc2);
    for (int o = L; o < 32; o <<= 1) acc = cadd(acc, shfl_xor_c(acc, o));
    if (seg == 0 && i < i1) out(i, acc);
  }
}

DV void share(int total, int parts, int p, int* b, int* e) {
  const int w = (total + parts - 1) / parts;
  *b = min(total, p * w);
  *e = min(total, *b + w);
}

// Chain q of the grid (one cluster each): 0 the prefix, 1 the suffix, 2 + 2 j
// + s the bracket of mode j and sign s.  env: L at [k], R at [d + 1 + k], the
// bracket (j, s) before mode k at [2 (d + 1) + (2 j + s) d + k], rmax apart.
__global__ void __launch_bounds__(kMomThreads)
moment_chains_kernel(const cplx* const* __restrict__ cores, const int* __restrict__ ranks, int d, int n, int rmax,
                     cplx* __restrict__ env, cplx* __restrict__ vals) {
  extern __shared__ __align__(16) unsigned char mom_sm[];
  cplx* vb = reinterpret_cast<cplx*>(mom_sm);  // [2][rmax]
  cg::cluster_group cl = cg::this_cluster();
  const int CS = cl.num_blocks(), p = cl.block_rank(), q = blockIdx.x / CS;
  const int c0 = n / 2;
  if (threadIdx.x == 0) vb[0] = mk(1, 0);
  cl.sync();
  int cur = 0;
  if (q == 1) {
    cplx* R = env + (size_t)(d + 1) * rmax;
    if (p == 0 && threadIdx.x == 0) R[(size_t)d * rmax] = mk(1, 0);
    for (int k = d - 1; k >= 0; --k, cur ^= 1) {
      const int a = ranks[k], c = ranks[k + 1];
      int b, e;
      share(a, CS, p, &b, &e);
      times_col(cores[k] + (size_t)a * c0, (size_t)a * n, c, vb + (size_t)cur * rmax, b, e, [&](int i, cplx x) {
        R[(size_t)k * rmax + i] = x;
        for (int t = 0; t < CS; ++t) cl.map_shared_rank(vb, t)[(size_t)(cur ^ 1) * rmax + i] = x;
      });
      cl.sync();
    }
    return;
  }
  const int jm = q == 0 ? -1 : (q - 2) / 2, off = q == 0 ? 0 : ((q & 1) ? -1 : 1);
  cplx* keep = q == 0 ? env : env + (size_t)(2 * (d + 1) + (q - 2) * d) * rmax;
  if (q == 0 && p == 0 && threadIdx.x == 0) keep[0] = mk(1, 0);
  for (int k = 0; k < d; ++k, cur ^= 1) {
    if (q != 0 && k == d - 1) break;  // the last mode belongs to the pairs
    const int a = ranks[k], c = ranks[k + 1];
    int b, e;
    share(c, CS, p, &b, &e);
    row_times(cores[k] + (size_t)a * (c0 + (k == jm ? off : 0)), (size_t)a * n, a, vb + (size_t)cur * rmax, b, e,
              [&](int j, cplx x) {
                if (q == 0) {
                  keep[(size_t)(k + 1) * rmax + j] = x;
                  if (k == d - 1) vals[0] = x;
                } else if (k >= jm) {
                  keep[(size_t)(k + 1) * rmax + j] = x;
                }
                for (int t = 0; t < CS; ++t) cl.map_shared_rank(vb, t)[(size_t)(cur ^ 1) * rmax + j] = x;
              });
    cl.sync();
  }
}

// One cluster per mode k and sign s': y = E_k^s' R_{k+1}, rows split over the
// cluster, then its products with L_k and with the brackets of every j < k.
__global__ void __launch_bounds__(kMomThreads)
moment_pairs_kernel(const cplx* const* __restrict__ cores, const int* __restrict__ ranks, int d, int n, int rmax,
                    const cplx* __restrict__ env, cplx* __restrict__ vals) {
  extern __shared__ __align__(16) unsigned char mom_sm[];
  cplx* rv = reinterpret_cast<cplx*>(mom_sm);  // R_{k+1} [rmax]
  cplx* y = rv + rmax;                         // own rows of y [rmax]
  cplx* part = y + rmax;                       // [2 d + 1] partial products
  cg::cluster_group cl = cg::this_cluster();
  const int CS = cl.num_blocks(), p = cl.block_rank(), q = blockIdx.x / CS;
  const int k = q >> 1, s = q & 1, c0 = n / 2 + (s ? -1 : 1);
  const int a = ranks[k], c = ranks[k + 1];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const cplx* R = env + (size_t)(d + 1 + k + 1) * rmax;
  for (int j = threadIdx.x; j < c; j += kMomThreads) rv[j] = R[j];
  __syncthreads();
  int b, e;
  share(a, CS, p, &b, &e);
  times_col(cores[k] + (size_t)a * c0, (size_t)a * n, c, rv, b, e, [&](int i, cplx x) { y[i] = x; });
  __syncthreads();
  for (int t = wid; t < 2 * k + 1; t += kMomThreads / 32) {
    const cplx* f = t == 0 ? env + (size_t)k * rmax : env + (size_t)(2 * (d + 1) + (t - 1) * d + k) * rmax;
    cplx acc = mk(0, 0);
    for (int i = b + lane; i < e; i += 32) acc = cfma(f[i], y[i], acc);
    acc = warp_sum(acc);
    if (lane == 0) part[t] = acc;
  }
  cl.sync();
  if (p == 0)
    for (int t = threadIdx.x; t < 2 * k + 1; t += kMomThreads) {
      cplx v = part[t];
      for (int o = 1; o < CS; ++o) v = cadd(v, cl.map_shared_rank(part, o)[t]);
      if (t == 0) {
        vals[1 + 2 * k + s] = v;
      } else {
        const int j = (t - 1) >> 1, sj = (t - 1) & 1;
        vals[1 + 2 * d + 4 * (j * d - j * (j + 1) / 2 + (k - j - 1)) + 2 * sj + s] = v;
      }
    }
  cl.sync();  // the other CTAs' partial products stay until they are read
}

template <class... A>
cudaError_t launch_cluster(void (*fn)(A...), int clusters, int cs, size_t smem, cudaStream_t s, A... args) {
  cudaError_t e = allow_smem((const void*)fn, smem);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(clusters * cs);
  cfg.blockDim = dim3(kMomThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = cs;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, fn, args...);
}

}  // namespace

size_t moment_env_elems(int d, int rmax) { return ((size_t)2 * (d + 1) + (size_t)2 * (d - 1) * d) * rmax; }

// CTAs per chain: a product's r^2 complex multiply-adds take 2 r^2 / CS cycles
// of the FP64 unit, the exchange about 1000; split while the product is the
// longer part and the chains still fit on the SMs at once (CS <= 8).
cudaError_t moment_values(const cplx* const* cores_dev, const int* ranks_dev, int d, int n, int rmax, cplx* env,
                          cplx* vals, cudaStream_t s) {
  int cs = 1;
  while (cs < 8 && (size_t)rmax * rmax / cs > 1024 && 2 * d * cs * 2 <= dev_info().sm_count) cs *= 2;
  const size_t vec = sizeof(cplx) * (size_t)rmax;
  cudaError_t e = launch_cluster(moment_chains_kernel, 2 * d, cs, 2 * vec, s, cores_dev, ranks_dev, d, n, rmax, env, vals);
  if (e != cudaSuccess) return e;
  return launch_cluster(moment_pairs_kernel, 2 * d, cs, 2 * vec + sizeof(cplx) * (2 * (size_t)d + 1), s, cores_dev,
                        ranks_dev, d, n, rmax, (const cplx*)env, vals);
}

}  // namespace hk
