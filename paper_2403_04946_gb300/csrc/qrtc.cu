// Blocked Householder QR and Q application whose dense products run on the
// tensor cores (tc.cu), for the mixed-precision rounding.
//
// The right-to-left sweep and the truncation sweep (App. A, Alg. 1/2
// mirrored, with Alg. 4's factor-then-SVD structure) spend their time in
// QR factorisations of tall flattenings, m x K with m = n p up to 49152 and
// K = 6 r = 384.  Here the columns are taken in outer panels of width
// kOuter = 128:
//   1. the panel is factored by the cooperative Householder kernel (qr.cu,
//      double-float arithmetic, FP64 scalars), leaving reflectors V (unit
//      lower trapezoidal) and tau;
//   2. the panel's Gram G = V^H V is formed on the tensor cores; with
//      D = diag(1/tau), T^{-1} = D + striu(G) is the triangular factor of the
//      compact WY form H_0 ... H_{b-1} = I - V T V^H;
//   3. the trailing columns A_t receive Q^H: W = V^H A_t (tensor cores,
//      split over the m rows in exact chunks), W2 = T^H W (forward
//      substitution on D-bar + striu(G)^H, FP64), A_t -= V W2 (tensor cores).
// Applying Q = H_0 ... H_{p-1} (ormqr_tc) walks the panels backwards with
// W2 = T W (back substitution on D + striu(G)).  G of every panel is kept
// by the caller between the two.
#include <algorithm>

#include "kernels.h"

namespace hk {

namespace {

constexpr int kOuter = 128;

// W2 = T^H W (forward) or T W (backward) for the compact WY factor given by
// G (v_s^H v_u in G[s + ldg u]; Hermitian) and tau: one warp per column l
// of W (nbk x nt, ldw), each lane holding rows s = lane + 32 q.  The
// recurrence runs in double-float arithmetic on the FP32 pipe (a chain of
// FP64 multiply-adds waits on this GPU's narrow FP64 pipe at every step);
// its ~2^-48 relative rounding is far below the tensor-core products'
// error.  The triangle of G it reads and tau are packed once per panel
// (wy_pack_kernel: negated, in double-float form, column u of the triangle
// holding -G[s, u] for s > u (forward) or s < u (backward)) and copied into
// shared memory by every CTA (the solve is a chain of nbk dependent steps;
// each step then reads shared memory, not L2).
constexpr int kWyWarps = 4;

DV int wy_off(int u, int nbk, int forward) {  // packed offset of column u
  return forward ? u * (2 * nbk - u - 1) / 2 : u * (u - 1) / 2;
}
HD size_t wy_packed_elems(int nbk) { return (size_t)nbk * (nbk - 1) / 2 + nbk; }

__global__ void wy_pack_kernel(const cplx* G, int ldg, const cplx* tau, int nbk, int forward, df2* packed) {
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= nbk * nbk) return;
  const int s = idx % nbk, u = idx / nbk;
  if (forward ? s > u : s < u) {
    const cplx gv = G[s + (size_t)ldg * u];
    packed[wy_off(u, nbk, forward) + (forward ? s - u - 1 : s)] = df_from(mk(-gv.x, -gv.y));
  }
  // forward: w2_u = conj(tau_u) (...); backward: w2_u = tau_u (...)
  if (s == u) packed[(size_t)nbk * (nbk - 1) / 2 + u] = df_from(forward ? cconj(tau[u]) : tau[u]);
}

__global__ void __launch_bounds__(32 * kWyWarps)
    wy_solve_kernel(const df2* packed, int nbk, const cplx* W, int ldw, int nt, cplx* W2, int ldw2, int forward) {
  extern __shared__ __align__(16) unsigned char wy_raw[];
  df2* tri = reinterpret_cast<df2*>(wy_raw);  // nbk (nbk - 1) / 2 packed
  df2* tsh = tri + (size_t)nbk * (nbk - 1) / 2;
  auto off = [&](int u) -> int { return wy_off(u, nbk, forward); };
  {
    // coalesced 16-byte loads, eight in flight per thread
    const float4* src = reinterpret_cast<const float4*>(packed);
    float4* dst = reinterpret_cast<float4*>(wy_raw);
    const int n16 = (int)wy_packed_elems(nbk);
    constexpr int U = 8;
    for (int e0 = threadIdx.x; e0 < n16; e0 += U * blockDim.x) {
      float4 v[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int e = e0 + u * blockDim.x;
        if (e < n16) v[u] = __ldg(src + e);
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int e = e0 + u * blockDim.x;
        if (e < n16) dst[e] = v[u];
      }
    }
  }
  __syncthreads();
  const int lane = threadIdx.x & 31;
  const int l = blockIdx.x * kWyWarps + (threadIdx.x >> 5);
  if (l >= nt) return;
  constexpr int Q = kOuter / 32;
  // the column scaled by a power of two to a maximum below one (the FP32
  // exponent range of the double-float parts is then never left; W2 = T^H W
  // is linear in W, so the scale comes back exactly at the end)
  cplx wv[Q];
  double mx = 0.0;
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    const int s = lane + 32 * q;
    wv[q] = (s < nbk) ? W[s + (size_t)ldw * l] : mk(0, 0);
    mx = fmax(mx, fmax(fabs(wv[q].x), fabs(wv[q].y)));
  }
  for (int o = 16; o >= 1; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  const int E = (mx > 0.0) ? ilogb(mx) + 1 : 0;
  df2 acc[Q], mine[Q];
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    acc[q] = df_from(mk(scalbn(wv[q].x, -E), scalbn(wv[q].y, -E)));
    mine[q] = df_zero();
  }
  for (int step = 0; step < nbk; ++step) {
    const int u = forward ? step : nbk - 1 - step;
    const int qu = u >> 5, lu = u & 31;
    df2 own = df_zero();
#pragma unroll
    for (int q = 0; q < Q; ++q)
      if (q == qu) own = acc[q];
    df2 w2 = df_zero();
    df_cmac(w2, tsh[u], own);  // valid on lane lu
    w2 = df2{__shfl_sync(0xffffffffu, w2.rh, lu), __shfl_sync(0xffffffffu, w2.ih, lu),
             __shfl_sync(0xffffffffu, w2.rl, lu), __shfl_sync(0xffffffffu, w2.il, lu)};
    if (lane == lu) {
#pragma unroll
      for (int q = 0; q < Q; ++q)
        if (q == qu) mine[q] = w2;
    }
    const df2* col = tri + off(u);
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      const int s = lane + 32 * q;
      if (s >= nbk) continue;
      // forward: (T^-H)[s, u] = conj(G[u, s]) = G[s, u] for s > u
      if (forward && s > u) df_cmac(acc[q], col[s - u - 1], w2);
      else if (!forward && s < u) df_cmac(acc[q], col[s], w2);
    }
  }
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    const int s = lane + 32 * q;
    if (s < nbk) {
      const cplx v = df_to(mine[q]);
      W2[s + (size_t)ldw2 * l] = mk(scalbn(v.x, E), scalbn(v.y, E));
    }
  }
}

// `packed` holds wy_packed_elems(nbk) double-float values of scratch.
cudaError_t wy_solve(const cplx* G, int ldg, const cplx* tau, int nbk, const cplx* W, int ldw, int nt, cplx* W2,
                     int ldw2, int forward, df2* packed, cudaStream_t s) {
  if (nt <= 0) return cudaSuccess;
  const size_t smem = sizeof(df2) * wy_packed_elems(nbk);
  static cudaError_t attr = cudaFuncSetAttribute(wy_solve_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                 (int)(sizeof(df2) * wy_packed_elems(kOuter)));
  if (attr != cudaSuccess) return attr;
  wy_pack_kernel<<<(nbk * nbk + 255) / 256, 256, 0, s>>>(G, ldg, tau, nbk, forward, packed);
  wy_solve_kernel<<<(nt + kWyWarps - 1) / kWyWarps, 32 * kWyWarps, smem, s>>>(packed, nbk, W, ldw, nt, W2, ldw2,
                                                                             forward);
  return cudaGetLastError();
}

// G[s, u] <- conj(G[u, s]) for s > u: the Gram exactly Hermitian, so that
// the forward solve (which reads the lower triangle, contiguous across the
// lanes) and the backward solve (the upper one) use the same numbers.
__global__ void hermitize_kernel(cplx* G, int ldg, int nb) {
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= nb * nb) return;
  const int s = idx % nb, u = idx / nb;
  if (s > u) G[s + (size_t)ldg * u] = cconj(G[u + (size_t)ldg * s]);
}

// Carves the scratch for one panel step out of ws.
struct Carve {
  unsigned char* p;
  size_t left;
  bool ok = true;
  void* take(size_t bytes) {
    bytes = (bytes + 255) & ~(size_t)255;
    if (bytes > left) {
      ok = false;
      return nullptr;
    }
    void* r = p;
    p += bytes;
    left -= bytes;
    return r;
  }
};

}  // namespace

int tc_outer_panel() { return kOuter; }

bool qr_tc_applies(int m, int p) { return m >= 4096 && p > 32; }

size_t qr_tc_scratch_bytes(int m, int k, int S) {
  const int Kc = tc_chunk(S);
  const int nt = std::max(k, 1);
  size_t b = 0;
  auto add = [&](size_t x) { b += (x + 255) & ~(size_t)255; };
  add(tc_operand_bytes(kOuter, m, S, Kc));  // V^H
  add(tc_operand_bytes(kOuter, m, S, Kc));  // V (as the Gram's second operand)
  add(tc_operand_bytes(nt, m, S, Kc));      // trailing columns / C
  add(tc_operand_bytes(m, kOuter, S, Kc));  // V
  add(tc_operand_bytes(nt, kOuter, S, Kc)); // W2
  add(std::max(tc_part_elems(kOuter, nt, m, S), tc_part_elems(kOuter, kOuter, m, S)) * sizeof(cplx));
  add((size_t)kOuter * nt * sizeof(cplx) * 2);  // W, W2
  add(wy_packed_elems(kOuter) * sizeof(df2));   // packed WY triangle
  return b + 1024;
}

size_t qr_tc_gram_elems(int k) { return (size_t)((k + kOuter - 1) / kOuter) * kOuter * kOuter; }

// Complex GEMM FLOPs (8 per complex multiply-add) of an M x N x K product.
static double zflops(double M, double N, double K) { return 8.0 * M * N * K; }

cudaError_t geqrf_tc(cplx* A, int lda, int m, int k, cplx* tau, cplx* Gout, void* scratch,
                     size_t scratch_bytes, const CoopWs& cws, int S, cudaStream_t s, const PhaseTimer& pt) {
  const int p = std::min(m, k);
  const int Kc = tc_chunk(S);
  cudaError_t e = cudaSuccess;
  for (int j0 = 0; j0 < p && e == cudaSuccess; j0 += kOuter) {
    const int nbk = std::min(kOuter, p - j0);
    const int mv = m - j0;
    cplx* Ap = A + j0 + (size_t)lda * j0;
    int nb = 32;
    int slot = pt.b();
    // without the record of the 32-column blocks: G below takes its place, and
    // the kernel leaves the last block's products and their barriers out
    e = geqrf(Ap, lda, mv, nbk, tau + j0, nullptr, &nb, cws, s, kQrMixed);
    pt.e(slot, pt.cls_panel, 8.0 * mv * (double)nbk * nbk - 8.0 * (double)nbk * nbk * nbk / 3.0, 1);
    if (e != cudaSuccess) break;
    Carve c{static_cast<unsigned char*>(scratch), scratch_bytes};
    void* bVH = c.take(tc_operand_bytes(nbk, mv, S, Kc));
    void* bVB = c.take(tc_operand_bytes(nbk, mv, S, Kc));
    const int nt = k - j0 - nbk;
    void* bX = c.take(tc_operand_bytes(std::max(nt, 1), mv, S, Kc));
    void* bV = c.take(tc_operand_bytes(mv, nbk, S, Kc));
    void* bW2 = c.take(tc_operand_bytes(std::max(nt, 1), nbk, S, Kc));
    const size_t npart = std::max(tc_part_elems(nbk, std::max(nt, 1), mv, S), tc_part_elems(nbk, nbk, mv, S));
    cplx* part = static_cast<cplx*>(c.take(npart * sizeof(cplx)));
    cplx* W = static_cast<cplx*>(c.take((size_t)nbk * std::max(nt, 1) * sizeof(cplx)));
    cplx* W2 = static_cast<cplx*>(c.take((size_t)nbk * std::max(nt, 1) * sizeof(cplx)));
    df2* packed = static_cast<df2*>(c.take(wy_packed_elems(nbk) * sizeof(df2)));
    if (!c.ok) return cudaErrorInvalidValue;
    // G = V^H V (reflector s along rows, entries i along K)
    TcOperand oVH, oVB, oX, oV, oW2;
    slot = pt.b();
    e = tc_split2(TcOperandView{Ap, lda, 1, nbk, mv, 1, 2, 0}, &oVH, bVH,
                  TcOperandView{Ap, lda, 1, nbk, mv, 0, 2, 0}, &oVB, bVB, S, s);
    cplx* G = Gout + (size_t)(j0 / kOuter) * kOuter * kOuter;
    if (e == cudaSuccess) e = tc_zgemm(oVH, oVB, G, 1, kOuter, 1.0, 0, part, npart, &cws.bar->err, s);
    if (e == cudaSuccess) {
      hermitize_kernel<<<(nbk * nbk + 255) / 256, 256, 0, s>>>(G, kOuter, nbk);
      e = cudaGetLastError();
    }
    // launches: the splits, the product, its chunk reduction (K > one chunk), hermitize
    pt.e(slot, pt.cls_tc, zflops(nbk, nbk, mv), 3 + (mv > Kc));
    if (e != cudaSuccess || nt <= 0) continue;
    // trailing columns: W = V^H A_t, W2 = T^H W, A_t -= V W2
    cplx* At = A + j0 + (size_t)lda * (j0 + nbk);
    slot = pt.b();
    e = tc_split(TcOperandView{At, lda, 1, nt, mv, 0, 0, 0}, S, &oX, bX, s);
    if (e == cudaSuccess) e = tc_zgemm(oVH, oX, W, 1, nbk, 1.0, 0, part, npart, &cws.bar->err, s);
    pt.e(slot, pt.cls_tc, zflops(nbk, nt, mv), 2 + (mv > Kc));
    slot = pt.b();
    if (e == cudaSuccess) e = wy_solve(G, kOuter, tau + j0, nbk, W, nbk, nt, W2, nbk, 1, packed, s);
    pt.e(slot, pt.cls_small, 0.0, 2);  // pack + solve
    slot = pt.b();
    if (e == cudaSuccess)
      e = tc_split2(TcOperandView{W2, nbk, 1, nt, nbk, 0, 0, 0}, &oW2, bW2,
                  TcOperandView{Ap, 1, lda, mv, nbk, 0, 3, 0}, &oV, bV, S, s);
    if (e == cudaSuccess) e = tc_zgemm(oV, oW2, At, 1, lda, -1.0, 1, nullptr, 0, &cws.bar->err, s);
    pt.e(slot, pt.cls_tc, zflops(mv, nt, nbk), 2);  // the splits, one chunk
  }
  return e;
}

cudaError_t ormqr_tc(const cplx* A, int lda, int m, int p, const cplx* tau, const cplx* Gin, cplx* C, int ldc, int q,
                     void* scratch, size_t scratch_bytes, int* err, int S, cudaStream_t s, const PhaseTimer& pt) {
  if (m <= 0 || p <= 0 || q <= 0) return cudaSuccess;
  const int Kc = tc_chunk(S);
  const int npanel = (p + kOuter - 1) / kOuter;
  cudaError_t e = cudaSuccess;
  for (int j = npanel - 1; j >= 0 && e == cudaSuccess; --j) {
    const int j0 = j * kOuter, nbk = std::min(kOuter, p - j0), mv = m - j0;
    const cplx* Ap = A + j0 + (size_t)lda * j0;
    cplx* Cj = C + j0;
    Carve c{static_cast<unsigned char*>(scratch), scratch_bytes};
    void* bVH = c.take(tc_operand_bytes(nbk, mv, S, Kc));
    void* bX = c.take(tc_operand_bytes(q, mv, S, Kc));
    void* bV = c.take(tc_operand_bytes(mv, nbk, S, Kc));
    void* bW2 = c.take(tc_operand_bytes(q, nbk, S, Kc));
    const size_t npart = tc_part_elems(nbk, q, mv, S);
    cplx* part = static_cast<cplx*>(c.take(std::max<size_t>(npart, 1) * sizeof(cplx)));
    cplx* W = static_cast<cplx*>(c.take((size_t)nbk * q * sizeof(cplx)));
    cplx* W2 = static_cast<cplx*>(c.take((size_t)nbk * q * sizeof(cplx)));
    df2* packed = static_cast<df2*>(c.take(wy_packed_elems(nbk) * sizeof(df2)));
    if (!c.ok) return cudaErrorInvalidValue;
    TcOperand oVH, oX, oV, oW2;
    int slot = pt.b();
    e = tc_split2(TcOperandView{Ap, lda, 1, nbk, mv, 1, 2, 0}, &oVH, bVH,
                  TcOperandView{Cj, ldc, 1, q, mv, 0, 0, 0}, &oX, bX, S, s);
    if (e == cudaSuccess) e = tc_zgemm(oVH, oX, W, 1, nbk, 1.0, 0, part, npart, err, s);
    pt.e(slot, pt.cls_tc, zflops(nbk, q, mv), 2 + (mv > Kc));
    slot = pt.b();
    if (e == cudaSuccess)
      e = wy_solve(Gin + (size_t)j * kOuter * kOuter, kOuter, tau + j0, nbk, W, nbk, q, W2, nbk, 0, packed, s);
    pt.e(slot, pt.cls_small, 0.0, 2);
    slot = pt.b();
    if (e == cudaSuccess)
      e = tc_split2(TcOperandView{W2, nbk, 1, q, nbk, 0, 0, 0}, &oW2, bW2,
                  TcOperandView{Ap, 1, lda, mv, nbk, 0, 3, 0}, &oV, bV, S, s);
    if (e == cudaSuccess) e = tc_zgemm(oV, oW2, Cj, 1, ldc, -1.0, 1, nullptr, 0, err, s);
    pt.e(slot, pt.cls_tc, zflops(mv, q, nbk), 2);
  }
  return e;
}

// ---- the same at FP64 accuracy ------------------------------------------------
namespace {

constexpr int kWidePanel = 32;

// W2 = T^H W (forward) or T W (backward) for a panel of at most 32 reflectors
// with Gram g (v_s^H v_u at g[s + nbk u]) and tau (NULL: g holds the panel's
// record instead, the strict upper triangle of the Gram with tau on the
// diagonal).  With t_s = conj(tau_s) (forward) or tau_s,
//   w2_s = t_s W_s - sum_u (t_s Gram[s, u]) w2_u
// over the u before s (forward) or after it: one warp per column, the scaled
// Gram in shared memory, so that a step of the chain is one exchange and one
// complex multiply-add (about 180 cycles).  The scaled Gram costs 2048 cycles
// of a CTA's FP64 unit and a load per entry: four warps load it with eight
// loads in flight each, and a CTA takes as many columns (four at most: their
// chains share the unit without waiting) as it needs for one CTA per SM.  With
// one warp per CTA loading entry after entry the kernel took 18.6 us, the
// 32 load latencies alone 10.  rec (may be NULL) receives the record.
constexpr int kWy64Cols = 4;  // warps, and columns at most, per CTA
__global__ void __launch_bounds__(32 * kWy64Cols)
wy_solve64_kernel(const cplx* __restrict__ g, const cplx* __restrict__ tau, int nbk, const cplx* __restrict__ W, int nt,
                  int cols, cplx* __restrict__ W2, int forward, cplx* __restrict__ rec) {
  // m[u * 33 + s] = -t_s Gram[s, u] for the pairs of the chain, else zero
  __shared__ cplx m[kWidePanel * (kWidePanel + 1)];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, l = blockIdx.x * cols + wid;
  const bool in = lane < nbk, mine = wid < cols && l < nt;
  const cplx tl = in ? (tau ? tau[lane] : g[lane + nbk * lane]) : mk(0, 0);
  const cplx wl = in && mine ? W[lane + (size_t)nbk * l] : mk(0, 0);
  const cplx t = forward ? cconj(tl) : tl;
  constexpr int Q = kWidePanel / kWy64Cols;
  cplx gv[Q];
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    // stored pair (min, max): Gram[s, u] itself for s < u, its conjugate else
    const int u = wid + kWy64Cols * q, lo = min(lane, u), hi = max(lane, u);
    gv[q] = in && u < nbk && u != lane ? g[lo + nbk * hi] : mk(0, 0);
  }
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    const int u = wid + kWy64Cols * q;
    cplx v = mk(0, 0);
    if (forward ? lane > u : lane < u) {
      const cplx p = cmul(t, forward ? cconj(gv[q]) : gv[q]);
      v = mk(-p.x, -p.y);
    }
    m[u * (kWidePanel + 1) + lane] = v;
    if (rec && blockIdx.x == 0 && in && u < nbk) rec[lane + nbk * u] = lane < u ? gv[q] : (lane == u ? tl : mk(0, 0));
  }
  __syncthreads();
  if (!mine) return;
  cplx acc = cmul(t, wl);
  for (int step = 0; step < nbk; ++step) {
    const int u = forward ? step : nbk - 1 - step;
    const cplx w = mk(__shfl_sync(0xffffffffu, acc.x, u), __shfl_sync(0xffffffffu, acc.y, u));
    acc = cfma(m[u * (kWidePanel + 1) + lane], w, acc);
  }
  if (in) W2[lane + (size_t)nbk * l] = acc;
}

cudaError_t wy_solve64(const cplx* g, const cplx* tau, int nbk, const cplx* W, int nt, cplx* W2, int forward, cplx* rec,
                       cudaStream_t s) {
  if (nt <= 0 && !rec) return cudaSuccess;
  const int sms = dev_info().sm_count, cols = std::min(kWy64Cols, std::max(1, (nt + sms - 1) / sms));
  wy_solve64_kernel<<<std::max(1, (nt + cols - 1) / cols), 32 * kWy64Cols, 0, s>>>(g, tau, nbk, W, nt, cols, W2, forward,
                                                                                  rec);
  return cudaGetLastError();
}

}  // namespace

// The panel kernel's own trailing update costs 16 m 32 FP64 operations per
// trailing column on all SMs together (1.1 TFLOP/s), the products about 100 us
// per panel in launches whatever the size.  Measured with both sides: from
// 2048 rows the products are ahead as soon as there is a second panel, from
// 1024 rows with two full panels (C2 steps 351 -> 345 ms, C3 278 -> 263 ms, the CDF
// workload's LQ factors 311 -> 265 ms); below that the C1 factors (336 x 96)
// are faster on the kernel alone.
bool qr_wide_applies(int m, int p) { return (m >= 2048 && p > kWidePanel) || (m >= 1024 && p >= 2 * kWidePanel); }

size_t qr_wide_scratch_bytes(int m, int k) {
  const int S = tc_wide_digits(), Kc = tc_chunk(S), nb = kWidePanel;
  size_t b = 0;
  auto add = [&](size_t x) { b += (x + 255) & ~(size_t)255; };
  add(tc_operand_bytes(nb, m, S, Kc));      // conj(V)
  add(tc_operand_bytes(k + nb, m, S, Kc));  // [V | trailing columns] / C
  add(tc_operand_bytes(m, nb, S, Kc));      // V
  add(tc_operand_bytes(std::max(k, 1), nb, S, Kc));  // W2
  add(tc_part_elems(k + nb, nb, m, S) * sizeof(cplx));
  add((size_t)nb * (k + nb) * sizeof(cplx));  // Gram and W
  add((size_t)nb * std::max(k, 1) * sizeof(cplx));
  return b + 1024;
}

cudaError_t geqrf_wide(cplx* A, int lda, int m, int k, cplx* tau, cplx* T, void* scratch, size_t scratch_bytes,
                       const CoopWs& cws, cudaStream_t s, const PhaseTimer& pt) {
  const int S = tc_wide_digits(), Kc = tc_chunk(S);
  const int p = std::min(m, k);
  cudaError_t e = cudaSuccess;
  for (int j0 = 0; j0 < p && e == cudaSuccess; j0 += kWidePanel) {
    const int nbk = std::min(kWidePanel, p - j0), mv = m - j0, nt = k - j0 - nbk;
    cplx* Ap = A + j0 + (size_t)lda * j0;
    int nb = kWidePanel;
    int slot = pt.b();
    e = geqrf(Ap, lda, mv, nbk, tau + j0, nullptr, &nb, cws, s, kQrFp64);
    pt.e(slot, pt.cls_panel, 8.0 * mv * (double)nbk * nbk - 8.0 * (double)nbk * nbk * nbk / 3.0, 1);
    if (e != cudaSuccess || (nt <= 0 && !T)) continue;
    Carve c{static_cast<unsigned char*>(scratch), scratch_bytes};
    void* bVH = c.take(tc_operand_bytes(nbk, mv, S, Kc));
    void* bX = c.take(tc_operand_bytes(nbk + nt, mv, S, Kc));
    void* bV = c.take(tc_operand_bytes(mv, nbk, S, Kc));
    void* bW2 = c.take(tc_operand_bytes(std::max(nt, 1), nbk, S, Kc));
    const size_t npart = tc_part_elems(nbk + nt, nbk, mv, S);
    cplx* part = static_cast<cplx*>(c.take(std::max<size_t>(npart, 1) * sizeof(cplx)));
    cplx* GW = static_cast<cplx*>(c.take((size_t)nbk * (nbk + nt) * sizeof(cplx)));
    cplx* W2 = static_cast<cplx*>(c.take((size_t)nbk * std::max(nt, 1) * sizeof(cplx)));
    if (!c.ok) return cudaErrorInvalidValue;
    // [G | W] = V^H [V | A_t], rows l of the product are the columns on the
    // right (128 to a tile), the reflectors its 32 columns
    TcOperand oVH, oX, oV, oW2;
    slot = pt.b();
    e = tc_split2(TcOperandView{Ap, lda, 1, nbk, mv, 1, 2, 0}, &oVH, bVH,
                  TcOperandView{Ap, lda, 1, nbk + nt, mv, 0, 4, nbk}, &oX, bX, S, s);
    if (e == cudaSuccess) e = tc_zgemm(oX, oVH, GW, nbk, 1, 1.0, 0, part, npart, &cws.bar->err, s);
    pt.e(slot, pt.cls_tc, zflops(nbk, nbk + nt, mv), 2 + (mv > Kc));
    slot = pt.b();
    cplx* rec = T ? T + (size_t)(j0 / kWidePanel) * kWidePanel * kWidePanel : nullptr;
    if (e == cudaSuccess) e = wy_solve64(GW, tau + j0, nbk, GW + (size_t)nbk * nbk, nt, W2, 1, rec, s);
    pt.e(slot, pt.cls_small, 0.0, 1);
    if (e != cudaSuccess || nt <= 0) continue;
    cplx* At = A + j0 + (size_t)lda * (j0 + nbk);
    slot = pt.b();
    e = tc_split2(TcOperandView{W2, nbk, 1, nt, nbk, 0, 0, 0}, &oW2, bW2,
                  TcOperandView{Ap, 1, lda, mv, nbk, 0, 3, 0}, &oV, bV, S, s);
    if (e == cudaSuccess) e = tc_zgemm(oV, oW2, At, 1, lda, -1.0, 1, nullptr, 0, &cws.bar->err, s);
    pt.e(slot, pt.cls_tc, zflops(mv, nt, nbk), 2);
  }
  return e;
}

cudaError_t ormqr_wide(const cplx* A, int lda, int m, int p, const cplx* T, cplx* C, int ldc, int q, void* scratch,
                       size_t scratch_bytes, int* err, cudaStream_t s, const PhaseTimer& pt) {
  if (m <= 0 || p <= 0 || q <= 0) return cudaSuccess;
  const int S = tc_wide_digits(), Kc = tc_chunk(S);
  const int npanel = (p + kWidePanel - 1) / kWidePanel;
  cudaError_t e = cudaSuccess;
  for (int j = npanel - 1; j >= 0 && e == cudaSuccess; --j) {
    const int j0 = j * kWidePanel, nbk = std::min(kWidePanel, p - j0), mv = m - j0;
    const cplx* Ap = A + j0 + (size_t)lda * j0;
    cplx* Cj = C + j0;
    Carve c{static_cast<unsigned char*>(scratch), scratch_bytes};
    void* bVH = c.take(tc_operand_bytes(nbk, mv, S, Kc));
    void* bX = c.take(tc_operand_bytes(q, mv, S, Kc));
    void* bV = c.take(tc_operand_bytes(mv, nbk, S, Kc));
    void* bW2 = c.take(tc_operand_bytes(q, nbk, S, Kc));
    const size_t npart = tc_part_elems(q, nbk, mv, S);
    cplx* part = static_cast<cplx*>(c.take(std::max<size_t>(npart, 1) * sizeof(cplx)));
    cplx* W = static_cast<cplx*>(c.take((size_t)nbk * q * sizeof(cplx)));
    cplx* W2 = static_cast<cplx*>(c.take((size_t)nbk * q * sizeof(cplx)));
    if (!c.ok) return cudaErrorInvalidValue;
    TcOperand oVH, oX, oV, oW2;
    int slot = pt.b();
    e = tc_split2(TcOperandView{Ap, lda, 1, nbk, mv, 1, 2, 0}, &oVH, bVH,
                  TcOperandView{Cj, ldc, 1, q, mv, 0, 0, 0}, &oX, bX, S, s);
    if (e == cudaSuccess) e = tc_zgemm(oX, oVH, W, nbk, 1, 1.0, 0, part, npart, err, s);
    pt.e(slot, pt.cls_tc, zflops(nbk, q, mv), 2 + (mv > Kc));
    slot = pt.b();
    if (e == cudaSuccess)
      e = wy_solve64(T + (size_t)j * kWidePanel * kWidePanel, nullptr, nbk, W, q, W2, 0, nullptr, s);
    pt.e(slot, pt.cls_small, 0.0, 1);
    slot = pt.b();
    if (e == cudaSuccess)
      e = tc_split2(TcOperandView{W2, nbk, 1, q, nbk, 0, 0, 0}, &oW2, bW2,
                  TcOperandView{Ap, 1, lda, mv, nbk, 0, 3, 0}, &oV, bV, S, s);
    if (e == cudaSuccess) e = tc_zgemm(oV, oW2, Cj, 1, ldc, -1.0, 1, nullptr, 0, err, s);
    pt.e(slot, pt.cls_tc, zflops(mv, q, nbk), 2);
  }
  return e;
}

}  // namespace hk
