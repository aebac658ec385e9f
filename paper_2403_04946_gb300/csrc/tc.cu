// Complex products on the tensor cores (tcgen05) with FP64-class accuracy.
//
// The mixed-precision rounding (App. A, Alg. 2 / Alg. 4: the QR trailing
// updates, the Q applications and the merges of the orthogonalisation sweep)
// needs products accurate to about 1e-12 of |A||B|, far beyond one BF16 or
// TF32 product.  Each operand is therefore cut into S digit planes
// (Ozaki-style splitting): per row r and per K-chunk, a power-of-two scale
// 2^e[r] brings the row below 1 in magnitude, and
//     x 2^-e = sum_j q_j 2^(-7-8j),   q_j integers with |q_j| <= 128,
// each q_j exactly representable in BF16.  A product of two digits is an
// integer below 2^14 in magnitude, so a K-chunk of at most 192 products per
// digit pair, summed over the pairs (i, j) of one level L = i + j (L + 1 <= 5
// pairs), stays below 2^24: the FP32 accumulation in tensor memory is exact.
// Levels L < S are kept (S (S + 1) / 2 digit products per real product); the
// dropped pairs weigh about S 2^(-8S) of |A||B| (5 digits: ~5e-12).
//
// Complex products use three real products (3M):
//     T1 = Ar Br,  T2 = Ai Bi,  T3 = (Ar + Ai)(Br + Bi),
//     C = (T1 - T2) + i (T3 - T1 - T2),
// each of Ar, Ai, Ar + Ai (and the same for B) split with its own scales.
//
// The product kernel: one CTA per 128 x 32 output tile and K-chunk.  Warp 8
// streams digit slabs (64 K-values, 128 B per row, 128-byte swizzle) into a
// two-stage shared-memory ring with TMA (cp.async.bulk.tensor); warp 9 issues
// tcgen05.mma (kind::f16, BF16 x BF16 -> FP32) into 15 accumulators
// (3 products x 5 levels x 32 columns) in tensor memory, one MMA per A digit
// plane covering all its levels; warps 0-7 (two per tensor-memory lane
// quadrant, 16 columns each) read the accumulators back (tcgen05.ld),
// combine levels, scales and the 3M terms in double-float, and write the
// complex result (overwritten, added, or as a per-chunk partial that a
// reduction kernel sums in a fixed order).
//
// Every wait is bounded (2 s of wall time): on expiry the kernel records
// the error in the grid-barrier record the host checks (HOPF_ETIMEOUT),
// stops issuing work, waits (bounded) for what it issued, frees its tensor
// memory and returns.
#include <cuda.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <mutex>

#include "kernels.h"
#include "tcgen05.cuh"

namespace hk {

namespace {

constexpr int kTcM = 128;        // rows of an output tile (one TMEM lane each)
constexpr int kTcN = 32;         // columns of an output tile
constexpr int kSlab = 64;        // K-values per digit slab (128 bytes of BF16)
constexpr int kMaxDigits = 5;    // 3 products x 5 levels x 32 columns = 480 TMEM columns
constexpr int kWideDigits = 8;   // FP64 products (tc_zgemm_wide_kernel): 63 bits per operand row
constexpr int kTmemCols = 512;
constexpr int kStages = 2;
constexpr int kTcThreads = 320;  // warps 0-7 epilogue, 8 producer, 9 MMA
constexpr uint64_t kWaitNs = kTcWaitNs;
static_assert(kTmaSlab == 64, "digit slabs are one 128-byte TMA box row");

__host__ __device__ constexpr int a_plane_bytes() { return kTcM * kSlab * 2; }  // 16 KB
__host__ __device__ constexpr int b_plane_bytes() { return kTcN * kSlab * 2; }  // 4 KB
__host__ __device__ int stage_bytes(int S) { return S * (a_plane_bytes() + b_plane_bytes()); }
size_t tc_smem_bytes(int S) { return (size_t)kStages * stage_bytes(S) + 1024; }



struct TcArgs {
  int M, N, K, S, Kc, nchunks;
  const int* eA;  // [3][nchunks][M] scale exponents of the A digits
  const int* eB;  // [3][nchunks][N]
  cplx* out;      // out[z * zstride + m + ldo * n]
  long long ldo, zstride;
  long long rso;  // wide kernel: out[z * zstride + rso * m + ldo * n]
  int alpha_exp, alpha_neg;  // alpha = (-1)^alpha_neg 2^alpha_exp: out = alpha * result (+ out if accumulate)
  int accumulate;
  int* err;       // expiry record (the context's grid-barrier err field)
  int n_first;    // this launch's columns begin here, those of out with them
};

__global__ void __launch_bounds__(kTcThreads, 1)
    tc_zgemm_kernel(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapB, TcArgs a) {
  extern __shared__ unsigned char smem_raw[];
  __shared__ __align__(8) uint64_t full_bar[kStages], empty_bar[kStages], acc_bar;
  __shared__ uint32_t tmem_slot;
  __shared__ int abort_flag;
  __shared__ int eb_sh[3][kTcN];
  // 1024-byte aligned stage ring (the swizzle atoms need it)
  unsigned char* smem =
      reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  const int S = a.S;
  const int sbytes = stage_bytes(S);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // N-tiles fastest: the CTAs that share an A-tile (the large digit planes)
  // run together and find it in L2
  const int m0 = blockIdx.y * kTcM, n0 = a.n_first + blockIdx.x * kTcN, z = blockIdx.z;
  const int k_begin = z * a.Kc;
  const int k_len = min(a.Kc, a.K - k_begin);
  const int nslab = (k_len + kSlab - 1) / kSlab;
  const int nstage = 3 * nslab;  // (slab, product) pairs

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(&full_bar[s], 1);
      mbar_init(&empty_bar[s], 1);
    }
    mbar_init(&acc_bar, 1);
    abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                 "r"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;
  volatile int* vabort = &abort_flag;

  if (warp == 8) {
    // ---- producer: one (slab, product) stage at a time ------------------
    if (lane == 0) {
      int issued = 0;
      for (int st = 0; st < nstage; ++st) {
        const int slot = st % kStages;
        if (st >= kStages && !mbar_wait(&empty_bar[slot], ((st / kStages) - 1) & 1, vabort, a.err)) break;
        const int c = st % 3, slab = st / 3;
        const int k0 = k_begin + slab * kSlab;
        unsigned char* base = smem + (size_t)slot * sbytes;
        mbar_expect_tx(&full_bar[slot], (uint32_t)sbytes);
        for (int j = 0; j < S; ++j) {
          tma_load_3d(base + (size_t)j * a_plane_bytes(), &mapA, &full_bar[slot], k0, m0, c * S + j);
          tma_load_3d(base + (size_t)S * a_plane_bytes() + (size_t)j * b_plane_bytes(), &mapB, &full_bar[slot], k0, n0,
                      c * S + j);
        }
        issued = st + 1;
      }
      // before leaving, every issued copy has landed (bounded): the stage
      // ring must not be written after the CTA exits
      for (int st = max(0, issued - kStages); st < issued; ++st) {
        uint64_t t0 = global_ns();
        while (!mbar_try_wait(&full_bar[st % kStages], (st / kStages) & 1))
          if (global_ns() - t0 > kWaitNs) break;
      }
    }
  } else if (warp == 9) {
    // ---- MMA issuer -------------------------------------------------------
    if (lane == 0) {
      for (int st = 0; st < nstage; ++st) {
        const int slot = st % kStages;
        if (!mbar_wait(&full_bar[slot], (st / kStages) & 1, vabort, a.err)) break;
        tc_fence_after();
        const int c = st % 3, slab = st / 3;
        const uint32_t abase = smem_u32(smem + (size_t)slot * sbytes);
        const uint64_t a0 = sw128_desc(abase), b0 = sw128_desc(abase + (uint32_t)(S * a_plane_bytes()));
        // A digit plane i against B planes 0 .. S-1-i in one product: the B
        // planes lie one after another (32 rows each), so together they are
        // one (S - i) x 32-row operand whose output columns are the level
        // accumulators L = i .. S-1, contiguous in tensor memory.  The
        // descriptors advance by adding the offset / 16 to their address
        // field (shared-memory addresses stay below 2^18).
        for (int i = 0; i < S; ++i) {
          const uint32_t acc = tmem + (uint32_t)((c * S + i) * kTcN);
          const uint32_t idesc = umma_idesc_bf16(kTcM, kTcN * (S - i));
#pragma unroll
          for (int kk = 0; kk < kSlab / 16; ++kk)
            umma(acc, a0 + (uint64_t)((i * a_plane_bytes() + kk * 32) >> 4), b0 + (uint64_t)(kk * 2), idesc,
                 (slab > 0 || i > 0 || kk > 0) ? 1u : 0u);
        }
        umma_commit(&empty_bar[slot]);  // the stage is free once these MMAs have read it
      }
      umma_commit(&acc_bar);  // all accumulators final (also after an abort)
    }
  } else {
    // ---- epilogue: warps 0-7, thread = output row of its lane quadrant ----
    // Every level accumulator is an exact FP32 integer; the levels, the
    // per-component scales and the 3M combination are summed in
    // double-float arithmetic on the FP32 pipe (error-free TwoSum steps),
    // and only the final value is converted to FP64 and scaled (on this GPU
    // the FP64 pipe is 1/64 of the FP32 one).
    // warp w reads tensor-memory lanes 32 (w % 4) .. +31 (its quadrant) and
    // columns 16 (w / 4) .. +15: two warps per quadrant share the rows
    const int quad = warp & 3, half = warp >> 2;
    const int m = m0 + 32 * quad + lane;
    cplx* out = a.out + z * a.zstride - a.ldo * a.n_first;
    // the tile's column exponents of B, staged while the MMAs run (named
    // barrier 1: the eight epilogue warps only)
    {
      const int t = threadIdx.x;
      if (t < 3 * kTcN) {
        const int c = t / kTcN, n = n0 + t % kTcN;
        eb_sh[c][t % kTcN] = (n < a.N) ? a.eB[(size_t)c * a.nchunks * a.N + (size_t)z * a.N + n] : 0;
      }
      asm volatile("bar.sync 1, 256;" ::: "memory");
    }
    // the values an accumulating product adds to, 8 columns at a time,
    // loaded ahead (independent loads in flight together): the first
    // quarter while the MMAs run, each next one before its accumulators are
    // read
    cplx pre[8];
    auto prefetch = [&](int h) {
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const int n = n0 + 8 * h + q;
        pre[q] = (a.accumulate && m < a.M && n < a.N) ? out[m + (size_t)a.ldo * n] : mk(0, 0);
      }
    };
    prefetch(2 * half);
    const bool ok = mbar_wait(&acc_bar, 0, vabort, a.err);
    tc_fence_after();
    if (ok && !*vabort) {
      const size_t eAs = (size_t)a.nchunks * a.M;
      int ea[3] = {0, 0, 0};
      if (m < a.M)
        for (int c = 0; c < 3; ++c) ea[c] = a.eA[c * eAs + (size_t)z * a.M + m];
      const uint32_t lane_base = tmem + ((uint32_t)(32 * quad) << 16);
#pragma unroll 1
      for (int h = 2 * half; h < 2 * half + 2; ++h) {
        if (h > 2 * half) prefetch(h);
        float th[3][8], tl[3][8];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          // all five level accumulators of product c (levels >= S are not
          // written by the MMAs and are skipped)
          float v[kMaxDigits][8];
          tmem_ld_levels8(lane_base + (uint32_t)(c * S * kTcN + 8 * h), v);
#pragma unroll
          for (int q = 0; q < 8; ++q) {
            th[c][q] = v[0][q] * pow2f(-14);  // exact: an integer below 2^24 times a power of two
            tl[c][q] = 0.f;
          }
#pragma unroll
          for (int L = 1; L < kMaxDigits; ++L) {
            if (L >= S) break;
            const float w = pow2f(-14 - 8 * L);
#pragma unroll
            for (int q = 0; q < 8; ++q) df_add_part(th[c][q], tl[c][q], v[L][q] * w, 0.f);
          }
        }
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          const int n = n0 + 8 * h + q;
          if (m >= a.M || n >= a.N) continue;
          int ex[3];
#pragma unroll
          for (int c = 0; c < 3; ++c) ex[c] = ea[c] + eb_sh[c][8 * h + q];
          const int E0 = max(ex[0], max(ex[1], ex[2]));
          // component values relative to 2^E0 (factors <= 1: exact scaling,
          // or below the double-float precision of the largest one)
          const float w0 = pow2f(ex[0] - E0), w1 = pow2f(ex[1] - E0), w2 = pow2f(ex[2] - E0);
          float h0 = th[0][q] * w0, l0 = tl[0][q] * w0;
          float h1 = th[1][q] * w1, l1 = tl[1][q] * w1;
          float h2 = th[2][q] * w2, l2 = tl[2][q] * w2;
          // re = T1 - T2, im = T3 - T1 - T2
          float rh = h0, rl = l0;
          df_add_part(rh, rl, -h1, -l1);
          float ih = h2, il = l2;
          df_add_part(ih, il, -h0, -l0);
          df_add_part(ih, il, -h1, -l1);
          // hi 2^E0 + lo 2^E0 as doubles built from the FP32 bit patterns
          // (exponent rebias plus E0 by integer arithmetic): one FP64
          // addition per part
          const int Es = E0 + a.alpha_exp;
          cplx r = mk(f2d_scaled(rh, Es, a.alpha_neg) + f2d_scaled(rl, Es, a.alpha_neg),
                      f2d_scaled(ih, Es, a.alpha_neg) + f2d_scaled(il, Es, a.alpha_neg));
          if (a.accumulate) r = cadd(pre[q], r);
          out[m + (size_t)a.ldo * n] = r;
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
  }
}

// ---- products at FP64 accuracy -----------------------------------------------
// The same product from kWideDigits = 8 digits per operand (63 bits below the
// row's power of two: every bit of entries down to 2^-10 of the row's largest;
// the dropped pairs weigh 8 2^-64 of |A||B|), so that the FP64 path's
// contractions leave the FP64 units, 1/800 of the tensor pipe.  (With seven
// digits a C2 step was 28 times further from a 64-bit reference than FP64
// products: the entries of a K-chunk decay, and the digits count from the
// largest.)  36 digit pairs per real product; a level sums at most 8 pairs, so
// a K-chunk of 128 stays within 8 2^7 2^14 = 2^24: exact.
//
// 8 levels x 32 columns are 256 tensor-memory columns, two of the three 3M
// products at a time: product c accumulates in half c mod 2 while the
// epilogue reads the previous one, the third waits until the first is read.
// A stage of all 8 + 8 planes would be 160 KB, so the ring holds single A
// planes (16 KB, nine of them) beside two sets of B planes (32 KB, one per
// K-slab); A plane i meets B planes 0 .. 7-i in one MMA of N = 32 (8 - i).
// The epilogue sums the integer levels exactly (64 + 16 bits), aligns the three
// products on the largest, combines them as integers and rounds once to FP64:
// no FP64 instruction but the addition to an accumulated output.  The component re + im of an operand is summed as
// fixed-point integers as well (split_kernel), not rounded to FP64 first.
constexpr int kWideA = 9;
constexpr int kWideChunk = 2 * kSlab;
__host__ __device__ constexpr int wide_b_bytes() { return kWideDigits * kTcN * kSlab * 2; }  // 32 KB
size_t wide_smem_bytes() { return (size_t)kWideA * a_plane_bytes() + 2 * wide_b_bytes() + 1024; }

DV void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// I 2^E as a double, rounded to nearest (ties away from zero), by integer
// arithmetic, over the whole range: gradual below 2^-1022, infinity from 2^1024.
// (The ends in a function of their own: inlined into the 32 values of a thread
// they cost the kernel a tenth of its time.)
__device__ __noinline__ double int_scaled_ends(long long I, int E) {
  const unsigned long long m0 = I < 0 ? 0ull - (unsigned long long)I : (unsigned long long)I;
  const unsigned long long sgn = I < 0 ? 1ull << 63 : 0ull;
  unsigned long long bits = 0x7FFull << 52;
  if (63 - __clzll((long long)m0) + E + 1023 <= 0) {  // units of 2^-1074: a carry into 2^-1022 comes out by itself
    const int d = -1074 - E;
    bits = d <= 0 ? m0 << -d : (d > 63 ? 0ull : (m0 + (1ull << (d - 1))) >> d);
  }
  return __longlong_as_double((long long)(sgn | bits));
}
DV double int_scaled(long long I, int E) {
  if (I == 0) return 0.0;
  const unsigned long long m0 = I < 0 ? 0ull - (unsigned long long)I : (unsigned long long)I;
  const int msb = 63 - __clzll((long long)m0), ex = msb + E + 1023;
  if ((unsigned)(ex - 1) >= 2046u) return int_scaled_ends(I, E);
  // m in [2^52, 2^53]: a carry moves into the exponent field by itself
  const unsigned long long m = msb > 52 ? (m0 + (1ull << (msb - 53))) >> (msb - 52) : m0 << (52 - msb);
  const unsigned long long sgn = I < 0 ? 1ull << 63 : 0ull;
  return __longlong_as_double((long long)(sgn | (((unsigned long long)ex << 52) + (m - (1ull << 52)))));
}

// I 2^-d rounded to nearest, d >= 0.
DV long long shift_round(long long I, int d) {
  if (d == 0) return I;
  return d > 62 ? 0 : (I + (1ll << (d - 1))) >> d;
}

// Exponent of a K-chunk of a row that holds an infinity or a NaN (wide digits):
// every output it enters becomes NaN, as in FP64 arithmetic.
constexpr int kNotFinite = 20000;

__global__ void __launch_bounds__(kTcThreads, 1)
    tc_zgemm_wide_kernel(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapB, TcArgs a) {
  extern __shared__ unsigned char smem_raw[];
  __shared__ __align__(8) uint64_t a_full[kWideA], a_empty[kWideA], b_full[2], b_empty[2], acc_full[3], acc_free, done;
  __shared__ uint32_t tmem_slot;
  __shared__ int abort_flag;
  __shared__ int eb_sh[3][kTcN];
  unsigned char* smem =
      reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  unsigned char* smem_b = smem + (size_t)kWideA * a_plane_bytes();
  constexpr int S = kWideDigits;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int m0 = blockIdx.y * kTcM, n0 = a.n_first + blockIdx.x * kTcN, z = blockIdx.z;
  const int k_begin = z * kWideChunk;
  const int k_len = min(kWideChunk, a.K - k_begin);
  const int nslab = (k_len + kSlab - 1) / kSlab;

  if (threadIdx.x == 0) {
    for (int i = 0; i < kWideA; ++i) {
      mbar_init(&a_full[i], 1);
      mbar_init(&a_empty[i], 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&b_full[i], 1);
      mbar_init(&b_empty[i], 1);
    }
    for (int i = 0; i < 3; ++i) mbar_init(&acc_full[i], 1);
    mbar_init(&acc_free, 256);
    mbar_init(&done, 1);
    abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                 "r"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;
  volatile int* vabort = &abort_flag;
  // units u = c * nslab + slab in order; A plane i of unit u is use u S + i
  const int nunit = 3 * nslab;

  if (warp == 8) {
    if (lane == 0) {
      int nb = 0, na = 0;  // B sets and A planes issued
      bool ok = true;
      for (int u = 0; u < nunit && ok; ++u) {
        const int c = u / nslab, k0 = k_begin + (u - c * nslab) * kSlab;
        const int sb = u & 1;
        if (u >= 2 && !mbar_wait(&b_empty[sb], ((u >> 1) - 1) & 1, vabort, a.err)) break;
        mbar_expect_tx(&b_full[sb], (uint32_t)wide_b_bytes());
        for (int j = 0; j < S; ++j)
          tma_load_3d(smem_b + (size_t)sb * wide_b_bytes() + (size_t)j * b_plane_bytes(), &mapB, &b_full[sb], k0, n0,
                      c * S + j);
        nb = u + 1;
        for (int i = 0; i < S; ++i) {
          const int w = u * S + i, sl = w % kWideA;
          if (w >= kWideA && !mbar_wait(&a_empty[sl], ((w / kWideA) - 1) & 1, vabort, a.err)) {
            ok = false;
            break;
          }
          mbar_expect_tx(&a_full[sl], (uint32_t)a_plane_bytes());
          tma_load_3d(smem + (size_t)sl * a_plane_bytes(), &mapA, &a_full[sl], k0, m0, c * S + i);
          na = w + 1;
        }
      }
      // every issued copy has landed before the CTA may exit (bounded)
      for (int u = max(0, nb - 2); u < nb; ++u) {
        const uint64_t t0 = global_ns();
        while (!mbar_try_wait(&b_full[u & 1], (u >> 1) & 1))
          if (global_ns() - t0 > kWaitNs) break;
      }
      for (int w = max(0, na - kWideA); w < na; ++w) {
        const uint64_t t0 = global_ns();
        while (!mbar_try_wait(&a_full[w % kWideA], (w / kWideA) & 1))
          if (global_ns() - t0 > kWaitNs) break;
      }
    }
  } else if (warp == 9) {
    if (lane == 0) {
      bool ok = true;
      for (int u = 0; u < nunit && ok; ++u) {
        const int c = u / nslab, slab = u - c * nslab, sb = u & 1;
        // the third product takes the first one's columns
        if (c == 2 && slab == 0 && !mbar_wait(&acc_free, 0, vabort, a.err)) break;
        if (!mbar_wait(&b_full[sb], (u >> 1) & 1, vabort, a.err)) break;
        const uint64_t b0 = sw128_desc(smem_u32(smem_b + (size_t)sb * wide_b_bytes()));
        const int nkk = min(kSlab, k_len - slab * kSlab + 15) / 16;  // 16-value steps that hold data
        const uint32_t acc = tmem + (uint32_t)((c & 1) * S * kTcN);
        for (int i = 0; i < S; ++i) {
          const int w = u * S + i, sl = w % kWideA;
          if (!mbar_wait(&a_full[sl], (w / kWideA) & 1, vabort, a.err)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint64_t a0 = sw128_desc(smem_u32(smem + (size_t)sl * a_plane_bytes()));
          const uint32_t idesc = umma_idesc_bf16(kTcM, kTcN * (S - i));
          for (int kk = 0; kk < nkk; ++kk)
            umma(acc + (uint32_t)(i * kTcN), a0 + (uint64_t)(kk * 2), b0 + (uint64_t)(kk * 2), idesc,
                 (slab > 0 || i > 0 || kk > 0) ? 1u : 0u);
          umma_commit(&a_empty[sl]);
        }
        if (!ok) break;
        umma_commit(&b_empty[sb]);
        if (slab == nslab - 1) umma_commit(&acc_full[c]);
      }
      // the MMAs issued have finished before the tensor memory is freed (bounded)
      umma_commit(&done);
      const uint64_t t0 = global_ns();
      while (!mbar_try_wait(&done, 0))
        if (global_ns() - t0 > kWaitNs) break;
    }
  } else {
    // ---- epilogue: warps 0-7; two per lane quadrant, 16 columns each -------
    const int quad = warp & 3, half = warp >> 2;
    const int m = m0 + 32 * quad + lane;
    cplx* out = a.out + z * a.zstride - a.ldo * a.n_first;
    {
      const int t = threadIdx.x;
      if (t < 3 * kTcN) {
        const int c = t / kTcN, n = n0 + t % kTcN;
        eb_sh[c][t % kTcN] = (n < a.N) ? a.eB[(size_t)c * a.nchunks * a.N + (size_t)z * a.N + n] : 0;
      }
      asm volatile("bar.sync 1, 256;" ::: "memory");
    }
    const size_t eAs = (size_t)a.nchunks * a.M;
    int ea[3] = {0, 0, 0};
    if (m < a.M)
#pragma unroll
      for (int c = 0; c < 3; ++c) ea[c] = a.eA[c * eAs + (size_t)z * a.M + m];
    const uint32_t lane_base = tmem + ((uint32_t)(32 * quad) << 16) + (uint32_t)(16 * half);
    // product c of column q: X 2^(ex - 54) + lo 2^(ex - 70), lo 16 bits
    long long X[3][16];
    unsigned int lo[3][8];
    bool ok = true;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      ok = ok && mbar_wait(&acc_full[c], 0, vabort, a.err);
      tc_fence_after();
      ok = __all_sync(0xffffffffu, ok);
      if (ok) {
#pragma unroll
        for (int h = 0; h < 4; ++h) {
          float v[8][4];
          tmem_ld_levels8x4(lane_base + (uint32_t)((c & 1) * S * kTcN + 4 * h), v);
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            long long x = __float2int_rn(v[0][q]);
#pragma unroll
            for (int L = 1; L < 6; ++L) x = x * 256 + __float2int_rn(v[L][q]);
            const long long low = (long long)__float2int_rn(v[6][q]) * 256 + __float2int_rn(v[7][q]);
            X[c][4 * h + q] = x + (low >> 16);
            const unsigned int l16 = (unsigned int)low & 0xFFFFu;
            unsigned int& w = lo[c][(4 * h + q) / 2];
            w = (q & 1) ? w | (l16 << 16) : l16;
          }
        }
      }
      if (c == 0) {  // read: its columns are free for the third product
        tc_fence_before();
        mbar_arrive(&acc_free);
      }
    }
    if (ok && !*vabort) {
      // the values an accumulating product adds to, two to four columns ahead (each
      // column's own load would otherwise wait out an L2 round trip: 16 us
      // of a tile's 26)
      cplx pre[2][2];
      auto prefetch = [&](int h) {
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          const int n = n0 + 16 * half + 2 * h + q;
          pre[h & 1][q] = (a.accumulate && m < a.M && n < a.N) ? out[(size_t)a.rso * m + (size_t)a.ldo * n] : mk(0, 0);
        }
      };
      prefetch(0);
#pragma unroll
      for (int q = 0; q < 16; ++q) {
        if (q % 2 == 0 && q < 14) prefetch(q / 2 + 1);
        const int n = n0 + 16 * half + q;
        if (m >= a.M || n >= a.N) continue;
        // all three at one unit, the largest at bit 60 (a zero product has no
        // scale): the sum is exact to 2^-60 of the largest product, whatever
        // the scales
        int ex[3], top = -100000;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          ex[c] = ea[c] + eb_sh[c][16 * half + q];
          const long long x = X[c][q];
          if (x != 0 || lo[c][q / 2] != 0)
            top = max(top, ex[c] + 63 - __clzll((x < 0 ? ~x : x) | 1ll));
        }
        long long T[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          const unsigned int l16 = (q & 1) ? lo[c][q / 2] >> 16 : lo[c][q / 2] & 0xFFFFu;
          const int up = 60 - top + ex[c];
          const long long x = X[c][q];
          if (x == 0 && l16 == 0) T[c] = 0;
          else if (up >= 0) T[c] = (x << up) + (long long)(up >= 16 ? (unsigned long long)l16 << (up - 16) : l16 >> (16 - up));
          else T[c] = shift_round(x, -up);
        }
        // re = T1 - T2, im = T3 - T1 - T2: each |T| <= 2^61, sums below 2^63
        long long re = T[0] - T[1], im = T[2] - T[0] - T[1];
        if (a.alpha_neg) {
          re = -re;
          im = -im;
        }
        const int Es = top - 114 + a.alpha_exp;
        cplx r = mk(int_scaled(re, Es), int_scaled(im, Es));
        if (max(ex[0], max(ex[1], ex[2])) > kNotFinite / 2) r = mk(__longlong_as_double(-1ll), __longlong_as_double(-1ll));
        if (a.accumulate) r = cadd(pre[(q / 2) & 1][q % 2], r);
        out[(size_t)a.rso * m + (size_t)a.ldo * n] = r;
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
  }
}

// ---- digit splitting ----------------------------------------------------------
// The operand view of TcOperandView (kernels.h), passed by value.
struct SplitView {
  const cplx* X;
  long long rs, ks;
  int R, K, conj;
  int tri_mode, tri;
  int group;        // rows per group (R: one group)
  long long gs;     // elements between groups
};
// A view and where its digits go.  top (may be NULL; wide digits): the column
// maxima of both operands (col_top_kernel), this one's side of the balance.
struct SplitJob {
  SplitView v;
  int nchunks, row_ctas;  // K-chunks; CTAs along the rows
  int* e;
  __nv_bfloat16* planes;
  long long ldk;
  const int* top;
  int side;
};

// What the view holds at an in-range (r, k): 0 the stored value, 1 zero
// (outside the triangle), 2 one (the unit diagonal of a reflector block).
DV int view_kind(const SplitView& v, int r, int k) {
  if (v.tri_mode == 1) return r > k + v.tri ? 1 : 0;
  // rows in groups: row i of group g is row i of an upper trapezoid's columns
  // from g tri on
  if (v.tri_mode == 5) return r % v.group > k + v.tri * (r / v.group) ? 1 : 0;
  // reflector s = r (rows of the view are reflector indices), entry i = k:
  // zero above the unit diagonal k < r + tri, one on it
  if (v.tri_mode == 2) return k < r + v.tri ? 1 : (k == r + v.tri ? 2 : 0);
  // same reflector block, view with rows = entry index i, columns = s
  if (v.tri_mode == 3) return r < k + v.tri ? 1 : (r == k + v.tri ? 2 : 0);
  // the first `tri` rows are such reflectors (r, entry k), the rest stored
  if (v.tri_mode == 4 && r < v.tri) return k < r ? 1 : (k == r ? 2 : 0);
  return 0;
}

// Splitting, one CTA per (16 rows, K-chunk): the chunk (16 x at most 192
// values, 48 KB) is staged once into shared memory by cp.async along
// whichever index is contiguous in memory (entries outside the view's
// triangle are written as their constants instead of read); pass 1 finds
// each row's per-component exponent e (max |x| 2^-e < 1) over the chunk,
// pass 2 cuts the digits, written as consecutive BF16 digits per row and
// plane.  Four CTAs per SM keep about 190 KB of loads in flight.  No FP64
// arithmetic beyond one addition (re + im): the magnitudes are compared as
// integers and the digits cut from the IEEE bit pattern (on this GPU the
// FP64 pipe retires two multiply-adds per clock per SM).
constexpr int kSplitRows = 16;
constexpr int kSplitThreads = 256;
constexpr int kSplitLd = 3 * kSlab + 1;  // one K-chunk and a zero pad per shared-memory row
size_t split_smem_bytes() { return (size_t)kSplitRows * kSplitLd * sizeof(cplx); }

DV void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
DV void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// |x| as an ordered integer key (the IEEE bits without the sign).
DV long long mag_key(double x) { return __double_as_longlong(x) & 0x7FFFFFFFFFFFFFFFll; }
// e with |x| 2^-e < 1 for the value whose key is given (ilogb + 1; 0 for 0).
DV int key_exponent(long long key) {
  if (key == 0) return 0;
  const int ex = (int)(key >> 52);
  return ex == 0 ? -1021 : ex - 1022;  // subnormal: below 2^-1022
}
// round(v 2^(nbits - e)) as an integer, |v| < 2^e: from v = M 2^E (M the
// 53-bit significand) by a rounding right shift.
DV long long fixed_point(double v, int e, int nbits) {
  const long long b = __double_as_longlong(v);
  const int ex = (int)((b >> 52) & 0x7FF);
  long long M = b & 0xFFFFFFFFFFFFFll;
  int E;
  if (ex == 0) {
    E = -1074;
  } else {
    M |= 1ll << 52;
    E = ex - 1075;
  }
  const int sh = E - e + nbits;
  long long X;
  if (M == 0 || sh < -62) X = 0;
  else if (sh >= 0) X = M << sh;  // only for nbits > 53: sh <= nbits - 53, X < 2^nbits
  else X = (M + (1ll << (-sh - 1))) >> (-sh);
  return b < 0 ? -X : X;
}

// ---- balance of a contraction (wide digits) -----------------------------------
// The digits count from the largest entry of a row, so a product is accurate
// against (largest of A's row) x (largest of B's row), not term by term.  If the
// columns of A grow with k and those of B shrink with it, the same tensor in
// another gauge of its bond, the terms are alike but every row is graded, and
// what lies 2^63 below its largest entry is cut: 1e-12 of the result where D and
// 1/D span 8 decades, 1e-8 for 12 (FP64 products: 1e-15).  So column k of A is
// multiplied by 2^s and that of B by 2^-s, exact, with s from the columns' largest
// exponents, half of their difference: then both are at the root of their
// product, and the error is of the largest term of |A||B| (1e-15 whatever the
// gauge).  A column that is zero on one side is left out on the other.
constexpr int kNoTop = -1000000;  // exponent of zero; a shift that leaves a value out

// e with |x| 2^-e < 1 (a power of two above it at most); kNoTop for 0.
DV int value_top(double x) {
  const int hi = __double2hiint(x) & 0x7fffffff;
  return (hi | __double2loint(x)) == 0 ? kNoTop : max(hi >> 20, 1) - 1022;
}
// Biased exponent of the larger part of what the view holds at (r, k), 0 for zero
// and for what is not finite.
DV int entry_top(const SplitView& v, int r, int k) {
  const int kind = view_kind(v, r, k);
  if (kind) return kind == 2 ? 1023 : 0;
  const cplx x = __ldg(v.X + (long long)k * v.ks + (long long)(r % v.group) * v.rs + (long long)(r / v.group) * v.gs);
  const int m = max(__double2hiint(x.x) & 0x7fffffff, __double2hiint(x.y) & 0x7fffffff);
  if (d_zero(x.x) && d_zero(x.y)) return 0;
  return m >= 0x7ff00000 ? 0 : max(m >> 20, 1);
}
// top[z * K + k] <- max over the rows of view z (0 or 1) of column k; zeroed
// before.  Lanes along whichever index is contiguous; bound by one read of the
// operands (8 to 10 us at 2048 to 8192 rows of 32 and 64 columns).
constexpr int kTopRows = 256;
__global__ void __launch_bounds__(256) col_top_kernel(SplitView a, SplitView b, int* __restrict__ top) {
  const SplitView& v = blockIdx.z ? b : a;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int ra = blockIdx.y * kTopRows, rb = min(v.R, ra + kTopRows);
  int* t = top + (size_t)blockIdx.z * v.K;
  int m = 0;
  if (v.rs == 1) {  // a column per warp
    const int k = blockIdx.x * 8 + w;
    if (k >= v.K) return;
#pragma unroll 4
    for (int r = ra + lane; r < rb; r += 32) m = max(m, entry_top(v, r, k));
    m = __reduce_max_sync(0xffffffffu, m);
    if (lane == 0 && m) atomicMax(t + k, m);
  } else {
    // eight columns per CTA here too; the rows over its 32 groups of eight lanes
    const int k = blockIdx.x * 8 + (threadIdx.x & 7);
    if (k < v.K)
#pragma unroll 4
      for (int r = ra + (threadIdx.x >> 3); r < rb; r += 32) m = max(m, entry_top(v, r, k));
    m = max(m, __shfl_xor_sync(0xffffffffu, m, 8));
    m = max(m, __shfl_xor_sync(0xffffffffu, m, 16));
    if (lane < 8 && k < v.K && m) atomicMax(t + k, m);
  }
}

// BF16 bits of a small integer (|d| <= 128: exact in BF16, so the upper
// half of its FP32 bits).
DV unsigned int bf16_bits(int d) { return __float_as_uint((float)d) >> 16; }

// The S balanced base-256 digits of two fixed-point values, digit j of both
// as one 32-bit word (first value in the low half) at dst[j * pstride].
// |X| <= 2^39 (S = 5): after the lowest digit the rest can reach 2^31 (a
// value within 2^-32 of its power-of-two scale), after the second it is
// below 2^24, so the first two steps run in 64 bits and the rest in 32.
DV void digit_pair(long long X0, long long X1, int S, unsigned int* dst, size_t pstride) {
  if (S == 1) {  // one digit: the value itself (|X| <= 128)
    dst[0] = bf16_bits((int)X0) | (bf16_bits((int)X1) << 16);
    return;
  }
  int d0 = (int)((X0 + 128) & 255) - 128, d1 = (int)((X1 + 128) & 255) - 128;
  X0 = (X0 - d0) >> 8;
  X1 = (X1 - d1) >> 8;
  dst[(size_t)(S - 1) * pstride] = bf16_bits(d0) | (bf16_bits(d1) << 16);
  if (S == 2) {
    dst[0] = bf16_bits((int)X0) | (bf16_bits((int)X1) << 16);
    return;
  }
  d0 = (int)((X0 + 128) & 255) - 128;
  d1 = (int)((X1 + 128) & 255) - 128;
  int y0 = (int)((X0 - d0) >> 8), y1 = (int)((X1 - d1) >> 8);
  dst[(size_t)(S - 2) * pstride] = bf16_bits(d0) | (bf16_bits(d1) << 16);
  for (int j = S - 3; j >= 1; --j) {
    d0 = ((y0 + 128) & 255) - 128;
    d1 = ((y1 + 128) & 255) - 128;
    y0 = (y0 - d0) >> 8;
    y1 = (y1 - d1) >> 8;
    dst[(size_t)j * pstride] = bf16_bits(d0) | (bf16_bits(d1) << 16);
  }
  dst[0] = bf16_bits(y0) | (bf16_bits(y1) << 16);
}

// The same for S = kWideDigits: |X| < 2^63, the first five digits are cut in
// 64 bits (below 2^24 is left), the rest in 32.
DV void digit_pair_wide(long long X0, long long X1, unsigned int* dst, size_t pstride) {
#pragma unroll
  for (int j = kWideDigits - 1; j >= 3; --j) {
    const int d0 = (int)((X0 + 128) & 255) - 128, d1 = (int)((X1 + 128) & 255) - 128;
    X0 = (X0 - d0) >> 8;
    X1 = (X1 - d1) >> 8;
    dst[(size_t)j * pstride] = bf16_bits(d0) | (bf16_bits(d1) << 16);
  }
  int y0 = (int)X0, y1 = (int)X1;
#pragma unroll
  for (int j = 2; j >= 1; --j) {
    const int d0 = ((y0 + 128) & 255) - 128, d1 = ((y1 + 128) & 255) - 128;
    y0 = (y0 - d0) >> 8;
    y1 = (y1 - d1) >> 8;
    dst[(size_t)j * pstride] = bf16_bits(d0) | (bf16_bits(d1) << 16);
  }
  dst[0] = bf16_bits(y0) | (bf16_bits(y1) << 16);
}

__global__ void __launch_bounds__(kSplitThreads)
    split_kernel(SplitJob j0, SplitJob j1, int Kc, int S) {
  extern __shared__ cplx tile[];  // [kSplitRows][kSplitLd]
  __shared__ int esh[4][kSplitRows];  // components' exponents; one above max(|re|, |im|)
  __shared__ int shift[kWideChunk];   // wide digits: column k is taken times 2^shift
  // the two jobs' CTAs one after the other
  int blk = blockIdx.x;
  const bool second = blk >= j0.row_ctas * j0.nchunks;
  if (second) blk -= j0.row_ctas * j0.nchunks;
  const SplitView v = second ? j1.v : j0.v;
  const int nchunks = second ? j1.nchunks : j0.nchunks, row_ctas = second ? j1.row_ctas : j0.row_ctas;
  int* e = second ? j1.e : j0.e;
  __nv_bfloat16* planes = second ? j1.planes : j0.planes;
  const long long ldk = second ? j1.ldk : j0.ldk;
  const int r0 = (blk % row_ctas) * kSplitRows, z = blk / row_ctas;
  const int kb = z * Kc, klen = min(v.K - kb, Kc);
  const int tid = threadIdx.x;
  const int nval = kSplitRows * klen;
  const bool rows_contiguous = v.rs == 1 && v.ks != 1;
  for (int idx = tid; idx < nval; idx += kSplitThreads) {
    int r, k;
    if (rows_contiguous) {
      r = idx % kSplitRows;
      k = idx / kSplitRows;
    } else {
      k = idx % klen;
      r = idx / klen;
    }
    cplx* dst = tile + r * kSplitLd + k;
    const int kind = (r0 + r < v.R) ? view_kind(v, r0 + r, kb + k) : 1;
    if (kind == 0) {
      const cplx* src = v.X + (long long)(kb + k) * v.ks;
      src += v.group < v.R ? (long long)((r0 + r) % v.group) * v.rs + (long long)((r0 + r) / v.group) * v.gs
                           : (long long)(r0 + r) * v.rs;
      cp_async16(dst, src);
    }
    else *dst = mk(kind == 2 ? 1.0 : 0.0, 0.0);
  }
  if ((klen & 1) && tid < kSplitRows) tile[tid * kSplitLd + klen] = mk(0, 0);  // second value of the last pair
  if (S == kWideDigits && tid < kWideChunk) {
    const int* top = second ? j1.top : j0.top;
    int sh = 0;
    if (top && tid < klen) {
      const int side = second ? j1.side : j0.side, own = top[(size_t)side * v.K + kb + tid],
                other = top[(size_t)(side ^ 1) * v.K + kb + tid];
      // (the same halving on both sides, so that the two shifts cancel)
      const int half = (side ? own - other : other - own) >> 1;
      sh = own == 0 || other == 0 ? kNoTop : (side ? -half : half);
    }
    shift[tid] = sh;
  }
  cp_async_wait_all();
  __syncthreads();
  const double sgn = v.conj ? -1.0 : 1.0;
  // pass 1: largest magnitude per row and component, a half-warp per row
  {
    const int r = tid >> 4, j = tid & 15;
    long long k0m = 0, k1m = 0, k2m = 0;
    int t0m = kNoTop, t1m = kNoTop, t2m = kNoTop;  // the same as exponents (wide digits)
    int bad = 0;  // an infinity or a NaN, by its exponent
    for (int k = j; k < klen; k += 16) {
      const cplx x = tile[r * kSplitLd + k];
      const double im = sgn * x.y;
      if (S == kWideDigits) {
        const int sh = shift[k], t0 = value_top(x.x), t1 = value_top(x.y);
        bad |= max(t0, t1) > 1024;
        t0m = max(t0m, t0 + sh);  // (a column left out stays far below any exponent)
        t1m = max(t1m, t1 + sh);
        t2m = max(t2m, value_top(x.x + im) + sh);
        continue;
      }
      k0m = max(k0m, mag_key(x.x));
      k1m = max(k1m, mag_key(im));
      k2m = max(k2m, mag_key(x.x + im));
    }
#pragma unroll
    for (int o = 8; o >= 1; o >>= 1) {
      k0m = max(k0m, __shfl_xor_sync(0xffffffffu, k0m, o));
      k1m = max(k1m, __shfl_xor_sync(0xffffffffu, k1m, o));
      k2m = max(k2m, __shfl_xor_sync(0xffffffffu, k2m, o));
      if (S == kWideDigits) {
        t0m = max(t0m, __shfl_xor_sync(0xffffffffu, t0m, o));
        t1m = max(t1m, __shfl_xor_sync(0xffffffffu, t1m, o));
        t2m = max(t2m, __shfl_xor_sync(0xffffffffu, t2m, o));
        bad |= __shfl_xor_sync(0xffffffffu, bad, o);
      }
    }
    if (j < 3) {
      const int t = j == 0 ? t0m : (j == 1 ? t1m : t2m);
      const int own = S == kWideDigits ? (t < kNoTop / 2 ? 0 : t) : key_exponent(j == 0 ? k0m : (j == 1 ? k1m : k2m));
      const int ex = bad ? kNotFinite : own;
      esh[j][r] = ex;
      if (j == 0) esh[3][r] = max(t0m, t1m) + 1;
      if (r0 + r < v.R) e[((size_t)j * nchunks + z) * v.R + r0 + r] = ex;
    }
  }
  __syncthreads();
  // pass 2: balanced base-256 digits of round(x 2^(8S-1)), |x| = |v| 2^-e < 1:
  // x ~ sum_j q_j 2^(-7-8j) with |q_j| <= 128.  Each thread cuts two
  // consecutive K-values of a row and stores each digit pair as one 32-bit
  // word (K-chunks start at even K, ldk is even).
  const size_t plane = (size_t)v.R * ldk;
  const int nbits = 8 * S - 1;
  const int nph = (klen + 1) >> 1;
  for (int pi = tid; pi < kSplitRows * nph; pi += kSplitThreads) {
    const int r = pi / nph, kk = 2 * (pi - r * nph);
    if (r0 + r >= v.R) break;
    const cplx x0 = tile[r * kSplitLd + kk], x1 = tile[r * kSplitLd + kk + 1];
    const double i0 = sgn * x0.y, i1 = sgn * x1.y;
    unsigned int* dst = reinterpret_cast<unsigned int*>(planes + (size_t)(r0 + r) * ldk + kb + kk);
    if (S == kWideDigits) {
      // round(v 2^(shift + nbits - e)); a column left out is zero
      const int sa = shift[kk], sb = kk + 1 < klen ? shift[kk + 1] : kNoTop;
      auto cut = [&](double v, int e, int sh) { return sh == kNoTop ? 0ll : fixed_point(v, e - sh, nbits); };
      digit_pair_wide(cut(x0.x, esh[0][r], sa), cut(x1.x, esh[0][r], sb), dst, plane / 2);
      digit_pair_wide(cut(i0, esh[1][r], sa), cut(i1, esh[1][r], sb), dst + (size_t)S * (plane / 2), plane / 2);
      // re + im as integers at a scale above both (exact to 2^-62 of the larger
      // one), then at the sum's own scale, which it does not exceed
      const int ec = esh[3][r], up = ec - esh[2][r];
      long long s0 = cut(x0.x, ec, sa) + cut(i0, ec, sa);
      long long s1 = cut(x1.x, ec, sb) + cut(i1, ec, sb);
      s0 = up < 63 ? s0 << max(up, 0) : 0;
      s1 = up < 63 ? s1 << max(up, 0) : 0;
      digit_pair_wide(s0, s1, dst + (size_t)(2 * S) * (plane / 2), plane / 2);
      continue;
    }
    const double c0[3] = {x0.x, i0, x0.x + i0};
    const double c1[3] = {x1.x, i1, x1.x + i1};
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      const int ex = esh[q][r];
      digit_pair(fixed_point(c0[q], ex, nbits), fixed_point(c1[q], ex, nbits), S, dst + (size_t)(q * S) * (plane / 2),
                 plane / 2);
    }
  }
}

// out[rso m + ldo n] = alpha * sum_z part[z * zstride + m + M n] (+ out), one
// thread per output, the partials in order (the narrow digits' results are
// kept to the last bit), eight loads in flight.
__global__ void reduce_parts_kernel(const cplx* __restrict__ part, int M, int N, int nz, long long zstride, double alpha,
                                    int accumulate, cplx* __restrict__ out, long long rso, long long ldo) {
  const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (long long)M * N) return;
  const int m = (int)(idx % M), n = (int)(idx / M);
  cplx s = mk(0, 0);
  for (int z0 = 0; z0 < nz; z0 += 8) {
    cplx v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) v[u] = z0 + u < nz ? part[(size_t)(z0 + u) * zstride + idx] : mk(0, 0);
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (z0 + u < nz) s = cadd(s, v[u]);
  }
  cplx* p = out + (size_t)rso * m + (size_t)ldo * n;
  cplx r = mk(alpha * s.x, alpha * s.y);
  if (accumulate) r = cadd(*p, r);
  *p = r;
}

// The same for the wide digits, whose chunks are shorter: eight threads per
// output take every eighth partial, four loads in flight, and their sums are
// added in a fixed order (384 partials of 49152 rows would be one chain of
// 384 dependent FP64 additions).
constexpr int kRedOut = 32;
constexpr int kRedZ = 8;
__global__ void __launch_bounds__(kRedOut * kRedZ)
    reduce_wide_kernel(const cplx* __restrict__ part, int M, int N, int nz, long long zstride, double alpha, int accumulate,
                       cplx* __restrict__ out, long long rso, long long ldo) {
  __shared__ cplx sums[kRedZ][kRedOut];
  const int o = threadIdx.x % kRedOut, zl = threadIdx.x / kRedOut;
  const long long idx = (long long)blockIdx.x * kRedOut + o, total = (long long)M * N;
  cplx s = mk(0, 0);
  if (idx < total) {
    const cplx* p = part + idx;
    int z = zl;
    for (; z + 3 * kRedZ < nz; z += 4 * kRedZ) {
      const cplx v0 = p[(size_t)z * zstride], v1 = p[(size_t)(z + kRedZ) * zstride],
                 v2 = p[(size_t)(z + 2 * kRedZ) * zstride], v3 = p[(size_t)(z + 3 * kRedZ) * zstride];
      s = cadd(cadd(s, v0), cadd(v1, cadd(v2, v3)));
    }
    for (; z < nz; z += kRedZ) s = cadd(s, p[(size_t)z * zstride]);
  }
  sums[zl][o] = s;
  __syncthreads();
  if (zl != 0 || idx >= total) return;
  for (int i = 1; i < kRedZ; ++i) s = cadd(s, sums[i][o]);
  const int m = (int)(idx % M), n = (int)(idx / M);
  cplx* q = out + (size_t)rso * m + (size_t)ldo * n;
  cplx r = mk(alpha * s.x, alpha * s.y);
  if (accumulate) r = cadd(*q, r);
  *q = r;
}

}  // namespace

// ---- host entry points ------------------------------------------------------------

size_t tc_operand_bytes(int R, int K, int S, int Kc) {
  const long long ldk = ((long long)K + kSlab - 1) / kSlab * kSlab;
  const int nchunks = (K + Kc - 1) / Kc;
  const size_t planes = (size_t)3 * S * R * ldk * sizeof(__nv_bfloat16);
  const size_t exps = (size_t)3 * nchunks * R * sizeof(int);
  return ((planes + 255) & ~(size_t)255) + exps + 256;
}

int tc_chunk(int S) { return S == kWideDigits ? kWideChunk : 3 * kSlab; }
int tc_max_digits() { return kMaxDigits; }
int tc_wide_digits() { return kWideDigits; }

static SplitJob split_job(const TcOperandView& ov, int S, TcOperand* out, void* buf) {
  const int Kc = tc_chunk(S);
  const long long ldk = ((long long)ov.K + kSlab - 1) / kSlab * kSlab;
  const int nchunks = (ov.K + Kc - 1) / Kc;
  const size_t planes = (size_t)3 * S * ov.R * ldk * sizeof(__nv_bfloat16);
  out->planes = buf;
  out->e = reinterpret_cast<int*>(reinterpret_cast<unsigned char*>(buf) + ((planes + 255) & ~(size_t)255));
  out->R = ov.R;
  out->K = ov.K;
  out->S = S;
  out->ldk = ldk;
  out->nchunks = nchunks;
  return SplitJob{SplitView{ov.X, ov.rs, ov.ks, ov.R, ov.K, ov.conj, ov.tri_mode, ov.tri,
                            ov.group > 0 ? ov.group : ov.R, ov.gs},
                  nchunks,
                  (ov.R + kSplitRows - 1) / kSplitRows, out->e, reinterpret_cast<__nv_bfloat16*>(buf), ldk, nullptr, 0};
}

// Two operands in one launch (a product's operands are split back to back, and
// most of these launches are short).
cudaError_t tc_split2(const TcOperandView& a, TcOperand* oa, void* bufa, const TcOperandView& b, TcOperand* ob, void* bufb,
                      int S, cudaStream_t s, int* top) {
  if (S < 1 || (S > kMaxDigits && S != kWideDigits) || a.R <= 0 || a.K <= 0 || b.R < 0 || (b.R > 0 && b.K <= 0))
    return cudaErrorInvalidValue;
  SplitJob j0 = split_job(a, S, oa, bufa);
  SplitJob j1{};
  if (b.R > 0) j1 = split_job(b, S, ob, bufb);
  if (top) {
    if (S != kWideDigits || b.R <= 0 || a.K != b.K) return cudaErrorInvalidValue;
    cudaError_t e = cudaMemsetAsync(top, 0, 2 * (size_t)a.K * sizeof(int), s);
    if (e != cudaSuccess) return e;
    const dim3 grid((a.K + 7) / 8, (std::max(a.R, b.R) + kTopRows - 1) / kTopRows, 2);
    if (grid.y > 65535) return cudaErrorInvalidValue;
    col_top_kernel<<<grid, 256, 0, s>>>(j0.v, j1.v, top);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    j0.top = j1.top = top;
    j1.side = 1;
  }
  const long long ctas = (long long)j0.row_ctas * j0.nchunks + (long long)j1.row_ctas * j1.nchunks;
  if (ctas > 0x7fffffffll) return cudaErrorInvalidValue;
  cudaError_t e = allow_smem((const void*)split_kernel, split_smem_bytes());
  if (e != cudaSuccess) return e;
  split_kernel<<<(unsigned)ctas, kSplitThreads, split_smem_bytes(), s>>>(j0, j1, tc_chunk(S), S);
  return cudaGetLastError();
}

cudaError_t tc_split(const TcOperandView& ov, int S, TcOperand* out, void* buf, cudaStream_t s) {
  return tc_split2(ov, out, buf, TcOperandView{}, nullptr, nullptr, S, s);
}

cudaError_t tc_zgemm(const TcOperand& A, const TcOperand& B, cplx* out, long long rso, long long ldo, double alpha,
                     int accumulate, cplx* part, size_t part_elems, int* err, cudaStream_t s) {
  if (A.K != B.K || A.S != B.S || A.nchunks != B.nchunks) return cudaErrorInvalidValue;
  const int M = A.R, N = B.R, K = A.K, S = A.S, nz = A.nchunks;
  const bool wide = S == kWideDigits;
  if (!wide && nz == 1 && rso != 1) return cudaErrorInvalidValue;
  CUtensorMap ma, mb;
  cudaError_t e = plane_map(&ma, static_cast<const __nv_bfloat16*>(A.planes), K, A.ldk, M, 3 * S, kTcM);
  if (e == cudaSuccess) e = plane_map(&mb, static_cast<const __nv_bfloat16*>(B.planes), K, B.ldk, N, 3 * S, kTcN);
  if (e != cudaSuccess) return e;
  const size_t smem = wide ? wide_smem_bytes() : tc_smem_bytes(S);
  e = allow_smem(wide ? (const void*)tc_zgemm_wide_kernel : (const void*)tc_zgemm_kernel, smem);
  if (e != cudaSuccess) return e;
  TcArgs a{};
  a.M = M;
  a.N = N;
  a.K = K;
  a.S = S;
  a.Kc = tc_chunk(S);
  a.nchunks = nz;
  a.eA = A.e;
  a.eB = B.e;
  a.err = err;
  // alpha must be a signed power of two (the callers use +-1)
  int aexp = 0;
  const double am = std::frexp(std::fabs(alpha), &aexp);
  if (am != 0.5) return cudaErrorInvalidValue;
  // the columns of one launch: as many as part holds the partial sums of
  long long cols = N;
  if (nz == 1) {
    a.rso = rso;
    a.ldo = ldo;
    a.alpha_exp = aexp - 1;
    a.alpha_neg = alpha < 0.0;
    a.accumulate = accumulate;
  } else {
    if (!part) return cudaErrorInvalidValue;
    if (part_elems < (size_t)nz * M * N) cols = (long long)(part_elems / ((size_t)nz * M)) / kTcN * kTcN;
    if (cols <= 0) return cudaErrorInvalidValue;
    a.out = part;
    a.rso = 1;
    a.ldo = M;
  }
  for (long long n0 = 0; n0 < N; n0 += cols) {
    const int nc = (int)std::min<long long>(cols, N - n0);
    const dim3 grid((nc + kTcN - 1) / kTcN, (M + kTcM - 1) / kTcM, nz);
    a.n_first = (int)n0;
    a.zstride = nz == 1 ? 0 : (long long)M * nc;
    if (nz == 1) a.out = out;
    if (wide) tc_zgemm_wide_kernel<<<grid, kTcThreads, smem, s>>>(ma, mb, a);
    else tc_zgemm_kernel<<<grid, kTcThreads, smem, s>>>(ma, mb, a);
    e = cudaGetLastError();
    if (e != cudaSuccess || nz == 1) return e;
    const long long n = (long long)M * nc;
    cplx* o = out + (size_t)ldo * n0;
    if (wide)
      reduce_wide_kernel<<<(unsigned)((n + kRedOut - 1) / kRedOut), kRedOut * kRedZ, 0, s>>>(
          part, M, nc, nz, a.zstride, alpha, accumulate, o, rso, ldo);
    else
      reduce_parts_kernel<<<(unsigned)((n + 127) / 128), 128, 0, s>>>(part, M, nc, nz, a.zstride, alpha, accumulate, o, rso,
                                                                      ldo);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// Partial sums take nz times the output: 20 times a core of 2560 columns.  Beyond
// 1 GiB a product runs in groups of columns instead, at least one tile's: a group
// is then a large launch by itself, and every sum has its order.
constexpr size_t kMaxPart = (size_t)1 << 26;
size_t tc_part_elems(int M, int N, int K, int S) {
  const size_t nz = (K + tc_chunk(S) - 1) / tc_chunk(S);
  return nz > 1 ? std::min(nz * M * N, std::max(kMaxPart, nz * M * kTcN)) : 0;
}

}  // namespace hk
