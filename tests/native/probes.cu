// Host entry points over device code that no public call reaches by itself,
// built by tests/native_probes.py beside the library's objects.  Every function
// takes host arrays and returns a cudaError_t (0: done).
#include <vector>

#include "kernels.h"


namespace {

struct Buf {  // device memory for the length of a call
  void* p = nullptr;
  cudaError_t e;
  explicit Buf(size_t bytes) { e = cudaMalloc(&p, bytes ? bytes : 1); }
  ~Buf() { cudaFree(p); }
  template <class T>
  T* as() { return static_cast<T*>(p); }
};

__global__ void reciprocal_kernel(int n, const double* x, double* rcp, double* rsq) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  rcp[i] = rcp_fast(x[i]);
  rsq[i] = rsqrt_fast(fabs(x[i]));
}

__global__ void house_kernel(int n, const cplx* alpha, const double* s2, cplx* out) {
  const int i = blockIdx.x;  // one warp each
  if (i < n) house_fast(alpha[i], s2[i], out + 3 * i);
}

}  // namespace

extern "C" {

// C[rso m + ldo n] (nc values, read first) = alpha A B^T (+ C), A M x K and B N x K
// row-major, from S digits (0: the wide ones); balance: with the contraction index
// balanced; max_part: elements of the buffer of partial sums (0: all it may take).
int probe_product(int M, int N, int K, const double* A, const double* B, double* C, long long nc, long long rso,
                  long long ldo, double alpha, int accumulate, int balance, int S, long long max_part) {
  if (S == 0) S = hk::tc_wide_digits();
  const int Kc = hk::tc_chunk(S);
  size_t np = hk::tc_part_elems(M, N, K, S);
  if (max_part > 0 && np > (size_t)max_part) np = max_part;
  Buf a(sizeof(cplx) * M * K), b(sizeof(cplx) * N * K), c(sizeof(cplx) * nc), pa(hk::tc_operand_bytes(M, K, S, Kc)),
      pb(hk::tc_operand_bytes(N, K, S, Kc)), part(sizeof(cplx) * np), top(2 * sizeof(int) * K), err(sizeof(int));
  for (const Buf* q : {&a, &b, &c, &pa, &pb, &part, &top, &err})
    if (q->e != cudaSuccess) return q->e;
  cudaMemcpy(a.p, A, sizeof(cplx) * M * K, cudaMemcpyHostToDevice);
  cudaMemcpy(b.p, B, sizeof(cplx) * N * K, cudaMemcpyHostToDevice);
  cudaMemcpy(c.p, C, sizeof(cplx) * nc, cudaMemcpyHostToDevice);
  cudaMemset(err.p, 0, sizeof(int));
  hk::TcOperand oa, ob;
  cudaError_t e = hk::tc_split2(hk::TcOperandView{a.as<cplx>(), K, 1, M, K, 0, 0, 0}, &oa, pa.p,
                                hk::TcOperandView{b.as<cplx>(), K, 1, N, K, 0, 0, 0}, &ob, pb.p, S, nullptr,
                                balance ? top.as<int>() : nullptr);
  if (e == cudaSuccess)
    e = hk::tc_zgemm(oa, ob, c.as<cplx>(), rso, ldo, alpha, accumulate, np ? part.as<cplx>() : nullptr, np, err.as<int>(),
                     nullptr);
  if (e == cudaSuccess) e = cudaDeviceSynchronize();
  if (e != cudaSuccess) return e;
  int expired = 0;
  cudaMemcpy(&expired, err.p, sizeof(int), cudaMemcpyDeviceToHost);
  if (expired) return cudaErrorUnknown;
  return cudaMemcpy(C, c.p, sizeof(cplx) * nc, cudaMemcpyDeviceToHost);
}

// C (M x N, column-major) = A R^H for A M x K and R N x (coff + K), column-major,
// upper trapezoidal, by the tiled kernels; uh: C = A^H R instead (A K x M, R K x N, full).
int probe_gemm(int M, int N, int K, const double* A, const double* R, double* C, int coff, int uh, int mixed) {
  const int rows = uh ? K : N, cols = uh ? N : coff + K;
  Buf a(sizeof(cplx) * M * K), r(sizeof(cplx) * rows * cols), c(sizeof(cplx) * M * N);
  for (const Buf* q : {&a, &r, &c})
    if (q->e != cudaSuccess) return q->e;
  cudaMemcpy(a.p, A, sizeof(cplx) * M * K, cudaMemcpyHostToDevice);
  cudaMemcpy(r.p, R, sizeof(cplx) * rows * cols, cudaMemcpyHostToDevice);
  cudaError_t e;
  if (uh) e = hk::gemm_uh_r(a.as<cplx>(), K, M, K, r.as<cplx>(), K, N, c.as<cplx>(), M, nullptr);
  else if (coff) e = hk::gemm_a_rblk_h(a.as<cplx>(), M, M, K, r.as<cplx>(), N, coff, N, c.as<cplx>(), M, nullptr, mixed);
  else e = hk::gemm_a_rh(a.as<cplx>(), M, M, K, r.as<cplx>(), N, N, c.as<cplx>(), M, 0, 1, 1, nullptr, mixed);
  if (e != cudaSuccess) return e;
  return cudaMemcpy(C, c.p, sizeof(cplx) * M * N, cudaMemcpyDeviceToHost);
}

// Bytes of partial sums a product asks for.
long long probe_part_bytes(int M, int N, int K, int S) {
  return (long long)(hk::tc_part_elems(M, N, K, S ? S : hk::tc_wide_digits()) * sizeof(cplx));
}

int probe_reciprocals(int n, const double* x, double* rcp, double* rsq) {
  Buf dx(8ull * n), dr(8ull * n), ds(8ull * n);
  if (dx.e || dr.e || ds.e) return cudaErrorMemoryAllocation;
  cudaMemcpy(dx.p, x, 8ull * n, cudaMemcpyHostToDevice);
  reciprocal_kernel<<<(n + 255) / 256, 256>>>(n, dx.as<double>(), dr.as<double>(), ds.as<double>());
  cudaMemcpy(rcp, dr.p, 8ull * n, cudaMemcpyDeviceToHost);
  return cudaMemcpy(rsq, ds.p, 8ull * n, cudaMemcpyDeviceToHost);
}

// out[3 i ..]: tau, scale and (beta, 0) of the reflector of (alpha_i, |x|^2 = s2_i)
int probe_house(int n, const double* alpha, const double* s2, double* out) {
  Buf da(16ull * n), ds(8ull * n), dout(48ull * n);
  if (da.e || ds.e || dout.e) return cudaErrorMemoryAllocation;
  cudaMemcpy(da.p, alpha, 16ull * n, cudaMemcpyHostToDevice);
  cudaMemcpy(ds.p, s2, 8ull * n, cudaMemcpyHostToDevice);
  house_kernel<<<n, 32>>>(n, da.as<cplx>(), ds.as<double>(), dout.as<cplx>());
  return cudaMemcpy(out, dout.p, 48ull * n, cudaMemcpyDeviceToHost);
}

}  // extern "C"
