// Screening stage (Sec. 3.3): Green's function on the real-space grid around
// the core hole along the imaginary frequency axis and the static RPA
// response from it,
//   G_j(r, r') = sum_K psi(r, K) conj(psi(r', K)) / (mu + i t_j - eps_K),
//   chi0(r, r') = (1/2 pi) sum_j w_j G_j(r, r') G_j(r', r),
// (Eqs. for chi^0 and G with omega' = mu + i t, d omega' = i dt), K = (n, k)
// running over bands and k-points.  G_j for all frequencies is one batched
// complex GEMM psi diag(d_j) psi^H in FP64 (tiles of psi staged in shared
// memory, the diagonal applied while staging); chi0 is an element-wise pass.
#include "bse_internal.cuh"

#include <algorithm>

namespace {

constexpr int GT = 32, GK = 16;   // output tile GT x GT, K chunk GK; 256 threads, 4 outputs each

__global__ void __launch_bounds__(256) green_kernel(const double2* __restrict__ psi, const double* __restrict__ eps,
                                                    int nr, int nkk, double mu, const double* __restrict__ t,
                                                    double2* __restrict__ G) {
  __shared__ double2 As[GT][GK + 1];   // psi(r, K) d_j(K)
  __shared__ double2 Bs[GT][GK + 1];   // conj(psi(r', K))
  const int j = blockIdx.z, r0 = blockIdx.y * GT, c0 = blockIdx.x * GT;
  const int tr = threadIdx.x / 8, tc = threadIdx.x % 8;   // rows r0 + tr, columns c0 + tc + 8 q
  const double tj = t[j];
  double ar[4] = {0, 0, 0, 0}, ai[4] = {0, 0, 0, 0};
  for (int k0 = 0; k0 < nkk; k0 += GK) {
    for (int e = threadIdx.x; e < GT * GK; e += blockDim.x) {
      const int rr = e / GK, kk = e % GK, r = r0 + rr, K = k0 + kk;
      double2 a = make_double2(0.0, 0.0), b = make_double2(0.0, 0.0);
      if (K < nkk) {
        // d = 1 / (mu - eps + i t) = (mu - eps - i t) / ((mu - eps)^2 + t^2)
        const double x = mu - eps[K], den = x * x + tj * tj;
        const double dr = x / den, di = -tj / den;
        if (r < nr) {
          const double2 p = psi[(size_t)r * nkk + K];
          a = make_double2(p.x * dr - p.y * di, p.x * di + p.y * dr);
        }
        const int c = c0 + rr;
        if (c < nr) {
          const double2 q = psi[(size_t)c * nkk + K];
          b = make_double2(q.x, -q.y);
        }
      }
      As[rr][kk] = a;
      Bs[rr][kk] = b;
    }
    __syncthreads();
#pragma unroll 4
    for (int kk = 0; kk < GK; ++kk) {
      const double2 a = As[tr][kk];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const double2 b = Bs[tc + 8 * q][kk];
        ar[q] += a.x * b.x - a.y * b.y;
        ai[q] += a.x * b.y + a.y * b.x;
      }
    }
    __syncthreads();
  }
  const int r = r0 + tr;
  if (r < nr) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int c = c0 + tc + 8 * q;
      if (c < nr) G[((size_t)j * nr + r) * nr + c] = make_double2(ar[q], ai[q]);
    }
  }
}

// chi0[r][c] = (1/2 pi) sum_j w_j G_j[r][c] G_j[c][r]
__global__ void chi0_kernel(const double2* __restrict__ G, const double* __restrict__ w, int nr, int nt,
                            double2* __restrict__ chi) {
  const size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  if (e >= (size_t)nr * nr) return;
  const int r = (int)(e / nr), c = (int)(e % nr);
  double sr = 0.0, si = 0.0;
  for (int j = 0; j < nt; ++j) {
    const double2 a = G[((size_t)j * nr + r) * nr + c], b = G[((size_t)j * nr + c) * nr + r];
    sr += w[j] * (a.x * b.x - a.y * b.y);
    si += w[j] * (a.x * b.y + a.y * b.x);
  }
  const double s = 1.0 / (2.0 * 3.14159265358979323846);
  chi[e] = make_double2(sr * s, si * s);
}

// d_j(K) = 1 / (mu - eps_K + i t_j)
__global__ void green_weights(const double* __restrict__ eps, int nkk, double mu, const double* __restrict__ t,
                              double2* __restrict__ d) {
  const int K = blockIdx.x * blockDim.x + threadIdx.x;
  if (K >= nkk) return;
  const double tj = t[blockIdx.y];
  const double x = mu - eps[K], den = x * x + tj * tj;
  d[(size_t)blockIdx.y * nkk + K] = make_double2(x / den, -tj / den);
}

// G of the elements that bse_oz_refused lists (j << 32 | r << 16 | r'), one warp each
__global__ void __launch_bounds__(256) green_repair(const double2* __restrict__ psi, const double2* __restrict__ d, int nr,
                                                    int nkk, const unsigned long long* __restrict__ list, unsigned cap,
                                                    const unsigned* __restrict__ count, double2* __restrict__ G) {
  const unsigned m = count[0] <= cap ? count[0] : min(count[1], cap), lane = threadIdx.x & 31;
  for (unsigned w = blockIdx.x * 8 + (threadIdx.x >> 5); w < m; w += gridDim.x * 8) {
    const unsigned j = (unsigned)(list[w] >> 32), r = (unsigned)(list[w] >> 16) & 0xffffu, c = (unsigned)list[w] & 0xffffu;
    const double2 *a = psi + (size_t)r * nkk, *b = psi + (size_t)c * nkk, *dj = d + (size_t)j * nkk;
    double2 s = make_double2(0.0, 0.0);
    for (int K = lane; K < nkk; K += 32) {
      const double2 p = a[K], q = b[K], e = dj[K];
      const double x = p.x * e.x - p.y * e.y, y = p.x * e.y + p.y * e.x;
      s.x = fma(x, q.x, fma(y, q.y, s.x));
      s.y = fma(y, q.x, fma(-x, q.y, s.y));
    }
    for (int off = 16; off > 0; off >>= 1) {
      s.x += __shfl_xor_sync(0xffffffffu, s.x, off);
      s.y += __shfl_xor_sync(0xffffffffu, s.y, off);
    }
    if (lane == 0) G[((size_t)j * nr + r) * nr + c] = s;
  }
}

struct Scratch {
  void* p = nullptr;
  ~Scratch() {
    if (p) cudaFree(p);
  }
};

// G_j on the tensor cores (k_oz.cu): the rows psi(r, :) d_j against the row
// pairs of psi(r', :), as many frequencies per pass as the scratch holds.
// *done = false (and nothing but G written) where the scratch or the kernel's
// set-up cannot be had, psi d_j holds Inf/NaN or a magnitude outside 2^+-400, a
// bounded wait gave up, or more than one element in 32 of a pass is refused
// (oz_accept; fewer are formed on the FP64 pipe).
bse_status green_tensor(const double2* psi, const double* eps, int nr, int nkk, double mu, const double* t, int nt,
                        double2* G, cudaStream_t st, bool* done) {
  *done = false;
  const int kp = bse_oz_kp(2 * nkk);
  const size_t per = bse_oz_digit_bytes(1, nr, kp), fixed = bse_oz_digit_bytes(1, 2 * nr, kp);
  const size_t budget = (size_t)512 << 20;
  int nj = (int)(budget / per);
  nj = nj < 1 ? 1 : (nj > nt ? nt : nj);
  const size_t bd = bse_oz_digit_bytes(nj, nr, kp);
  const size_t tab = ((size_t)nt * nkk * sizeof(double2) + 255) / 256 * 256;
  const size_t sca = ((size_t)nj * nr * sizeof(double) + 255) / 256 * 256;
  const size_t scb = ((size_t)2 * nr * sizeof(double) + 255) / 256 * 256;
  const size_t nma = ((size_t)nj * nr * sizeof(float2) + 255) / 256 * 256, nmb = ((size_t)nr * sizeof(float2) + 255) / 256 * 256;
  const size_t cap = std::min<size_t>((size_t)nj * nr * nr / 32 + 1024, (size_t)1 << 22);
  const size_t lst = (cap * sizeof(unsigned long long) + 255) / 256 * 256;
  Scratch sc;
  if (cudaMalloc(&sc.p, bd + fixed + tab + sca + scb + nma + nmb + lst + 256) != cudaSuccess) {
    cudaGetLastError();
    sc.p = nullptr;
    return BSE_OK;
  }
  char* q = (char*)sc.p;
  bse_oz_operand a, b;
  a.digits = q, q += bd;
  b.digits = q, q += fixed;
  double2* d = (double2*)q;
  q += tab;
  a.scale = (double*)q, q += sca;
  b.scale = (double*)q, q += scb;
  a.norm = (float2*)q, q += nma;
  b.norm = (float2*)q, q += nmb;
  unsigned long long* list = (unsigned long long*)q;
  q += lst;
  int* word = (int*)q;   // {wait gave up, out of range or too many refused, elements refused (two)}
  a.rows = nr, b.rows = 2 * nr;
  a.kp = b.kp = kp;
  cudaMemsetAsync(word, 0, 2 * sizeof(int), st);
  green_weights<<<dim3((unsigned)((nkk + 255) / 256), (unsigned)nt), 256, 0, st>>>(eps, nkk, mu, t, d);
  bse_status s = bse_oz_split_rows(psi, nr, nkk, nullptr, 1, 1, b, word + 1, st);
  for (int j = 0; j < nt && s == BSE_OK; j += nj) {
    const int n = nt - j < nj ? nt - j : nj;
    a.batches = n;
    s = bse_oz_split_rows(psi, nr, nkk, d + (size_t)j * nkk, n, 0, a, word + 1, st);
    if (s == BSE_OK)
      s = bse_oz_gemm(a, b, n, 1.0, (double*)(G + (size_t)j * nr * nr), 2ll * nr * nr, 4ll * nr, 2ll * nr, 1, word, st);
    if (s == BSE_OK) s = bse_oz_refused(a, b, n, list, (unsigned)cap, (unsigned*)word + 2, word + 1, st);
    if (s == BSE_OK)
      green_repair<<<608, 256, 0, st>>>(psi, d + (size_t)j * nkk, nr, nkk, list, (unsigned)cap, (unsigned*)word + 2,
                                        G + (size_t)j * nr * nr);
  }
  int hw[2] = {0, 0};
  if (s == BSE_OK && (cudaMemcpyAsync(hw, word, sizeof(hw), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
                      cudaStreamSynchronize(st) != cudaSuccess))
    s = BSE_ERR_CUDA;
  if (s != BSE_OK) {
    cudaStreamSynchronize(st);   // before the scratch goes
    return s == BSE_ERR_UNSUPPORTED ? BSE_OK : s;
  }
  *done = hw[0] == 0 && hw[1] == 0;
  return BSE_OK;
}

}  // namespace

bse_status bse_screening_device(const double2* psi, const double* eps, int nr, int nkk, double mu, const double* t,
                                const double* w, int nt, double2* G, double2* chi, cudaStream_t st) {
  // from 2^22 complex products on (FP64 kernel: about 0.1 ms) the tensor-core
  // form; K is bounded by its 64-bit partial sums
  bool done = false;
  if ((double)nr * nr * nkk * nt >= 4194304.0 && nkk <= (1 << 20)) {
    const bse_status s = green_tensor(psi, eps, nr, nkk, mu, t, nt, G, st, &done);
    if (s != BSE_OK) return s;
  }
  if (!done) {
    const dim3 g((unsigned)((nr + GT - 1) / GT), (unsigned)((nr + GT - 1) / GT), (unsigned)nt);
    green_kernel<<<g, 256, 0, st>>>(psi, eps, nr, nkk, mu, t, G);
  }
  const size_t n = (size_t)nr * nr;
  chi0_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(G, w, nr, nt, chi);
  return cudaGetLastError() == cudaSuccess ? BSE_OK : BSE_ERR_CUDA;
}
