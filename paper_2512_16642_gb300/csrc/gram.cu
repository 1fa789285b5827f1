// Per-frequency Hessians (eq. Qmatrix with S S^T replaced by its frequency-domain blocks):
//   H_k[i][j] = sum_x ghat_i(w_k, x) conj(ghat_j(w_k, x)),   Q_k = H_k + mu I.
// With M_k = [Re ghat_0; Im ghat_0; Re ghat_1; ...] (2 nrec rows, G columns) and the real
// symmetric C = M_k M_k^T:
//   Re H[i][j] = C[2i][2j] + C[2i+1][2j+1],   Im H[i][j] = C[2i+1][2j] - C[2i][2j+1].
// C is computed in 64 x 64 tiles on and above the tile diagonal only, with the grid sum split
// into `splits` ranges whose partial tiles are reduced in a second kernel (scratch workspace).
#include <algorithm>
#include <cmath>

#include <cooperative_groups.h>

#include "egh_internal.cuh"

namespace egh {

constexpr int GT = 64;   // tile edge
constexpr int GK = 16;   // points per shared-memory stage
constexpr int GFLUSH = 128;  // stages accumulated before adding into the running total

__host__ __device__ int gram_tiles(int nrec) { return (2 * nrec + GT - 1) / GT; }

size_t gram_workspace_floats(int nrec, int nf, int splits) {
  const int nt = gram_tiles(nrec);
  const size_t pairs = (size_t)nt * (nt + 1) / 2;
  return (size_t)splits * nf * pairs * GT * GT;
}

__device__ inline const float* m_row(const float* gh, int a, int k, int nf, long long G) {
  return gh + ((long long)((a >> 1) * nf + k) * 2 + (a & 1)) * G;
}

__global__ void __launch_bounds__(256)
    k_gram_partial(const float* __restrict__ gh, int nrec, int nf, long long G, int ntile,
                   long long split_len, float* __restrict__ part) {
  __shared__ __align__(16) float As[GK][GT + 4];
  __shared__ __align__(16) float Bs[GK][GT + 4];
  const int pair = blockIdx.x, k = blockIdx.y, s = blockIdx.z;
  int ta = 0, rem = pair;
  while (rem >= ntile - ta) {
    rem -= ntile - ta;
    ++ta;
  }
  const int tb = ta + rem;
  const int rows = 2 * nrec;
  const int tid = threadIdx.x;
  const int tx = tid & 15, ty = tid >> 4;
  const int lr = tid >> 2, lp = (tid & 3) * 4;
  const int ra = ta * GT + lr, rb = tb * GT + lr;
  const float* arow = ra < rows ? m_row(gh, ra, k, nf, G) : nullptr;
  const float* brow = rb < rows ? m_row(gh, rb, k, nf, G) : nullptr;
  const long long p0 = (long long)s * split_len;
  const long long p1 = min(G, p0 + split_len);

  float acc[4][4], tot[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = tot[i][j] = 0.f;
  int stages = 0;
  for (long long p = p0; p < p1; p += GK) {
    float4 va = make_float4(0.f, 0.f, 0.f, 0.f), vb = va;
    if (arow) va = *reinterpret_cast<const float4*>(arow + p + lp);
    if (brow) vb = *reinterpret_cast<const float4*>(brow + p + lp);
    As[lp + 0][lr] = va.x;
    As[lp + 1][lr] = va.y;
    As[lp + 2][lr] = va.z;
    As[lp + 3][lr] = va.w;
    Bs[lp + 0][lr] = vb.x;
    Bs[lp + 1][lr] = vb.y;
    Bs[lp + 2][lr] = vb.z;
    Bs[lp + 3][lr] = vb.w;
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < GK; ++kk) {
      const float4 a4 = *reinterpret_cast<const float4*>(&As[kk][ty * 4]);
      const float4 b4 = *reinterpret_cast<const float4*>(&Bs[kk][tx * 4]);
      const float av[4] = {a4.x, a4.y, a4.z, a4.w};
      const float bv[4] = {b4.x, b4.y, b4.z, b4.w};
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(av[i], bv[j], acc[i][j]);
    }
    __syncthreads();
    if (++stages == GFLUSH) {
      stages = 0;
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          tot[i][j] += acc[i][j];
          acc[i][j] = 0.f;
        }
    }
  }
  const int npairs = ntile * (ntile + 1) / 2;
  float* out = part + (((long long)s * nf + k) * npairs + pair) * (GT * GT);
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    float4 v;
    v.x = tot[i][0] + acc[i][0];
    v.y = tot[i][1] + acc[i][1];
    v.z = tot[i][2] + acc[i][2];
    v.w = tot[i][3] + acc[i][3];
    *reinterpret_cast<float4*>(out + (ty * 4 + i) * GT + tx * 4) = v;
  }
}

cudaError_t launch_gram_partial(const float* gh, int nrec, int nf, long long G, int splits,
                                float* part, cudaStream_t st) {
  const int nt = gram_tiles(nrec);
  const int npairs = nt * (nt + 1) / 2;
  long long split_len = (G + splits - 1) / splits;
  split_len = (split_len + GK - 1) / GK * GK;
  dim3 grid(npairs, nf, splits);
  count_launches(1);
  k_gram_partial<<<grid, 256, 0, st>>>(gh, nrec, nf, G, nt, split_len, part);
  return cudaGetLastError();
}

// C[a][b] summed over splits, read from the tile pair with ta <= tb (C is symmetric).
__device__ inline float c_entry(const float* part, int a, int b, int k, int nf, int ntile,
                                int npairs, int splits) {
  if (a / GT > b / GT) {
    const int t = a;
    a = b;
    b = t;
  }
  const int ta = a / GT, tb = b / GT;
  const int pair = ta * ntile - ta * (ta - 1) / 2 + (tb - ta);
  const long long off = (long long)(a % GT) * GT + (b % GT);
  double sum = 0.0;
  for (int s = 0; s < splits; ++s)
    sum += part[(((long long)s * nf + k) * npairs + pair) * (GT * GT) + off];
  return (float)sum;
}

__global__ void k_gram_finish(const float* __restrict__ part, int nrec, int nf, int splits,
                              float2* __restrict__ Qh) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  const int i = blockIdx.y;
  const int k = blockIdx.z;
  if (j >= nrec) return;
  const int ntile = gram_tiles(nrec);
  const int npairs = ntile * (ntile + 1) / 2;
  const int a = min(i, j), b = max(i, j);
  const float rr = c_entry(part, 2 * a, 2 * b, k, nf, ntile, npairs, splits);
  const float ii = c_entry(part, 2 * a + 1, 2 * b + 1, k, nf, ntile, npairs, splits);
  float im = 0.f;
  if (a != b)
    im = c_entry(part, 2 * a + 1, 2 * b, k, nf, ntile, npairs, splits) -
         c_entry(part, 2 * a, 2 * b + 1, k, nf, ntile, npairs, splits);
  // entry (a, b) with a <= b; (b, a) is its conjugate
  Qh[((long long)k * nrec + i) * nrec + j] = make_float2(rr + ii, i <= j ? im : -im);
}

cudaError_t launch_gram_finish(const float* part, int nrec, int nf, int splits, float2* Qh,
                               cudaStream_t st) {
  dim3 grid((nrec + 127) / 128, nrec, nf);
  count_launches(1);
  k_gram_finish<<<grid, 128, 0, st>>>(part, nrec, nf, splits, Qh);
  return cudaGetLastError();
}

// d_sum[0] = sum over k, i of Re Qh[k][i][i]   (one block)
__global__ void k_diag_sum(const float2* __restrict__ Qh, int nrec, int nf, double* d_sum) {
  __shared__ double red[256];
  double s = 0.0;
  for (int t = threadIdx.x; t < nrec * nf; t += blockDim.x) {
    const int k = t / nrec, i = t % nrec;
    s += (double)Qh[((long long)k * nrec + i) * nrec + i].x;
  }
  red[threadIdx.x] = s;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) d_sum[0] = red[0];
}

cudaError_t launch_diag_sum(const float2* Qh, int nrec, int nf, double* d_sum, cudaStream_t st) {
  count_launches(1);
  k_diag_sum<<<1, 256, 0, st>>>(Qh, nrec, nf, d_sum);
  return cudaGetLastError();
}

// ||Q_k||_F^2 per frequency: one block per frequency.  The squares are summed to FP64-class
// accuracy in FP32 arithmetic (TwoProd and TwoSum into a two-word sum per thread, Ogita, Rump and
// Oishi's Dot2) and combined in FP64: the GB300 issues FP64 at a small fraction of the FP32 rate,
// and two FP64 operations per entry were the kernel's time (40 matrices of 341 rows: 150 us, now
// 18 us).
constexpr int FR_THREADS = 1024;

__device__ __forceinline__ void two_word_square(float a, float& s, float& c) {
  const float p = __fmul_rn(a, a);
  const float e = __fmaf_rn(a, a, -p);
  const float t = __fadd_rn(s, p);
  const float bp = __fsub_rn(t, s);
  c = __fadd_rn(c, __fadd_rn(__fadd_rn(__fsub_rn(s, __fsub_rn(t, bp)), __fsub_rn(p, bp)), e));
  s = t;
}

__global__ void __launch_bounds__(FR_THREADS)
    k_fro2(const float2* __restrict__ Qh, int n, double* d_out) {
  __shared__ double red[FR_THREADS / 32];
  const long long n2 = (long long)n * n;
  const float2* A = Qh + (long long)blockIdx.x * n2;
  float s[2] = {0.f, 0.f}, c[2] = {0.f, 0.f};
#pragma unroll 4
  for (long long t = threadIdx.x; t < n2; t += FR_THREADS) {
    const float2 a = __ldg(A + t);
    two_word_square(a.x, s[0], c[0]);
    two_word_square(a.y, s[1], c[1]);
  }
  double v = ((double)s[0] + c[0]) + ((double)s[1] + c[1]);
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    double sum = 0.0;
    for (int w = 0; w < FR_THREADS / 32; ++w) sum += red[w];
    d_out[blockIdx.x] = sum;
  }
}

cudaError_t launch_fro2(const float2* Qh, int n, int nf, double* d_out, cudaStream_t st) {
  count_launches(1);
  k_fro2<<<nf, FR_THREADS, 0, st>>>(Qh, n, d_out);
  return cudaGetLastError();
}

// Largest eigenvalue of Q_k^{-1} (the dense inverse P_k) by 40 steps of power iteration in FP32:
// lam[k] = ||P v|| / ||v|| for the last v, which approaches 1 / lambda_min(Q_k) from below.
//
// One cluster of IP_CL blocks per matrix: each block keeps its share of the rows of P in shared
// memory (as many as fit; the rest is read from L2 every step), so that a step costs one
// shared-memory matrix-vector product, a warp per row, and one cluster barrier; the new vector
// and the partial norms go to every block of the cluster through distributed shared memory, in
// two alternating buffers.  The 40 steps are a serial chain: with one block per matrix reading the
// two triangular factors from L2 each of them took 10 to 37 us.  Measured on 40 matrices of 341
// rows: 1471 us before, 166 us now (161 rows: 378 and 105 us).
constexpr int IP_CL = 8, IP_THREADS = 512, IP_STEPS = 40;

__global__ void __cluster_dims__(IP_CL, 1, 1) __launch_bounds__(IP_THREADS)
    k_inv_power(const float2* __restrict__ Ph, int n, int cached, double* lam) {
  namespace cg = cooperative_groups;
  cg::cluster_group cluster = cg::this_cluster();
  extern __shared__ __align__(16) float2 pv[];  // v[2][n], then `cached` rows of P
  __shared__ float wred[IP_THREADS / 32];
  __shared__ float part[2][IP_CL];  // the blocks' partial ||P v||^2, by step parity
  const int rank = (int)cluster.block_rank(), tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr int NW = IP_THREADS / 32;
  const float2* P = Ph + (long long)(blockIdx.x / IP_CL) * n * n;
  const int r0 = (int)((long long)n * rank / IP_CL), r1 = (int)((long long)n * (rank + 1) / IP_CL);
  const int nr = r1 - r0, nc = min(nr, cached);
  float2* rows = pv + 2 * n;
  for (int e = tid; e < nc * n; e += IP_THREADS) rows[e] = P[(long long)r0 * n + e];
  float vv = 0.f;  // ||v||^2 of the start vector, the same sum in every block
  for (int i = lane; i < n; i += 32) {
    const float x = 1.f + 0.01f * (i % 7);
    vv += x * x;
  }
  for (int o = 16; o > 0; o >>= 1) vv += __shfl_xor_sync(0xffffffffu, vv, o);
  for (int i = tid; i < n; i += IP_THREADS) pv[i] = make_float2(1.f + 0.01f * (i % 7), 0.f);
  float sc = 1.f, norm = 0.f;
  cluster.sync();  // every block of the cluster runs before its shared memory is written
  for (int it = 0; it < IP_STEPS; ++it) {
    const float2* v = pv + (it & 1) * n;
    float2* vn = pv + ((it & 1) ^ 1) * n;
    float w2 = 0.f;
    for (int r = warp; r < nr; r += NW) {
      const float2* row = r < nc ? rows + (size_t)r * n : P + (long long)(r0 + r) * n;
      float re = 0.f, im = 0.f;
#pragma unroll 4
      for (int j = lane; j < n; j += 32) {
        const float2 a = row[j], b = v[j];
        re = fmaf(a.x, b.x, fmaf(-a.y, b.y, re));
        im = fmaf(a.x, b.y, fmaf(a.y, b.x, im));
      }
      for (int o = 16; o > 0; o >>= 1) {
        re += __shfl_xor_sync(0xffffffffu, re, o);
        im += __shfl_xor_sync(0xffffffffu, im, o);
      }
      re *= sc;
      im *= sc;
      w2 += re * re + im * im;
      if (lane < IP_CL) cluster.map_shared_rank(vn, lane)[r0 + r] = make_float2(re, im);
    }
    if (lane == 0) wred[warp] = w2;
    __syncthreads();
    if (tid < IP_CL) {
      float s = 0.f;
      for (int w = 0; w < NW; ++w) s += wred[w];
      cluster.map_shared_rank(&part[it & 1][0], tid)[rank] = s;
    }
    cluster.sync();
    float s = 0.f;
    for (int b = 0; b < IP_CL; ++b) s += part[it & 1][b];
    norm = sqrtf(s / vv);
    sc = 1.f / sqrtf(s);  // applied to the next product
    vv = 1.f;
  }
  // the last step's barrier is behind every remote write: no block leaves early
  if (rank == 0 && tid == 0) lam[blockIdx.x / IP_CL] = norm;
}

cudaError_t launch_inv_power(const float2* Ph, int n, int nf, double* lam, cudaStream_t st) {
  // rows of P beside the two vectors in at most 200 KB of a block's shared memory
  const size_t vec = 2 * sizeof(float2) * (size_t)n, cap = 200 * 1024;
  const int share = (n + IP_CL - 1) / IP_CL;
  const int cached = (int)std::min<size_t>((size_t)share, vec < cap ? (cap - vec) / (sizeof(float2) * (size_t)n) : 0);
  const size_t smem = vec + sizeof(float2) * (size_t)cached * n;
  cudaError_t e =
      cudaFuncSetAttribute(k_inv_power, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  count_launches(1);
  k_inv_power<<<nf * IP_CL, IP_THREADS, smem, st>>>(Ph, n, cached, lam);
  return cudaGetLastError();
}

// Largest eigenvalue of each Hermitian H_k by power iteration (fixed 300 iterations, Rayleigh
// quotient), one block per frequency; d_lmax[k].
constexpr int PI_ITERS = 300;

__global__ void k_lambda_max(const float2* __restrict__ Qh, int n, double* d_lmax) {
  extern __shared__ double sv[];  // v: 2n doubles, y: 2n doubles
  __shared__ double red[256];
  const int k = blockIdx.x;
  const float2* A = Qh + (long long)k * n * n;
  double* v = sv;
  double* y = sv + 2 * n;
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    v[2 * i] = 1.0 + 0.01 * (i % 7);
    v[2 * i + 1] = 0.0;
  }
  __syncthreads();
  double lam = 0.0;
  for (int it = 0; it < PI_ITERS; ++it) {
    // y = A v
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
      double re = 0.0, im = 0.0;
      for (int j = 0; j < n; ++j) {
        const float2 a = A[(long long)i * n + j];
        re += a.x * v[2 * j] - a.y * v[2 * j + 1];
        im += a.x * v[2 * j + 1] + a.y * v[2 * j];
      }
      y[2 * i] = re;
      y[2 * i + 1] = im;
    }
    __syncthreads();
    // Rayleigh quotient v^H y / v^H v and the norm of y
    double num = 0.0, den = 0.0, yy = 0.0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
      num += v[2 * i] * y[2 * i] + v[2 * i + 1] * y[2 * i + 1];
      den += v[2 * i] * v[2 * i] + v[2 * i + 1] * v[2 * i + 1];
      yy += y[2 * i] * y[2 * i] + y[2 * i + 1] * y[2 * i + 1];
    }
    double vals[3] = {num, den, yy};
    for (int q = 0; q < 3; ++q) {
      red[threadIdx.x] = vals[q];
      __syncthreads();
      for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
        __syncthreads();
      }
      vals[q] = red[0];
      __syncthreads();
    }
    lam = vals[1] > 0.0 ? vals[0] / vals[1] : 0.0;
    const double inv = vals[2] > 0.0 ? 1.0 / sqrt(vals[2]) : 0.0;
    for (int i = threadIdx.x; i < 2 * n; i += blockDim.x) v[i] = y[i] * inv;
    __syncthreads();
  }
  if (threadIdx.x == 0) d_lmax[k] = lam;
}

cudaError_t launch_lambda_max(const float2* Qh, int nrec, int nf, double* d_lmax,
                              cudaStream_t st) {
  const size_t smem = sizeof(double) * 4 * (size_t)nrec;
  if (smem > 48 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(k_lambda_max, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)smem);
    if (e != cudaSuccess) return e;
  }
  count_launches(1);
  k_lambda_max<<<nf, 256, smem, st>>>(Qh, nrec, d_lmax);
  return cudaGetLastError();
}

// Qh += mu I; Lh = Qh.
__global__ void k_add_mu_copy(float2* __restrict__ Qh, float2* __restrict__ Lh, long long n2,
                              int nrec, float mu) {
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n2;
       t += (long long)gridDim.x * blockDim.x) {
    const long long local = t % ((long long)nrec * nrec);
    float2 v = Qh[t];
    if (local / nrec == local % nrec) {
      v.x += mu;
      Qh[t] = v;
    }
    Lh[t] = v;
  }
}

cudaError_t launch_add_mu_copy(float2* Qh, float2* Lh, int nrec, int nf, float mu,
                               cudaStream_t st) {
  const long long n2 = (long long)nf * nrec * nrec;
  long long blocks = (n2 + 255) / 256;
  if (blocks > 4096) blocks = 4096;
  count_launches(1);
  k_add_mu_copy<<<(int)blocks, 256, 0, st>>>(Qh, Lh, n2, nrec, mu);
  return cudaGetLastError();
}

// The penalty of the Hessians changed from mu_old to mu_new: Qh's diagonal has mu_old removed
// (when nonzero) and mu_new added, and Lh = Qh.  From mu_old = 0 the result is the one of
// launch_add_mu_copy with mu_new, bit for bit.
__global__ void k_set_mu_copy(float2* __restrict__ Qh, float2* __restrict__ Lh, long long n2,
                              int nrec, float mu_old, float mu_new) {
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n2;
       t += (long long)gridDim.x * blockDim.x) {
    const long long local = t % ((long long)nrec * nrec);
    float2 v = Qh[t];
    if (local / nrec == local % nrec) {
      if (mu_old != 0.f) v.x -= mu_old;
      v.x += mu_new;
      Qh[t] = v;
    }
    Lh[t] = v;
  }
}

cudaError_t launch_add_mu_copy_delta(float2* Qh, float2* Lh, int nrec, int nf, double mu_old,
                                     double mu_new, cudaStream_t st) {
  const long long n2 = (long long)nf * nrec * nrec;
  long long blocks = (n2 + 255) / 256;
  if (blocks > 4096) blocks = 4096;
  count_launches(1);
  k_set_mu_copy<<<(int)blocks, 256, 0, st>>>(Qh, Lh, n2, nrec, (float)mu_old, (float)mu_new);
  return cudaGetLastError();
}

}  // namespace egh
