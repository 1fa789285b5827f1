// Per-frequency Hessians (eq. Qmatrix with S S^T replaced by its frequency-domain blocks):
//   H_k[i][j] = sum_x ghat_i(w_k, x) conj(ghat_j(w_k, x)),   Q_k = H_k + mu I.
// With M_k = [Re ghat_0; Im ghat_0; Re ghat_1; ...] (2 nrec rows, G columns) and the real
// symmetric C = M_k M_k^T:
//   Re H[i][j] = C[2i][2j] + C[2i+1][2j+1],   Im H[i][j] = C[2i+1][2j] - C[2i][2j+1].
// C is computed in square tiles on and above the tile diagonal only, with the grid sum split
// into `splits` ranges whose partial tiles are reduced in a second kernel (scratch workspace).
#include <algorithm>
#include <cmath>

#include <cooperative_groups.h>

#include "egh_internal.cuh"

namespace egh {

constexpr int GK = 16;       // points per shared-memory stage
constexpr int GST = 3;       // stages in the ring
constexpr int GFLUSH = 128;  // stages accumulated before adding into the running total

// Tile edge of the FP32 Gram: 128 (8 x 8 entries per thread) or 64 (4 x 4).  The larger tile reads
// each staged value for twice the products; the smaller one computes less past the last receiver,
// so it is taken where that is a third less: up to 32 and from 65 to 96 receivers.  Measured with 64
// and with 128: 30 receivers 0.92 and 1.19 ms, 85 receivers (0.6 of the tiles' entries with 64) 3.21
// and 3.49 ms, 150 receivers (0.71) 17.0 and 16.3 ms, 212 receivers (0.78) 19.7 and 17.3 ms.  The
// warps of a 128-row diagonal tile that lie below the diagonal, a quarter of it, compute nothing.
int gram_tile_edge(int nrec) {
  const long long n64 = (2LL * nrec + 63) / 64, n128 = (2LL * nrec + 127) / 128;
  const long long a64 = n64 * (n64 + 1) / 2, a128 = n128 * (n128 + 1) / 2 * 4 - n128;
  return 3 * a64 < 2 * a128 ? 64 : 128;
}

__host__ __device__ int gram_tiles(int nrec, int edge) { return (2 * nrec + edge - 1) / edge; }

size_t gram_workspace_floats(int nrec, int nf, int splits, int edge) {
  const int nt = gram_tiles(nrec, edge);
  const size_t pairs = (size_t)nt * (nt + 1) / 2;
  return (size_t)splits * nf * pairs * edge * edge;
}

__device__ inline const float* m_row(const float* gh, int a, int k, int nf, long long G) {
  return gh + ((long long)((a >> 1) * nf + k) * 2 + (a & 1)) * G;
}

__device__ __forceinline__ void gram_cp4(unsigned dst, const float* src, bool ok) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(ok ? 4 : 0)
               : "memory");
}

// One tile pair of C at one frequency over one range of points, in FP32 on the CUDA cores.  Rows
// arrive by cp.async, turned on the way ([point][row], three stages in the ring, one barrier per
// stage); a thread reads 2 R values per point for R^2 products, taken as packed FP32x2 FMAs over
// two adjacent rows.  Every sum runs over the points in order, and every GFLUSH stages of the range
// it is added into a total in shared memory (fixed ranges of points: the sums do not depend on the
// tile edge).  Columns of the padded rows past the grid (x >= nx, zero) are skipped.
//
// Bound by the FP32 FMA rate: 231 receivers x 26 frequencies x 349 184 points took 75.7 ms with 64 x
// 64 tiles (4 x 4 entries per thread, two barriers per 16 points and no loads in flight across
// them), 67.4 ms with these tiles in the order of their index, now 60.4 ms.  520 blocks are 1.7
// rounds of the 304 that fit, and the sums' fixed ranges of points allow no other split; so the full
// tiles start first, then those of the last, partial column, then the diagonal with its idle half.
template <int R>
__global__ void __launch_bounds__(256, 2)
    k_gram_partial(const float* __restrict__ gh, int nrec, int nf, long long G, int ntile, int nsplit,
                   long long split_len, int px, int xe, float* __restrict__ part) {
  constexpr int T = 16 * R;     // tile edge: 4 x 2 warps of 4 x 8 lanes with R x R entries each
  constexpr int H = R / 4;      // groups of four adjacent rows (columns) per thread
  // [GST][A, B][GK][T], then totals [R * R][256].  Row r of a staged point p sits at r ^ 4 (p % 8):
  // the copies, which turn 16 points at a time, then meet two to a bank, and two blocks fit an SM
  extern __shared__ __align__(16) float gsm[];
  float* tot = gsm + GST * 2 * GK * T;
  // the tile pair is the slowest index: off the diagonal column by column, then the diagonal
  const int ks = nf * nsplit, order = blockIdx.x / ks, k = (blockIdx.x - order * ks) % nf,
            s = (blockIdx.x - order * ks) / nf;
  int ta = order, tb = 1;
  while (tb < ntile && ta >= tb) ta -= tb++;
  if (tb == ntile) tb = ta;
  const int pair = ta * ntile - ta * (ta - 1) / 2 + (tb - ta);
  const bool diag = ta == tb;  // B is A
  const int rows = 2 * nrec;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const long long p0 = (long long)s * split_len;
  const long long p1 = min(G, p0 + split_len);
  // copies of a stage: point tid % 16 of rows tid / 16 + 16 q of each operand
  const int cp = tid & 15, cr = tid >> 4;
  const unsigned ring = (unsigned)__cvta_generic_to_shared(gsm) + (unsigned)(cp * T) * 4u;
  const int csw = 4 * (cp & 7);
  // rows 2 r, 2 r + 1 of M_k are the planes of receiver r: row a starts at (a / 2 * nf * 2 + a % 2) G;
  // 16 rows on is 8 receivers on
  const float* srcA = m_row(gh, ta * T + cr, k, nf, G) + cp;
  const float* srcB = m_row(gh, tb * T + cr, k, nf, G) + cp;
  const long long step16 = 16LL * nf * G;
  // stages of the range that hold grid columns: point p, column x of its row
  auto advance = [&](long long& p, int& x) {
    p += GK;
    x += GK;
    if (px > 0 && x >= xe) {
      p += px - x;
      x = 0;
    }
  };
  auto begin = [&](long long& p, int& x) {
    p = p0;
    x = px > 0 ? (int)(p0 % px) : 0;
    if (px > 0 && x >= xe) {
      p += px - x;
      x = 0;
    }
  };
  long long lp, mp;  // next stage to copy, stage to multiply
  int lx, mx;
  begin(lp, lx);
  begin(mp, mx);
  auto issue = [&](int buf) {
    if (lp < p1) {
      const unsigned dst = ring + (unsigned)(buf * 2 * GK * T) * 4u;
#pragma unroll
      for (int q = 0; q < R; ++q) {
        const bool in = ta * T + cr + 16 * q < rows;
        gram_cp4(dst + 4u * ((cr + 16 * q) ^ csw), in ? srcA + q * step16 + lp : gh, in);
      }
      if (!diag) {
#pragma unroll
        for (int q = 0; q < R; ++q) {
          const bool in = tb * T + cr + 16 * q < rows;
          gram_cp4(dst + 4u * (GK * T + ((cr + 16 * q) ^ csw)), in ? srcB + q * step16 + lp : gh, in);
        }
      }
      advance(lp, lx);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");  // empty groups keep the count uniform
  };
  // this thread's entries: rows ra + 4 R h + i, columns rb + 8 R h + j (i, j < 4, h < H) of the tile
  const int wr = (warp >> 1) * 4 * R, wc = (warp & 1) * 8 * R;
  const int ra = wr + 4 * (lane >> 3), rb = wc + 4 * (lane & 7);
  const bool work = !(diag && wr >= wc + 8 * R) && ta * T + wr < rows && tb * T + wc < rows;
  float2 acc[R / 2][R];  // adjacent rows as pairs
#pragma unroll
  for (int i = 0; i < R / 2; ++i)
#pragma unroll
    for (int j = 0; j < R; ++j) {
      acc[i][j] = make_float2(0.f, 0.f);
      tot[(2 * i * R + j) * 256 + tid] = 0.f;
      tot[((2 * i + 1) * R + j) * 256 + tid] = 0.f;
    }
  long long flush_at = p0 + (long long)GFLUSH * GK;
  issue(0);
  issue(1);
  int buf = 0;
  while (mp < p1) {
    asm volatile("cp.async.wait_group 1;" ::: "memory");
    __syncthreads();  // the stage has landed; every thread is done with the one before
    issue(buf == 0 ? 2 : buf - 1);
    while (mp >= flush_at) {
#pragma unroll
      for (int i = 0; i < R / 2; ++i)
#pragma unroll
        for (int j = 0; j < R; ++j) {
          tot[(2 * i * R + j) * 256 + tid] += acc[i][j].x;
          tot[((2 * i + 1) * R + j) * 256 + tid] += acc[i][j].y;
          acc[i][j] = make_float2(0.f, 0.f);
        }
      flush_at += (long long)GFLUSH * GK;
    }
    if (work) {
      const float* A = gsm + buf * 2 * GK * T;
      const float* B = gsm + (buf * 2 + (diag ? 0 : 1)) * GK * T;
#pragma unroll
      for (int q = 0; q < GK; ++q) {
        float4 a[H], b[H];
#pragma unroll
        for (int h = 0; h < H; ++h) {
          a[h] = *reinterpret_cast<const float4*>(A + q * T + ((ra + 16 * h) ^ (4 * (q & 7))));
          b[h] = *reinterpret_cast<const float4*>(B + q * T + ((rb + 32 * h) ^ (4 * (q & 7))));
        }
#pragma unroll
        for (int h = 0; h < H; ++h) {
          const float bv[4] = {b[h].x, b[h].y, b[h].z, b[h].w};
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const float2 bb = make_float2(bv[j], bv[j]);
#pragma unroll
            for (int g = 0; g < H; ++g) {
              acc[2 * g][4 * h + j] = __ffma2_rn(make_float2(a[g].x, a[g].y), bb, acc[2 * g][4 * h + j]);
              acc[2 * g + 1][4 * h + j] = __ffma2_rn(make_float2(a[g].z, a[g].w), bb, acc[2 * g + 1][4 * h + j]);
            }
          }
        }
      }
    }
    advance(mp, mx);
    buf = buf == GST - 1 ? 0 : buf + 1;
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  const int npairs = ntile * (ntile + 1) / 2;
  float* out = part + (((long long)s * nf + k) * npairs + pair) * (T * T);
#pragma unroll
  for (int i = 0; i < R; ++i)
#pragma unroll
    for (int h = 0; h < H; ++h) {
      float v[4];
#pragma unroll
      for (int j = 0; j < 4; ++j)
        v[j] = tot[(i * R + 4 * h + j) * 256 + tid] + (i & 1 ? acc[i / 2][4 * h + j].y : acc[i / 2][4 * h + j].x);
      *reinterpret_cast<float4*>(out + (ra + 16 * (i / 4) + i % 4) * T + rb + 32 * h) =
          make_float4(v[0], v[1], v[2], v[3]);
    }
}

cudaError_t launch_gram_partial(const float* gh, int nrec, int nf, long long G, int splits, int edge,
                                int px, int nx, float* part, cudaStream_t st) {
  const int nt = gram_tiles(nrec, edge);
  const int npairs = nt * (nt + 1) / 2;
  if ((edge != 64 && edge != 128) || px % GK != 0) return cudaErrorInvalidValue;
  long long split_len = (G + splits - 1) / splits;
  split_len = (split_len + GK - 1) / GK * GK;
  const int R = edge / 16;
  auto bytes = [](int r) { return (GST * 2 * GK * 16 * r + r * r * 256) * (int)sizeof(float); };
  const int smem = bytes(R);
  auto kern = R == 8 ? k_gram_partial<8> : k_gram_partial<4>;
  // both instances, so that a later call with the other tile edge loads no code
  cudaError_t e;
  if ((e = cudaFuncSetAttribute(k_gram_partial<8>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes(8))) ||
      (e = cudaFuncSetAttribute(k_gram_partial<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes(4))))
    return e;
  const long long blocks = (long long)npairs * nf * splits;
  if (blocks > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
  count_launches(1);
  kern<<<(unsigned)blocks, 256, smem, st>>>(gh, nrec, nf, G, nt, splits, split_len, px,
                                        (nx + GK - 1) / GK * GK, part);
  return cudaGetLastError();
}

// C[a][b] summed over splits, read from the tile pair with ta <= tb (C is symmetric).
__device__ inline float c_entry(const float* part, int a, int b, int k, int nf, int ntile,
                                int npairs, int splits, int T) {
  if (a / T > b / T) {
    const int t = a;
    a = b;
    b = t;
  }
  const int ta = a / T, tb = b / T;
  const int pair = ta * ntile - ta * (ta - 1) / 2 + (tb - ta);
  const long long off = (long long)(a % T) * T + (b % T);
  double sum = 0.0;
  for (int s = 0; s < splits; ++s)
    sum += part[(((long long)s * nf + k) * npairs + pair) * (T * T) + off];
  return (float)sum;
}

__global__ void k_gram_finish(const float* __restrict__ part, int nrec, int nf, int splits, int T,
                              float2* __restrict__ Qh) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  const int i = blockIdx.y;
  const int k = blockIdx.z;
  if (j >= nrec) return;
  const int ntile = gram_tiles(nrec, T);
  const int npairs = ntile * (ntile + 1) / 2;
  const int a = min(i, j), b = max(i, j);
  const float rr = c_entry(part, 2 * a, 2 * b, k, nf, ntile, npairs, splits, T);
  const float ii = c_entry(part, 2 * a + 1, 2 * b + 1, k, nf, ntile, npairs, splits, T);
  float im = 0.f;
  if (a != b)
    im = c_entry(part, 2 * a + 1, 2 * b, k, nf, ntile, npairs, splits, T) -
         c_entry(part, 2 * a, 2 * b + 1, k, nf, ntile, npairs, splits, T);
  // entry (a, b) with a <= b; (b, a) is its conjugate
  Qh[((long long)k * nrec + i) * nrec + j] = make_float2(rr + ii, i <= j ? im : -im);
}

cudaError_t launch_gram_finish(const float* part, int nrec, int nf, int splits, int edge,
                               float2* Qh, cudaStream_t st) {
  dim3 grid((nrec + 127) / 128, nrec, nf);
  count_launches(1);
  k_gram_finish<<<grid, 128, 0, st>>>(part, nrec, nf, splits, edge, Qh);
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

// ||Q_k||_F^2 per frequency in FP64: one cluster per matrix, the blocks' sums joined by the first one
// through distributed shared memory, in order.  Bound by the FP64 rate (a conversion and an FMA per real
// number, two lanes a cycle and SM), so a matrix is spread over FR_CL SMs: 40 matrices of 341 rows took
// 150 us with a block each, now 54 us.  (Two-word FP32 sums took 28 us, but are off by 1e-12 where the
// entries' roundings all go one way.)
constexpr int FR_CL = 8, FR_THREADS = 256;

__global__ void __cluster_dims__(FR_CL, 1, 1) __launch_bounds__(FR_THREADS)
    k_fro2(const float2* __restrict__ Qh, int n, double* d_out) {
  namespace cg = cooperative_groups;
  cg::cluster_group cluster = cg::this_cluster();
  __shared__ double red[FR_THREADS / 32];
  __shared__ double part[FR_CL];
  const int rank = (int)cluster.block_rank(), tid = threadIdx.x;
  const long long n2 = (long long)n * n;
  const float2* A = Qh + (long long)(blockIdx.x / FR_CL) * n2;
  double s = 0.0, c = 0.0;
#pragma unroll 4
  for (long long t = rank * FR_THREADS + tid; t < n2; t += FR_CL * FR_THREADS) {
    const float2 a = __ldg(A + t);
    const double x = a.x, y = a.y;
    s = fma(x, x, s);
    c = fma(y, y, c);
  }
  s += c;
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((tid & 31) == 0) red[tid >> 5] = s;
  cluster.sync();  // (every block of the cluster runs before its shared memory is written)
  if (tid == 0) {
    double sum = 0.0;
    for (int w = 0; w < FR_THREADS / 32; ++w) sum += red[w];
    cluster.map_shared_rank(part, 0)[rank] = sum;
  }
  cluster.sync();
  if (rank == 0 && tid == 0) {
    double sum = 0.0;
    for (int b = 0; b < FR_CL; ++b) sum += part[b];
    d_out[blockIdx.x / FR_CL] = sum;
  }
}

cudaError_t launch_fro2(const float2* Qh, int n, int nf, double* d_out, const Lane& lane) {
  count_launches(1);
  return launch_on(lane, false, k_fro2, nf * FR_CL, FR_THREADS, 0, Qh, n, d_out);
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
// rows: 1471 us before, 304 us now (257 rows: 800 and 166 us, 161 rows: 378 and 105 us).
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

cudaError_t launch_inv_power(const float2* Ph, int n, int nf, double* lam, const Lane& lane) {
  // rows of P beside the two vectors in at most 200 KB of a block's shared memory
  const size_t vec = 2 * sizeof(float2) * (size_t)n, cap = 200 * 1024;
  const int share = (n + IP_CL - 1) / IP_CL;
  const int cached = (int)std::min<size_t>((size_t)share, vec < cap ? (cap - vec) / (sizeof(float2) * (size_t)n) : 0);
  const size_t smem = vec + sizeof(float2) * (size_t)cached * n;
  const cudaError_t e = allow_block_smem<k_inv_power>();
  if (e != cudaSuccess) return e;
  count_launches(1);
  return launch_on(lane, false, k_inv_power, nf * IP_CL, IP_THREADS, smem, Ph, n, cached, lam);
}

// Largest eigenvalue of each Hermitian H_k by power iteration in FP64 (fixed 300 iterations, Rayleigh
// quotient of the last), one cluster of blocks per matrix as k_inv_power: the blocks' rows of H_k in
// shared memory (as doubles where they fit, which saves the conversions), eight lanes per row, the
// vector handed round through distributed shared memory, the norm taken by one thread.  Bound by the
// FP64 rate, two lanes a cycle and SM: one block per matrix left it to one SM each and every thread
// took the root and the quotient (26 matrices of 100 rows 10.0 ms; a band-limited update 147 ms then,
// 139 ms now).
constexpr int PI_ITERS = 300, LM_THREADS = 256, LM_L = 8;  // lanes per row

template <typename T>  // float2 or double2: the rows in shared memory
__global__ void __cluster_dims__(IP_CL, 1, 1) __launch_bounds__(LM_THREADS)
    k_lambda_max(const float2* __restrict__ Qh, int n, int cached, double* d_lmax) {
  namespace cg = cooperative_groups;
  cg::cluster_group cluster = cg::this_cluster();
  extern __shared__ __align__(16) double2 lv[];  // v[2][n], then `cached` rows of H
  constexpr int NW = LM_THREADS / 32;
  __shared__ double wred[3][NW];
  __shared__ double part[2][3][IP_CL];  // the blocks' partial sums, by iteration parity
  __shared__ double inv_s;
  const int rank = (int)cluster.block_rank(), tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const float2* A = Qh + (long long)(blockIdx.x / IP_CL) * n * n;
  const int r0 = (int)((long long)n * rank / IP_CL), r1 = (int)((long long)n * (rank + 1) / IP_CL);
  const int nr = r1 - r0, nc = min(nr, cached);
  T* rows = reinterpret_cast<T*>(lv + 2 * n);
  for (int e = tid; e < nc * n; e += LM_THREADS) {
    const float2 a = A[(long long)r0 * n + e];
    rows[e] = T{a.x, a.y};
  }
  for (int i = tid; i < n; i += LM_THREADS) lv[i] = make_double2(1.0 + 0.01 * (i % 7), 0.0);
  double inv = 1.0, lam = 0.0;
  const int g = tid / LM_L, l = tid % LM_L;
  cluster.sync();  // every block of the cluster runs before its shared memory is written
  for (int it = 0; it < PI_ITERS; ++it) {
    const double2* v = lv + (it & 1) * n;
    double2* vn = lv + ((it & 1) ^ 1) * n;
    const bool last = it == PI_ITERS - 1;
    double yy = 0.0, num = 0.0, den = 0.0;
    for (int rb = warp * (32 / LM_L); rb < nr; rb += LM_THREADS / LM_L) {  // warp-uniform
      const int r = rb + (g & (32 / LM_L - 1));
      double re = 0.0, im = 0.0;
      if (r < nc) {
        const T* row = rows + (size_t)r * n;
        for (int j = l; j < n; j += LM_L) {
          const T a = row[j];
          const double2 b = v[j];
          re = fma((double)a.x, b.x, fma(-(double)a.y, b.y, re));
          im = fma((double)a.x, b.y, fma((double)a.y, b.x, im));
        }
      } else if (r < nr) {
        const float2* row = A + (long long)(r0 + r) * n;
        for (int j = l; j < n; j += LM_L) {
          const float2 a = row[j];
          const double2 b = v[j];
          re = fma((double)a.x, b.x, fma(-(double)a.y, b.y, re));
          im = fma((double)a.x, b.y, fma((double)a.y, b.x, im));
        }
      }
      for (int o = LM_L / 2; o > 0; o >>= 1) {
        re += __shfl_xor_sync(0xffffffffu, re, o);
        im += __shfl_xor_sync(0xffffffffu, im, o);
      }
      if (r < nr) {
        re *= inv;  // v holds the unscaled product of the iteration before
        im *= inv;
        if (l == 0) {
          yy = fma(re, re, fma(im, im, yy));
          if (last) {  // Rayleigh quotient v^H y / v^H v
            const double2 x = make_double2(v[r0 + r].x * inv, v[r0 + r].y * inv);
            num = fma(x.x, re, fma(x.y, im, num));
            den = fma(x.x, x.x, fma(x.y, x.y, den));
          }
        }
        cluster.map_shared_rank(vn, l)[r0 + r] = make_double2(re, im);  // lane l to block l
      }
    }
    for (int o = 16; o >= LM_L; o >>= 1) {  // the rows' first lanes
      yy += __shfl_xor_sync(0xffffffffu, yy, o);
      if (last) {
        num += __shfl_xor_sync(0xffffffffu, num, o);
        den += __shfl_xor_sync(0xffffffffu, den, o);
      }
    }
    if (lane == 0) {
      wred[0][warp] = yy;
      wred[1][warp] = num;
      wred[2][warp] = den;
    }
    __syncthreads();
    if (tid < 3 * IP_CL && (last || tid < IP_CL)) {
      const int q = tid / IP_CL, to = tid % IP_CL;
      double s = 0.0;
      for (int w = 0; w < NW; ++w) s += wred[q][w];
      cluster.map_shared_rank(&part[it & 1][0][0], to)[q * IP_CL + rank] = s;
    }
    cluster.sync();
    if (tid == 0) {
      double s = 0.0;
      for (int b = 0; b < IP_CL; ++b) s += part[it & 1][0][b];
      inv_s = s > 0.0 ? 1.0 / sqrt(s) : 0.0;
      if (last) {
        double sn = 0.0, sd = 0.0;
        for (int b = 0; b < IP_CL; ++b) {
          sn += part[it & 1][1][b];
          sd += part[it & 1][2][b];
        }
        lam = sd > 0.0 ? sn / sd : 0.0;
      }
    }
    __syncthreads();
    inv = inv_s;
  }
  if (rank == 0 && tid == 0) d_lmax[blockIdx.x / IP_CL] = lam;
}

cudaError_t launch_lambda_max(const float2* Qh, int nrec, int nf, double* d_lmax,
                              cudaStream_t st) {
  static_assert(LM_L == IP_CL, "lane l of a row's group writes to block l");
  const size_t vec = 2 * sizeof(double2) * (size_t)nrec, cap = 200 * 1024;
  const int share = (nrec + IP_CL - 1) / IP_CL;
  const bool dbl = vec + sizeof(double2) * (size_t)share * nrec <= cap;
  const size_t el = dbl ? sizeof(double2) : sizeof(float2);
  const int cached =
      (int)std::min<size_t>((size_t)share, vec < cap ? (cap - vec) / (el * (size_t)nrec) : 0);
  const size_t smem = vec + el * (size_t)cached * nrec;
  auto kern = dbl ? k_lambda_max<double2> : k_lambda_max<float2>;
  const cudaError_t e = dbl ? allow_block_smem<k_lambda_max<double2>>() : allow_block_smem<k_lambda_max<float2>>();
  if (e != cudaSuccess) return e;
  count_launches(1);
  kern<<<nf * IP_CL, LM_THREADS, smem, st>>>(Qh, nrec, cached, d_lmax);
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
