// Cholesky factorisation of every frequency's Hessian, Q_k = L_k L_k^H, in one launch
// (Algorithm 2 inverts each frequency's matrix; here the Hermitian positive-definite blocks
// are factored and kept resident instead).  One block per frequency, right-looking:
// for each column j the pivot is checked (non-positive or non-finite -> status[k] = j + 1 and the
// block stops, no trap), the column is scaled and cached in shared memory, and each warp updates
// whole rows of the trailing lower triangle with coalesced row accesses.  The upper triangle is
// zeroed at the end.
#include <algorithm>
#include <cmath>

#include "egh_internal.cuh"

namespace egh {

constexpr int CH_THREADS = 512;

// piv64: the diagonal is carried in FP64 (dg[i] = Q[i][i] - sum_l |L[i][l]|^2 accumulated in
// double from the stored FP32 columns) and each pivot is taken from it, so the pivots of
// ill-conditioned matrices do not inherit the FP32 cancellation of the trailing updates; the
// off-diagonal entries stay FP32.
// Factors one n x n matrix in place with the calling block (status: 0 or failing pivot + 1).
__device__ void potrf_block(float2* __restrict__ A, int n, int* __restrict__ status_k, int piv64,
                            float2* col, double* dg, int& bad) {
  const int tid = threadIdx.x;
  const int lane = tid & 31, warp = tid >> 5, nwarps = blockDim.x >> 5;
  if (tid == 0) bad = 0;
  __syncthreads();
  if (piv64)
    for (int i = tid; i < n; i += blockDim.x) dg[i] = (double)A[(long long)i * n + i].x;
  __syncthreads();
  for (int j = 0; j < n; ++j) {
    if (tid == 0) {
      const double d = piv64 ? dg[j] : (double)A[(long long)j * n + j].x;
      if (!(d > 0.0) || !isfinite(d)) {
        bad = j + 1;
      } else {
        const float s = piv64 ? (float)sqrt(d) : sqrtf((float)d);
        A[(long long)j * n + j] = make_float2(s, 0.f);
        col[j] = make_float2(s, 0.f);
      }
    }
    __syncthreads();
    if (bad) break;
    const float inv = 1.f / col[j].x;
    for (int i = j + 1 + tid; i < n; i += blockDim.x) {
      float2 v = A[(long long)i * n + j];
      v.x *= inv;
      v.y *= inv;
      A[(long long)i * n + j] = v;
      col[i] = v;
      if (piv64) dg[i] -= (double)v.x * v.x + (double)v.y * v.y;
    }
    __syncthreads();
    // A[i][l] -= col[i] * conj(col[l]),  j < l <= i
    for (int i = j + 1 + warp; i < n; i += nwarps) {
      const float2 ci = col[i];
      float2* rowp = A + (long long)i * n;
      for (int l = j + 1 + lane; l <= i; l += 32) {
        const float2 cl = col[l];
        float2 a = rowp[l];
        a.x -= ci.x * cl.x + ci.y * cl.y;
        a.y -= ci.y * cl.x - ci.x * cl.y;
        rowp[l] = a;
      }
    }
    __syncthreads();
  }
  if (tid == 0) *status_k = bad;
  if (!bad) {
    for (long long t = tid; t < (long long)n * n; t += blockDim.x) {
      const int i = (int)(t / n), l = (int)(t % n);
      if (l > i) A[t] = make_float2(0.f, 0.f);
    }
  }
}

// Blocked form (matrices whose 32-column panel fits in shared memory).  A panel of rows p0 .. n-1
// and columns p0 .. p0+31 sits in shared memory:
//   - its diagonal tile is factored by one warp, a lane holding 8 columns of a row in registers and
//     each new column passed on by shuffles;
//   - every row below is solved against that tile by one thread, 8 columns at a time in registers,
//     the tile read as broadcasts (rows are independent: no barrier per column; 32 columns at a
//     time make straight-line code of 4000 instructions, which a single warp fetches more slowly
//     than it runs: the launch then takes 825 us);
//   - the trailing lower triangle takes the panel's rank-32 update in one pass over global memory,
//     A[i][l] -= sum_c P[i][c] conj(P[l][c]), in 16 x 32 tiles per warp with 4 x 4 entries per lane
//     (16 FMAs per shared-memory read).
// Same pivot rule and FP64 diagonal as the column form, and every entry takes the same operations in
// the same order for any block size (the solves of ill-conditioned sets magnify a changed rounding
// of the factor by their condition).  One block factors one matrix, so the time
// of the largest matrix bounds a launch; it was three barriers per column and two shared-memory
// reads per four FMAs: 120 matrices of 161, 257 and 341 rows in mixed precision took 933 us (1024
// threads a block), now 605 us (512 threads).
constexpr int CH_PB = 32, CH_PS = CH_PB + 1;  // panel width, panel row stride (float2)
constexpr int CH_PANEL_NMAX = 800;            // panel of n x 33 float2 + n doubles in 227 KB

// (float)sqrt(d) of a positive double.  The float root with one Newton correction, its residual taken
// in double, is within 2.6e-14 of the root (half the square of the start's 9e-8, the correction's
// roundings, 4 x 2^-24 of 9e-8); where both ends of a wider range round to one float, so does the
// double root between them, and its long chain of FP64 operations is only taken next to the middle of
// two floats, once in some 10^6 pivots.  (The root stands in the chain of columns: the range's ends in
// FP64 cost 75 us of the 2.50 ms of three patches.)
__device__ __forceinline__ float root_to_float(double d) {
  const float f = (float)d;
  if (!(f > 1e-30f) || !(f < 1e30f)) return (float)sqrt(d);
  const float s = sqrtf(f);
  const float c = (float)fma(-(double)s, (double)s, d) * (0.5f / s), t = 3.2e-14f * s;
  const float lo = s + (c - t), hi = s + (c + t);
  return lo == hi ? lo : (float)sqrt(d);
}

constexpr int CH_SB = 8;  // columns a thread holds at a time (unrolled code, run 4 times a panel)

struct alignas(16) PotrfShared {
  float2 LT[CH_PB][CH_PB];  // LT[j][c] = the diagonal tile's entry (c, j), c > j
  float inv[CH_PB];         // reciprocal pivots
};

// x[q] -= y conj(l[q]) for the CH_SB columns at l
__device__ __forceinline__ void rank1_sub(float2 (&x)[CH_SB], float2 y, const float4* l) {
#pragma unroll
  for (int h = 0; h < CH_SB / 2; ++h) {
    const float4 v = l[h];
    x[2 * h].x -= y.x * v.x + y.y * v.y;
    x[2 * h].y -= y.y * v.x - y.x * v.y;
    x[2 * h + 1].x -= y.x * v.z + y.y * v.w;
    x[2 * h + 1].y -= y.y * v.z - y.x * v.w;
  }
}

__device__ void potrf_block_panel(float2* __restrict__ A, int n, int* __restrict__ status_k,
                                  int piv64, float2* P, double* dg, PotrfShared& sh, int& bad_s) {
  const int tid = threadIdx.x;
  const int lane = tid & 31, warp = tid >> 5, nwarps = blockDim.x >> 5;
  if (tid == 0) bad_s = 0;
  for (int i = tid; i < n; i += blockDim.x) dg[i] = (double)A[(long long)i * n + i].x;
  __syncthreads();
  for (int p0 = 0; p0 < n; p0 += CH_PB) {
    const int pw = min(CH_PB, n - p0), R = n - p0;
    // panel rows p0 .. n-1, columns p0 .. p0+pw-1 (zero beyond; entries above the diagonal are
    // not used)
    for (int r = warp; r < R; r += nwarps)
      P[r * CH_PS + lane] = lane < pw ? A[(long long)(p0 + r) * n + p0 + lane] : make_float2(0.f, 0.f);
    __syncthreads();
    if (warp == 0) {
      const bool in = lane < pw;  // a row of the tile (the panel has only these when n is small)
      double d = in ? dg[p0 + lane] : 1.0;
      int bad = 0;
      for (int j0 = 0; j0 < pw && !bad; j0 += CH_SB) {  // all warp-uniform
        float2 a[CH_SB];
#pragma unroll
        for (int q = 0; q < CH_SB; ++q) a[q] = in ? P[lane * CH_PS + j0 + q] : make_float2(0.f, 0.f);
        // the columns before, in order
        for (int c = 0; c < j0; ++c)
          rank1_sub(a, in ? P[lane * CH_PS + c] : make_float2(0.f, 0.f),
                    reinterpret_cast<const float4*>(&sh.LT[c][j0]));
#pragma unroll
        for (int q = 0; q < CH_SB; ++q) {
          if (j0 + q < pw && !bad) {
            const double dj = piv64 ? __shfl_sync(0xffffffffu, d, j0 + q)
                                    : (double)__shfl_sync(0xffffffffu, a[q].x, j0 + q);
            if (!(dj > 0.0) || !isfinite(dj)) {
              bad = p0 + j0 + q + 1;
            } else {
              const float s = piv64 ? root_to_float(dj) : sqrtf((float)dj), inv = 1.f / s;
              if (lane == j0 + q) {
                a[q] = make_float2(s, 0.f);
              } else {
                a[q].x *= inv;
                a[q].y *= inv;
              }
              if (lane == 0) sh.inv[j0 + q] = inv;
              if (piv64 && lane > j0 + q) d -= (double)a[q].x * a[q].x + (double)a[q].y * a[q].y;
#pragma unroll
              for (int c = q + 1; c < CH_SB; ++c) {  // a[c] of lanes above row j0 + c is not used
                const float cx = __shfl_sync(0xffffffffu, a[q].x, j0 + c);
                const float cy = __shfl_sync(0xffffffffu, a[q].y, j0 + c);
                a[c].x -= a[q].x * cx + a[q].y * cy;
                a[c].y -= a[q].y * cx - a[q].x * cy;
              }
            }
          }
        }
#pragma unroll
        for (int q = 0; q < CH_SB; ++q) {
          if (in) P[lane * CH_PS + j0 + q] = a[q];
          sh.LT[j0 + q][lane] = a[q];
        }
        __syncwarp();
      }
      if (bad && lane == 0) bad_s = bad;
    }
    __syncthreads();
    if (bad_s) break;
    // rows below the tile: x L^H = a, CH_SB columns at a time: the earlier columns in order, then
    // each new entry at once subtracted from the later ones (pw = 32 whenever there are rows below)
    for (int r = CH_PB + tid; r < R; r += blockDim.x) {
      float2* row = P + r * CH_PS;
      double d = dg[p0 + r];
      for (int j0 = 0; j0 < CH_PB; j0 += CH_SB) {
        float2 x[CH_SB];
#pragma unroll
        for (int q = 0; q < CH_SB; ++q) x[q] = row[j0 + q];
#pragma unroll 2
        for (int c = 0; c < j0; ++c)
          rank1_sub(x, row[c], reinterpret_cast<const float4*>(&sh.LT[c][j0]));
#pragma unroll
        for (int q = 0; q < CH_SB; ++q) {
          const float inv = sh.inv[j0 + q];
          x[q].x *= inv;
          x[q].y *= inv;
          if (piv64) d -= (double)x[q].x * x[q].x + (double)x[q].y * x[q].y;
#pragma unroll
          for (int c = q + 1; c < CH_SB; ++c) {
            const float2 l = sh.LT[j0 + q][j0 + c];
            x[c].x -= x[q].x * l.x + x[q].y * l.y;
            x[c].y -= x[q].y * l.x - x[q].x * l.y;
          }
          row[j0 + q] = x[q];
        }
      }
      dg[p0 + r] = d;
    }
    __syncthreads();
    // the factored panel back to A (lower part only)
    for (int r = warp; r < R; r += nwarps)
      if (lane < pw && lane <= r) A[(long long)(p0 + r) * n + p0 + lane] = P[r * CH_PS + lane];
    // trailing rank-32 update: rows and columns q0 .. n-1, tiles of 16 rows x 32 columns that
    // touch the lower triangle
    const int q0 = p0 + CH_PB, m = n - q0;
    if (m > 0) {
      const int tx = lane & 7, ty = lane >> 3;
      const int nti = (m + 15) / 16;
      // row tile ti (16 rows) needs the column tiles 0 .. ti / 2
      int ti = 0, tj = warp;
      while (true) {
        while (ti < nti && tj > ti / 2) {
          tj -= ti / 2 + 1;
          ++ti;
        }
        if (ti >= nti) break;
        const int ib = 16 * ti + ty, lb = 32 * tj + tx;  // first row and column of this lane
        float2 v[4][4], s[4][4];
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
          for (int b = 0; b < 4; ++b) {
            const int i = ib + 4 * a, l = lb + 8 * b;
            v[a][b] = (i < m && l <= i) ? A[(long long)(q0 + i) * n + q0 + l] : make_float2(0.f, 0.f);
            s[a][b] = make_float2(0.f, 0.f);
          }
        int ra[4], rb[4];  // panel rows, kept inside the panel (the sums past m are not stored)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          ra[q] = (CH_PB + min(ib + 4 * q, m - 1)) * CH_PS;
          rb[q] = (CH_PB + min(lb + 8 * q, m - 1)) * CH_PS;
        }
#pragma unroll 2
        for (int c = 0; c < CH_PB; ++c) {
          float2 x[4], y[4];
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            x[q] = P[ra[q] + c];
            y[q] = P[rb[q] + c];
          }
#pragma unroll
          for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b) {
              s[a][b].x = fmaf(x[a].x, y[b].x, fmaf(x[a].y, y[b].y, s[a][b].x));
              s[a][b].y = fmaf(x[a].y, y[b].x, fmaf(-x[a].x, y[b].y, s[a][b].y));
            }
        }
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
          for (int b = 0; b < 4; ++b) {
            const int i = ib + 4 * a, l = lb + 8 * b;
            if (i < m && l <= i)
              A[(long long)(q0 + i) * n + q0 + l] =
                  make_float2(v[a][b].x - s[a][b].x, v[a][b].y - s[a][b].y);
          }
        tj += nwarps;
      }
    }
    __syncthreads();
  }
  if (tid == 0) *status_k = bad_s;
  if (!bad_s) {
    for (int i = warp; i < n; i += nwarps)
      for (int l = i + 1 + lane; l < n; l += 32) A[(long long)i * n + l] = make_float2(0.f, 0.f);
  }
}

// shared memory for every matrix size up to nmax: the blocked form for n <= CH_PANEL_NMAX needs
// the panel and its diagonal tile, the column form beyond it one column; a batch may hold both kinds
// (225.9 KB for the panel of an 800-row matrix)
constexpr size_t potrf_smem(int nmax) {
  const size_t np = (size_t)std::min(nmax, CH_PANEL_NMAX);
  const size_t panel = sizeof(PotrfShared) + sizeof(float2) * np * CH_PS + sizeof(double) * np;
  if (nmax <= CH_PANEL_NMAX) return panel;
  const size_t column = sizeof(float2) * (size_t)(nmax + (nmax & 1)) + sizeof(double) * (size_t)nmax;
  return std::max(panel, column);
}

// the column form's 14527 rows, and the panel's, fit a block beside the status word
static_assert(potrf_smem(14527) + sizeof(int) <= kBlockSmem && potrf_smem(CH_PANEL_NMAX) + sizeof(int) <= kBlockSmem);

__device__ inline void potrf_any(float2* A, int n, int* status_k, int piv64, float2* buf, int& bad) {
  if (n <= CH_PANEL_NMAX) {
    PotrfShared& sh = *reinterpret_cast<PotrfShared*>(buf);
    float2* P = reinterpret_cast<float2*>(&sh + 1);
    potrf_block_panel(A, n, status_k, piv64, P, reinterpret_cast<double*>(P + (size_t)n * CH_PS), sh, bad);
  } else {
    potrf_block(A, n, status_k, piv64, buf, reinterpret_cast<double*>(buf + n + (n & 1)), bad);
  }
}

__global__ void __launch_bounds__(CH_THREADS)
    k_potrf(float2* __restrict__ Lh, int n, int* __restrict__ status, int piv64) {
  extern __shared__ __align__(16) float2 pbuf[];  // panel (or column) cache, then the FP64 diagonal
  __shared__ int bad;
  const int k = blockIdx.x;
  potrf_any(Lh + (long long)k * n * n, n, status + k, piv64, pbuf, bad);
}

// Batched form: every matrix of a list (several survey patches x all their frequencies, of
// different sizes) in one persistent launch; block b factors matrices b, b + gridDim.x, ...
template <int THREADS>
__global__ void __launch_bounds__(THREADS)
    k_potrf_many(const PotrfItem* __restrict__ items, int count, int piv64) {
  extern __shared__ __align__(16) float2 col[];  // sized for the largest matrix
  __shared__ int bad;
  for (int m = blockIdx.x; m < count; m += gridDim.x) {
    const PotrfItem it = items[m];
    potrf_any(it.A, it.n, it.status, piv64, col, bad);
    __syncthreads();
  }
}

cudaError_t potrf_many_prepare(int nmax) {
  if (potrf_smem(nmax) + sizeof(int) > (size_t)kBlockSmem) return cudaErrorInvalidValue;
  const cudaError_t e = allow_block_smem<k_potrf_many<256>>();
  return e ? e : allow_block_smem<k_potrf_many<512>>();
}

cudaError_t launch_potrf_many(const PotrfItem* items, int count, int nmax, int blocks, int threads,
                              int piv64, const Lane& lane) {
  const size_t smem = potrf_smem(nmax);
  if (threads != 256 && threads != 512) return cudaErrorInvalidValue;
  count_launches(1);
  return launch_on(lane, false, threads == 256 ? k_potrf_many<256> : k_potrf_many<512>, blocks, threads, smem,
                   items, count, piv64);
}

cudaError_t launch_potrf(float2* Lh, int n, int nf, int* status, cudaStream_t st, int piv64) {
  const size_t smem = potrf_smem(n);
  if (smem > 47 * 1024) {  // (beside the status word)
    const cudaError_t e = allow_block_smem<k_potrf>();
    if (e != cudaSuccess) return e;
  }
  count_launches(1);
  k_potrf<<<nf, CH_THREADS, smem, st>>>(Lh, n, status, piv64);
  return cudaGetLastError();
}

}  // namespace egh
