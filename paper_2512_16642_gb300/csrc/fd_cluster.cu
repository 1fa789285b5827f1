// Finite-difference solver for small grids: one thread-block cluster per receiver pair, the whole
// wavefield of the pair in the cluster's shared memory for a chunk of steps (Section "Direct
// Hessian-inverse computation": one wave-equation solve per receiver, eq. wave_eq; the scheme is
// the one of fd.cu, the same operations in the same order, so both give identical levels).
//
// On a small grid the per-step kernel is bound by a launch and by its warps' first rows, not by
// work: the 141 x 141 padded grid with 16 receivers takes 4.5 us a step on 36 of 152 SMs.  Here
// the padded rows are split evenly over the CL blocks of a cluster, each block holds both levels
// of its rows (4 halo rows above and below, 4 zero columns on each side) and, where they fit, the
// coefficients; a unit is (2 adjacent columns, SR rows) and its thread marches down the rows with
// the z first differences in registers, as fd.cu does.  The new level overwrites u^{n-1} in
// place; the rows a neighbour needs go to its halo through distributed shared memory as they are
// computed, and one cluster barrier ends the step (a halo written in a step belongs to the buffer
// that no block reads before that barrier).  The snapshot of a level is written by the step after
// it, which has the values in registers anyway, so that the barrier's release does not wait for
// fresh global stores.  A batch's clusters run side by side; no block waits for another cluster.
//
// Bound by shared-memory reads (8 of 16 bytes per 2 points of a pair and row) and the barrier.
// 101 x 101 grid, 21 receivers x 1000 steps, 5 frequencies: the whole model update 11.4 ms with the
// per-step kernel as it was, 9.4 ms as it is now, 3.5 ms with this one.
#include <cuda_bf16.h>

#include <algorithm>

#include <cooperative_groups.h>

#include "egh_internal.cuh"
#include "tc.cuh"

namespace egh {

namespace {

constexpr int CL = 8;  // blocks per cluster (the largest portable size)

__device__ __forceinline__ float2 csub2(float2 a, float2 b) {
  return __ffma2_rn(b, make_float2(-1.f, -1.f), a);  // a - b, one rounding
}

__device__ __forceinline__ unsigned cbf2(__nv_bfloat162 v) { return *reinterpret_cast<unsigned*>(&v); }

__device__ __forceinline__ void csplit(float a, float b, unsigned& hi, unsigned& lo) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
  const float2 hf = __bfloat1622float2(h);
  const float2 r = csub2(make_float2(a, b), hf);
  hi = cbf2(h);
  lo = cbf2(__floats2bfloat162_rn(r.x, r.y));
}

// the first-difference Laplacian of fd.cu (same operation order)
__device__ __forceinline__ float2 clap2(const float2 (&dz)[8], const float2* e, const float2 (&cz)[4],
                                        const float2 (&cx)[4]) {
  float2 l = __fmul2_rn(cz[0], csub2(dz[4], dz[3]));
  l = __ffma2_rn(cz[1], csub2(dz[5], dz[2]), l);
  l = __ffma2_rn(cz[2], csub2(dz[6], dz[1]), l);
  l = __ffma2_rn(cz[3], csub2(dz[7], dz[0]), l);
  l = __ffma2_rn(cx[0], csub2(e[4], e[3]), l);
  l = __ffma2_rn(cx[1], csub2(e[5], e[2]), l);
  l = __ffma2_rn(cx[2], csub2(e[6], e[1]), l);
  l = __ffma2_rn(cx[3], csub2(e[7], e[0]), l);
  return l;
}

struct ClArgs {
  float2* lev;         // [3][pslot][F] state slots (level t in slot t mod 3)
  long long F;         // float2 per level per pair
  int pslot;           // pairs per state slot
  long long org;       // padded point (0, 0) inside a level
  int NZ, NX, PX;
  const float2* coef;  // (c1, c3) per padded point, pitched like a level
  int ta, nsteps;      // levels ta .. ta + nsteps - 1 are computed
  int t0, decim, sbase;  // snapshot of level t: ring slot sbase + (t - t0) / decim if t % decim == 0
  __nv_bfloat16* snap;   // ring base (hi plane of slot 0)
  long long sslot, splane, srec;  // elements per ring slot, hi -> lo plane, per receiver
  const float* wav;    // wavelet samples (level t takes sample t - 1), or null
  int nw;              // their number
  const int* pts;      // each receiver's point (offset inside a level)
  int nrec;            // receivers of the batch
  float scale;         // 1 / (dx dz)
  int rows;            // rows per block at most
  Stencil C;           // cumulative weights C_j
};

// two values of one receiver pair at two adjacent points, split, to the snapshot planes
__device__ __forceinline__ void snap_store(__nv_bfloat16* sp, long long plane, long long rec, float2 v0,
                                           float2 v1) {
  unsigned ha, la, hb, lb;
  csplit(v0.x, v1.x, ha, la);
  csplit(v0.y, v1.y, hb, lb);
  __stcs(reinterpret_cast<unsigned*>(sp), ha);
  __stcs(reinterpret_cast<unsigned*>(sp + plane), la);
  __stcs(reinterpret_cast<unsigned*>(sp + rec), hb);
  __stcs(reinterpret_cast<unsigned*>(sp + rec + plane), lb);
}

template <int SR, bool CSM>
__global__ void __launch_bounds__(512, 1) k_fd_cluster(const ClArgs a) {
  namespace cg = cooperative_groups;
  cg::cluster_group cluster = cg::this_cluster();
  extern __shared__ __align__(16) float4 csm[];
  const int tid = threadIdx.x, nthr = blockDim.x;
  const int rank = (int)cluster.block_rank(), pair = blockIdx.x / CL;
  const int NXH = (a.NX + 1) >> 1, RS = NXH + 4;  // float4 per row: 2 zero ones on each side
  const int LV = (a.rows + 8) * RS;               // float4 per level
  const int z0 = a.NZ * rank / CL, VR = a.NZ * (rank + 1) / CL - z0;
  float4* cf = csm + 2 * LV;                      // [rows][NXH]
  const long long pb = (long long)pair * a.F + a.org;
  // both levels with their halos (rows outside the grid and columns past it stay zero)
  for (int b = 0; b < 2; ++b) {
    const int s = b == 0 ? (a.ta - 1) % 3 : (a.ta - 2 + 3) % 3;
    const float2* src = a.lev + (long long)s * a.pslot * a.F + pb;
    for (int e = tid; e < LV; e += nthr) {
      const int r = e / RS - 4, z = z0 + r, x = 2 * (e % RS - 2);
      float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
      // (column NX of an odd grid is padding of the level, zero)
      if (r < VR + 4 && z >= 0 && z < a.NZ && x >= 0 && x < a.NX)
        v = __ldcg(reinterpret_cast<const float4*>(src + (long long)z * a.PX + x));
      csm[b * LV + e] = v;
    }
  }
  if (CSM)
    for (int e = tid; e < VR * NXH; e += nthr)
      cf[e] = __ldg(reinterpret_cast<const float4*>(a.coef + a.org + (long long)(z0 + e / NXH) * a.PX +
                                                    2 * (e % NXH)));
  // this pair's source points (rows of this block, columns)
  int sr_[2] = {-1, -1}, sx_[2] = {-1, -1};
  if (a.wav)
    for (int u = 0; u < 2; ++u)
      if (2 * pair + u < a.nrec) {
        const int p = a.pts[2 * pair + u] - (int)a.org;
        sr_[u] = p / a.PX - z0;
        sx_[u] = p % a.PX;
      }
  float2 cz2[4], cx2[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    cz2[j] = make_float2(a.C.cz[j], a.C.cz[j]);
    cx2[j] = make_float2(a.C.cx[j], a.C.cx[j]);
  }
  // the neighbours' copies of row r of a level: above holds my rows 0..3 below its own rows, below
  // holds my last four rows above its own
  const int VRa = rank > 0 ? z0 - a.NZ * (rank - 1) / CL : 0;
  float4* above = rank > 0 ? cluster.map_shared_rank(csm, rank - 1) : nullptr;
  float4* below = rank + 1 < CL ? cluster.map_shared_rank(csm, rank + 1) : nullptr;
  const int nseg = (VR + SR - 1) / SR, nunits = NXH * nseg;
  cluster.sync();
  for (int it = 0; it < a.nsteps; ++it) {
    const int t = a.ta + it;
    const int bc = it & 1, bn = bc ^ 1;  // current level, previous level (overwritten by the new)
    // the current level's snapshot (the first one was written before this launch)
    __nv_bfloat16* sl = nullptr;
    if (it > 0 && (t - 1) % a.decim == 0)
      sl = a.snap + (long long)(a.sbase + (t - 1 - a.t0) / a.decim) * a.sslot + (long long)(2 * pair) * a.srec;
    const float amp = a.wav && t - 1 < a.nw ? a.wav[t - 1] : 0.f;
    for (int u = tid; u < nunits; u += nthr) {
      const int q = u % NXH, r0 = (u / NXH) * SR;
      const float4* cu = csm + bc * LV + q;  // slot q + 2 of row r + 4 is the unit's centre
      float4* pv = csm + bn * LV + q + 2;
      const int x = 2 * q;
      const bool ok1 = x + 1 < a.NX;
      float2 dz[2][8], ul[2];
      {
        const float4 v = cu[r0 * RS + 2];
        ul[0] = make_float2(v.x, v.y);
        ul[1] = make_float2(v.z, v.w);
      }
#pragma unroll
      for (int k = 1; k < 8; ++k) {
        const float4 v = cu[(r0 + k) * RS + 2];
        const float2 nv[2] = {make_float2(v.x, v.y), make_float2(v.z, v.w)};
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          dz[i][k] = csub2(nv[i], ul[i]);
          ul[i] = nv[i];
        }
      }
#pragma unroll
      for (int ii = 0; ii < SR; ++ii) {
        const int r = r0 + ii;
        if (r >= VR) break;
        {
          const float4 v = cu[(r + 8) * RS + 2];
          const float2 nv[2] = {make_float2(v.x, v.y), make_float2(v.z, v.w)};
#pragma unroll
          for (int i = 0; i < 2; ++i) {
#pragma unroll
            for (int m = 0; m < 7; ++m) dz[i][m] = dz[i][m + 1];
            dz[i][7] = csub2(nv[i], ul[i]);
            ul[i] = nv[i];
          }
        }
        // u^n at row r, points x - 4 .. x + 5 (both receivers of the pair)
        const float4* xr = cu + (r + 4) * RS;
        const float4 A0 = xr[0], A1 = xr[1], A2 = xr[2], A3 = xr[3], A4 = xr[4];
        const float2 w[10] = {make_float2(A0.x, A0.y), make_float2(A0.z, A0.w), make_float2(A1.x, A1.y),
                              make_float2(A1.z, A1.w), make_float2(A2.x, A2.y), make_float2(A2.z, A2.w),
                              make_float2(A3.x, A3.y), make_float2(A3.z, A3.w), make_float2(A4.x, A4.y),
                              make_float2(A4.z, A4.w)};
        if (sl) snap_store(sl + (long long)(z0 + r) * a.PX + x, a.splane, a.srec, w[4], w[5]);
        float2 e[9];
#pragma unroll
        for (int m = 0; m < 9; ++m) e[m] = csub2(w[m + 1], w[m]);
        const float4 uo = pv[(r + 4) * RS];
        const float4 cc = CSM ? cf[r * NXH + q]
                              : __ldg(reinterpret_cast<const float4*>(a.coef + a.org + (long long)(z0 + r) * a.PX + x));
        const float2 l0 = clap2(dz[0], e, cz2, cx2), l1 = clap2(dz[1], e + 1, cz2, cx2);
        // u^{n+1} = c3 L u + c1 (u - u^{n-1}) + u^{n-1}
        const float2 o0 = make_float2(uo.x, uo.y), o1 = make_float2(uo.z, uo.w);
        float2 v0 = __ffma2_rn(make_float2(cc.y, cc.y), l0,
                               __ffma2_rn(make_float2(cc.x, cc.x), csub2(w[4], o0), o0));
        float2 v1 = __ffma2_rn(make_float2(cc.w, cc.w), l1,
                               __ffma2_rn(make_float2(cc.z, cc.z), csub2(w[5], o1), o1));
        if (!ok1) v1 = make_float2(0.f, 0.f);
        if (amp != 0.f) {  // the wavelet sample at the receivers' points
          if (r == sr_[0]) {
            if (x == sx_[0]) v0.x = v0.x + cc.y * amp * a.scale;
            if (x + 1 == sx_[0]) v1.x = v1.x + cc.w * amp * a.scale;
          }
          if (r == sr_[1]) {
            if (x == sx_[1]) v0.y = v0.y + cc.y * amp * a.scale;
            if (x + 1 == sx_[1]) v1.y = v1.y + cc.w * amp * a.scale;
          }
        }
        const float4 v = make_float4(v0.x, v0.y, v1.x, v1.y);
        pv[(r + 4) * RS] = v;
        if (r < 4 && above) above[bn * LV + (VRa + 4 + r) * RS + q + 2] = v;
        if (r >= VR - 4 && below) below[bn * LV + (r - (VR - 4)) * RS + q + 2] = v;
      }
    }
    cluster.sync();
  }
  // the last level's snapshot, and the last two levels back to their state slots
  const int t1 = a.ta + a.nsteps;
  const int bl = a.nsteps & 1;  // buffer of level t1 - 1
  if ((t1 - 1) % a.decim == 0) {
    __nv_bfloat16* sl = a.snap + (long long)(a.sbase + (t1 - 1 - a.t0) / a.decim) * a.sslot +
                        (long long)(2 * pair) * a.srec;
    for (int e = tid; e < VR * NXH; e += nthr) {
      const int r = e / NXH, q = e % NXH;
      const float4 v = csm[bl * LV + (r + 4) * RS + q + 2];
      snap_store(sl + (long long)(z0 + r) * a.PX + 2 * q, a.splane, a.srec, make_float2(v.x, v.y),
                 make_float2(v.z, v.w));
    }
  }
  for (int b = 0; b < 2; ++b) {
    const int s = (t1 - 1 - b) % 3;
    float2* dst = a.lev + (long long)s * a.pslot * a.F + pb;
    for (int e = tid; e < VR * NXH; e += nthr) {
      const int r = e / NXH, q = e % NXH;
      __stcg(reinterpret_cast<float4*>(dst + (long long)(z0 + r) * a.PX + 2 * q),
             csm[(bl ^ b) * LV + (r + 4) * RS + q + 2]);
    }
  }
}

constexpr int kSR[] = {2, 3, 4, 6, 8, 11};

template <bool CSM>
void* kernel_of(int sr) {
  switch (sr) {
    case 2: return (void*)k_fd_cluster<2, CSM>;
    case 3: return (void*)k_fd_cluster<3, CSM>;
    case 4: return (void*)k_fd_cluster<4, CSM>;
    case 6: return (void*)k_fd_cluster<6, CSM>;
    case 8: return (void*)k_fd_cluster<8, CSM>;
    default: return (void*)k_fd_cluster<11, CSM>;
  }
}

}  // namespace

bool fd_cluster_plan(const Layout& L, ClGeom* out) {
  if (L.NZ < 4 * CL) return false;  // a neighbour's halo comes from one block: four rows at least
  int dev = 0, optin = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess)
    return false;
  ClGeom g{};
  g.rows = (L.NZ + CL - 1) / CL;
  const int NXH = (L.NX + 1) / 2;
  const size_t lev = sizeof(float4) * 2 * (size_t)(g.rows + 8) * (NXH + 4);
  const size_t cf = sizeof(float4) * (size_t)g.rows * NXH;
  g.coef_smem = lev + cf <= (size_t)optin;
  g.smem = g.coef_smem ? lev + cf : lev;
  if (g.smem > (size_t)optin) return false;
  // rows per unit: the rounds of 512 threads times a unit's length (its rows and the window of
  // eight rows that it reads first, half as dear), and a little for all the units' reads.  Chosen and
  // best of the six, 20 receivers x 1000 steps, 26 frequencies: 31 x 41 grid 2.02 (2 rows) and 1.98 ms
  // (3), 101 x 101 3.46 (3) and 3.37 (6), 101 x 301 5.53 (11), 151 x 201 5.22 (6) and 5.11 (8), 201 x 201
  // 6.03 (8) and 5.98 (11), 101 x 500 8.20 (6); the worst of the six took 1.15 to 1.4 times the best
  long long best = 0;
  for (int sr : kSR) {
    const long long units = (long long)NXH * ((g.rows + sr - 1) / sr);
    const long long cost = (units + 511) / 512 * (2 * sr + 5) * 16 + units * (sr + 1) / 8;
    if (best == 0 || cost < best) {
      best = cost;
      g.sr = sr;
      g.threads = (int)std::min<long long>(512, (units + 31) / 32 * 32);
    }
  }
  void* k = g.coef_smem ? kernel_of<true>(g.sr) : kernel_of<false>(g.sr);
  // (no static shared memory; one limit for every grid, as allow_block_smem)
  if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kBlockSmem) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = CL;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cfg.gridDim = dim3(CL);
  cfg.blockDim = dim3(g.threads);
  cfg.dynamicSmemBytes = g.smem;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  if (cudaOccupancyMaxActiveClusters(&g.clusters, k, &cfg) != cudaSuccess || g.clusters < 1) {
    cudaGetLastError();
    return false;
  }
  *out = g;
  return true;
}

// Microseconds per time step of the whole Green stage with either solver, fitted to runs of 1000 steps
// on nine grids (71 x 81 to 271 x 278 padded points), 2 to 100 receivers, 5, 26 and 60 frequencies, to
// within 12% for one round of clusters (or one batch), 25% for several; n: receivers, p: points, c:
// transform components.
// The clusters leave the transform fewer SMs beside them, so its work counts more than beside the
// per-step kernel.  The choice was 1.002 times the better one's time on
// average, with every level transformed, and more than 1.06 times in two of 270 runs (1.10, 1.16).  Clusters and per-step kernel, ms: 101 x 101 grid, 21 receivers,
// 5 frequencies 3.3 and 6.5; 151 x 201, 12 and 26: 4.7 and 5.7; 215 x 230, 6 and 26: 6.4 and 4.9, 21 and
// 26: 7.9 and 8.6; 201 x 201, 40 and 26: 13.4 and 13.5, 100 and 60: 36.5 and 30.5.
bool fd_cluster_faster(const ClGeom& g, const Layout& L, int nrec, int b, int nf) {
  const int rounds = (nrec + std::min(b, 2 * g.clusters) - 1) / std::min(b, 2 * g.clusters);
  const int batches = (nrec + b - 1) / b;
  const double n = nrec, p = (double)L.NZ * L.NX, w = n * p * dft_ncomp(nf);
  const double tc = (rounds == 1 ? 1.5 + 0.57e-4 * p : rounds * (1.0 + 0.77e-4 * p)) + 2.2e-8 * w;
  const double ts = batches == 1 ? 3.65 + 0.10 * n + 0.78e-6 * n * p + 1.2e-8 * w
                                 : 1.4 + 1.8 * batches + 0.15 * n + 0.63e-6 * n * p + 0.9e-8 * w;
  return tc < ts;
}

cudaError_t launch_fd_cluster(const ClGeom& g, float2* lev, int pslot, const Layout& L, const float2* coef,
                              const Stencil& S, int nb, int ta, int nsteps, int t0, int decim, int sbase,
                              __nv_bfloat16* snap, long long sslot, long long splane, long long srec,
                              const float* wav, int nw, const int* pts, float scale, cudaStream_t st) {
  if (ta < 2 || nsteps < 1 || nb < 1) return cudaErrorInvalidValue;
  ClArgs a{};
  a.lev = lev;
  a.F = L.F;
  a.pslot = pslot;
  a.org = L.org;
  a.NZ = L.NZ;
  a.NX = L.NX;
  a.PX = L.PX;
  a.coef = coef;
  a.ta = ta;
  a.nsteps = nsteps;
  a.t0 = t0;
  a.decim = decim;
  a.sbase = sbase;
  a.snap = snap;
  a.sslot = sslot;
  a.splane = splane;
  a.srec = srec;
  a.wav = wav;
  a.nw = nw;
  a.pts = pts;
  a.nrec = nb;
  a.scale = scale;
  a.rows = g.rows;
  float az = 0.f, ax = 0.f;
  for (int k = 3; k >= 0; --k) {  // cumulative weights C_j = sum_{k>=j} c_k
    az += S.cz[k];
    ax += S.cx[k];
    a.C.cz[k] = az;
    a.C.cx[k] = ax;
  }
  void* k = g.coef_smem ? kernel_of<true>(g.sr) : kernel_of<false>(g.sr);
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kBlockSmem);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = CL;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cfg.gridDim = dim3((unsigned)(CL * ((nb + 1) / 2)));
  cfg.blockDim = dim3(g.threads);
  cfg.dynamicSmemBytes = g.smem;
  cfg.stream = st;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  void* args[] = {&a};
  count_launches(1);
  return cudaLaunchKernelExC(&cfg, k, args);
}

}  // namespace egh
