// Per-frequency Hessians on the tensor cores (eq. Qmatrix with S S^T replaced by its
// frequency-domain blocks; Section "Direct Hessian-inverse computation", Algorithm 2):
//   H_k[i][j] = sum_x ghat_i(w_k, x) conj(ghat_j(w_k, x)).
// With M_k = [Re ghat_0; Im ghat_0; Re ghat_1; ...] (2 nrec rows, G columns) and the real symmetric
// C = M_k M_k^T:
//   Re H[i][j] = C[2i][2j] + C[2i+1][2j+1],   Im H[i][j] = C[2i+1][2j] - C[2i][2j+1].
//
// C is formed in 128 x 256 blocks (64 x 128 receivers x re/im; 128 x 128 at the last panel)
// covering exactly the panel pairs on and above the diagonal, by tcgen05 `kind::f16` MMAs in
// bf16x3: each entry of M_k is stored by the transform's
// last chunk as hi = bf16(g), lo = bf16(g - hi), and C = Hi Hi^T + Hi Lo^T + Lo Hi^T accumulates in
// FP32 in TMEM (the dropped Lo Lo^T and the split are ~2^-17 relative).  Operands arrive by bulk
// copies of 32 points x up to 128 receivers x re/im, stored so that they land as rows of 64 bytes in
// the K-major 64-byte-swizzled layout the MMA reads: the kernel does no conversion.  The grid
// sum is split into `splits` ranges; each CTA writes its FP32 tile to a workspace and a second
// kernel adds the splits (in double) and forms Q_k.
#include <cuda_bf16.h>

#include <algorithm>

#include "egh_internal.cuh"
#include "tc.cuh"

namespace egh {

constexpr int GC_M = 128;            // block rows of C (64 receivers x re/im)
constexpr int GC_N = 256;            // block columns of C (128 receivers x re/im)
constexpr int GC_P = 64;   // point ranges are multiples of it
constexpr int GC_K = 32;   // points per stage and block of the layout: 64-byte rows (64-byte swizzle)
constexpr int GC_ST = 4;   // stages in flight (4 x 48 KB: the copies run three stages ahead)
constexpr unsigned GC_BOX = 128u * GC_K * 2;  // one operand box: 64 receivers x re/im = 128 rows
constexpr unsigned GC_STAGE = 6 * GC_BOX;  // A hi, A lo (1 box each), B hi, B lo (2 boxes each)

// Blocks (ta, j) of C: rows of 64-receiver panel ta (128 rows), columns of panels ta + 2j and
// ta + 2j + 1 (256 columns; a "half" block when the second panel is past the last), j = 0, 1, ...
// -- exactly the panel pairs on and above the diagonal.  Block (ta, 0) is "inner": its A panel is
// the first half of its B panels.
__host__ __device__ inline int gram_tc_panels64(int nrec) { return (nrec + 63) / 64; }
__host__ __device__ inline int gram_tc_blocks_before(int ta, int n64) {
  int s = 0;
  for (int t = 0; t < ta; ++t) s += (n64 - t + 1) / 2;
  return s;
}
__host__ __device__ int gram_tc_blocks(int nrec) {
  const int n64 = gram_tc_panels64(nrec);
  return gram_tc_blocks_before(n64, n64);
}

size_t gram_tc_workspace_floats(int nrec, int nf, int splits) {
  return (size_t)splits * nf * gram_tc_blocks(nrec) * GC_M * GC_N;
}

size_t gram_tc_smem() { return 1024 + (size_t)GC_ST * GC_STAGE; }

// The Gram's bf16 operands from FP32 transforms gh[nrec][nf][re/im][G]: hi = bf16(g),
// lo = bf16(g - hi), blocked by 32 points as ghb[nf][G/32][hi/lo][nrec x re/im][32] (the layout the
// transform's last chunk writes, from the same values).  Within a row the 16-byte runs are swapped as
// the MMA's 64-byte swizzle has them (run c of row R at c ^ (R / 2 % 4), R / 2 the receiver), so that a
// panel's rows are one contiguous run that a bulk copy lands as the operand.
// A thread converts one run: two 16-byte reads, a 16-byte write to each plane (231 receivers x 4
// frequencies x 267 008 points, the import with its copy: 3.10 ms with a point per thread, 1.55 ms now).
__global__ void k_gh_to_ghb(const float* __restrict__ gh, int nrec, int nf, long long G,
                            __nv_bfloat16* __restrict__ ghb) {
  const long long runs = G >> 3, total = (long long)nrec * nf * 2 * runs;
  const long long rows = 2LL * nrec;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < total;
       t += (long long)gridDim.x * blockDim.x) {
    const long long p = t % runs * 8, c2 = (t / runs) % (2LL * nf), r = t / (2LL * nf * runs);
    const float4 a = __ldcs(reinterpret_cast<const float4*>(gh) + 2 * t);
    const float4 b = __ldcs(reinterpret_cast<const float4*>(gh) + 2 * t + 1);
    const float v[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
    __align__(16) __nv_bfloat16 h[8], l[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      h[i] = __float2bfloat16_rn(v[i]);
      l[i] = __float2bfloat16_rn(v[i] - __bfloat162float(h[i]));
    }
    __nv_bfloat16* q = ghb + (((c2 >> 1) * (G >> 5) + (p >> 5)) * 2 * rows + 2 * r + (c2 & 1)) * 32 +
                       ((p & 31) ^ ((r & 3) << 3));
    *reinterpret_cast<uint4*>(q) = *reinterpret_cast<const uint4*>(h);
    *reinterpret_cast<uint4*>(q + rows * 32) = *reinterpret_cast<const uint4*>(l);
  }
}

cudaError_t launch_gh_to_ghb(const float* gh, int nrec, int nf, long long G, __nv_bfloat16* ghb,
                             cudaStream_t st) {
  if (G % 32 != 0) return cudaErrorInvalidValue;
  const long long total = (long long)nrec * nf * 2 * (G / 8);
  const long long blocks = std::min<long long>((total + 255) / 256, 152LL * 16);
  count_launches(1);
  k_gh_to_ghb<<<(unsigned)blocks, 256, 0, st>>>(gh, nrec, nf, G, ghb);
  return cudaGetLastError();
}

// One CTA: block (ta, tb) of C at frequency k over points [p0, p1), as M128 x N256 MMAs (each
// A row group read from shared memory serves 256 columns, which halves the operand traffic per
// product against square 128 x 128 tiles).  One thread of warp 8 issues the copies of a
// GC_ST-stage ring, one of warp 9 the MMAs.  The tensor core's FP32 accumulation of a long sum drifts
// (its rounding is not round-to-nearest: about 2^-24 relative per accumulation, measured 1e-3 over
// 87 000 points), so the MMAs accumulate into one of two 256-column TMEM buffers for blocks of
// GC_J stages only, and warps 0..7 (lane quarter w % 4, column half w / 4) drain each finished
// block into FP32 register totals with round-to-nearest adds while the MMAs fill the other
// buffer.  Every wait is bounded (on expiry: error flag, the copies in flight awaited, TMEM freed,
// CTA leaves).
//
// Bound by the MMAs (231 receivers x 26 frequencies: 5.09 ms, 7.6e12 issued flop, 1490 TFLOP/s) and
// their operands in shared memory beside the copies' writes.  There 7.68 ms with tensor boxes of
// 64-byte rows and one thread for copies and MMAs; 7.56 with the last panel's columns ending with its
// rows (in the MMA's steps of 16); 6.69 with the operands stored swizzled and copied as contiguous
// runs; 5.09 with the copies on a thread of their own, which no MMA issue holds up.  Stages of
// 32 points (48 KB) keep four in the ring (against two 96 KB stages of 64 points: 9.6 -> 8.1 ms).
constexpr int GC_J = 8 * (GC_P / GC_K);  // stages per TMEM accumulation block (96 accumulations)

// K-major shared-memory descriptor of the 64-byte swizzle (8-row groups 512 bytes apart)
__device__ __forceinline__ uint64_t gc_desc(unsigned saddr) { return tc::sdesc_sw64(saddr); }

__global__ void __launch_bounds__(320)
    k_gram_tc(const __nv_bfloat16* __restrict__ ghb, int nrec, long long split_len, long long G,
              float* __restrict__ part, int* __restrict__ err) {
  extern __shared__ __align__(1024) unsigned char dsm[];
  unsigned char* sm = dsm + ((1024 - (tc::smem_u32(dsm) & 1023)) & 1023);
  // full[GC_ST], empty[GC_ST], blockdone[2], drained[2]
  __shared__ __align__(8) unsigned long long bars[2 * GC_ST + 4];
  __shared__ unsigned tslot;
  __shared__ int fail;
  const int blkid = blockIdx.x, k = blockIdx.y, sp = blockIdx.z, nf = gridDim.y;
  const int n64 = gram_tc_panels64(nrec);
  int ta = 0;
  while (ta + 1 < n64 && gram_tc_blocks_before(ta + 1, n64) <= blkid) ++ta;
  const int bp = ta + 2 * (blkid - gram_tc_blocks_before(ta, n64));  // first B panel
  const bool inner = bp == ta;         // the A panel is the first half of the B panels
  const bool half = bp + 1 >= n64;     // one B panel only
  // columns: those of rows that exist, in the MMA's steps of 16 (the last panel is seldom full)
  const int last = (2 * nrec - GC_M * (n64 - 1) + 15) & ~15;
  const int N = half ? last : bp + 2 == n64 ? GC_M + last : GC_N;
  const long long p0 = (long long)sp * split_len;
  const long long p1 = min(G, p0 + split_len);
  const int nst = p1 > p0 ? (int)((p1 - p0 + GC_K - 1) / GC_K) : 0;
  const int nblk = (nst + GC_J - 1) / GC_J;
  const int tid = threadIdx.x, warp = tid >> 5;
  if (warp == 0) tc::tmem_alloc(&tslot, 2 * GC_N);
  const unsigned bar0 = tc::smem_u32(&bars[0]);
  auto full = [&](int i) { return bar0 + 8u * i; };
  auto empty = [&](int i) { return bar0 + 8u * (GC_ST + i); };
  auto blockdone = [&](int i) { return bar0 + 8u * (2 * GC_ST + i); };
  auto drained = [&](int i) { return bar0 + 8u * (2 * GC_ST + 2 + i); };
  if (tid == 0) {
    for (int i = 0; i < 2 * GC_ST + 2; ++i) tc::mbar_init(bar0 + 8u * i, 1);
    tc::mbar_init(drained(0), 256);
    tc::mbar_init(drained(1), 256);
    fail = 0;
    tc::mbar_init_fence();
  }
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  const unsigned tmem = tslot;
  // stage buffer: [A_hi][A_lo][B_hi: 2 boxes][B_lo: 2 boxes]
  auto stage_addr = [&](int b) { return tc::smem_u32(sm + (size_t)b * GC_STAGE); };
  if (warp == 8) {
    if (tid == 256) {
      // rows of the panels (the last may be partial; rows of a stage past them stay what they were and
      // reach no entry that is read)
      const int rows = 2 * nrec;
      const unsigned ab = (unsigned)min(GC_M, rows - GC_M * ta) * (GC_K * 2);
      const unsigned bb = (unsigned)min(GC_N, rows - GC_M * bp) * (GC_K * 2);
      const long long plane = (long long)rows * GC_K;  // elements per point block and plane
      const __nv_bfloat16* src = ghb + ((long long)k * (G / GC_K) + p0 / GC_K) * 2 * plane;
      int s = 0;
      for (; s < nst; ++s) {
        const int b = s % GC_ST;
        if (s >= GC_ST && !tc::mbar_wait(empty(b), (s / GC_ST - 1) & 1)) {
          fail = 1;
          atomicExch(err, 1);
          break;
        }
        const unsigned base = stage_addr(b);
        tc::mbar_expect_tx(full(b), 2 * (bb + (inner ? 0 : ab)));
        for (int hl = 0; hl < 2; ++hl) {
          const __nv_bfloat16* q = src + (2LL * s + hl) * plane;
          if (!inner) tc::bulk_g2s(base + hl * GC_BOX, q + GC_M * GC_K * ta, ab, full(b));
          tc::bulk_g2s(base + (2 + 2 * hl) * GC_BOX, q + GC_M * GC_K * bp, bb, full(b));
        }
      }
      // no copy outlives the block
      for (int i = max(0, s - GC_ST); i < s; ++i) tc::mbar_wait(full(i % GC_ST), (i / GC_ST) & 1);
    }
    __syncwarp();
  } else if (warp == 9) {
    if (tid == 288) {
      const unsigned idesc = tc::idesc_bf16(GC_M, N, 0, 0);
      bool ok = true;
      for (int s = 0; s < nst; ++s) {
        const int b = s % GC_ST;
        const int blk = s / GC_J;
        const bool first = s % GC_J == 0;
        // a block reuses the TMEM buffer of block blk - 2 once the drain warps have read it
        ok = !(first && blk >= 2) || tc::mbar_wait(drained(blk & 1), ((blk >> 1) - 1) & 1);
        ok = ok && tc::mbar_wait(full(b), (s / GC_ST) & 1);
        if (!ok) break;
        tc::tc_fence_after();
        const unsigned dt = tmem + (unsigned)((blk & 1) * GC_N);
        const unsigned bh = stage_addr(b) + 2 * GC_BOX, bl = stage_addr(b) + 4 * GC_BOX;
        // an inner block's A rows are the first 128 B rows
        const unsigned ah = inner ? bh : stage_addr(b);
        const unsigned al = inner ? bl : ah + GC_BOX;
#pragma unroll
        for (int ks = 0; ks < GC_K / 16; ++ks) {
          const unsigned o = 32u * ks;
          const uint64_t dah = gc_desc(ah + o), dal = gc_desc(al + o);
          const uint64_t dbh = gc_desc(bh + o), dbl = gc_desc(bl + o);
          tc::mma_bf16(dt, dah, dbh, idesc, !(first && ks == 0));
          tc::mma_bf16(dt, dah, dbl, idesc, true);
          tc::mma_bf16(dt, dal, dbh, idesc, true);
        }
        tc::mma_commit(empty(b));
        if (s % GC_J == GC_J - 1 || s == nst - 1) tc::mma_commit(blockdone(blk & 1));
      }
      if (!ok) {
        fail = 1;
        atomicExch(err, 1);
        // wake the drain warps: every MMA issued so far completes before these arrivals
        tc::mma_commit(blockdone(0));
        tc::mma_commit(blockdone(1));
      }
    }
    __syncwarp();
  } else {
    // warps 0..7: TMEM lanes 32 (w % 4) .. = rows of the block, columns 128 (w / 4) ..
    const int q = warp & 3, h = warp >> 2;
    float tot[128];
#pragma unroll
    for (int c = 0; c < 128; ++c) tot[c] = 0.f;
    bool ok = true;
    const int nc = min(128, N - h * 128);  // this warp's columns (none: nothing to drain)
    for (int blk = 0; blk < nblk; ++blk) {
      const bool got = tc::mbar_wait(blockdone(blk & 1), (blk >> 1) & 1);
      if (!__all_sync(0xffffffffu, got && !fail)) {  // warp-uniform: TMEM loads are collective
        ok = false;
        break;
      }
      tc::tc_fence_after();
      const unsigned base =
          tmem + ((unsigned)(q * 32) << 16) + (unsigned)((blk & 1) * GC_N + h * 128);
#pragma unroll
      for (int c0 = 0; c0 < 128; c0 += 32) {
        if (c0 < nc) {
          float v[32];
          tc::tmem_ld32(base + (unsigned)c0, v);
#pragma unroll
          for (int i = 0; i < 32; ++i) tot[c0 + i] += v[i];
        }
      }
      tc::tc_fence_before();
      tc::mbar_arrive(drained(blk & 1));
    }
    if (ok && !fail) {
      const int row = q * 32 + (tid & 31);
      float* out = part +
                   (((long long)sp * nf + k) * gram_tc_blocks(nrec) + blkid) * (GC_M * GC_N) +
                   (long long)row * GC_N + h * 128;
#pragma unroll
      for (int i = 0; i < 128; i += 4)
        if (i < nc)
          *reinterpret_cast<float4*>(out + i) = make_float4(tot[i], tot[i + 1], tot[i + 2], tot[i + 3]);
    } else if ((tid & 31) == 0) {
      atomicExch(err, 1);
    }
  }
  tc::tc_fence_before();
  __syncthreads();
  if (warp == 0) tc::tmem_dealloc(tmem, 2 * GC_N);
}

int gram_tc_splits(int nrec, int nf, long long G) {
  // one CTA per SM (shared memory); about sixteen waves of short point ranges keep the CTAs of
  // one frequency close together in the grid sum, so that their shared panels meet in L2
  // (measured on 231 receivers x 26 frequencies: 6 splits 11.1 ms, 16 splits 10.5 ms)
  const long long blocks = (long long)gram_tc_blocks(nrec) * nf;
  long long s = (16LL * 152 + blocks - 1) / blocks;
  s = std::max(1LL, std::min(s, G / (16LL * GC_P)));
  return (int)s;
}

cudaError_t launch_gram_tc(const __nv_bfloat16* ghb, int nrec, int nf, long long G, int splits,
                           float* part, int* err, cudaStream_t st) {
  if (G % GC_P != 0 || splits < 1) return cudaErrorInvalidValue;
  long long split_len = (G + splits - 1) / splits;
  split_len = (split_len + GC_P - 1) / GC_P * GC_P;
  const size_t smem = gram_tc_smem();
  cudaError_t e =
      cudaFuncSetAttribute(k_gram_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  count_launches(1);
  k_gram_tc<<<dim3(gram_tc_blocks(nrec), nf, splits), 320, smem, st>>>(ghb, nrec, split_len, G,
                                                                       part, err);
  return cudaGetLastError();
}

// Q_k from the tiles: entry (i, j), i <= j, from the block that holds row 2i and column 2j of C (the
// panel of i is not past the panel of j), its four values as two 8-byte loads per split, the splits
// summed in order in double; (j, i) is its conjugate.  Bound by the tiles' bytes (231 receivers x 26
// frequencies, 16 splits, with the sum of the diagonal after it: 0.44 ms with every entry read at its
// own place, half of them down a column, now 0.30 ms).
__global__ void k_gram_tc_finish(const float* __restrict__ part, int nrec, int nf, int splits,
                                 float2* __restrict__ Qh) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  const int i = blockIdx.y;
  const int k = blockIdx.z;
  if (j >= nrec || j < i) return;
  const int n64 = gram_tc_panels64(nrec), nblocks = gram_tc_blocks(nrec);
  const int pa = i / 64, pb = j / 64;
  const int blk = gram_tc_blocks_before(pa, n64) + (pb - pa) / 2;
  const float* t = part + ((long long)k * nblocks + blk) * (GC_M * GC_N) + (2 * i % GC_M) * GC_N +
                   ((pb - pa) & 1) * GC_M + 2 * j % GC_M;
  const long long step = (long long)nf * nblocks * (GC_M * GC_N);
  double rr = 0.0, ri = 0.0, ir = 0.0, ii = 0.0;
#pragma unroll 8
  for (int s = 0; s < splits; ++s) {
    const float2 re = __ldcs(reinterpret_cast<const float2*>(t + s * step));
    const float2 im = __ldcs(reinterpret_cast<const float2*>(t + s * step + GC_N));
    rr += re.x;
    ri += re.y;
    ir += im.x;
    ii += im.y;
  }
  const float re = (float)(rr + ii), im = i == j ? 0.f : (float)(ir - ri);
  Qh[((long long)k * nrec + i) * nrec + j] = make_float2(re, im);
  if (i != j) Qh[((long long)k * nrec + j) * nrec + i] = make_float2(re, -im);
}

cudaError_t launch_gram_tc_finish(const float* part, int nrec, int nf, int splits, float2* Qh,
                                  cudaStream_t st) {
  dim3 grid((nrec + 127) / 128, nrec, nf);
  count_launches(1);
  k_gram_tc_finish<<<grid, 128, 0, st>>>(part, nrec, nf, splits, Qh);
  return cudaGetLastError();
}

}  // namespace egh
