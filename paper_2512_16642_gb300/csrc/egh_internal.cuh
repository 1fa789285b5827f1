// Internal declarations of the egh library (not part of the ABI).
//
// Device data layout (all float32 unless stated):
//   wavefield level: [NZ + 2*GUARD][PX], rows z = -GUARD .. NZ+GUARD-1, row pitch PX >= NX + 4
//     (multiple of 64).  Guard rows and columns x >= NX are zero and never written, so the
//     eighth-order stencil reads them as the u = 0 boundary without any bounds test;
//   FD state of a batch of B receivers in pairs: [3][B/2][F] float2, F = (NZ + 2*GUARD) * PX,
//     level n in slot n mod 3 (float2 = receivers 2i, 2i+1 at one point);
//   snapshot ring of the transform: [2 planes hi/lo][2K slots][Bp receivers][G] bf16, level n of
//     a chunk in slot (chunk parity) * K + n mod K, point p = z*PX + x (x >= NX and p >= NZ*PX
//     stay zero); u = hi + lo;
//   Green transforms gh: [nrec][nf][2][G], planes re/im, G = NZ*PX rounded up to 256, point
//     p = z*PX + x (entries with x >= NX or p >= NZ*PX are zero);
//   Hessians Qh, factors Lh: [nf][nrec][nrec] float2 (complex64).
#pragma once
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "egh.h"

#include <atomic>
#include <complex>
#include <cstdint>
#include <string>
#include <tuple>
#include <utility>
#include <vector>

namespace egh {

constexpr int GUARD = 4;  // stencil radius of the eighth-order Laplacian

// Counts kernel launches (every launch_* wrapper adds its launches); read by egh_get_stats.
void count_launches(int n);
long long launches_so_far();
// Message returned by egh_last_error(NULL) for calls that have no context.
void set_context_free_error(const std::string& msg);

// Lets kernel K take all the dynamic shared memory a block can have (227 KB with its static part).
// The limit belongs to the kernel in the whole process, not to a call: a launch that set it to its
// own size would lower it under another host thread's launch, or under a captured one.  So a kernel
// whose size differs from call to call has this one value set, whatever the call.
constexpr int kBlockSmem = 227 * 1024;
template <auto K>
cudaError_t allow_block_smem() {
  static std::atomic<int> dynamic{0};
  int d = dynamic.load(std::memory_order_relaxed);
  if (d == 0) {
    cudaFuncAttributes fa;
    const cudaError_t e = cudaFuncGetAttributes(&fa, K);
    if (e != cudaSuccess) return e;
    dynamic.store(d = kBlockSmem - (int)fa.sharedSizeBytes, std::memory_order_relaxed);
  }
  return cudaFuncSetAttribute(K, cudaFuncAttributeMaxDynamicSharedMemorySize, d);
}

// Where a launch goes: to a stream, or into a graph under construction, after the node *last (if it is
// not null), which the new one then replaces.  Graphs are built from nodes and not captured: while a
// stream captures, any host thread's cudaDeviceSynchronize fails and ends the capture, and contexts of
// different threads are independent.
struct Lane {
  Lane(cudaStream_t s) : stream(s) {}
  Lane(cudaGraph_t g, cudaGraphNode_t* l) : graph(g), last(l) {}
  cudaStream_t stream = nullptr;
  cudaGraph_t graph = nullptr;
  cudaGraphNode_t* last = nullptr;
};
// early: programmatic launch, the kernel may start when the one before it allows it (griddepcontrol)
cudaError_t lane_launch(const Lane& lane, const void* kernel, dim3 grid, dim3 block, size_t smem,
                        void** args, bool early);
template <typename... P, typename... A>
cudaError_t launch_on(const Lane& lane, bool early, void (*kernel)(P...), dim3 grid, dim3 block,
                      size_t smem, const A&... a) {
  std::tuple<P...> p(a...);  // converted to the kernel's parameter types
  return std::apply(
      [&](auto&... x) {
        void* args[] = {const_cast<void*>(static_cast<const void*>(&x))...};
        return lane_launch(lane, (const void*)kernel, grid, block, smem, args, early);
      },
      p);
}

struct Stencil {
  float cx[4];  // c_k / dx^2, k = 1..4
  float cz[4];  // c_k / dz^2
};

struct Layout {
  int nz, nx, ns;  // physical grid and sponge width
  int NZ, NX, PX;  // padded grid and pitch
  long long F;     // floats per wavefield level (with guard rows)
  long long org;   // offset of padded point (0, 0) inside a level: GUARD * PX
  long long G;     // Gram contraction length
};

// ---- egh_api.cu (host helpers shared with the serving loop) -----------------------------------
std::vector<float2> twiddle_table(const std::vector<double>& f, double dt, int len);
std::vector<float> synthesis_weights(const std::vector<double>& f, double dt, int nt);

// ---- fd.cu ------------------------------------------------------------------------------------
// Paired levels: float2 per grid point = (receiver 2i, receiver 2i+1); coef = (c1, c3).
// Snapshot output of one level: hi plane of its slot (receiver 0, point 0) or nullptr for none.
struct SnapOut {
  __nv_bfloat16* lvl;
  long long plane;  // elements from the hi plane to the lo plane
  long long rec;    // elements between receivers (G)
};
cudaError_t launch_check_velocity(const float* vel, long long n, float* d_vmax_bad, cudaStream_t st);
cudaError_t launch_build_coef(const float* vel, const Layout& L, double dz, double dx, double dt,
                              double R, const float* d_vmax, float2* coef, cudaStream_t st);
// What a step does besides: the sample amp into the new level at the points pts (null: none), and the
// current level's values at rec_pts as sample t of the traces (null: none).
struct FdAux {
  const int* pts;
  int nb;  // receivers (sources) of the batch
  float amp, scale;
  const int* rec_pts;
  int nrec;
  float* traces;  // [nb][nrec][nt]
  int nt, t;
};
// tz: rows per warp (12, 16, 18, 20, 24 or 32; 0 = default)
cudaError_t launch_fd_step(const float2* ucur, const float2* uprev, float2* unext,
                           const float2* coef, const Layout& L, const Stencil& S, int npairs,
                           const SnapOut& so, const Lane& lane, int tz, const FdAux* aux = nullptr);
int fd_rows_one_wave(const Layout& L, int npairs);
int fd_rows_per_warp_default();
cudaError_t fd_prepare(int nf);  // once per context, before any capture
cudaError_t launch_inject(float2* u, long long pstride, const int* pts, const float2* coef, int nb,
                          float amp, float scale, long long org, const SnapOut& so,
                          cudaStream_t st);
cudaError_t launch_record(const float2* u, long long pstride, const int* rec_pts, int nrec, int nb,
                          float* traces, int nt, int t, cudaStream_t st);
int dft_ncomp(int nf);
size_t dft_smem(int nf);
std::vector<unsigned char> dft_twiddle_tiles(const std::vector<double>& f, double dt, int nt,
                                             const std::vector<std::complex<double>>* scale = nullptr);
cudaError_t make_snap_tmap(CUtensorMap* tm, void* base, long long G, int Bp, int nslot);
// per_sm: CTAs per SM of the persistent transform (1 beside the FD steps, more when it runs
// alone; 0: one CTA per tile); beside_smem: shared memory (reserved parts included) of the FD
// CTAs an SM holds beside the transform (0: none), which sizes the transform's CTAs so that an
// SM holds one of them next to the FD CTAs and never two; last: the launch completes the totals, which
// are then multiplied by `down` (and written to ghb too, unless that is null)
cudaError_t launch_dft_tc(const CUtensorMap& tmap, const unsigned char* twt, int nf, int slot0,
                          int kcount, int n0, const Layout& L, float* gh, __nv_bfloat16* ghb,
                          int last, int rec0, int nvalid, int nrec_all, int* err, int expire,
                          int per_sm, long long beside_smem, float down, cudaStream_t st);
// n floats (a multiple of four) times scale, in place
cudaError_t launch_scale_totals(float* g, long long n, float scale, int per_sm, cudaStream_t st);
// dynamic shared memory of one k_fd_step CTA for npairs receiver pairs
int fd_block_smem(int npairs);
// shared memory (reserved parts included) of the k_fd_step CTAs of npairs pairs and tz rows per
// warp that one SM holds at once; 0 if it cannot be queried
long long fd_sm_smem(int npairs, int tz);

// ---- fd_resident.cu ---------------------------------------------------------------------------
// The padded grid as TR x TC tiles of TZ x TX points (TX % 4 == 0), one block per tile, all
// resident at once; P receiver pairs of a batch held in each block's shared memory.
struct ResGeom {
  int TR, TC, TZ, TX;
  int P;
  size_t smem;  // dynamic shared memory per block
};
// Tile grid with the most pairs (<= want_pairs, <= 8) whose state fits a block's shared memory,
// then the smallest tile; false if not even one pair fits.
bool fd_resident_plan(const Layout& L, int want_pairs, ResGeom* g);
size_t fd_resident_xbuf_float4(const ResGeom& g);  // halo exchange buffer (float4)
size_t fd_resident_flags(const ResGeom& g);        // step counters + abort flag (ints)
int fd_resident_sr_default();                         // rows per z-march segment
bool fd_resident_sr_valid(int sr);                    // 6, 8, 11 or 16
// shared-memory limit of every instance, and a check that the grid is co-resident (sr, np:
// the launch's segment rows and pairs, which set its block size)
cudaError_t fd_resident_prepare(const ResGeom& g, int sr, int np);
// Levels ta .. ta+nsteps-1 of np pairs (ta >= 2), from the state slots of levels ta-1, ta-2 of
// lev ([3][pslot][F]) to the slots of the last two levels; level t's bf16 hi/lo snapshot goes to
// ring slot sbase + (t - t0) / decim when t % decim == 0 (snap: hi plane of ring slot 0, or
// null).  flags: fd_resident_flags(g) ints (zeroed here).  Cooperative launch.
cudaError_t launch_fd_resident(const ResGeom& g, int sr, float2* lev, int pslot, const Layout& L,
                               const float2* coef, const Stencil& S, int np, int ta, int nsteps,
                               int t0, int decim, int sbase, __nv_bfloat16* snap, long long sslot,
                               long long splane, long long srec, float4* xbuf, int* flags,
                               int* err, int expire, cudaStream_t st);

// ---- fd_cluster.cu ----------------------------------------------------------------------------
// Small grids: a cluster of blocks per receiver pair, both levels of its rows in each block's
// shared memory.
struct ClGeom {
  int rows;        // grid rows per block at most
  int sr;          // rows per unit
  int threads;     // per block
  int clusters;    // clusters that the GPU holds at once
  bool coef_smem;  // coefficients in shared memory too
  size_t smem;     // dynamic shared memory per block
};
bool fd_cluster_plan(const Layout& L, ClGeom* g);  // false if the grid does not fit
// whether nrec receivers, at most b in a batch, and nf frequencies take less time than with the
// per-step kernel
bool fd_cluster_faster(const ClGeom& g, const Layout& L, int nrec, int b, int nf);
// Levels ta .. ta+nsteps-1 (ta >= 2) of nb receivers from the state slots of levels ta-1, ta-2 to
// the slots of the last two; level t's snapshot to ring slot sbase + (t - t0) / decim when
// t % decim == 0; wav (device, may be null): level t takes sample t - 1 < nw at the receivers' points
cudaError_t launch_fd_cluster(const ClGeom& g, float2* lev, int pslot, const Layout& L, const float2* coef,
                              const Stencil& S, int nb, int ta, int nsteps, int t0, int decim, int sbase,
                              __nv_bfloat16* snap, long long sslot, long long splane, long long srec,
                              const float* wav, int nw, const int* pts, float scale, cudaStream_t st);

// ---- gram_tc.cu -------------------------------------------------------------------------------
// Gram on the tensor cores from the bf16 hi/lo transforms ghb[nf][G/32][hi/lo][nrec x re/im][32].
__host__ __device__ int gram_tc_blocks(int nrec);
size_t gram_tc_workspace_floats(int nrec, int nf, int splits);
int gram_tc_splits(int nrec, int nf, long long G);
cudaError_t launch_gram_tc(const __nv_bfloat16* ghb, int nrec, int nf, long long G, int splits,
                           float* part, int* err, cudaStream_t st);
cudaError_t launch_gh_to_ghb(const float* gh, int nrec, int nf, long long G, __nv_bfloat16* ghb,
                             cudaStream_t st);
cudaError_t launch_gram_tc_finish(const float* part, int nrec, int nf, int splits, float2* Qh,
                                  cudaStream_t st);

// ---- gram.cu ----------------------------------------------------------------------------------
// edge: tile edge of C, 64 or 128 (gram_tile_edge: the better one for nrec); px, nx: row pitch of
// the points and columns that are not zero (px a multiple of 16; 0: every point counts)
int gram_tile_edge(int nrec);
__host__ __device__ int gram_tiles(int nrec, int edge);
size_t gram_workspace_floats(int nrec, int nf, int splits, int edge);
cudaError_t launch_gram_partial(const float* gh, int nrec, int nf, long long G, int splits, int edge,
                                int px, int nx, float* part, cudaStream_t st);
cudaError_t launch_gram_finish(const float* part, int nrec, int nf, int splits, int edge,
                               float2* Qh, cudaStream_t st);
cudaError_t launch_diag_sum(const float2* Qh, int nrec, int nf, double* d_sum, cudaStream_t st);
cudaError_t launch_lambda_max(const float2* Qh, int nrec, int nf, double* d_lmax, cudaStream_t st);
cudaError_t launch_add_mu_copy(float2* Qh, float2* Lh, int nrec, int nf, float mu, cudaStream_t st);
cudaError_t launch_add_mu_copy_delta(float2* Qh, float2* Lh, int nrec, int nf, double mu_old,
                                     double mu_new, cudaStream_t st);

// ---- chol.cu ----------------------------------------------------------------------------------
// piv64: FP64 diagonal and pivots (mixed precision)
struct PotrfItem {
  float2* A;    // n x n, factored in place
  int n;
  int* status;  // 0, or the failing pivot + 1
};
cudaError_t potrf_many_prepare(int nmax);
cudaError_t launch_potrf_many(const PotrfItem* items, int count, int nmax, int blocks, int threads,
                              int piv64, const Lane& lane);
cudaError_t launch_potrf(float2* Lh, int n, int nf, int* status, cudaStream_t st, int piv64);

// ---- deblur.cu --------------------------------------------------------------------------------
// spectra of ntr = nrec * ns traces into columns s0 .. s0+ns-1 of D[nf][nrec][ld] on the tensor
// cores; twt: the transform's twiddle tiles for at least nt_d levels; err: the flag a bounded
// wait sets (both required; nf <= 64); expire: test hook, the first CTA's first wait runs out
// dev_in: resid is device memory (not a mapping of host memory), which the TMA form needs;
// scratch: device memory of scratch_bytes for the block sums of calls with few traces (used when
// trace_scratch_bytes asks for some and it is large enough)
cudaError_t launch_trace_dft(const float* resid, int ntr, int nt_d, int nf, int nrec, int ld,
                             int s0, float2* Dh, cudaStream_t st, const unsigned char* twt,
                             int* err, int expire = 0, bool dev_in = false, void* scratch = nullptr,
                             size_t scratch_bytes = 0);
size_t trace_scratch_bytes(int nf, long long ntr, int nt_d);
// the most that any call of at most nt_d levels asks for
size_t trace_scratch_most(int nf, int nrec, int nt_d);
cudaError_t launch_trsm(const float2* Lh, int n, int nf, float2* Dh, int ns, cudaStream_t st);
// W = L^{-1} per frequency
cudaError_t launch_trtri(const float2* Lh, int n, int nf, float2* Wh, const Lane& lane);
// Q^{-1}_k = W_k^H W_k (dense) from the inverse factors
cudaError_t launch_gram_inverse(const float2* Wh, int n, int nf, float2* Ph, const Lane& lane);
// operand images of A_k (n x n complex64 per frequency) for launch_cmm_tc: cmm_image_bytes(n, nf)
size_t cmm_image_bytes(int n, int nf);
cudaError_t launch_cmm_images(const float2* A, int n, int nf, unsigned char* img, const Lane& lane);
// C_k = A_k B_k (complex, A_k n x n as images, B_k and C_k n x ld, row-major; C must not alias B) on
// the tensor cores with FP32-class products (three-term bf16 splits), for the nk frequencies of the
// device list kl (all when null); err: the flag a bounded wait sets (solve_tc.cu)
cudaError_t launch_cmm_tc(const unsigned char* Aimg, int n, int nk, const float2* B, int ld, float2* C,
                          const int* kl, int* err, cudaStream_t st);
// diagonal-Hessian baseline: D_k[r][s] /= Q_k[r][r]
cudaError_t launch_diag_solve(const float2* Qh, int n, int nf, float2* Dh, int ns, cudaStream_t st);
// refinement residual R = D - Q X: FP64 arithmetic (fp64) or the compensated FP32 dot product;
// frequencies of the device list kl (nf of them), all when kl is null
cudaError_t launch_resid(const float2* Qh, int n, int nf, const float2* Xh, const float2* Dh,
                         int ns, float2* Rh, bool fp64, cudaStream_t st, const int* kl = nullptr);
inline bool prec_mixed(int prec) { return prec == EGH_PREC_MIXED || prec == EGH_PREC_MIXED_FP64; }
// X_k += R_k (m elements per frequency) for the nk frequencies of kl (all when kl is null)
cudaError_t launch_add_correction(float2* X, const float2* R, long long m, int nk, cudaStream_t st,
                                  const int* kl = nullptr);
// ||Q_k||_F^2 per frequency (FP64 sums) into d_out[nf]
cudaError_t launch_fro2(const float2* Qh, int n, int nf, double* d_out, const Lane& lane);
// lambda_max(P_k) = 1 / lambda_min(Q_k), P_k = Q_k^{-1}, by power iteration (from below) into lam[nf]
cudaError_t launch_inv_power(const float2* Ph, int n, int nf, double* lam, const Lane& lane);
// Condition bound of a factorisation from ||Q||_F^2, the power estimate of 1/lambda_min (with a
// margin for its approach from below) and, when known (> 0), mu <= lambda_min.
inline double cond_bound(double fro2, double inv_lmin, double mu) {
  double c = 1.25 * sqrt(fro2) * inv_lmin;
  if (mu > 0 && sqrt(fro2) / mu < c) c = sqrt(fro2) / mu;
  return c;
}
// Frequencies whose solves get one step of iterative refinement: condition bound above this
// threshold.  The products with the inverse factor give solutions with a relative error of about
// 1e-8 cond (measured on the 101x101 case, cond 200-1800) and the bound exceeds cond about
// twofold, so unrefined solutions stay near or below 1e-4, a tenth of the multipliers' tolerance.
constexpr double kRefineCond = 1e4;
// (on the tensor cores when tws, the synthesis twiddle tiles for at least nt_d samples, and err
// are given and 2 nf <= 64; else on the CUDA cores)
// dev_out: mult is device memory (not a mapping of host memory), which the TMA-store form needs;
// scratch: device memory of scratch_bytes for the synthesis operand images (used when at least
// synth_operands_bytes(nf, nrec * ns) and 16-byte aligned; else the kernel gathers them itself)
cudaError_t launch_synth(const float2* Dh, int nrec, int ns, int ld, int s0, int nf, const float* w,
                         const float2* tw, int nt_d, float* mult, cudaStream_t st,
                         const unsigned char* tws = nullptr, int* err = nullptr,
                         bool dev_out = false, unsigned char* scratch = nullptr,
                         size_t scratch_bytes = 0);
size_t synth_operands_bytes(int nf, long long ntr);
std::vector<unsigned char> synth_twiddle_tiles(const std::vector<double>& f, double dt, int nt);

}  // namespace egh
