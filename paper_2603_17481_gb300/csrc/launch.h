// launch.h -- host-side launchers of the liblbm kernels (internal to the library).
#pragma once

#include <utility>

#include "lbm_device.cuh"

namespace lbm {

// Launches a step kernel with programmatic stream serialization (see pdl_enter).
template <typename... KArgs, typename... Args>
cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, Args &&...args) {
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}

// Kernel modes of the hydrodynamic kernel.
enum HydroMode { kStep = 0, kMoments = 1 };

// The near-contact list of one phi buffer: the 32 x 8 x 4 tiles (3D; 32 x 16 in 2D) holding a
// gated cell, their count, and one mark per tile of the grid, set while the tile is listed.
struct TileList {
  int *tiles = nullptr;
  int *count = nullptr;
  int *mark = nullptr;
};

// Buffers of the near-contact pass besides the normals and forces: for every row of 32 cells of a
// listed tile the masks of its gated cells by the direction of their normals (8 words, 6 or 4 used);
// in 3D the component ranges of the gated normals of every 4x4x4 brick, as halves lo0 lo1 lo2 - hi0
// hi1 hi2 - (lo rounded down, hi up); the half tiles that may hold a facing pair (2 * tile + half),
// and their count.
struct NciAux {
  unsigned *masks = nullptr;
  uint4 *bricks = nullptr;
  int *scan_units = nullptr;
  int *nscan = nullptr;
};
bool nci_prefilter_applies(int dim, const KParams &P);
size_t nci_brick_count(const KParams &P);
size_t nci_mask_bytes(const KParams &P);

// Most blocks that share one scanned unit (1 where several cases share the device).
constexpr int kNciParts = 8;

// The near-contact pass over the listed tiles on phi: normals of the gated cells into nrm, zero force
// at them, then the force at the cells that have a partner. list.tiles == nullptr: over every tile, with
// zero force (and no partner, where partner is given) at every other cell too.
// list_blocks: blocks per kernel are at most a few times this (the device's SMs, or fewer).
// reset_other (listed tiles, may be null): the count of the other phi buffer's list, whose tiles
// were consumed by the previous step; the normals pass sets it to zero, so that the phase pass of
// this step starts that buffer's list empty.
cudaError_t launch_nci(int dim, const KParams &P, const int32_t *phi, float4 *nrm, float4 *frep, int32_t *partner,
                       const TileList &list, int list_blocks, cudaStream_t s, const NciAux &aux,
                       int *reset_other = nullptr, int max_parts = kNciParts);
int nci_list_blocks();
cudaError_t phase_prepare(int dim);

// src/dst are population buffers of the store type; MODE kStep writes dst and u, kMoments writes
// u and pstar only.
cudaError_t launch_hydro(int Q, int store, int mode, const KParams &P, const void *src, void *dst,
                         const int32_t *phi, const float4 *frep, float *u, float *pstar, cudaStream_t s);

// The hydrodynamic step split in two launches around the near-contact pass (3D, nx even,
// Q N <= 2^32: the paired kernel). part 0 updates every 32 x 2 x 4 tile whose near-contact
// tile is not marked in `listed` (those cells are not gated, so they never read frep, and it may
// run while the near-contact pass writes frep); part 1 walks the listed tiles on 2 `blocks`
// resident blocks and updates the rest, after the near-contact pass. Each cell is written by
// exactly one part, with the arithmetic of launch_hydro.
bool hydro_split_applies(int Q, const KParams &P);
cudaError_t launch_hydro_split(int part, int Q, int store, const KParams &P, const void *src, void *dst,
                               const int32_t *phi, const float4 *frep, float *u, const TileList &listed, int blocks,
                               cudaStream_t s);

// Also builds `next` (if its tiles are not null): appends the tiles of phi_out that hold an
// interfacial cell, using next.mark (all zero on entry) in 3D so that each is appended once.
// In 3D the marks of `prev` (the list of phi, consumed by this step's near-contact and
// hydrodynamic passes) are cleared, so that buffer's marks are zero when its list is built again.
cudaError_t launch_phase(int dim, const KParams &P, const int32_t *phi, const float *u, int32_t *phi_out,
                         const TileList &next, const TileList &prev, cudaStream_t s);
// Lists (and in 3D marks) the tiles holding an interfacial cell of phi (after the state is set
// from the host); the count and the marks are zero on entry.
cudaError_t launch_gate_tiles(int dim, const KParams &P, const int32_t *phi, const TileList &list, cudaStream_t s);
int tile_count(int dim, const KParams &P);

// Geometry of the 3D phase-field register march (phase3_march.cuh).
struct March3 {
  static constexpr int OUT = 28;       // output columns per warp
  static constexpr int WARPS = 4;      // warps per block
  static constexpr int NT = 32 * WARPS;
  // fewest planes per warp before the grid is shrunk: a run of n planes takes n + 4 iterations, and
  // a small grid is bound by the time of one run, not by the work (a 48^3 pass: 18.5 us with runs of
  // 8, 10.3 with runs of 2; its whole step 33.6 us with 2, 36.2 with 1, 35.4 with 3)
  static constexpr int MIN_RUN = 2;
};

// Batched passes over many independent cases (the sweep of uneven collision cases). One
// BatchCase per case and buffer parity: where the pass reads and writes, and its tile grids.
struct __align__(16) BatchCase {
  KParams P;
  const void *src;      // populations of the current state
  void *dst;            // populations of the next state
  const int32_t *phi;   // phi^n
  int32_t *phi_out;     // phi^{n+1}
  const float4 *frep;   // near-contact force at the gated cells of phi^n
  float *u;             // velocity, written by the hydrodynamic pass, read by the phase pass
  TileList next;        // near-contact list of phi^{n+1}, built by the phase pass (tiles null: none)
  TileList prev;        // near-contact list of phi^n, whose marks the phase pass clears
  int ncx;              // x segments of the phase march
};
// The paired hydrodynamic kernel over a list of (case, bx, by, bz) tile items of 32 x ty x tz cells
// (ty x tz = 8; all cases D3Q19 or D3Q27 per Q, one store type, nx even, Q N <= 2^32), on a grid of
// `blocks` resident blocks walking the list.
cudaError_t launch_hydro_batch(int Q, int store, int ty, const BatchCase *cases, const int4 *items, int nitems,
                               int blocks, cudaStream_t s);
int hydro_batch_blocks(int Q, int store, int ty);  // resident blocks of the device (SMs x per SM)
// The phase march over the concatenated (column, plane) units of every case (uoff: ncases + 1
// prefix offsets); rows = 2 or 4 rows of y per thread.
cudaError_t launch_phase_batch(int rows, const BatchCase *cases, const long long *uoff, int ncases, int blocks,
                               cudaStream_t s);
int phase_batch_blocks(int rows);

// Conversions between host-layout FP64 staging buffers and the device state.
cudaError_t launch_phi_in(const KParams &P, const double *phi64, int32_t *phi, cudaStream_t s);
cudaError_t launch_phi_out(const KParams &P, const int32_t *phi, double *phi64, cudaStream_t s);
cudaError_t launch_f32_out(long long n, const float *src, double *dst, cudaStream_t s);
cudaError_t launch_init_pops(int Q, int store, const KParams &P, const double *u64, const double *ps64,
                             void *pops, cudaStream_t s);
cudaError_t launch_set_pops(int Q, int store, const KParams &P, const double *f64, void *pops, cudaStream_t s);
cudaError_t launch_get_pops(int Q, int store, const KParams &P, const void *pops, double *f64, cudaStream_t s);
cudaError_t launch_partner_frep_out(const KParams &P, int dim, const float4 *frep, double *frep64,
                                    cudaStream_t s);

// FP64 / exact-integer reductions over the current fields.
struct ReduceOut {
  long long phi_q30;  // exact sum of the fixed-point phi
  double mom[3];      // sum of rho(phi) u
  long long nonfinite;
};
constexpr int kReduceBlocks = 608;  // 4 per SM of a 152-SM GB300
// The phi sum (exact), the non-finite count of u (u may be null when mom is false) and, with mom,
// the FP64 momentum sum of rho(phi) u.
cudaError_t launch_reduce(const KParams &P, const int32_t *phi, const float *u, ReduceOut *partials,
                          ReduceOut *out, cudaStream_t s, bool mom = true);
// The same reduction on a grid of nblocks blocks (nblocks partial slots).
cudaError_t launch_reduce_n(const KParams &P, const int32_t *phi, const float *u, ReduceOut *partials,
                            int nblocks, ReduceOut *out, cudaStream_t s);

// Near-contact film statistics (Sec. 3.3): over the cells with a partner (frep.w = 1 at gated
// cells), V_film, sum |F_rep.n|, sum |F_cap.n|, max |F_rep|, sum |F_rep| in FP64, fixed order.
struct DiagOut {
  double v[5];
};
cudaError_t launch_nci_diag(int dim, const KParams &P, const int32_t *phi, const float4 *frep, DiagOut *partials,
                            DiagOut *out, cudaStream_t s);

// Interfacial mean curvature kappa = div n (Sec. 3.4, Eq. 78): normals of every cell into nrm, then
// over the band q >= q_th a histogram of kappa on [kmin, kmax) (nbins <= kMaxCurvBins, integer
// counts) and the band's cell count and sum of kappa (FP64, fixed order): out = {count, sum}.
constexpr int kMaxCurvBins = 4096;

// Carrier-phase kinetic-energy spectrum (Sec. 3.4) of the velocity u (3N) into E_dev (nshells
// doubles on the device), synchronous on s. Returns 0, 1 (bad nshells), 2 (CUDA error or out of
// memory) or 3 (cuFFT failure). Allocates about 8N bytes plus the transform's workspace per call.
constexpr int kMaxSpectrumShells = 1024;
int spectrum_compute(const KParams &P, const int32_t *phi, const float *u, int nshells, double *E_dev,
                     cudaStream_t s);
cudaError_t launch_curvature(int dim, const KParams &P, const int32_t *phi, float4 *nrm, float kmin, float kmax,
                             int nbins, unsigned long long *hist, double *partials, double *out, cudaStream_t s);

}  // namespace lbm
