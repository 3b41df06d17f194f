// kernels_phase.cu -- the phase-field half of a time step (Sec. 2.1.1): Eq. 28,
//   phi^{n+1} = phi^n - div_h(u phi) + D lap_h(phi) + S_comp,
// with MUSCL-minmod face fluxes (Eqs. 29-34), the isotropic Laplacian (Eq. 23) and the
// isotropic compressive divergence S_comp = -(kappa / cs^2) sum_i w_i c_i . a(x + c_i),
// a = phi (1 - phi) n, kappa = 4 D / eps (Eqs. 26, 35).
//
// Face-flux form. The D2Q9 and D3Q27 weights are tensor products of the 1D weights
// (1, 4, 1) / 6, w_i = s(c_x) s(c_y) [s(c_z)] / 6^d with s(0) = 4, s(+-1) = 1. Writing s = 6 + d2
// (d2 the 1D second difference), the isotropic Laplacian 6 (sum_i w_i phi(x + c_i) - phi) expands
// into sum_a d2_a(B_a phi) with, in 3D, B_x = s_y s_z / 36, B_y = s_z / 6, B_z = 1 (2D: B_x = s_y / 6,
// B_y = 1), and the isotropic divergence sum_i w_i c_i . a(x + c_i) into a difference of face
// sums with weights s_b s_c / 216 (2D: s_b / 36) over the two transverse axes. Hence
//   phi^{n+1}(x) - phi^n(x) = sum_a [ tau_a(x - e_a / 2) - tau_a(x + e_a / 2) ],
//   tau_a(x + e_a/2) = u_f phi_up + D B_a (phi(x) - phi(x + e_a))
//                      + 3 kappa W_a (a_a(x) + a_a(x + e_a)),   W_a = s_b s_c / 216 (2D s_b / 36),
// which equals Eq. 28 term by term in exact arithmetic. Each face transfer tau is computed once
// per block (the cells of a tile plus the faces on its low boundary), rounded once to the 2^-30
// fixed-point phi grid and applied with opposite signs on its two cells, so sum(phi) is exactly
// conserved. The kernel also lists the tiles of the near-contact kernel (same tiling) that hold an
// interfacial cell of phi^{n+1}, so the next near-contact pass visits only those.
// This file holds the 2D kernel (one block per tile, shared-memory face transfers) and the
// launchers; the 3D update is the register march of phase3_march.cuh.
#include "launch.h"
#include "phase3_march.cuh"

namespace lbm {

// Tile shapes of the near-contact lists (2D: also of the phase kernel).
template <int DIM> struct PhaseGeom {
  static constexpr int TX = PhaseTile<DIM>::X, TY = PhaseTile<DIM>::Y, TZ = PhaseTile<DIM>::Z;
  static constexpr int NT = TX * TY * TZ;
};
// The 2D phase kernel's shared-memory boxes and face transfers.
struct Phase2 : PhaseGeom<2> {
  static_assert(TZ == 1, "a plane");
  static constexpr int HX = TX + 4, HY = TY + 4, NB = HX * HY;  // phi, halo 2
  static constexpr int AX = TX + 2, AY = TY + 2, NA = AX * AY;  // a, halo 1
  // face transfers: faces of the tile cells on their high side plus the low boundary faces
  static constexpr int FX = (TX + 1) * TY, FY = TX * (TY + 1);
};

__device__ __forceinline__ int32_t minmod_i(int32_t a, int32_t b) {
  if (a > 0 && b > 0) return a < b ? a : b;
  if (a < 0 && b < 0) return a > b ? a : b;
  return 0;
}

// Transfer across the face between cells p and p + e_AX (tile-local coordinates, p may be one
// cell below the tile). s_phi has halo 2, s_a halo 1.
template <int AXIS>
__device__ __forceinline__ int32_t face_transfer(const KParams &P, const int32_t *s_phi, const float *s_a,
                                                 const float *__restrict__ u, int px, int py, int gx, int gy) {
  using G = Phase2;
  constexpr int SX = 1, SY = G::HX;    // phi-box strides
  constexpr int AXS = 1, AYS = G::AX;  // a-box strides
  constexpr int E = AXIS == 0 ? SX : SY;
  constexpr int EA = AXIS == 0 ? AXS : AYS;
  const int b = (py + 2) * SY + px + 2;
  const int ba = (py + 1) * AYS + px + 1;
  const int32_t v0 = s_phi[b], v1 = s_phi[b + E];

  // diffusion D B_a (phi(p) - phi(p + e)) with exact integer differences
  float dif;
  if (AXIS == 0) {
    // B = s_y / 6
    float acc = __fmul_rn(4.f, dphi_of(v0, v1));
    acc = __fadd_rn(acc, dphi_of(s_phi[b - SY], s_phi[b - SY + E]));
    acc = __fadd_rn(acc, dphi_of(s_phi[b + SY], s_phi[b + SY + E]));
    dif = __fmul_rn(acc, 1.0f / 6.0f);
  } else {
    dif = dphi_of(v0, v1);
  }
  float tau = __fmul_rn(P.Dlap * (1.0f / 6.0f), dif);  // Dlap = 6 D

  // compressive transfer 3 kappa W_a (a_a(p) + a_a(p + e)), W_a = s_b / 36
  {
    const float *sa = s_a + AXIS * G::NA;
    constexpr int T1 = AXIS == 0 ? AYS : AXS;
    float acc = __fmul_rn(4.f, __fadd_rn(sa[ba], sa[ba + EA]));
    acc = __fadd_rn(acc, __fadd_rn(sa[ba - T1], sa[ba - T1 + EA]));
    acc = __fadd_rn(acc, __fadd_rn(sa[ba + T1], sa[ba + T1 + EA]));
    acc = __fmul_rn(acc, 1.0f / 36.0f);
    tau = __fadd_rn(tau, __fmul_rn(P.kc * kCs2 * 3.0f, acc));  // kc = kappa / cs^2 -> 3 kappa
  }

  // MUSCL face flux u_f phi_up (Eqs. 30-34)
  {
    const int32_t vm = s_phi[b - E], vp = s_phi[b + 2 * E];
    const int32_t s0 = minmod_i(v0 - vm, v1 - v0);
    const int32_t s1 = minmod_i(v1 - v0, vp - v1);
    // global cells p and p + e (periodic)
    int qx = gx, qy = gy;
    if (AXIS == 0) qx = qx == P.nx - 1 ? 0 : qx + 1;
    if (AXIS == 1) qy = qy == P.ny - 1 ? 0 : qy + 1;
    const long long N = P.N;
    const float ua = __ldg(u + AXIS * N + gx + (long long)P.nx * gy);
    const float ub = __ldg(u + AXIS * N + qx + (long long)P.nx * qy);
    const float uf = __fmul_rn(0.5f, __fadd_rn(ua, ub));
    // upwind state; exact integer slopes, FP32 sum (no 64-bit conversion, which runs on the FP64 pipe)
    const float pup = uf >= 0.0f ? (__int2float_rn(v0) + 0.5f * __int2float_rn(s0)) * kInvQ30
                                 : (__int2float_rn(v1) - 0.5f * __int2float_rn(s1)) * kInvQ30;
    tau = __fadd_rn(tau, __fmul_rn(uf, pup));
  }
  return __float2int_rn(__fmul_rn(tau, kQ30));
}

__global__ void __launch_bounds__(Phase2::NT)
k_phase2(const KParams P, const int32_t *__restrict__ phi, const float *__restrict__ u,
         int32_t *__restrict__ phi_out, const TileList next) {
  pdl_enter();
  using G = Phase2;
  using SL = StencilOf<2>::type;
  __shared__ int32_t s_phi[G::NB];
  __shared__ float s_a[2 * G::NA];
  __shared__ int32_t s_tx[G::FX], s_ty[G::FY];

  const int tx = threadIdx.x, ty = threadIdx.y;
  const int tid = tx + G::TX * ty;
  const int x0 = blockIdx.x * G::TX, y0 = blockIdx.y * G::TY;
  const int nx = P.nx, ny = P.ny;

  // stage phi (halo 2) row by row: rows of HX = TX + 4 values
  int32_t some = 0;
  {
    const int xl = wrapn(x0 - 2 + tx, nx);
    const int xr = wrapn(x0 + 30 + (tx & 3), nx);
    for (int r = ty; r < G::HY; r += G::TY) {
      const int32_t *row = phi + (long long)nx * wrapn(y0 + r - 2, ny);
      some |= s_phi[r * G::HX + tx] = row[xl];
      if (tx < 4) some |= s_phi[r * G::HX + 32 + tx] = row[xr];
    }
  }
  // Where phi is exactly zero in the tile and its halo (gas further from every interface than the
  // profiles and their diffusive tails reach), each transfer of the tile is zero, since phi, its
  // differences and the compressive vector are: phi stays zero and holds no interfacial cell. The tails
  // grow as 3 sqrt(t) cells at first and slow down as they round to zero, so the gain lasts but shrinks.
  // A step of 1021 x 509 with two droplets of radius 96, with the test and without it: at step 100 27.1
  // and 31.1 us (773 of 1024 tiles empty), at 4000 28.0 and 31.2 (559), at 16000 29.0 and 30.8 (355); on
  // 2048 x 2048 106.5 and 162.5, at step 16000 110 and 162.
  // (In the 3D march the same test did not pay: it gained 9 % of the pass on 256 x 128 x 128 and cost a third of
  // it on 160 x 96 x 96, and both grids are full after about 50 steps.)
  if (!__syncthreads_or(some)) {
    const int x = x0 + tx, y = y0 + ty;
    if (x < nx && y < ny) phi_out[(long long)x + (long long)nx * y] = 0;
    if (next.tiles && tid == 0) next.mark[blockIdx.x + gridDim.x * blockIdx.y] = 0;
    return;
  }

  // compressive vector a = phi (1 - phi) grad(phi) / (|grad(phi)| + eps_n) on the tile + 1 halo
  for (int t = tid; t < G::NA; t += G::NT) {
    const int b = (t / G::AX + 1) * G::HX + t % G::AX + 1;
    float g0 = 0.f, g1 = 0.f;
#pragma unroll
    for (int i = 1; i < SL::Q; i++) {
      if (!positive<SL>(i)) continue;
      const int o = SL::c(i, 0) + G::HX * SL::c(i, 1);
      const float d = SL::w(i) * dphi_of(s_phi[b + o], s_phi[b - o]);
      g0 += SL::c(i, 0) * d;
      g1 += SL::c(i, 1) * d;
    }
    g0 *= 3.0f; g1 *= 3.0f;
    const float ph = phi_of(s_phi[b]);
    const float s = ph * (1.0f - ph) / (sqrtf(g0 * g0 + g1 * g1) + P.eps_n);
    s_a[t] = g0 * s;
    s_a[G::NA + t] = g1 * s;
  }
  __syncthreads();

  // face transfers: x faces (TX + 1) x TY with the low face of the tile first
  for (int t = tid; t < G::FX; t += G::NT) {
    const int px = t % (G::TX + 1) - 1, fy = t / (G::TX + 1);  // px: left cell, tile-local
    s_tx[t] = face_transfer<0>(P, s_phi, s_a, u, px, fy, wrapn(x0 + px, nx), wrapn(y0 + fy, ny));
  }
  for (int t = tid; t < G::FY; t += G::NT) {
    const int fx = t % G::TX, py = t / G::TX - 1;
    s_ty[t] = face_transfer<1>(P, s_phi, s_a, u, fx, py, wrapn(x0 + fx, nx), wrapn(y0 + py, ny));
  }
  __syncthreads();

  const int x = x0 + tx, y = y0 + ty;
  bool gated = false;
  if (x < nx && y < ny) {
    int32_t acc = s_tx[tx + (G::TX + 1) * ty] - s_tx[tx + 1 + (G::TX + 1) * ty];
    acc += s_ty[tx + G::TX * ty] - s_ty[tx + G::TX * (ty + 1)];
    const int32_t vn = s_phi[(ty + 2) * G::HX + tx + 2] + acc;
    phi_out[(long long)x + (long long)nx * y] = vn;
    gated = q_gate_value(vn) >= P.q_th;
  }
  if (next.tiles) {  // one block per tile: it sets the tile's mark either way
    const int any = __syncthreads_or(gated);
    if (tid == 0) {
      const int tile = blockIdx.x + gridDim.x * blockIdx.y;
      next.mark[tile] = any != 0;
      if (any) next.tiles[atomicAdd(next.count, 1)] = tile;
    }
  }
}

static cudaError_t launch_phase2(const KParams &P, const int32_t *phi, const float *u, int32_t *phi_out,
                                 const TileList &next, cudaStream_t s) {
  using G = Phase2;
  dim3 grid((P.nx + G::TX - 1) / G::TX, (P.ny + G::TY - 1) / G::TY);
  return launch_pdl(k_phase2, grid, dim3(G::TX, G::TY), 0, s, P, phi, u, phi_out, next);
}

// Records once, at context creation, how many k_phase3m blocks the device holds at once (SMs x
// resident blocks), so that the launches make no non-stream CUDA call (they may be captured).
static int g_march_slots2 = 0, g_march_slots4 = 0;  // two and four rows of y per thread

cudaError_t phase_prepare(int dim) {
  static bool done = false;
  if (dim != 3 || done) return cudaSuccess;
  int dev = 0, sms = 0, per2 = 0, per4 = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per2, k_phase3m<2>, March3::NT, 0);
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per4, k_phase3m<4>, March3::NT, 0);
  if (e == cudaSuccess) {
    g_march_slots2 = sms * (per2 > 0 ? per2 : 1);
    g_march_slots4 = sms * (per4 > 0 ? per4 : 1);
    done = true;
  }
  return e;
}

// One resident wave of warps sharing the (column, plane) units equally, at least MIN_RUN planes each.
template <int M, class Off = unsigned>
static cudaError_t launch_march(const KParams &P, const int32_t *phi, const float *u, int32_t *phi_out,
                                const TileList &next, const TileList &prev, int slots, cudaStream_t s) {
  const int ncx = (P.nx + March3::OUT - 1) / March3::OUT, ncy = (P.ny + M - 1) / M;
  const long long units = (long long)ncx * ncy * P.nz;
  const long long want = (units + March3::MIN_RUN - 1) / March3::MIN_RUN;
  long long blocks = (want + March3::WARPS - 1) / March3::WARPS;
  if (blocks > slots) blocks = slots;
  if (blocks < 1) blocks = 1;
  const TileList none{};
  return launch_pdl(k_phase3m<M, Off>, dim3((unsigned)blocks), dim3(March3::NT), 0, s, P, phi, u, phi_out,
                    next.tiles ? next : none, next.tiles ? prev : none, ncx, units);
}

// Two rows per thread up to 44 planes per warp of the four-row kernel, four beyond. A whole step with
// four and with two: 64^3 40.0 and 36.5 us, 96^3 66.8 and 64.2, 128^3 117.8 and 115.3, 256 x 128 x 128 (34 planes)
// 210.8 and 207.7, 192^3 (53 planes) 348.5 and 349.2, 256^3 798 and 805, 384^3 2717 and 2754.
static cudaError_t launch_phase3(const KParams &P, const int32_t *phi, const float *u, int32_t *phi_out,
                                 const TileList &next, const TileList &prev, cudaStream_t s) {
  const cudaError_t e = phase_prepare(3);
  if (e != cudaSuccess) return e;
  if (march_wide(P))
    return launch_march<4, unsigned long long>(P, phi, u, phi_out, next, prev, g_march_slots4, s);
  const long long units4 = (long long)((P.nx + March3::OUT - 1) / March3::OUT) * ((P.ny + 3) / 4) * P.nz;
  if (units4 <= 44LL * March3::WARPS * g_march_slots4)
    return launch_march<2>(P, phi, u, phi_out, next, prev, g_march_slots2, s);
  return launch_march<4>(P, phi, u, phi_out, next, prev, g_march_slots4, s);
}

cudaError_t launch_phase(int dim, const KParams &P, const int32_t *phi, const float *u, int32_t *phi_out,
                         const TileList &next, const TileList &prev, cudaStream_t s) {
  return dim == 2 ? launch_phase2(P, phi, u, phi_out, next, s)
                  : launch_phase3(P, phi, u, phi_out, next, prev, s);
}

// Lists the tiles holding an interfacial cell of phi (used after the state is set from the host).
template <int DIM>
__global__ void __launch_bounds__(PhaseGeom<DIM>::NT)
k_gate_tiles(const KParams P, const int32_t *__restrict__ phi, int *__restrict__ tiles, int *__restrict__ ntiles,
             int *__restrict__ mark) {
  using G = PhaseGeom<DIM>;
  const int x = blockIdx.x * G::TX + threadIdx.x, y = blockIdx.y * G::TY + threadIdx.y,
            z = blockIdx.z * G::TZ + threadIdx.z;
  bool gated = false;
  if (x < P.nx && y < P.ny && z < P.nz)
    gated = q_gate_value(phi[(long long)x + (long long)P.nx * (y + (long long)P.ny * z)]) >= P.q_th;
  const int any = __syncthreads_or(gated);
  if (any && threadIdx.x == 0 && threadIdx.y == 0 && threadIdx.z == 0) {
    const int tile = blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * blockIdx.z);
    tiles[atomicAdd(ntiles, 1)] = tile;
    mark[tile] = 1;
  }
}

cudaError_t launch_gate_tiles(int dim, const KParams &P, const int32_t *phi, const TileList &list, cudaStream_t s) {
  if (dim == 2) {
    using G = PhaseGeom<2>;
    dim3 grid((P.nx + G::TX - 1) / G::TX, (P.ny + G::TY - 1) / G::TY, 1);
    k_gate_tiles<2><<<grid, dim3(G::TX, G::TY, G::TZ), 0, s>>>(P, phi, list.tiles, list.count, list.mark);
  } else {
    using G = PhaseGeom<3>;
    dim3 grid((P.nx + G::TX - 1) / G::TX, (P.ny + G::TY - 1) / G::TY, (P.nz + G::TZ - 1) / G::TZ);
    k_gate_tiles<3><<<grid, dim3(G::TX, G::TY, G::TZ), 0, s>>>(P, phi, list.tiles, list.count, list.mark);
  }
  return cudaGetLastError();
}

}  // namespace lbm
