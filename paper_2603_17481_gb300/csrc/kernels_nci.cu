// kernels_nci.cu -- near-contact interaction (Sec. 2.3): interfacial gate (Eqs. 58-59), bounded
// window pairing (Eqs. 60-65), closed-form proximity indicator and repulsive force (Eqs. 66-73).
//
// Passes over the tiles that hold an interfacial (gated) cell, as listed by the phase-field kernel
// of the previous step (or over every tile for the diagnostic read-back):
//   k_nci_normals3 / k_nci_normals2  the normal n = grad(phi) / (|grad(phi)| + eps_n) of every gated
//                  cell (Eq. 57, isotropic gradient of Eq. 22), computed once and stored as a float4;
//                  zero force at every gated cell (listed tiles); for every row of 32 cells six
//                  (2D: four) 32-bit masks of its gated cells by the direction of their normals; in
//                  3D also the normal ranges of each 4x4x4 brick;
//   k_nci_prefilter (3D, sides multiples of 4) per listed tile, a lower bound of n(x).n(y) from the
//                  brick ranges; only the half tiles where the facing gate can hold go on to the scan;
//   k_nci_scan     per unit (half a tile in 3D): the cells that have a possible partner in their
//                  window by the masks, then one warp per such cell tests its possible partners,
//                  keeps the nearest accepted one and writes the force. On 3D sides that are not
//                  multiples of 4 its blocks also make the brick test.
// The masks are exact: for a cell whose normal's largest component is n_a > 0, a partner with
// n(x).n(y) <= cos_opp (Eq. 62) has a component m_a below a bound that cos_opp fixes (face_t of the
// parameters; 0.03 at the paper's -0.8, so partners point the other way along a), and likewise for
// n_a < 0: class 2 a holds the gated cells with m_a <= face_t, class 2 a + 1 those with m_a >= -face_t.
// One word answers which cells of a window row may face a cell, so an interface that faces nothing
// costs 49 words per cell, and the accepted-partner test (Eqs. 59, 61, 62, 65) reads the normals of the
// few cells that remain.
// The pass is bound by latency: few units are scanned (20 on 48^3, 60 on 256 x 128 x 128), and a unit is
// one chain of dependent reads at 700 to 1000 cycles each. So lists are read with their counts,
// a unit's masks, normals and phi together, and a warp reads several possible partners at once.
// Staging phi and the normals of a unit + 3 halo in shared memory took 12000 to 15000 cycles alone,
// and one list of all cells, a warp per cell over all SMs, 7000 to 9000 cycles per cell.
// The force is written only at gated cells; the hydrodynamic kernel reads it exactly there (same
// gate function).
#include "launch.h"

namespace lbm {

// Window radius bound, words of a mask record (one per row of 32 cells) and direction classes.
constexpr int kWin = 3, kMaskWords = 8;
template <int DIM> constexpr int kClasses = 2 * DIM;

// The scan's unit of work: half a near-contact tile in 3D (32 x 4 x 4 cells), a tile in 2D.
template <int DIM> struct NciGeom {
  static constexpr int TX = NciTile<DIM>::X, TY = DIM == 3 ? NciTile<DIM>::Y / 2 : NciTile<DIM>::Y, TZ = NciTile<DIM>::Z;
  static constexpr int UNITS = DIM == 3 ? 2 : 1;  // units of a tile, along y
  static constexpr int NT = TX * TY * TZ, NW = NT / 32;
};

// The masks of the rows around a unit: 38 columns (bit j of a row: column x0 - 3 + j, in two words),
// TY + 6 by TZ + 6 rows (2D: one plane).
template <int DIM> struct MaskBox {
  using G = NciGeom<DIM>;
  static constexpr int COLS = 32 + 2 * kWin, HY = G::TY + 2 * kWin, HZ = DIM == 3 ? G::TZ + 2 * kWin : 1, ROWS = HY * HZ;
  uint2 m[kClasses<DIM>][ROWS];
};

// The direction class whose members may face a cell with normal n: the axis of its largest component.
template <int DIM> __device__ __forceinline__ int facing_class(const float4 &n) {
  const float a0 = fabsf(n.x), a1 = fabsf(n.y), a2 = fabsf(n.z);
  if (DIM == 3 && a2 > a0 && a2 > a1) return 4 + (n.z > 0.0f ? 0 : 1);
  if (a1 > a0) return 2 + (n.y > 0.0f ? 0 : 1);
  return n.x > 0.0f ? 0 : 1;
}

// Writes the mask record of one row of 32 cells (the warp's; g: this lane's cell is gated, n its normal).
template <int DIM>
__device__ __forceinline__ void store_masks(const KParams &P, unsigned *__restrict__ rec, bool g, float n0, float n1,
                                            float n2, int lane) {
  const float a[3] = {n0, n1, n2};
  unsigned mine = 0;
  if (__any_sync(0xffffffffu, g)) {
#pragma unroll
    for (int c = 0; c < kClasses<DIM>; c++) {
      const unsigned m = __ballot_sync(0xffffffffu, g && ((c & 1) ? a[c >> 1] >= -P.face_t : a[c >> 1] <= P.face_t));
      if (lane == c) mine = m;
    }
  }
  if (lane < kClasses<DIM>) rec[lane] = mine;
}

// Fills the mask box (all zero on entry) of the unit at (x0, y0, z0), threads tid of nt. A row of 38 columns of
// the periodic grid is made of pieces that end at a word's or the grid's edge, three where nx is a
// multiple of 32; each thread takes one piece of a row, so all reads are in flight together. A piece
// in a tile that is not listed has no gated cell (its record is of an older step); mark == nullptr:
// every tile is listed.
template <int DIM>
__device__ __forceinline__ void stage_masks(const KParams &P, MaskBox<DIM> &box, const unsigned *__restrict__ masks,
                                            const int *__restrict__ mark, int gtx, int gty, int x0, int y0, int z0,
                                            int tid, int nt) {
  using M = MaskBox<DIM>;
  const int nx = P.nx, s = wrapn(x0 - kWin, nx);
  // pieces per row: a word's piece is at least 32 columns except at the ends and at the grid's edge
  const int pieces = nx % 32 == 0 ? 3 : 3 + 2 * (M::COLS / nx + 1);
  for (int it = tid; it < pieces * M::ROWS; it += nt) {
    const int r = it % M::ROWS, k = it / M::ROWS;
    int col = s, pos = 0, take = 0;
    for (int j = 0;; j++) {
      take = min(min(32 - (col & 31), nx - col), M::COLS - pos);
      if (j == k || take == 0) break;
      pos += take;
      col += take;
      if (col == nx) col = 0;
    }
    if (take == 0) continue;
    const int y = wrapn(y0 - kWin + r % M::HY, P.ny), z = DIM == 3 ? wrapn(z0 - kWin + r / M::HY, P.nz) : 0;
    const uint4 *rec = reinterpret_cast<const uint4 *>(masks) +
                       kMaskWords / 4 * ((col >> 5) + gtx * (y + (long long)P.ny * z));
    const uint4 a = rec[0];
    const uint2 b = DIM == 3 ? *reinterpret_cast<const uint2 *>(rec + 1) : make_uint2(0u, 0u);
    if (mark && !mark[(col >> 5) + gtx * (y / NciTile<DIM>::Y + gty * (z / NciTile<DIM>::Z))]) continue;
    const unsigned w[6] = {a.x, a.y, a.z, a.w, b.x, b.y};
#pragma unroll
    for (int c = 0; c < kClasses<DIM>; c++) {
      const unsigned v = take == 32 ? w[c] : (w[c] >> (col & 31)) & ((1u << take) - 1u);
      if (!v) continue;
      const unsigned long long p = (unsigned long long)v << pos;
      if ((unsigned)p) atomicOr(&box.m[c][r].x, (unsigned)p);
      if (p >> 32) atomicOr(&box.m[c][r].y, (unsigned)(p >> 32));
    }
  }
}

// The possible partners (7 columns x - 3 .. x + 3, bits above are not cleared) of the cell in column cx in
// a row of its class.
__device__ __forceinline__ unsigned window_bits(const uint2 &row, int cx) { return __funnelshift_r(row.x, row.y, cx); }

// Whether the cell in column tx, row (ty, tz) of the unit, with normal n, has a possible partner in its
// window of radius W.
template <int DIM, int W>
__device__ __forceinline__ bool may_face(const MaskBox<DIM> &box, const float4 &n, int tx, int ty, int tz) {
  using M = MaskBox<DIM>;
  const uint2 *m = box.m[facing_class<DIM>(n)] + (DIM == 3 ? (tz + kWin) * M::HY : 0) + ty + kWin;
  unsigned any = 0;
#pragma unroll
  for (int dz = DIM == 3 ? -W : 0; dz <= (DIM == 3 ? W : 0); dz++)
#pragma unroll
    for (int dy = -W; dy <= W; dy++) any |= window_bits(m[dz * M::HY + dy], tx);
  return (any & (((1u << (2 * W + 1)) - 1u) << (kWin - W))) != 0u;
}

template <int DIM>
__device__ __forceinline__ void tile_of(int tile, int gtx, int gty, int &bx, int &by, int &bz) {
  bx = tile % gtx;
  by = (tile / gtx) % gty;
  bz = tile / (gtx * gty);
}

// Normals, masks and zero force of the gated cells of the listed tiles (or normals and masks of every
// tile when tiles == nullptr), 2D: a warp per row of a tile.
__global__ void __launch_bounds__(NciGeom<2>::NT)
k_nci_normals2(const KParams P, const int32_t *__restrict__ phi, float4 *__restrict__ nrm, float4 *__restrict__ frep,
               const int *__restrict__ tiles, const int *__restrict__ ntiles, int total, int gtx, int gty,
               unsigned *__restrict__ masks, int *__restrict__ reset_other) {
  pdl_enter();
  if (reset_other && blockIdx.x == 0 && threadIdx.x == 0 && threadIdx.y == 0) *reset_other = 0;
  using G = NciGeom<2>;
  using SL = StencilOf<2>::type;
  const int first = tiles ? tiles[blockIdx.x] : 0;  // in flight with the count (the list has room for every tile)
  const int n = tiles ? *ntiles : total;
  const int nx = P.nx, ny = P.ny;
  for (int t = blockIdx.x; t < n; t += gridDim.x) {
    int bx, by, bz;
    tile_of<2>(!tiles ? t : (t == (int)blockIdx.x ? first : tiles[t]), gtx, gty, bx, by, bz);
    const int x = bx * G::TX + threadIdx.x, y = by * G::TY + threadIdx.y;
    if (y >= ny) continue;  // the whole warp
    const long long idx = (long long)x + (long long)nx * y;
    const bool g = x < nx && q_gate_value(phi[idx]) >= P.q_th;
    float g0 = 0.f, g1 = 0.f;
    if (g) {
      const int X[3] = {x == 0 ? nx - 1 : x - 1, x, x == nx - 1 ? 0 : x + 1};
      const int Y[3] = {y == 0 ? ny - 1 : y - 1, y, y == ny - 1 ? 0 : y + 1};
#pragma unroll
      for (int i = 1; i < SL::Q; i++) {
        if (!positive<SL>(i)) continue;
        const int c0 = SL::c(i, 0), c1 = SL::c(i, 1);
        const float d = SL::w(i) * dphi_of(__ldg(phi + X[1 + c0] + (long long)nx * Y[1 + c1]),
                                           __ldg(phi + X[1 - c0] + (long long)nx * Y[1 - c1]));
        g0 += c0 * d;
        g1 += c1 * d;
      }
      g0 *= 3.0f; g1 *= 3.0f;
      const float inv = 1.0f / (sqrtf(g0 * g0 + g1 * g1) + P.eps_n);
      g0 = g0 * inv; g1 = g1 * inv;
      nrm[idx] = make_float4(g0, g1, 0.0f, 0.0f);
      if (tiles) frep[idx] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    store_masks<2>(P, masks + (long long)kMaskWords * (bx + (long long)gtx * y), g, g0, g1, 0.f, threadIdx.x);
  }
}

// Normals of the gated cells of the listed tiles (or of every tile when tiles == nullptr), 3D.
// One 128-thread block per half tile (32 x 4 x 4 cells, eight 4x4x4 bricks side by side in x):
// phi of the half tile + 1 halo (34 x 6 x 6) is staged in shared memory, then warp w takes the 4
// rows of plane z0 + w (a thread per cell spends more on the bricks than it gains in latency: 414
// against 164 us on the 384^3 swarm, 13.9 against 7.2 on 256 x 128 x 128). The gradient is the
// isotropic D3Q27 one of Eq. 22, summed over the 13 links in the same order as everywhere else.
// On listed tiles every gated cell's force is set to zero here (it is overwritten where a partner is
// found) and, with the bricks, the component ranges of the gated normals of each brick are stored (empty bricks as [+inf, -inf]; cells beyond the grid in the last brick of a side
// that is not a multiple of 4 count as not gated).
constexpr int kNrmThreads = 128;
struct NrmBox {
  static constexpr int X = 34, Y = 6, Z = 6, ROWS = Y * Z;  // warp w stages rows w, w + 4, ...
};

__global__ void __launch_bounds__(kNrmThreads)
k_nci_normals3(const KParams P, const int32_t *__restrict__ phi, float4 *__restrict__ nrm, float4 *__restrict__ frep,
               const int *__restrict__ tiles, const int *__restrict__ ntiles, int total, int gtx, int gty,
               const NciAux aux, int *__restrict__ reset_other) {
  pdl_enter();
  using G = NciGeom<3>;
  using SL = StencilOf<3>::type;
  using B = NrmBox;
  static_assert(G::TX == 32 && G::TY == 4 && G::TZ == 4, "half a near-contact tile");
  __shared__ int32_t s_box[B::ROWS * B::X];
  __shared__ float s_part[4][8][6];  // [warp][brick][lo0..hi2]
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const bool bricks = aux.bricks != nullptr;  // uniform over the grid
  const int first = tiles ? tiles[blockIdx.x >> 1] : 0;  // in flight with the count (the list has room for every tile)
  const int n = tiles ? *ntiles : total;
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    if (reset_other) *reset_other = 0;
    if (bricks) *aux.nscan = 0;
  }
  const int nx = P.nx, ny = P.ny, nz = P.nz;
  const float inf = __int_as_float(0x7f800000);
  for (int item = blockIdx.x; item < 2 * n; item += gridDim.x) {
    const int tile = !tiles ? (item >> 1) : (item == (int)blockIdx.x ? first : tiles[item >> 1]);
    const int half = item & 1;
    int bx, by, bz;
    tile_of<3>(tile, gtx, gty, bx, by, bz);
    const int x0 = bx * G::TX, y0 = by * NciTile<3>::Y + 4 * half, z0 = bz * G::TZ;
    {
      const int xa = wrapn(x0 - 1 + lane, nx), xb = wrapn(x0 + 31 + (lane & 1), nx);
      int32_t va[9], vb[9];
#pragma unroll
      for (int j = 0; j < 9; j++) {
        const int r = warp + 4 * j, ry = r % B::Y, rz = r / B::Y;
        const long long row = (long long)nx * (wrapn(y0 - 1 + ry, ny) + (long long)ny * wrapn(z0 - 1 + rz, nz));
        va[j] = phi[row + xa];
        if (lane < 2) vb[j] = phi[row + xb];
      }
#pragma unroll
      for (int j = 0; j < 9; j++) {
        const int r = warp + 4 * j;
        s_box[r * B::X + lane] = va[j];
        if (lane < 2) s_box[r * B::X + 32 + lane] = vb[j];
      }
    }
    __syncthreads();
    const int x = x0 + lane, z = z0 + warp;
    const bool xin = x < nx && z < nz;
    float lo0 = inf, lo1 = inf, lo2 = inf, hi0 = -inf, hi1 = -inf, hi2 = -inf;
#pragma unroll
    for (int r = 0; r < 4; r++) {
      const int y = y0 + r;
      const int o = ((warp + 1) * B::Y + r + 1) * B::X + lane + 1;
      const bool g = xin && y < ny && q_gate_value(s_box[o]) >= P.q_th;
      float g0 = 0.f, g1 = 0.f, g2 = 0.f;
      if (g) {
#pragma unroll
        for (int i = 1; i < SL::Q; i++) {
          if (!positive<SL>(i)) continue;
          const int c0 = SL::c(i, 0), c1 = SL::c(i, 1), c2 = SL::c(i, 2);
          const int off = c0 + B::X * (c1 + B::Y * c2);
          const float d = SL::w(i) * dphi_of(s_box[o + off], s_box[o - off]);
          g0 += c0 * d;
          g1 += c1 * d;
          g2 += c2 * d;
        }
        g0 *= 3.0f; g1 *= 3.0f; g2 *= 3.0f;
        const float inv = 1.0f / (sqrtf(g0 * g0 + g1 * g1 + g2 * g2) + P.eps_n);
        g0 *= inv; g1 *= inv; g2 *= inv;
        const long long idx = (long long)x + (long long)nx * (y + (long long)ny * z);
        nrm[idx] = make_float4(g0, g1, g2, 0.0f);
        if (tiles) frep[idx] = make_float4(0.f, 0.f, 0.f, 0.f);
        lo0 = fminf(lo0, g0); lo1 = fminf(lo1, g1); lo2 = fminf(lo2, g2);
        hi0 = fmaxf(hi0, g0); hi1 = fmaxf(hi1, g1); hi2 = fmaxf(hi2, g2);
      }
      if (y < ny && z < nz)  // the whole warp
        store_masks<3>(P, aux.masks + (long long)kMaskWords * (bx + (long long)gtx * (y + (long long)ny * z)), g, g0, g1,
                       g2, lane);
    }
    if (bricks) {  // lanes 4k..4k+3 of each warp share brick k; the four planes meet in shared memory
#pragma unroll
      for (int sh = 1; sh <= 2; sh <<= 1) {
        lo0 = fminf(lo0, __shfl_xor_sync(0xffffffffu, lo0, sh));
        lo1 = fminf(lo1, __shfl_xor_sync(0xffffffffu, lo1, sh));
        lo2 = fminf(lo2, __shfl_xor_sync(0xffffffffu, lo2, sh));
        hi0 = fmaxf(hi0, __shfl_xor_sync(0xffffffffu, hi0, sh));
        hi1 = fmaxf(hi1, __shfl_xor_sync(0xffffffffu, hi1, sh));
        hi2 = fmaxf(hi2, __shfl_xor_sync(0xffffffffu, hi2, sh));
      }
      if ((lane & 3) == 0) {
        float *sp = s_part[warp][lane >> 2];
        sp[0] = lo0; sp[1] = lo1; sp[2] = lo2; sp[3] = hi0; sp[4] = hi1; sp[5] = hi2;
      }
    }
    __syncthreads();  // s_part complete; s_box and s_part are free for the next item after this
    if (bricks) {
      const int k = threadIdx.x;
      const int gbx = 8 * bx + k, gby = 2 * by + half;
      if (k < 8 && gbx < ((nx + 3) >> 2) && gby < ((ny + 3) >> 2)) {
        float v[6];
#pragma unroll
        for (int c = 0; c < 6; c++) {
          v[c] = s_part[0][k][c];
#pragma unroll
          for (int w = 1; w < 4; w++) v[c] = c < 3 ? fminf(v[c], s_part[w][k][c]) : fmaxf(v[c], s_part[w][k][c]);
        }
        const auto h = [](__half q) { return (unsigned)__half_as_ushort(q); };
        uint4 o;
        o.x = h(__float2half_rd(v[0])) | (h(__float2half_rd(v[1])) << 16);
        o.y = h(__float2half_rd(v[2]));
        o.z = h(__float2half_ru(v[3])) | (h(__float2half_ru(v[4])) << 16);
        o.w = h(__float2half_ru(v[5]));
        aux.bricks[(long long)gbx + (long long)((nx + 3) >> 2) * (gby + (long long)((ny + 3) >> 2) * bz)] = o;
      }
    }
  }
}

// Component ranges of the gated normals of some cells: lo0..2, hi0..2.
struct NrmRange {
  float v[6];
};

// The union of the ranges of the bricks that hold the cells 4 jx .. 4 jx + 3 (and likewise in y and z) of
// the periodic grid; a brick of a tile that is not listed holds no gated cell and counts as empty.
// Where a side is a multiple of 4 the four cells are one brick; elsewhere they may touch up to three
// (the last brick of the side is short). At most one axis in four starts a new brick per cell, so
// the loops below run once per distinct brick. ALIGNED: every side is a multiple of 4.
template <bool ALIGNED>
__device__ __forceinline__ NrmRange brick_range(const KParams &P, const uint4 *__restrict__ bricks,
                                                const int *__restrict__ mark, int gtx, int gty, int jx, int jy, int jz) {
  const float inf = __int_as_float(0x7f800000);
  NrmRange r{{inf, inf, inf, -inf, -inf, -inf}};
  const int nbx = (P.nx + 3) >> 2, nby = (P.ny + 3) >> 2;
  const bool ax = !ALIGNED && (P.nx & 3), ay = !ALIGNED && (P.ny & 3), az = !ALIGNED && (P.nz & 3);
  int pz = -1;
  for (int cz = 0; cz < (az ? 4 : 1); cz++) {
    const int bz = ALIGNED ? wrapn(jz, P.nz >> 2) : wrapn(4 * jz + cz, P.nz) >> 2;
    if (bz == pz) continue;
    pz = bz;
    int py = -1;
    for (int cy = 0; cy < (ay ? 4 : 1); cy++) {
      const int by = ALIGNED ? wrapn(jy, P.ny >> 2) : wrapn(4 * jy + cy, P.ny) >> 2;
      if (by == py) continue;
      py = by;
      int px = -1;
      for (int cx = 0; cx < (ax ? 4 : 1); cx++) {
        const int bx = ALIGNED ? wrapn(jx, P.nx >> 2) : wrapn(4 * jx + cx, P.nx) >> 2;
        if (bx == px) continue;
        px = bx;
        const uint4 w = bricks[(long long)bx + (long long)nbx * (by + (long long)nby * bz)];
        if (!mark[(bx >> 3) + gtx * ((by >> 1) + gty * bz)]) continue;
        const auto lo = [](unsigned u) { return __half2float(__ushort_as_half((unsigned short)(u & 0xffffu))); };
        const auto hi = [](unsigned u) { return __half2float(__ushort_as_half((unsigned short)(u >> 16))); };
        r.v[0] = fminf(r.v[0], lo(w.x)); r.v[1] = fminf(r.v[1], hi(w.x)); r.v[2] = fminf(r.v[2], lo(w.y));
        r.v[3] = fmaxf(r.v[3], lo(w.z)); r.v[4] = fmaxf(r.v[4], hi(w.z)); r.v[5] = fmaxf(r.v[5], lo(w.w));
      }
    }
  }
  return r;
}

// A lower bound of n(x).n(y) over the cells x of the brick whose ranges are entry rc of the staged box
// (s_r[component][entry], entries RX wide and RY high) and every gated cell y of their windows, along
// axis a. Every window offset of the scan (each component |r_a| <= 3) stays inside the 27 entries
// around the brick, so with [L, H] their union
//   n(x).n(y) >= sum_a min(lo_a L_a, lo_a H_a, hi_a L_a, hi_a H_a)
// (the product is bilinear, so its minimum over the two boxes is at a corner).
template <int RX, int RY, int NR>
__device__ __forceinline__ float brick_bound(const float (*s_r)[NR], int a, int rc) {
  const float inf = __int_as_float(0x7f800000);
  float L = inf, H = -inf;
#pragma unroll
  for (int dz = -1; dz <= 1; dz++)
#pragma unroll
    for (int dy = -1; dy <= 1; dy++)
#pragma unroll
      for (int dx = -1; dx <= 1; dx++) {
        const int r = rc + dx + RX * (dy + RY * dz);
        L = fminf(L, s_r[a][r]);
        H = fmaxf(H, s_r[3 + a][r]);
      }
  const float lo = s_r[a][rc], hi = s_r[3 + a][rc];
  return fminf(fminf(lo * L, lo * H), fminf(hi * L, hi * H));
}

// One 128-thread block per listed tile (3D, sides multiples of 4). The tile's sixteen bricks are
// tested against the union of the normal ranges of their 27 neighbouring bricks, a 10x4x3 box of
// bricks. Where the bound exceeds cos_opp + 1e-5 for all eight bricks of a half tile, none of its
// cells can meet the facing gate (Eq. 62) and the half keeps the zero force written by the normals
// pass; otherwise it goes to the scan list. mark: the tiles listed for this phi.
__global__ void __launch_bounds__(128, 12)
k_nci_prefilter(const KParams P, const NciAux aux, const int *__restrict__ mark, const int *__restrict__ tiles,
                const int *__restrict__ ntiles, int gtx, int gty) {
  pdl_enter();
  constexpr int RX = 10, RY = 4, RZ = 3, NR = RX * RY * RZ;
  __shared__ float s_r[6][NR];
  __shared__ float s_b[48];
  const int tid = threadIdx.x;
  const int first = tiles[blockIdx.x];  // in flight with the count (the list has room for every tile)
  const int n = *ntiles;
  const int nbx = P.nx >> 2, nby = P.ny >> 2;
  const float thr = P.cos_opp + 1e-5f;
  for (int t = blockIdx.x; t < n; t += gridDim.x) {
    const int tile = t == (int)blockIdx.x ? first : tiles[t];
    int bx, by, bz;
    tile_of<3>(tile, gtx, gty, bx, by, bz);
    if (tid < NR) {
      const int rx = tid % RX, ry = (tid / RX) % RY, rz = tid / (RX * RY);
      const NrmRange r = brick_range<true>(P, aux.bricks, mark, gtx, gty, 8 * bx - 1 + rx, 2 * by - 1 + ry, bz - 1 + rz);
#pragma unroll
      for (int c = 0; c < 6; c++) s_r[c][tid] = r.v[c];
    }
    __syncthreads();
    const int rc = ((tid & 7) + 1) + RX * (((tid >> 3) & 1) + 1 + RY);
    if (tid < 48) s_b[tid] = brick_bound<RX, RY, NR>(s_r, tid >> 4, rc);
    __syncthreads();
    if (tid < 32) {
      const int b = tid & 15;
      const bool has = tid < 16 && 8 * bx + (tid & 7) < nbx && 2 * by + (tid >> 3) < nby && s_r[0][rc] <= s_r[3][rc];
      const unsigned need = __ballot_sync(0xffffffffu, has && s_b[b] + s_b[16 + b] + s_b[32 + b] <= thr);
      if (tid < 2 && ((need >> (8 * tid)) & 0xffu)) aux.scan_units[atomicAdd(aux.nscan, 1)] = 2 * tile + tid;
    }
    __syncthreads();  // s_r and s_b are free for the next tile
  }
}

// The window of radius W: row r of a cell's window is (dy, dz), entry r * (2 W + 1) + dx + W in canonical order.
template <int DIM, int W> struct Window {
  static constexpr int SIDE = 2 * W + 1, ROWS = DIM == 3 ? SIDE * SIDE : SIDE;
  static constexpr int CELLS = SIDE * ROWS;
  __device__ static int dy(int r) { return r % SIDE - W; }
  __device__ static int dz(int r) { return DIM == 3 ? r / SIDE - W : 0; }
};
// The cell at a window offset of (x, y, z), periodic.
template <int DIM>
__device__ __forceinline__ long long window_cell(const KParams &P, int x, int y, int z, int dx, int dy, int dz) {
  return (long long)wrapn(x + dx, P.nx) +
         (long long)P.nx * (wrapn(y + dy, P.ny) + (long long)P.ny * (DIM == 3 ? wrapn(z + dz, P.nz) : 0));
}

// The partner of one cell (Eqs. 59-65), by a warp: candidate criteria Eqs. 59, 61, 62; the winner is the
// nearest accepted candidate, then the largest facing score, then the first in the window's canonical
// order, which the packed key |r|^2 - 31 bits of the score - 9 bits of the entry orders exactly; all
// ones: none. m: the cell's row of its class (pitch HY in z); list: room for the window's cells. The
// possible partners are listed first, so that every lane reads as many as the others.
template <int DIM, int W>
__device__ __forceinline__ unsigned long long pair_of(const KParams &P, const int32_t *__restrict__ phi,
                                                      const float4 *__restrict__ nrm, int x, int y, int z,
                                                      const float4 &me, const int32_t vx, int lane, const uint2 *m, int cx,
                                                      unsigned short *list) {
  using Win = Window<DIM, W>;
  int cand = 0;
#pragma unroll
  for (int k = 0; k < (Win::ROWS + 31) / 32; k++) {
    const int r = lane + 32 * k;
    unsigned b = 0;
    if (r < Win::ROWS) {
      const int dz = Win::dz(r), dy = Win::dy(r);
      b = (window_bits(m[(DIM == 3 ? dz * MaskBox<DIM>::HY : 0) + dy], cx) >> (kWin - W)) & ((1u << Win::SIDE) - 1u);
      if (dy == 0 && dz == 0) b &= ~(1u << W);  // the cell itself
    }
    // entries of the lanes before this one
    int at = __popc(b);
    const int own = at;
#pragma unroll
    for (int sh = 1; sh < 32; sh <<= 1) {
      const int o = __shfl_up_sync(0xffffffffu, at, sh);
      if (lane >= sh) at += o;
    }
    const int all = __shfl_sync(0xffffffffu, at, 31);
    at += cand - own;
    cand += all;
    while (b) {
      list[at++] = (unsigned short)(r * Win::SIDE + __ffs(b) - 1);
      b &= b - 1u;
    }
  }
  __syncwarp();
  const float n0 = me.x, n1 = me.y, n2 = me.z, qxc = q_gate_value(vx);
  const float sim = __fmul_rn(P.eta, fmaxf(qxc, P.eps_q));
  unsigned long long best = ~0ull;
  constexpr int AT = 4;  // read together
  for (int i0 = lane; i0 < cand; i0 += 32 * AT) {
    int e[AT];
    int32_t vy[AT];
    float4 o[AT];
#pragma unroll
    for (int j = 0; j < AT; j++) {
      const int i = i0 + 32 * j;
      e[j] = i < cand ? list[i] : -1;
      if (e[j] >= 0) {
        const int r = e[j] / Win::SIDE, dx = e[j] % Win::SIDE - W;
        const long long q = window_cell<DIM>(P, x, y, z, dx, Win::dy(r), Win::dz(r));
        vy[j] = phi[q];
        o[j] = __ldg(nrm + q);
      }
    }
#pragma unroll
    for (int j = 0; j < AT; j++) {
      if (e[j] < 0) continue;
      const float qy = q_gate_value(vy[j]);
      if (fabsf(__fsub_rn(qy, qxc)) <= sim) {
        const float dot = __fadd_rn(__fadd_rn(__fmul_rn(n0, o[j].x), __fmul_rn(n1, o[j].y)), __fmul_rn(n2, o[j].z));
        if (dot <= P.cos_opp) {
          const float ff = fmaxf(-dot, 0.0f);
          const int r = e[j] / Win::SIDE, dx = e[j] % Win::SIDE - W, dy = Win::dy(r), dz = Win::dz(r);
          const unsigned long long key = ((unsigned long long)(dx * dx + dy * dy + dz * dz) << 40) |
                                         ((unsigned long long)(0x7fffffffu - __float_as_uint(ff)) << 9) |
                                         (unsigned long long)e[j];
          best = key < best ? key : best;
        }
      }
    }
  }
  __syncwarp();  // the list is free for the warp's next cell
  if (__any_sync(0xffffffffu, best != ~0ull)) {
#pragma unroll
    for (int sh = 16; sh > 0; sh >>= 1) {
      const unsigned long long other = __shfl_xor_sync(0xffffffffu, best, sh);
      best = other < best ? other : best;
    }
  }
  return best;
}

// The force of a cell on its partner's key (Eqs. 66-73), and the partner where asked for.
template <int DIM, int W>
__device__ __forceinline__ void pair_force(const KParams &P, const int32_t *__restrict__ phi,
                                           const float4 *__restrict__ nrm, float4 *__restrict__ frep,
                                           int32_t *__restrict__ partner, int x, int y, int z, const float4 &me,
                                           const int32_t vx, const unsigned long long best) {
  using Win = Window<DIM, W>;
  const float n0 = me.x, n1 = me.y, n2 = me.z, qxc = q_gate_value(vx);
  const long long gidx = window_cell<DIM>(P, x, y, z, 0, 0, 0);
  const int bj = (int)(best & 511ull), od2 = (int)(best >> 40), r = bj / Win::SIDE;
  const int dx = bj % Win::SIDE - W, dy = Win::dy(r), dz = Win::dz(r);
  const float ff = __uint_as_float(0x7fffffffu - (unsigned)((best >> 9) & 0x7fffffffull));
  const long long gy = window_cell<DIM>(P, x, y, z, dx, dy, dz);
  const int32_t vy = phi[gy];
  const float4 o = __ldg(nrm + gy);
  const float m0 = o.x, m1 = o.y, m2 = o.z;
  const float qy = q_gate_value(vy);
  // paired indicator and clamp, Eqs. 66-67
  const float qpair = 0.5f * (qxc + qy);
  const float qcl = fminf(fmaxf(qpair, P.eps_q), 0.25f - P.eps_q);
  // proximity indicator, Eq. 70, as eps * artanh(sqrt(1 - 4 q)): the same value, and
  // 1 - 4 q_pair = ((1 - 2 phi_x)^2 + (1 - 2 phi_y)^2) / 2 has no cancellation
  float mm;
  if (qcl == qpair) {
    const float ax = 1.0f - 2.0f * fminf(fmaxf(phi_of(vx), 0.f), 1.f);
    const float ay = 1.0f - 2.0f * fminf(fmaxf(phi_of(vy), 0.f), 1.f);
    mm = 0.5f * (ax * ax + ay * ay);
  } else {
    mm = 1.0f - 4.0f * qcl;
  }
  const float h = P.eps * atanhf(sqrtf(mm));
  const float tt = h / P.h0;
  const float tp = (P.p == 4.0f) ? (tt * tt) * (tt * tt) : powf(tt, P.p);
  const float wh = 1.0f / (1.0f + tp);  // Eq. 71
  // symmetric normal, Eq. 69, line-of-centres fallback, oriented toward the partner
  const float rn = sqrtf((float)od2);
  const float r0 = dx / rn, r1 = dy / rn, r2 = dz / rn;
  float s0 = n0 - m0, s1 = n1 - m1, s2 = n2 - m2;
  const float sn = sqrtf(s0 * s0 + s1 * s1 + s2 * s2);
  if (sn < 1e-8f) {
    s0 = r0; s1 = r1; s2 = r2;
  } else {
    const float is = 1.0f / (sn + P.eps_n);
    s0 *= is; s1 *= is; s2 *= is;
  }
  if (r0 * s0 + r1 * s1 + r2 * s2 < 0.0f) {
    s0 = -s0; s1 = -s1; s2 = -s2;
  }
  // flux and force density with the facing factor of Eq. 68, Eqs. 72-73
  const float rho = P.rho_g + P.drho * phi_of(vx);
  const float amp = rho * P.A_rep * qcl * wh * ff;
  frep[gidx] = make_float4(amp * s0, amp * s1, DIM == 3 ? amp * s2 : 0.0f, 1.0f);
  if (partner) {
    partner[3 * gidx] = dx;
    partner[3 * gidx + 1] = dy;
    partner[3 * gidx + 2] = dz;
  }
}

// list: the units to scan (tile * UNITS + half), or with per_tile the tiles whose units to scan, and their
// count; nullptr: every unit, with zero force and no partner first written at every cell (the
// read-back). With bricks (3D) each unit is first tested against the ranges of the bricks around it,
// as in the prefilter. mark: the tiles listed for this phi (nullptr: all).
template <int DIM, int W>
__global__ void __launch_bounds__(NciGeom<DIM>::NT, 2)
k_nci_scan(const KParams P, const int32_t *__restrict__ phi, const float4 *__restrict__ nrm,
           float4 *__restrict__ frep, int32_t *__restrict__ partner, const int *__restrict__ list,
           const int *__restrict__ count, bool per_tile, int total, int gtx, int gty, const unsigned *__restrict__ masks,
           const uint4 *__restrict__ bricks, const int *__restrict__ mark, const int max_parts) {
  using G = NciGeom<DIM>;
  using M = MaskBox<DIM>;
  constexpr int RX = 10, RY = 3, RZ = 3, NR = RX * RY * RZ;
  __shared__ M s_box;
  __shared__ float s_r[DIM == 3 ? 6 : 1][NR];
  __shared__ float s_b[24];
  __shared__ int s_list[G::NT];
  __shared__ float4 s_n[G::NT];  // normals of the listed cells
  __shared__ int32_t s_v[G::NT];  // and their phi
  __shared__ unsigned long long s_best[G::NT];  // and their partners
  __shared__ unsigned short s_cand[G::NW][Window<DIM, W>::CELLS];
  __shared__ int s_count;
  const int tx = threadIdx.x, ty = threadIdx.y, tz = threadIdx.z;
  const int tid = tx + G::TX * (ty + G::TY * tz), lane = tid & 31, warp = tid >> 5;
  const int nx = P.nx, ny = P.ny, nz = P.nz;
  pdl_enter();
  const int per = per_tile ? G::UNITS : 1;
  const int n = list ? *count * per : total;
  // Where there are fewer units than blocks several blocks take the same one, each a share of its cells
  // by position (a film's 70 cells are then one round of the block's 16 warps instead of five: 48^3 35.2 ->
  // 34.0 us a step); the tests before that are repeated by each, in the time one of them takes. max_parts
  // is 1 where other cases use the SMs meanwhile (a batch: nine film cases 222 us with 8, 211 with 1).
  int parts = 1;
  while (parts < max_parts && 2 * parts * n <= (int)gridDim.x) parts *= 2;

  for (int item = blockIdx.x; item < n * parts; item += gridDim.x) {
    const int t = item / parts, part = item - t * parts;
    int u = list ? list[t / per] : t;
    if (per_tile) u = u * G::UNITS + t % G::UNITS;
    const int half = u % G::UNITS;
    int bx, by, bz;
    tile_of<DIM>(u / G::UNITS, gtx, gty, bx, by, bz);
    if constexpr (DIM == 3) {
      if (bricks) {
        if (tid < NR) {
          const int rx = tid % RX, ry = (tid / RX) % RY, rz = tid / (RX * RY);
          const NrmRange r =
              brick_range<false>(P, bricks, mark, gtx, gty, 8 * bx - 1 + rx, 2 * by + half - 1 + ry, bz - 1 + rz);
#pragma unroll
          for (int c = 0; c < 6; c++) s_r[c][tid] = r.v[c];
        }
        __syncthreads();
        const int rc = ((tid & 7) + 1) + RX * (1 + RY);
        if (tid < 24) s_b[tid] = brick_bound<RX, RY, NR>(s_r, tid >> 3, rc);
        __syncthreads();
        const bool has = tid < 8 && 32 * bx + 4 * tid < nx && 8 * by + 4 * half < ny && s_r[0][rc] <= s_r[3][rc];
        const bool need = has && s_b[tid] + s_b[8 + tid] + s_b[16 + tid] <= P.cos_opp + 1e-5f;
        if (!__syncthreads_or(need)) continue;  // uniform over the block
      }
    }
    const int x0 = bx * G::TX, y0 = by * NciTile<DIM>::Y + half * G::TY, z0 = bz * G::TZ;
    const int x = x0 + tx, y = y0 + ty, z = z0 + tz;
    const bool inb = x < nx && y < ny && z < nz;
    const long long idx = inb ? (long long)x + (long long)nx * (y + (long long)ny * z) : 0;
    const int32_t v = phi[idx];
    const float4 nv = __ldg(nrm + idx);  // used where gated
    for (int i = tid; i < kClasses<DIM> * M::ROWS; i += G::NT) (&s_box.m[0][0])[i] = make_uint2(0u, 0u);
    if (tid == 0) s_count = 0;
    __syncthreads();
    stage_masks<DIM>(P, s_box, masks, mark, gtx, gty, x0, y0, z0, tid, G::NT);
    const bool gated = inb && q_gate_value(v) >= P.q_th;
    if (!list && inb && ((tx + ty + tz) & (parts - 1)) == part) {
      frep[idx] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (partner) partner[3 * idx] = partner[3 * idx + 1] = partner[3 * idx + 2] = INT32_MIN;
    }
    __syncthreads();
    {  // list the cells with a possible partner
      const bool scan = gated && ((tx + ty + tz) & (parts - 1)) == part && may_face<DIM, W>(s_box, nv, tx, ty, tz);
      const unsigned m = __ballot_sync(0xffffffffu, scan);
      int base = 0;
      if (lane == 0 && m) base = atomicAdd(&s_count, __popc(m));
      base = __shfl_sync(0xffffffffu, base, 0);
      if (scan) {
        const int k = base + __popc(m & ((1u << lane) - 1u));
        s_list[k] = tid;
        s_n[k] = nv;
        s_v[k] = v;
      }
    }
    __syncthreads();
    const int ncell = s_count;
    for (int k = warp; k < ncell; k += G::NW) {
      const int c = s_list[k];
      const int cx = c % G::TX, cy = (c / G::TX) % G::TY, cz = c / (G::TX * G::TY);
      const float4 me = s_n[k];
      const unsigned long long best =
          pair_of<DIM, W>(P, phi, nrm, x0 + cx, y0 + cy, z0 + cz, me, s_v[k], lane,
                          s_box.m[facing_class<DIM>(me)] + (DIM == 3 ? (cz + kWin) * M::HY : 0) + cy + kWin, cx, s_cand[warp]);
      if (lane == 0) s_best[k] = best;
    }
    __syncthreads();
    if (tid < ncell && s_best[tid] != ~0ull) {  // a thread per cell; without a partner the force stays zero
      const int c = s_list[tid];
      pair_force<DIM, W>(P, phi, nrm, frep, partner, x0 + c % G::TX, y0 + (c / G::TX) % G::TY, z0 + c / (G::TX * G::TY),
                         s_n[tid], s_v[tid], s_best[tid]);
    }
    __syncthreads();  // the next unit reuses the shared buffers
  }
}

template <int DIM>
static cudaError_t launch_nci_dim(const KParams &P, const int32_t *phi, float4 *nrm, float4 *frep, int32_t *partner,
                                  const TileList &list, int list_blocks, cudaStream_t s, const NciAux &aux,
                                  int *reset_other, int max_parts) {
  using G = NciGeom<DIM>;
  const int *tiles = list.tiles, *ntiles = list.count;
  const int gtx = (P.nx + NciTile<DIM>::X - 1) / NciTile<DIM>::X, gty = (P.ny + NciTile<DIM>::Y - 1) / NciTile<DIM>::Y,
            gtz = (P.nz + NciTile<DIM>::Z - 1) / NciTile<DIM>::Z;
  const int total = gtx * gty * gtz, units = G::UNITS * total;
  // grid-stride blocks walk the lists, at most 16 (normals, prefilter) or 2 (scan) per list block; a small
  // grid has fewer items than that
  const int most = 16 * list_blocks, scan_blocks = units < 2 * list_blocks ? units : 2 * list_blocks;
  const dim3 block(G::TX, G::TY, G::TZ);
  int *reset = tiles ? reset_other : nullptr;
  cudaError_t e;
  if constexpr (DIM == 2) {
    e = launch_pdl(k_nci_normals2, dim3(total < most ? total : most), block, 0, s, P, phi, nrm, frep, tiles, ntiles, total,
                   gtx, gty, aux.masks, reset);
  } else {
    NciAux a = aux;
    if (!tiles) a.bricks = nullptr;
    e = launch_pdl(k_nci_normals3, dim3(2 * total < most ? 2 * total : most), dim3(kNrmThreads), 0, s, P, phi, nrm, frep,
                   tiles, ntiles, total, gtx, gty, a, reset);
  }
  if (e != cudaSuccess) return e;
  const unsigned *masks = aux.masks;
  const float4 *normals = nrm;
  const uint4 *bricks = nullptr;
  const int *mark = tiles ? list.mark : nullptr, *items = tiles, *count = ntiles;
  bool per_tile = tiles != nullptr;
  if (tiles && nci_prefilter_applies(DIM, P)) {
    e = launch_pdl(k_nci_prefilter, dim3(total < most ? total : most), dim3(128), 0, s, P, aux, mark, tiles, ntiles, gtx,
                   gty);
    if (e != cudaSuccess) return e;
    items = aux.scan_units;
    count = aux.nscan;
    per_tile = false;
  } else if (tiles) {
    // Where a side is not a multiple of 4 an entry of the brick test reads several bricks, and the test is
    // made by the scan's own blocks: the pass has no prefilter kernel.
    bricks = aux.bricks;
  }
  const auto scan = P.w == 3 ? k_nci_scan<DIM, 3> : (P.w == 2 ? k_nci_scan<DIM, 2> : k_nci_scan<DIM, 1>);
  return launch_pdl(scan, dim3(scan_blocks), block, 0, s, P, phi, normals, frep, partner, items, count, per_tile, units,
                    gtx, gty, masks, bricks, mark, max_parts);
}

cudaError_t launch_nci(int dim, const KParams &P, const int32_t *phi, float4 *nrm, float4 *frep, int32_t *partner,
                       const TileList &list, int list_blocks, cudaStream_t s, const NciAux &aux, int *reset_other,
                       int max_parts) {
  return dim == 2 ? launch_nci_dim<2>(P, phi, nrm, frep, partner, list, list_blocks, s, aux, reset_other, max_parts)
                  : launch_nci_dim<3>(P, phi, nrm, frep, partner, list, list_blocks, s, aux, reset_other, max_parts);
}

bool nci_prefilter_applies(int dim, const KParams &P) {
  return dim == 3 && P.nx % 4 == 0 && P.ny % 4 == 0 && P.nz % 4 == 0;
}

size_t nci_brick_count(const KParams &P) {
  return (size_t)((P.nx + 3) / 4) * (size_t)((P.ny + 3) / 4) * (size_t)((P.nz + 3) / 4);
}

size_t nci_mask_bytes(const KParams &P) {
  return sizeof(unsigned) * kMaskWords * (size_t)((P.nx + 31) / 32) * (size_t)P.ny * (size_t)P.nz;
}

// SMs of the device: the near-contact kernels are launched with a number of blocks per SM.
int nci_list_blocks() {
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 0;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
  return sms;
}

}  // namespace lbm
