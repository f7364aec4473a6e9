// Several time steps of a small lattice in one launch (Liu & He, arXiv 1311.7239, Eqs. 6-20, and Eq. B.2
// for the temperature), in shared memory.
//
// A lattice that fits in L2 spends its steps on launches: 64^2 takes 3.9 us per step and 512^2 5.1,
// nearly all of it launch and memory latency.  Here a CTA loads a tile of 64 columns and up to `rows`
// rows with a halo of T cells, takes T steps on it in shared memory (two buffers, one barrier per
// step, each step on one cell less on every side that is not a side of the lattice) and stores the
// cells that are then still valid.  A warp owns a row: two cells per lane, the one-cell shifts are
// shuffles.  The halo is computed more than once, which costs nothing while the chip is not full.  What
// bounds it: the latency of a step (512^2 FP32: an instruction in 44 % of the active cycles, waits on the
// pipe and at the barrier) and, per launch, of the tile's loads and stores.
// The next launch starts early and waits for this one's results only (programmatic dependent launch).
#include "lbm_internal.h"
#include "rows.cuh"

namespace lbm {

constexpr int kTileCells = 64;  // columns of a tile: 32 lanes of two cells
constexpr int kTileWarps = 16;
constexpr int kTileSmem = 220 * 1024;

struct Tile {
  int strips;  // tiles of a row
  int halo;    // T of the geometry (even): columns and rows of halo
  int height;  // rows that a tile stores
  int wrap;    // x sides are periodic
  int steps;   // steps of this launch, at most halo
};

__host__ __device__ inline int tile_out(int halo) { return kTileCells - 2 * halo; }
__host__ __device__ inline int tile_strips(int nx, int halo, bool wrap) {
  const int out = tile_out(halo);
  if (wrap) return (nx + out - 1) / out;
  return nx <= kTileCells ? 1 : 1 + (nx - kTileCells + out - 1) / out;
}
__host__ __device__ inline int tile_x0(int strip, int halo, bool wrap) { return strip * tile_out(halo) - (wrap ? halo : 0); }

template <int PREC, bool HET, bool THERMAL, bool EDGE, bool PRESS>
struct TileRow : RowOps<PREC, HET, THERMAL, 2, EDGE, EDGE, PRESS> {
  using Ops = RowOps<PREC, HET, THERMAL, 2, EDGE, EDGE, PRESS>;
  using typename Ops::E;
  using typename Ops::V;
  using Ops::lane;
  using Ops::x0;
  static constexpr int kPlanes = THERMAL ? 13 : 8;
  static constexpr int kSpan = kTileCells * (int)sizeof(E);  // bytes of a plane's row
  static constexpr int kRow = kPlanes * kSpan;               // bytes of a row

  __device__ __forceinline__ explicit TileRow(const StepParams& p) : Ops(p) {}

  __device__ __forceinline__ V at(const char* row, int plane) const {
    return load_cells<PREC, 2>(reinterpret_cast<const E*>(row + plane * kSpan) + lane * 2);
  }

  // One step of row y (in memory), held at `row` between its neighbours; medium at med.
  __device__ __forceinline__ float step(const char* row, int y, const float* med, V w[8], V gw[5]) const {
    const char* down = row - kRow;
    const char* up = row + kRow;
    const bool lo = Ops::low(y), hi = Ops::high(y);
    w[0] = at(row, 0);
    w[2] = at(row, 2);
    w[1] = lo ? at(row, 3) : at(down, 1);
    w[4] = lo ? at(row, 6) : at(down, 4);
    w[5] = lo ? at(row, 7) : at(down, 5);
    w[3] = hi ? at(row, 1) : at(up, 3);
    w[6] = hi ? at(row, 4) : at(up, 6);
    w[7] = hi ? at(row, 5) : at(up, 7);
    if constexpr (THERMAL) {
      gw[0] = at(row, 8);
      gw[1] = at(row, 9);
      gw[3] = at(row, 11);
      gw[2] = lo ? at(row, 12) : at(down, 10);
      gw[4] = hi ? at(row, 10) : at(up, 12);
    }
    uint32_t own[3] = {0u, 0u, 0u}, og = 0u;
    if constexpr (EDGE) {
      if (Ops::any_left || Ops::any_right) {  // (every lane reads; the side column's lane uses it)
        const bool l = Ops::left;
        const V a = at(row, l ? 2 : 0), b = at(row, l ? 6 : 7), c = at(row, l ? 5 : 4);
        const int k = l ? 0 : Ops::cr;
        own[0] = k ? cell_bits<PREC, 2>(a, 1) : cell_bits<PREC, 2>(a, 0);
        own[1] = k ? cell_bits<PREC, 2>(b, 1) : cell_bits<PREC, 2>(b, 0);
        own[2] = k ? cell_bits<PREC, 2>(c, 1) : cell_bits<PREC, 2>(c, 0);
        if constexpr (THERMAL) {
          const V t = at(row, l ? 11 : 9);
          og = k ? cell_bits<PREC, 2>(t, 1) : cell_bits<PREC, 2>(t, 0);
        }
      }
    }
    float ph[2], k[2];
    if constexpr (HET) {
      const float2 a = *reinterpret_cast<const float2*>(med + lane * 2), b = *reinterpret_cast<const float2*>(med + kTileCells + lane * 2);
      ph[0] = a.x; ph[1] = a.y;
      k[0] = b.x; k[1] = b.y;
    }
    Ops::shift(y, w, gw);
    return Ops::collide_row(y, ph, k, own, og, w, gw);
  }
};

template <int PREC, bool HET, bool THERMAL, bool PRESS>
__global__ void __launch_bounds__(kTileWarps * 32, 1) k_tile(const __grid_constant__ StepParams P, const __grid_constant__ Tile M) {
  extern __shared__ __align__(16) char smem[];
  using Inner = TileRow<PREC, HET, THERMAL, false, false>;
  using Edge = TileRow<PREC, HET, THERMAL, true, PRESS>;
  using E = typename Inner::E;
  using V = typename Inner::V;
  launch_dependents();
  const int nx = P.nx, ny = P.ny, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int strip = blockIdx.x % M.strips, seg = blockIdx.x / M.strips;
  const bool walls = P.bc_y == BC_WALL;
  const int xs = tile_x0(strip, M.halo, M.wrap);
  const int ya = seg * M.height, yb = min(ya + M.height, ny);
  // rows held: [y0, y1), unwrapped
  const int y0 = walls ? max(ya - M.steps, 0) : ya - M.steps, y1 = walls ? min(yb + M.steps, ny) : yb + M.steps;
  const int rows = y1 - y0;
  // one spare row below and above (read by a wall row's unused neighbour only)
  char* const buf0 = smem + Inner::kRow;
  char* const buf1 = buf0 + (rows + 2) * Inner::kRow;
  float* const med = reinterpret_cast<float*>(buf1 + (rows + 1) * Inner::kRow);
  const bool edge = xs < 4 || xs + kTileCells > (nx - 1) / 4 * 4;
  Inner inner(P);
  Edge side(P);
  inner.set_lane(xs, M.wrap);
  side.set_lane(xs, M.wrap);
  wait_prerequisites();  // (nothing above reads memory)
  if (!dbg_check(P, ya < yb && M.steps >= 1 && M.steps <= M.halo) || !dbg_shared(P, smem, med + (HET ? rows * 2 * kTileCells : 0))) return;
  const int x0 = inner.x0;
  const bool first = !M.wrap && strip == 0, last = !M.wrap && strip == M.strips - 1;
  const bool out = (first || lane * 2 >= M.halo) && (last || lane * 2 < kTileCells - M.halo) && x0 < nx;
  auto memory_row = [&](int y) { return side.in_rows(y < 0 ? y + ny : (y >= ny ? y - ny : y)); };

  // the tile (columns past the lattice are clamped: never part of a stored result)
  if constexpr (HET) {
    for (int j = warp; j < rows; j += kTileWarps) {
      const int64_t o = (int64_t)memory_row(y0 + j) * P.pitch;
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        med[j * 2 * kTileCells + lane * 2 + c] = __ldg(P.phi + o + side.in_cols(side.col(c), 1));
        med[j * 2 * kTileCells + kTileCells + lane * 2 + c] = __ldg(P.K + o + side.in_cols(side.col(c), 1));
      }
    }
  }
  for (int j = warp; j < rows; j += kTileWarps) {
    const int64_t o = (int64_t)memory_row(y0 + j) * P.pitch;
    char* d = buf0 + j * Inner::kRow + lane * 2 * (int)sizeof(E);
    const int xl = min(x0, P.pitch - 2);
#pragma unroll
    for (int p = 0; p < Inner::kPlanes; ++p) {
      const E* row = (p >= 8 ? static_cast<const E*>(P.gsrc) + (p - 8) * P.plane : static_cast<const E*>(P.src) + p * P.plane) + o;
      if (!side.slow) {
        if constexpr (PREC == PREC_FP32) copy_async8(d + p * Inner::kSpan, row + side.in_cols(xl, 2));
        else copy_async4(d + p * Inner::kSpan, row + side.in_cols(xl, 2));
      } else if constexpr (PREC == PREC_FP32) {
        copy_async4(d + p * Inner::kSpan, row + side.in_cols(side.col(0), 1));
        copy_async4(d + p * Inner::kSpan + 4, row + side.in_cols(side.col(1), 1));
      } else {
        copy_async4(d + p * Inner::kSpan, row + side.in_cols(min(side.col(0), P.pitch - 2), 2));  // (nx is a multiple of 4)
      }
    }
  }
  copy_commit();
  side.read_wall();
  copy_wait<0>();
  __syncthreads();

  float check = 0.0f;
  for (int s = 1; s <= M.steps; ++s) {
    const char* in = (s & 1) ? buf0 : buf1;
    char* res = (s & 1) ? buf1 : buf0;
    const int reach = M.steps - s;
    const int lo = (walls ? max(ya - reach, 0) : ya - reach) - y0, hi = (walls ? min(yb + reach, ny) : yb + reach) - y0;
    for (int j = lo + warp; j < hi; j += kTileWarps) {
      if (!dbg_check(P, j >= 0 && j < rows)) continue;
      const int y = memory_row(y0 + j);
      V w[8], gw[5];
      const char* row = in + j * Inner::kRow;
      const float* m = med + j * 2 * kTileCells;
      float u;
      if (edge || (walls && (y == 0 || y == ny - 1))) u = side.step(row, y, m, w, gw);
      else u = inner.step(row, y, m, w, gw);
      if (y0 + j >= ya && y0 + j < yb) check += u;
      if (s < M.steps) {
        char* d = res + j * Inner::kRow + lane * 2 * (int)sizeof(E);
#pragma unroll
        for (int p = 0; p < 8; ++p) store_cells<PREC, 2>(reinterpret_cast<E*>(d + p * Inner::kSpan), w[p]);
        if constexpr (THERMAL) {
#pragma unroll
          for (int p = 0; p < 5; ++p) store_cells<PREC, 2>(reinterpret_cast<E*>(d + (8 + p) * Inner::kSpan), gw[p]);
        }
      } else if (out && dbg_check(P, x0 >= 0 && x0 + 2 <= P.pitch)) {
        if (x0 + 1 >= nx) {  // row padding holds zeros
#pragma unroll
          for (int p = 0; p < 8; ++p) put_bits<PREC, 2>(w[p], 1, 0u);
          if constexpr (THERMAL) {
#pragma unroll
            for (int p = 0; p < 5; ++p) put_bits<PREC, 2>(gw[p], 1, 0u);
          }
        }
        const int64_t o = (int64_t)y * P.pitch + x0;
#pragma unroll
        for (int p = 0; p < 8; ++p) store_cells<PREC, 2>(static_cast<E*>(P.dst) + p * P.plane + o, w[p]);
        if constexpr (THERMAL) {
#pragma unroll
          for (int p = 0; p < 5; ++p) store_cells<PREC, 2>(static_cast<E*>(P.gdst) + p * P.plane + o, gw[p]);
        }
      }
    }
    if (s < M.steps) __syncthreads();
  }
  if (out && !(check < 1e30f)) atomicOr(P.err, 1u);
}

static size_t tile_bytes(int prec, bool het, bool thermal, int rows) {
  const size_t row = (size_t)(thermal ? 13 : 8) * kTileCells * (prec == PREC_FP32 ? 4 : 2);
  return 2 * (size_t)(rows + 2) * row + (het ? (size_t)rows * 2 * kTileCells * 4 : 0);
}

// Steps per launch, and the tiles' height: one wave of CTAs, one per SM (more waves wait for each
// other's loads and were slower than single steps: 640^2 FP32 6.3 us per step against 5.9).  Four steps
// per launch: 64^2 FP32 takes 1.5 / 1.2 / 1.25 / 1.8 us per step with 2 / 4 / 8 / 16 (a launch costs
// about 0.6 us, a step in shared memory 1; beyond 4 the halo's rows cost more than the launches
// saved), 512^2 4.9 / 3.6 / 5.3.  False where the lattice is left to the other kernels: above one wave,
// and for the sides and widths that they treat differently (march_takes).
static bool tile_shape(const StepParams& P, int prec, bool het, bool thermal, Tile& M) {
  if (P.inplace || P.nx < 16 || P.ny < 16 || P.bc_x > BC_PRESSURE || P.bc_y > BC_WALL) return false;
  if (P.bc_x == BC_PRESSURE && (prec != PREC_FP32 || thermal)) return false;
  if (P.bc_x == BC_PERIODIC && prec != PREC_FP32 && (P.nx & 3)) return false;
  if (het && thermal) return false;
  M.wrap = P.bc_x == BC_PERIODIC;
  M.halo = 4;
  M.strips = tile_strips(P.nx, M.halo, M.wrap);
  int segs = sm_count() / M.strips;
  if (segs < 1) return false;
  if (segs > P.ny) segs = P.ny;
  M.height = (P.ny + segs - 1) / segs;
  // (16-bit storage, with its slower frame groups, falls behind single steps above 48 rows: 600^2 FP16
  // with a per-cell medium 8.4 us per step against 7.2, 512^2 6.2 against 6.7)
  const int rows = M.height + 2 * M.halo;
  return tile_bytes(prec, het, thermal, rows) <= (size_t)kTileSmem && (prec == PREC_FP32 || rows <= 48);
}

int tile_steps(const StepParams& P, int prec, bool het, bool thermal) {
  Tile M;
  return tile_shape(P, prec, het, thermal, M) ? M.halo : 0;
}

template <int PREC, bool HET, bool THERMAL>
static cudaError_t launch_tile_t(const StepParams& P, const Tile& M, int prec, cudaStream_t s) {
  const size_t bytes = tile_bytes(prec, HET, THERMAL, M.height + 2 * M.halo);
  auto fn = k_tile<PREC, HET, THERMAL, false>;
  if constexpr (PREC == PREC_FP32 && !THERMAL) {
    if (P.bc_x == BC_PRESSURE) fn = k_tile<PREC, HET, THERMAL, true>;
  }
  cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kTileSmem);
  if (e != cudaSuccess) return e;
  return launch_early(fn, dim3(M.strips * ((P.ny + M.height - 1) / M.height)), dim3(kTileWarps * 32), bytes, s, P, M);
}

template <int PREC>
static cudaError_t launch_tile_p(const StepParams& P, const Tile& M, bool het, bool thermal, cudaStream_t s) {
  if (thermal) return launch_tile_t<PREC, false, true>(P, M, PREC, s);
  return het ? launch_tile_t<PREC, true, false>(P, M, PREC, s) : launch_tile_t<PREC, false, false>(P, M, PREC, s);
}

cudaError_t launch_tile(const StepParams& P, int prec, bool het, bool thermal, int steps, cudaStream_t s) {
  Tile M;
  if (!tile_shape(P, prec, het, thermal, M) || steps < 1 || steps > M.halo) return cudaErrorInvalidValue;
  M.steps = steps;
  switch (prec) {
    case PREC_FP32: return launch_tile_p<PREC_FP32>(P, M, het, thermal, s);
    case PREC_FP16: return launch_tile_p<PREC_FP16>(P, M, het, thermal, s);
    default: return launch_tile_p<PREC_BF16>(P, M, het, thermal, s);
  }
}

}  // namespace lbm
