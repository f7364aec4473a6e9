// Two time steps of the fused stream-collide update (Liu & He, arXiv 1311.7239, Eqs. 6-20, and Eq. B.2
// for the temperature) in one pass over the populations.
//
// A single step reads and writes every population once and is bound by HBM (64 bytes per cell and
// step with FP32 storage; 98 % of the measured copy rate).  Two steps at once halve that: each warp
// marches up a strip of 32 C columns, takes the first step on row r and, from the rows it has just
// computed, the second step on row r - 1, so the state between the two never leaves the registers
// (of the last rows only the populations that the next row pulls are kept: 3 + 3 moving up, 2
// sideways).  One lane of halo on either side and one row above and below are computed twice (7 %
// and 2 of `rows` rows).  The rows of the first step arrive in shared memory two rows ahead
// (cp.async), which costs no registers and keeps enough bytes in flight at 12-16 warps per SM:
// 4096^2 FP32, interior alone, 183 GLUPS against 161 with the rows prefetched in registers.
// The collisions run on packed FP32 pairs (collide_d2q8_pair, collide_pair): with scalar ones the
// pass was bound by instruction issue (79 %, 195 thread instructions per cell and step).
// Measured (GLUPS, one step per pass -> two): FP32 4096^2 104 -> 183, per-cell medium 91 -> 151,
// temperature (2048^2) 59 -> 89, FP16 4096^2 176 -> 207.  What bounds it now: HBM at 32 bytes per cell and
// step (86 % of the measured copy rate), with 16-bit storage latency and issue (2048^2: an instruction in
// 56 % of the active cycles from 9 warps per SM, DRAM at a quarter of its rate).  Every cell is rounded as by k_step: the results are the same bits.
#include "lbm_internal.h"
#include "rows.cuh"

namespace lbm {

// Strips and segments of one lattice (see k_march).
struct March {
  int strips;   // strips of a row
  int s0, s1;   // strips [s0, s1) have no side within reach
  int wrap;     // x sides are periodic
  int segs, rows;            // segments of `rows` rows between the first and the last kMarchSide rows
  int side_segs, side_rows;  // the same for the strips with an x side
};

constexpr int kMarchThreads = 128;
constexpr int kMarchSide = 4;  // rows of the bottom and top segments, which have a y side within reach

// Lanes of halo on either side of a strip: one (C >= 2 cells, the reach of two steps), or with
// periodic x sides as many as keep every strip's first column on a 16-byte boundary.
template <int PREC, int C>
__host__ __device__ constexpr int march_halo(bool wrap) {
  return !wrap ? 1 : (PREC == PREC_FP32 ? 4 : 8) / C;
}
template <int PREC, int C>
__host__ __device__ constexpr int march_out(bool wrap) {
  return (32 - 2 * march_halo<PREC, C>(wrap)) * C;
}
template <int PREC, int C>
__host__ __device__ inline int march_strips(int nx, bool wrap) {
  const int out = march_out<PREC, C>(wrap);
  if (wrap) return (nx + out - 1) / out;
  return nx <= 32 * C ? 1 : 1 + (nx - 32 * C + out - 1) / out;
}
template <int PREC, int C>
__host__ __device__ inline int march_x0(int strip, bool wrap) {
  return strip * march_out<PREC, C>(wrap) - (wrap ? march_halo<PREC, C>(true) * C : 0);
}

// One warp's march over the rows [ya, yb) of a strip.  XE: the strip has an x side (or, with 16-bit
// storage, a frame group) within reach; YE: the rows have a y side within reach.
template <int PREC, bool HET, bool THERMAL, int C, int STAGES, bool XE, bool YE, bool PRESS = false>
struct Marcher : RowOps<PREC, HET, THERMAL, C, XE, YE, PRESS> {
  using Ops = RowOps<PREC, HET, THERMAL, C, XE, YE, PRESS>;
  using typename Ops::E;
  using typename Ops::V;
  using Ops::EDGE;
  using Ops::P;
  using Ops::lane;
  using Ops::x0;
  using Ops::slow;
  using Ops::left;
  using Ops::right;
  using Ops::wrap_y;
  using Ops::low;
  using Ops::high;
  using Ops::col;
  using Ops::in_rows;
  using Ops::in_cols;
  using Ops::shift;
  using Ops::collide_row;
  using Ops::pick;
  static constexpr int kPlanes = THERMAL ? 13 : 8;
  static constexpr int kRow = 32 * C * (int)sizeof(E);      // bytes of a plane's row
  static constexpr int kMed = 32 * C * (int)sizeof(float);  // bytes of a medium field's row
  static constexpr int kStage = kPlanes * kRow + (HET ? 2 * kMed : 0);
  static constexpr int kChunks = kRow / 16, kMedChunks = kMed / 16;
  static constexpr int kCopies = (kPlanes * kChunks + 31) / 32;

  char* buf;     // the warp's STAGES stages in shared memory
  int xs;        // column of the warp's first cell
  bool out;      // the lane stores its cells
  uint32_t at[kCopies]; // (EDGE: unused)
  uint32_t e[3], eg;    // XE: own populations of the lane's side column that bounce back there, of the row loaded next

  __device__ __forceinline__ Marcher(const StepParams& p, char* b) : Ops(p), buf(b) {}

  // Start of plane p's row that the pull into row y (in memory) reads.  At a wall row the populations
  // that come through the wall are the row's own opposite ones.
  __device__ __forceinline__ const E* source(int p, int y) const {
    const bool heat = THERMAL && p >= 8;
    int i = heat ? p - 8 : p;
    int dy;
    if (heat) dy = i == 2 ? -1 : (i == 4 ? 1 : 0);
    else dy = -ey_of(i);
    if constexpr (YE) {
      if ((dy < 0 && low(y)) || (dy > 0 && high(y))) {
        i = heat ? opp5(i) : opp_of(i);
        dy = 0;
      }
    }
    return static_cast<const E*>(heat ? P.gsrc : P.src) + (int64_t)i * P.plane + (int64_t)in_rows(wrap_y(y + dy)) * P.pitch;
  }

  // Starts the copies of the rows that the pull into row r reads into a stage.
  __device__ __forceinline__ void fill(char* st, int r) {
    const int y = wrap_y(r);
    if (XE && slow) {
#pragma unroll
      for (int p = 0; p < kPlanes; ++p) {
        const E* row = source(p, y);
        char* d = st + p * kRow + lane * C * (int)sizeof(E);
        if constexpr (PREC == PREC_FP32) {
#pragma unroll
          for (int c = 0; c < C; ++c) copy_async4(d + 4 * c, row + in_cols(col(c), 1));
        } else {
          copy_async8(d, row + in_cols(col(0), C));  // (nx is a multiple of 4)
        }
      }
      if constexpr (HET) {
        char* d = st + kPlanes * kRow + lane * C * 4;
#pragma unroll
        for (int c = 0; c < C; ++c) {
          copy_async4(d + 4 * c, P.phi + (int64_t)in_rows(y) * P.pitch + in_cols(col(c), 1));
          copy_async4(d + kMed + 4 * c, P.K + (int64_t)in_rows(y) * P.pitch + in_cols(col(c), 1));
        }
      }
    } else if constexpr (EDGE) {
#pragma unroll
      for (int j = 0; j < (kPlanes * kChunks + 31) / 32; ++j) {
        const int q = j * 32 + lane, p = q / kChunks;
        if ((j + 1) * 32 <= kPlanes * kChunks || p < kPlanes) {
          const int x = min(xs + (q - p * kChunks) * (16 / (int)sizeof(E)), P.pitch - 16 / (int)sizeof(E));
          copy_async16(st + q * 16, source(p, y) + in_cols(x, 16 / (int)sizeof(E)));
        }
      }
      if constexpr (HET) {
#pragma unroll
        for (int j = 0; j < 2 * kMedChunks / 32; ++j) {
          const int q = j * 32 + lane, p = q / kMedChunks;
          const int x = min(xs + (q - p * kMedChunks) * 4, P.pitch - 4);
          copy_async16(st + kPlanes * kRow + q * 16, (p ? P.K : P.phi) + (int64_t)in_rows(y) * P.pitch + in_cols(x, 4));
        }
      }
    } else if (dbg_check(P, r >= 1 && r < P.ny - 1 && xs >= 0 && xs + 32 * C <= P.pitch)) {
      // 16-byte units from the start of the flow or temperature planes in 32 bits (march_takes checks):
      // the lane's part `at` of each copy is kept, the row's part is the same for the warp
      const uint32_t row = (uint32_t)r * ((uint32_t)P.pitch * (uint32_t)sizeof(E) / 16);
      char* d = st + lane * 16;
#pragma unroll
      for (int j = 0; j < kCopies; ++j) {
        const char* base = static_cast<const char*>(32 * j >= 8 * kChunks ? P.gsrc : P.src);
        const uint32_t unit = at[j] + row;
        if (((j + 1) * 32 <= kPlanes * kChunks || lane < kPlanes * kChunks - j * 32) &&
            dbg_check(P, ((uint64_t)unit + 1) * 16 <= (32 * j >= 8 * kChunks ? 5 : 8) * (uint64_t)P.plane * sizeof(E)))
          copy_async16(d + j * 512, base + (uint64_t)unit * 16);
      }
      if constexpr (HET) {
        const uint32_t mrow = (uint32_t)r * ((uint32_t)P.pitch / 4);
#pragma unroll
        for (int j = 0; j < 2 * kMedChunks / 32; ++j) {
          const int q = j * 32 + lane, p = q / kMedChunks;
          const uint32_t x = (uint32_t)(xs / 4 + q - p * kMedChunks) + mrow;
          if (dbg_check(P, ((int64_t)x + 1) * 4 <= P.plane))
            copy_async16(st + kPlanes * kRow + q * 16, reinterpret_cast<const char*>(p ? P.K : P.phi) + (uint64_t)x * 16);
        }
      }
    }
  }

  // the lane's parts of the copies (see fill)
  __device__ __forceinline__ void set_copies() {
    if constexpr (!EDGE) {
#pragma unroll
      for (int j = 0; j < kCopies; ++j) {
        const int q = j * 32 + lane, p = min(q / kChunks, kPlanes - 1);
        const bool heat = THERMAL && p >= 8;
        const int i = heat ? p - 8 : p;
        const int dy = heat ? (i == 2 ? -1 : (i == 4 ? 1 : 0)) : -ey_of(i);
        at[j] = (uint32_t)(((int64_t)i * P.plane + (int64_t)dy * P.pitch + xs) * (int64_t)sizeof(E) / 16 + (q - p * kChunks));
      }
    }
  }

  // the side columns' own populations of row r (prefetched: plain loads, used one row later)
  __device__ __forceinline__ void fetch_own(int r) {
    if (XE && (left || right)) {
      const int y = in_rows(wrap_y(r));
      const E* own = static_cast<const E*>(P.src) + (int64_t)y * P.pitch + (left ? 0 : P.nx - 1);
      e[0] = raw_bits<PREC>(own + (left ? 2 : 0) * P.plane);
      e[1] = raw_bits<PREC>(own + (left ? 6 : 7) * P.plane);
      e[2] = raw_bits<PREC>(own + (left ? 5 : 4) * P.plane);
      if constexpr (THERMAL) {
        const E* og = static_cast<const E*>(P.gsrc) + (int64_t)y * P.pitch + (left ? 0 : P.nx - 1);
        eg = raw_bits<PREC>(og + (left ? 3 : 1) * P.plane);
      }
    }
  }

  __device__ __forceinline__ void store(int y, V w[8], V gw[5]) const {
    if (!dbg_check(P, y >= 0 && y < P.ny && x0 >= 0 && x0 + C <= P.pitch)) return;
    if (XE && x0 + C > P.nx) {  // row padding holds zeros
#pragma unroll
      for (int c = 0; c < C; ++c) {
        if (x0 + c >= P.nx) {
#pragma unroll
          for (int i = 0; i < 8; ++i) put_bits<PREC, C>(w[i], c, 0u);
          if constexpr (THERMAL) {
#pragma unroll
            for (int i = 0; i < 5; ++i) put_bits<PREC, C>(gw[i], c, 0u);
          }
        }
      }
    }
    // (offset of the lane's cells in vectors of C cells, formed anew for each row rather than kept as pointers)
    uint32_t o = (uint32_t)y * ((uint32_t)P.pitch / C) + (uint32_t)(x0 / C);
    asm volatile("" : "+r"(o));
    const uint64_t at_b = (uint64_t)o * (C * sizeof(E)), pb = (uint64_t)P.plane * sizeof(E);
    char* dst = static_cast<char*>(P.dst);
#pragma unroll
    for (int i = 0; i < 8; ++i) store_cells<PREC, C>(reinterpret_cast<E*>(dst + i * pb + at_b), w[i]);
    if constexpr (THERMAL) {
      char* gdst = static_cast<char*>(P.gdst);
#pragma unroll
      for (int i = 0; i < 5; ++i) store_cells<PREC, C>(reinterpret_cast<E*>(gdst + i * pb + at_b), gw[i]);
    }
  }

  __device__ __forceinline__ void run(const March& M, int strip, int ya, int yb) {
    if (!dbg_check(P, strip >= 0 && strip < M.strips && ya >= 0 && yb <= P.ny)) return;
    if (!dbg_shared(P, buf - (threadIdx.x >> 5) * (STAGES * kStage), buf + STAGES * kStage)) return;
    xs = march_x0<PREC, C>(strip, M.wrap);
    Ops::set_lane(xs, M.wrap);
    Ops::read_wall();
    const int halo = march_halo<PREC, C>(M.wrap);
    const bool first = XE && !M.wrap && strip == 0, last = XE && !M.wrap && strip == M.strips - 1;
    out = (lane >= halo || first) && (lane < 32 - halo || last) && (!XE || x0 < P.nx);
    const bool walls = YE && P.bc_y == BC_WALL;
    const int lo = walls && ya == 0 ? 0 : ya - 1, hi = walls && yb == P.ny ? yb : yb + 1;  // rows of the first step
    float check = 0.0f;
    // of the state after the first step: the upward populations of the last two rows and the sideways
    // ones of the last row; with walls, the downward diagonal of the last row's side column
    V up2[3], up1[3], z1[2], gup2, gup1, gz1[3];
    float ph1[HET ? C : 1], k1[HET ? C : 1];
    uint32_t keep = 0;
    set_copies();
#pragma unroll
    for (int j = 0; j < STAGES - 1; ++j) {
      if (lo + j < hi) fill(buf + j * kStage, lo + j);
      copy_commit();
    }
    fetch_own(lo);
    int slot = 0;
#pragma unroll 1
    for (int r = lo; r <= yb; ++r) {  // first step on row r, second on row r - 1
      V w[8], gw[5];
      float ph[HET ? C : 1], k[HET ? C : 1];
      if (!EDGE || r < hi) {
        const int ahead = slot == 0 ? STAGES - 1 : slot - 1;  // the stage that row r - 1 left
        if (r + STAGES - 1 < hi) fill(buf + ahead * kStage, r + STAGES - 1);
        copy_commit();
        copy_wait<STAGES - 1>();
        __syncwarp();
        const char* st = buf + slot * kStage;
#pragma unroll
        for (int i = 0; i < 8; ++i) w[i] = load_cells<PREC, C>(reinterpret_cast<const E*>(st + i * kRow) + lane * C);
        if constexpr (THERMAL) {
#pragma unroll
          for (int i = 0; i < 5; ++i) gw[i] = load_cells<PREC, C>(reinterpret_cast<const E*>(st + (8 + i) * kRow) + lane * C);
        }
        if constexpr (HET) {
          const float* m = reinterpret_cast<const float*>(st + kPlanes * kRow) + lane * C;
#pragma unroll
          for (int c = 0; c < C; ++c) {
            ph[c] = m[c];
            k[c] = m[32 * C + c];
          }
        }
        __syncwarp();
        slot = slot == STAGES - 1 ? 0 : slot + 1;
        const int y = wrap_y(r);
        uint32_t own[3] = {0u, 0u, 0u}, og = 0u;
        if constexpr (XE) {
          own[0] = e[0]; own[1] = e[1]; own[2] = e[2];
          og = eg;
          if (r + 1 < hi) fetch_own(r + 1);
        }
        shift(y, w, gw);
        const float s = collide_row(y, ph, k, own, og, w, gw);
        if (r >= ya && r < yb) check += s;
      }
      if (r > ya) {
        const int y = r - 1;
        V q[8], gq[5];
        const bool hiy = high(y);
        q[0] = z1[0]; q[2] = z1[1];
        q[1] = up2[0]; q[4] = up2[1]; q[5] = up2[2];
        q[3] = hiy ? up1[0] : w[3];
        q[6] = hiy ? up1[1] : w[6];
        q[7] = hiy ? up1[2] : w[7];
        if constexpr (THERMAL) {
          gq[0] = gz1[0]; gq[1] = gz1[1]; gq[2] = gup2; gq[3] = gz1[2];
          gq[4] = hiy ? gup1 : gw[4];
        }
        uint32_t own[3] = {0u, 0u, 0u}, og = 0u;
        if constexpr (XE) {
          if (left) {
            own[0] = cell_bits<PREC, C>(z1[1], 0);
            own[2] = cell_bits<PREC, C>(up1[2], 0);
            if constexpr (THERMAL) og = cell_bits<PREC, C>(gz1[2], 0);
          } else if (right) {
            own[0] = pick(z1[0]);
            own[2] = pick(up1[1]);
            if constexpr (THERMAL) og = pick(gz1[1]);
          }
          own[1] = keep;
        }
        shift(y, q, gq);
        check += collide_row(y, ph1, k1, own, og, q, gq);
        if (out) store(y, q, gq);
      }
      if (low(r)) {  // the wall sends the row's own downward populations back up
        up2[0] = w[3]; up2[1] = w[6]; up2[2] = w[7];
        if constexpr (THERMAL) gup2 = gw[4];
      } else {
#pragma unroll
        for (int j = 0; j < 3; ++j) up2[j] = up1[j];
        if constexpr (THERMAL) gup2 = gup1;
      }
      up1[0] = w[1]; up1[1] = w[4]; up1[2] = w[5];
      z1[0] = w[0]; z1[1] = w[2];
      if constexpr (THERMAL) { gup1 = gw[2]; gz1[0] = gw[0]; gz1[1] = gw[1]; gz1[2] = gw[3]; }
      if constexpr (HET) {
#pragma unroll
        for (int c = 0; c < C; ++c) { ph1[c] = ph[c]; k1[c] = k[c]; }
      }
      if constexpr (XE) {
        if (left) keep = cell_bits<PREC, C>(w[6], 0);
        else if (right) keep = pick(w[7]);
      }
    }
    if (out && !(check < 1e30f)) atomicOr(P.err, 1u);
  }
};

// The warps at the sides: the bottom and top segments, then the strips with an x side in pieces of
// `rows` rows.  A kernel of its own, so that the rules at the sides cost the main one no registers;
// it lets the main kernel start at once (the two write different cells).
template <int PREC, bool HET, bool THERMAL, int C, int STAGES, bool PRESS>
__global__ void __launch_bounds__(kMarchThreads) k_march_side(const __grid_constant__ StepParams P, const __grid_constant__ March M) {
  extern __shared__ __align__(16) char smem[];
  launch_dependents();
  constexpr int kBytes = STAGES * Marcher<PREC, HET, THERMAL, C, STAGES, false, false>::kStage;
  int item = (int)((blockIdx.x * kMarchThreads + threadIdx.x) >> 5);
  char* buf = smem + (threadIdx.x >> 5) * kBytes;
  const int ny = P.ny, sides = M.strips - (M.s1 - M.s0);
  if (item < 2 * M.strips) {
    const int top = item >= M.strips;
    Marcher<PREC, HET, THERMAL, C, STAGES, true, true, PRESS> m(P, buf);
    m.run(M, top ? item - M.strips : item, top ? ny - kMarchSide : 0, top ? ny : kMarchSide);
    return;
  }
  item -= 2 * M.strips;
  if (item >= sides * M.side_segs) return;
  const int seg = item / sides;
  int strip = item - seg * sides;
  if (strip >= M.s0) strip += M.s1 - M.s0;
  const int ya = kMarchSide + seg * M.side_rows, yb = min(ya + M.side_rows, ny - kMarchSide);
  Marcher<PREC, HET, THERMAL, C, STAGES, true, false, PRESS> m(P, buf);
  m.run(M, strip, ya, yb);
}

// The strips and rows that no side comes near.  Launched to run beside k_march_side; it ends only
// after that one has (the next kernel on the stream waits for this one alone).
template <int PREC, bool HET, bool THERMAL, int C, int STAGES, int CTAS>
__global__ void __launch_bounds__(kMarchThreads, CTAS) k_march(const __grid_constant__ StepParams P, const __grid_constant__ March M) {
  extern __shared__ __align__(16) char smem[];
  using Inner = Marcher<PREC, HET, THERMAL, C, STAGES, false, false>;
  const int item = (int)((blockIdx.x * kMarchThreads + threadIdx.x) >> 5), n = M.s1 - M.s0;
  const int seg = item / n;
  if (seg < M.segs) {
    const int ya = kMarchSide + seg * M.rows;
    Inner m(P, smem + (threadIdx.x >> 5) * (STAGES * Inner::kStage));
    m.run(M, M.s0 + item - seg * n, ya, min(ya + M.rows, P.ny - kMarchSide));
  }
  wait_prerequisites();
}

// Which contexts take their steps in pairs.  Periodic and halfway-wall sides, and with FP32 storage
// pressure columns; with 16-bit storage and
// periodic x sides the halo must be whole groups of four cells (k_step's frame groups round
// differently).  Below the size of L2 (129 MB) single steps do not go to HBM and their many small
// warps win: 1024^2 FP32 8.6 us per step against 9.8 in pairs, 1536^2 24.6 against 17.0; with
// temperature 1024^2 (109 MB) 16.5 against 11.6.  16-bit storage is bound by the collisions rather
// than by HBM: the uniform medium gains from the size of L2 on (2048^2 FP16 26.3 -> 24.0 us, 1536^2
// 13.4 -> 15.7), a per-cell medium or the temperature does not (4096^2 per-cell 111 -> 114, 2048^2
// temperature 40.8 -> 45.5).
bool march_takes(const StepParams& P, int prec, bool het, bool thermal) {
  const uint64_t bytes = 2 * (uint64_t)(thermal ? 13 : 8) * (uint64_t)P.nx * P.ny * (prec == PREC_FP32 ? 4 : 2);
  if (bytes < (prec == PREC_FP32 ? kMarchBytes : 120ull << 20)) return false;
  if (prec != PREC_FP32 && (het || thermal)) return false;
  return march_shape(P, prec, het, thermal);
}

// The sides and sizes that the pair kernels handle.
bool march_shape(const StepParams& P, int prec, bool het, bool thermal) {
  if (P.inplace || P.nx < 16 || P.ny < 16) return false;
  if (P.bc_x > BC_PRESSURE || P.bc_y > BC_WALL || (P.bc_x == BC_PRESSURE && (prec != PREC_FP32 || thermal))) return false;
  if (P.bc_x == BC_PERIODIC && prec != PREC_FP32 && (P.nx & 3)) return false;
  if (het && thermal) return false;
  return 8 * (uint64_t)P.plane * (prec == PREC_FP32 ? 4 : 2) / 16 < (1ull << 32);  // (fill's 32-bit offsets)
}

int sm_count() {
  int dev = 0, n = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n < 1) {
    cudaGetLastError();
    return 152;
  }
  return n;
}

// Strips and segments for CTAS resident CTAs per SM.
template <int PREC, int C, int CTAS>
static March march_of(const StepParams& P) {
  March M;
  M.wrap = P.bc_x == BC_PERIODIC;
  M.strips = march_strips<PREC, C>(P.nx, M.wrap);
  auto xs = [&](int k) { return march_x0<PREC, C>(k, M.wrap); };
  auto inner_strip = [&](int k) { return xs(k) >= 4 && xs(k) + 32 * C <= (P.nx - 1) / 4 * 4; };
  for (M.s0 = 0; M.s0 < M.strips && !inner_strip(M.s0);) ++M.s0;
  for (M.s1 = M.s0; M.s1 < M.strips && inner_strip(M.s1);) ++M.s1;
  // Rows per segment: whole waves of resident warps, at most 24 rows (longer segments drift apart and
  // lose the halo columns from L2: 4096^2 FP32 93.5 us at 25 rows, 102 at 50), at least 12.  The strips
  // at the sides, whose warps are slower, take short segments.
  const int ny = P.ny - 2 * kMarchSide, strips = M.s1 - M.s0 > 0 ? M.s1 - M.s0 : 1;
  const int64_t resident = (int64_t)sm_count() * CTAS * (kMarchThreads / 32);
  M.rows = ny;
  for (int64_t wave = 1; M.rows > 24; ++wave) {
    const int64_t segs = wave * resident / strips;
    if (segs > 0) M.rows = (int)((ny + segs - 1) / segs);
  }
  if (M.rows < 12) M.rows = 12;
  M.side_rows = 8;
  M.segs = (ny + M.rows - 1) / M.rows;
  M.side_segs = (ny + M.side_rows - 1) / M.side_rows;
  return M;
}

template <int PREC, bool HET, bool THERMAL, int C, int STAGES, int CTAS>
static cudaError_t launch_march_t(const StepParams& P, cudaStream_t s) {
  const March M = march_of<PREC, C, CTAS>(P);
  const size_t bytes = (kMarchThreads / 32) * STAGES * Marcher<PREC, HET, THERMAL, C, STAGES, false, false>::kStage;
  auto side = k_march_side<PREC, HET, THERMAL, C, STAGES, false>;
  if constexpr (PREC == PREC_FP32 && !THERMAL) {
    if (P.bc_x == BC_PRESSURE) side = k_march_side<PREC, HET, THERMAL, C, STAGES, true>;
  }
  auto main = k_march<PREC, HET, THERMAL, C, STAGES, CTAS>;
  cudaError_t e = cudaFuncSetAttribute(side, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(main, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  if (e != cudaSuccess) return e;
  const int side_items = 2 * M.strips + (M.strips - (M.s1 - M.s0)) * M.side_segs;
  side<<<(side_items + 3) / 4, kMarchThreads, bytes, s>>>(P, M);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  const int items = (M.s1 - M.s0) * M.segs;
  if (items > 0 && (e = launch_early(main, dim3((items + 3) / 4), dim3(kMarchThreads), bytes, s, P, M)) != cudaSuccess) return e;
  return cudaGetLastError();
}

// cells per lane and CTAs per SM: the widest forms that hold their registers without a spill (any
// spill costs more than a missing CTA: local memory shares the little L1 that the stages leave)
template <int PREC>
static cudaError_t launch_march_p(const StepParams& P, bool het, bool thermal, cudaStream_t s) {
  if constexpr (PREC == PREC_FP32) {
    if (thermal) return launch_march_t<PREC, false, true, 2, 3, 4>(P, s);
    return het ? launch_march_t<PREC, true, false, 2, 3, 4>(P, s) : launch_march_t<PREC, false, false, 4, 3, 3>(P, s);
  } else {
    return launch_march_t<PREC, false, false, 4, 3, 3>(P, s);
  }
}

// kernels of launch_march: the sides', and the main one where the lattice has strips without a side
int march_kernels(const StepParams& P, int prec, bool het, bool thermal) {
  const March M = prec == PREC_FP32 ? (het || thermal ? march_of<PREC_FP32, 2, 4>(P) : march_of<PREC_FP32, 4, 3>(P))
                                    : march_of<PREC_FP16, 4, 3>(P);
  return M.s1 > M.s0 ? 2 : 1;
}

cudaError_t launch_march(const StepParams& P, int prec, bool het, bool thermal, cudaStream_t s) {
  switch (prec) {
    case PREC_FP32: return launch_march_p<PREC_FP32>(P, het, thermal, s);
    case PREC_FP16: return launch_march_p<PREC_FP16>(P, het, thermal, s);
    default: return launch_march_p<PREC_BF16>(P, het, thermal, s);
  }
}

// --------------------------------------------------------------------------------------------
// Batched ensembles (FP32, per-cell media): the same pairs of steps for all lattices of a batch in one
// launch of each kernel (48 lattices of 64..1024 cells a side: 84 -> 104 GLUPS, 109 since the side warps of
// batches without pressure columns leave their rules out; segments of 24 rows, 8 at the sides: 32 and 16
// rows gave 106 against the 104, but 72 against 76 on lattices up to 512).  A CTA's four warps take four items of one lattice, whose parameters are
// staged in shared memory; the items of a lattice are padded to whole CTAs.
// --------------------------------------------------------------------------------------------
constexpr int kBatchC = 2, kBatchStages = 3;

template <bool SIDE, bool PRESS>
__global__ void __launch_bounds__(kMarchThreads, SIDE ? 1 : 4)
    k_march_batch(const StepParams* __restrict__ Pd, const MarchItem* __restrict__ items) {
  extern __shared__ __align__(16) char smem[];
  __shared__ StepParams sP;
  using Inner = Marcher<PREC_FP32, true, false, kBatchC, kBatchStages, false, false>;
  if (SIDE) launch_dependents();
  const MarchItem it = items[blockIdx.x * (kMarchThreads / 32) + (threadIdx.x >> 5)];
  static_assert(sizeof(StepParams) % 8 == 0, "parameters are copied as 8-byte words");
  const unsigned long long* from = reinterpret_cast<const unsigned long long*>(Pd + it.lattice);
  for (int i = threadIdx.x; i < (int)(sizeof(StepParams) / 8); i += kMarchThreads) reinterpret_cast<unsigned long long*>(&sP)[i] = from[i];
  __syncthreads();
  char* buf = smem + (threadIdx.x >> 5) * (kBatchStages * Inner::kStage);
  March M;
  M.strips = it.strips;
  M.wrap = it.wrap;
  if (it.ya < it.yb) {
    if constexpr (!SIDE) {
      Inner m(sP, buf);
      m.run(M, it.strip, it.ya, it.yb);
    } else if (it.ya == 0 || it.yb == sP.ny) {
      Marcher<PREC_FP32, true, false, kBatchC, kBatchStages, true, true, PRESS> m(sP, buf);
      m.run(M, it.strip, it.ya, it.yb);
    } else {
      Marcher<PREC_FP32, true, false, kBatchC, kBatchStages, true, false, PRESS> m(sP, buf);
      m.run(M, it.strip, it.ya, it.yb);
    }
  }
  if (!SIDE) wait_prerequisites();
}

// Items of one lattice, in whole CTAs (kMarchThreads / 32 items).
void march_items(const StepParams& P, int lattice, std::vector<MarchItem>& side, std::vector<MarchItem>& main) {
  const bool wrap = P.bc_x == BC_PERIODIC;
  const int strips = march_strips<PREC_FP32, kBatchC>(P.nx, wrap), ny = P.ny, rows = 24, side_rows = 8;
  auto pad = [&](std::vector<MarchItem>& v) {
    while (v.size() % (kMarchThreads / 32)) v.push_back(MarchItem{lattice, 0, 0, 0, strips, wrap});
  };
  for (int k = 0; k < strips; ++k) {
    const int x = march_x0<PREC_FP32, kBatchC>(k, wrap);
    const bool inner = x >= 4 && x + 32 * kBatchC <= (P.nx - 1) / 4 * 4;
    side.push_back(MarchItem{lattice, k, 0, kMarchSide, strips, wrap});
    side.push_back(MarchItem{lattice, k, ny - kMarchSide, ny, strips, wrap});
    const int step = inner ? rows : side_rows;
    for (int y = kMarchSide; y < ny - kMarchSide; y += step)
      (inner ? main : side).push_back(MarchItem{lattice, k, y, y + step < ny - kMarchSide ? y + step : ny - kMarchSide, strips, wrap});
  }
  pad(side);
  pad(main);
}

cudaError_t launch_march_batch(const StepParams* Pd, const MarchItem* side, int n_side, const MarchItem* main, int n_main, bool pressure,
                               cudaStream_t s) {
  const size_t bytes = (kMarchThreads / 32) * kBatchStages * Marcher<PREC_FP32, true, false, kBatchC, kBatchStages, false, false>::kStage;
  auto sides = pressure ? k_march_batch<true, true> : k_march_batch<true, false>;
  auto inner = k_march_batch<false, false>;
  cudaError_t e = cudaFuncSetAttribute(sides, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(inner, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  if (e != cudaSuccess) return e;
  sides<<<n_side / 4, kMarchThreads, bytes, s>>>(Pd, side);
  if ((e = cudaGetLastError()) != cudaSuccess || n_main == 0) return e;
  return launch_early(inner, dim3(n_main / 4), dim3(kMarchThreads), bytes, s, Pd, main);
}

}  // namespace lbm
