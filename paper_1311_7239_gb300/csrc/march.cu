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
// Measured (GLUPS, one step per pass -> two): FP32 4096^2 104 -> 178, per-cell medium 90 -> 147,
// temperature (2048^2) 59 -> 95.  Every cell is rounded as by k_step: the results are the same bits.
#include "lbm_device.cuh"
#include "lbm_internal.h"
#include "tiles.cuh"

namespace lbm {

// C consecutive cells of one population as stored: floats, or 32-bit words of two 16-bit values.
template <int PREC, int C>
struct Cells {
  static_assert(C == 2 || C == 4, "cells per lane");
  static constexpr int N = PREC == PREC_FP32 ? C : C / 2;
  uint32_t v[N];
};

template <int PREC, int C>
__device__ __forceinline__ Cells<PREC, C> load_cells(const typename Store<PREC>::T* __restrict__ p) {
  Cells<PREC, C> r;
  if constexpr (Cells<PREC, C>::N == 4) {
    const uint4 q = *reinterpret_cast<const uint4*>(p);
    r.v[0] = q.x; r.v[1] = q.y; r.v[2] = q.z; r.v[3] = q.w;
  } else if constexpr (Cells<PREC, C>::N == 2) {
    const uint2 q = *reinterpret_cast<const uint2*>(p);
    r.v[0] = q.x; r.v[1] = q.y;
  } else {
    r.v[0] = *reinterpret_cast<const uint32_t*>(p);
  }
  return r;
}

template <int PREC, int C>
__device__ __forceinline__ void store_cells(typename Store<PREC>::T* __restrict__ p, const Cells<PREC, C>& r) {
  if constexpr (Cells<PREC, C>::N == 4) *reinterpret_cast<uint4*>(p) = make_uint4(r.v[0], r.v[1], r.v[2], r.v[3]);
  else if constexpr (Cells<PREC, C>::N == 2) *reinterpret_cast<uint2*>(p) = make_uint2(r.v[0], r.v[1]);
  else *reinterpret_cast<uint32_t*>(p) = r.v[0];
}

// cell c in true units
template <int PREC, int C>
__device__ __forceinline__ float get_cell(const Cells<PREC, C>& r, int c, float inv) {
  if constexpr (PREC == PREC_FP32) {
    return __uint_as_float(r.v[c]);
  } else {
    const float2 p = Store<PREC>::w2f(r.v[c >> 1]);
    return ((c & 1) ? p.y : p.x) * inv;
  }
}

// bits of one stored value
template <int PREC>
__device__ __forceinline__ uint32_t raw_bits(const typename Store<PREC>::T* p) {
  if constexpr (PREC == PREC_FP32) return __float_as_uint(*p);
  else return Store<PREC>::bits(*p);
}

template <int PREC, int C>
__device__ __forceinline__ void put_bits(Cells<PREC, C>& r, int c, uint32_t b) {
  if constexpr (PREC == PREC_FP32) r.v[c] = b;
  else r.v[c >> 1] = (c & 1) ? __byte_perm(r.v[c >> 1], b, 0x5410) : __byte_perm(b, r.v[c >> 1], 0x7610);
}

template <int PREC, int C>
__device__ __forceinline__ void put_cell(Cells<PREC, C>& r, int c, float v, float sc) {
  if constexpr (PREC == PREC_FP32) {
    r.v[c] = __float_as_uint(v);
  } else {
    const typename Store<PREC>::T e = Store<PREC>::enc(v, sc);
    put_bits<PREC, C>(r, c, Store<PREC>::bits(e));
  }
}

// bits of cell c
template <int PREC, int C>
__device__ __forceinline__ uint32_t cell_bits(const Cells<PREC, C>& r, int c) {
  if constexpr (PREC == PREC_FP32) return r.v[c];
  else return (c & 1) ? r.v[c >> 1] >> 16 : r.v[c >> 1] & 0xffffu;
}

// one stored value in true units
template <int PREC>
__device__ __forceinline__ float true_value(uint32_t bits, float inv) {
  if constexpr (PREC == PREC_FP32) return __uint_as_float(bits);
  else return Store<PREC>::w2f(bits).x * inv;
}

// the cells x - SH of the row whose cells x a warp holds (the first / last lane's outer cell repeats its own)
template <int PREC, int C, int SH>
__device__ __forceinline__ Cells<PREC, C> shift_cells(const Cells<PREC, C>& r) {
  constexpr int N = Cells<PREC, C>::N;
  Cells<PREC, C> o;
  if constexpr (SH == 0) {
    o = r;
  } else if constexpr (SH == 1) {
    const uint32_t l = __shfl_up_sync(kFull, r.v[N - 1], 1);
#pragma unroll
    for (int k = N - 1; k >= 0; --k) {
      const uint32_t below = k ? r.v[k - 1] : l;
      o.v[k] = PREC == PREC_FP32 ? below : __byte_perm(below, r.v[k], 0x5432);
    }
  } else {
    const uint32_t g = __shfl_down_sync(kFull, r.v[0], 1);
#pragma unroll
    for (int k = 0; k < N; ++k) {
      const uint32_t above = k < N - 1 ? r.v[k + 1] : g;
      o.v[k] = PREC == PREC_FP32 ? above : __byte_perm(r.v[k], above, 0x5432);
    }
  }
  return o;
}

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

__device__ __forceinline__ void copy_async16(void* smem, const void* gmem) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(smem)), "l"(gmem) : "memory");
}
__device__ __forceinline__ void copy_async8(void* smem, const void* gmem) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((uint32_t)__cvta_generic_to_shared(smem)), "l"(gmem) : "memory");
}
__device__ __forceinline__ void copy_async4(void* smem, const void* gmem) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((uint32_t)__cvta_generic_to_shared(smem)), "l"(gmem) : "memory");
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void copy_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// One warp's march over the rows [ya, yb) of a strip.  XE: the strip has an x side (or, with 16-bit
// storage, a frame group) within reach; YE: the rows have a y side within reach.
template <int PREC, bool HET, bool THERMAL, int C, int STAGES, bool XE, bool YE>
struct Marcher {
  using S = Store<PREC>;
  using E = typename S::T;
  using V = Cells<PREC, C>;
  static constexpr bool EDGE = XE || YE;
  static constexpr int kPlanes = THERMAL ? 13 : 8;
  static constexpr int kRow = 32 * C * (int)sizeof(E);      // bytes of a plane's row
  static constexpr int kMed = 32 * C * (int)sizeof(float);  // bytes of a medium field's row
  static constexpr int kStage = kPlanes * kRow + (HET ? 2 * kMed : 0);
  static constexpr int kChunks = kRow / 16, kMedChunks = kMed / 16;
  static constexpr int kCopies = (kPlanes * kChunks + 31) / 32;

  const StepParams& P;
  char* buf;     // the warp's STAGES stages in shared memory
  int lane, xs;  // xs: column of the warp's first cell
  int x0;        // (unwrapped) column of the lane's first cell
  bool out;      // the lane stores its cells
  // XE only
  bool slow;            // (uniform) the strip crosses a periodic side
  bool left, right;     // the lane holds the first / last column, between walls
  bool frame;           // 16-bit storage: the lane's cells are a frame group of k_step, which takes the FP32 collision
  int cr;               // component of the last column
  float dot[3];         // e_i . u_w of the side wall of the lane's first / last column
  uint32_t at[kCopies]; // (EDGE: unused)
  uint32_t e[3], eg;    // own populations of that column that bounce back there, of the row loaded next

  __device__ __forceinline__ Marcher(const StepParams& p, char* b) : P(p), buf(b) {}

  __device__ __forceinline__ int wrap_x(int x) const { return x < 0 ? x + P.nx : (x >= P.nx ? x - P.nx : x); }
  __device__ __forceinline__ int wrap_y(int y) const { return !YE ? y : y < 0 ? y + P.ny : (y >= P.ny ? y - P.ny : y); }
  __device__ __forceinline__ bool low(int y) const { return YE && P.bc_y == BC_WALL && y == 0; }
  __device__ __forceinline__ bool high(int y) const { return YE && P.bc_y == BC_WALL && y == P.ny - 1; }
  // column of the lane's cell c in memory (clamped where the cell is never part of a stored result)
  __device__ __forceinline__ int col(int c) const {
    if constexpr (!XE) return x0 + c;
    const int x = slow ? wrap_x(x0 + c) : x0 + c;
    return x < P.nx ? x : P.nx - 1;
  }

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
    return static_cast<const E*>(heat ? P.gsrc : P.src) + (int64_t)i * P.plane + (int64_t)wrap_y(y + dy) * P.pitch;
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
          for (int c = 0; c < C; ++c) copy_async4(d + 4 * c, row + col(c));
        } else {
          copy_async8(d, row + col(0));  // (nx is a multiple of 4)
        }
      }
      if constexpr (HET) {
        char* d = st + kPlanes * kRow + lane * C * 4;
#pragma unroll
        for (int c = 0; c < C; ++c) {
          copy_async4(d + 4 * c, P.phi + (int64_t)y * P.pitch + col(c));
          copy_async4(d + kMed + 4 * c, P.K + (int64_t)y * P.pitch + col(c));
        }
      }
    } else if constexpr (EDGE) {
#pragma unroll
      for (int j = 0; j < (kPlanes * kChunks + 31) / 32; ++j) {
        const int q = j * 32 + lane, p = q / kChunks;
        if ((j + 1) * 32 <= kPlanes * kChunks || p < kPlanes) {
          const int x = min(xs + (q - p * kChunks) * (16 / (int)sizeof(E)), P.pitch - 16 / (int)sizeof(E));
          copy_async16(st + q * 16, source(p, y) + x);
        }
      }
      if constexpr (HET) {
#pragma unroll
        for (int j = 0; j < 2 * kMedChunks / 32; ++j) {
          const int q = j * 32 + lane, p = q / kMedChunks;
          const int x = min(xs + (q - p * kMedChunks) * 4, P.pitch - 4);
          copy_async16(st + kPlanes * kRow + q * 16, (p ? P.K : P.phi) + (int64_t)y * P.pitch + x);
        }
      }
    } else {
      // 16-byte units from the start of the flow or temperature planes in 32 bits (march_takes checks):
      // the lane's part `at` of each copy is kept, the row's part is the same for the warp
      const uint32_t row = (uint32_t)r * ((uint32_t)P.pitch * (uint32_t)sizeof(E) / 16);
      char* d = st + lane * 16;
#pragma unroll
      for (int j = 0; j < kCopies; ++j) {
        const char* base = static_cast<const char*>(32 * j >= 8 * kChunks ? P.gsrc : P.src);
        if ((j + 1) * 32 <= kPlanes * kChunks || lane < kPlanes * kChunks - j * 32) copy_async16(d + j * 512, base + (uint64_t)(at[j] + row) * 16);
      }
      if constexpr (HET) {
        const uint32_t mrow = (uint32_t)r * ((uint32_t)P.pitch / 4);
#pragma unroll
        for (int j = 0; j < 2 * kMedChunks / 32; ++j) {
          const int q = j * 32 + lane, p = q / kMedChunks;
          const uint32_t x = (uint32_t)(xs / 4 + q - p * kMedChunks) + mrow;
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
      const int y = wrap_y(r);
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

  // the one-cell x shifts of the pull into row y (none for populations that came back from a wall row)
  __device__ __forceinline__ void shift(int y, V f[8], V g[5]) const {
    f[0] = shift_cells<PREC, C, 1>(f[0]);
    f[2] = shift_cells<PREC, C, -1>(f[2]);
    if (!low(y)) {
      f[4] = shift_cells<PREC, C, 1>(f[4]);
      f[5] = shift_cells<PREC, C, -1>(f[5]);
    }
    if (!high(y)) {
      f[6] = shift_cells<PREC, C, -1>(f[6]);
      f[7] = shift_cells<PREC, C, 1>(f[7]);
    }
    if constexpr (THERMAL) {
      g[1] = shift_cells<PREC, C, 1>(g[1]);
      g[3] = shift_cells<PREC, C, -1>(g[3]);
    }
  }

  // One cell in true units with its wall links patched: d, g pulled (wall links: the own opposite population).
  __device__ __forceinline__ void patch_cell(int c, int y, const uint32_t e[3], uint32_t eg, float d[8], float g[5]) const {
    const bool lo = low(y), hi = high(y);
    if (lo) {
      d[1] = bounce<PREC>(P, d[1], 1, wall_dot(P, 1, 2));
      d[4] = bounce<PREC>(P, d[4], 4, wall_dot(P, 4, 2));
      d[5] = bounce<PREC>(P, d[5], 5, wall_dot(P, 5, 2));
      if constexpr (THERMAL) g[2] = heat_bounce<PREC>(P, g[2], 2);
    }
    if (hi) {
      d[3] = bounce<PREC>(P, d[3], 3, wall_dot(P, 3, 3));
      d[6] = bounce<PREC>(P, d[6], 6, wall_dot(P, 6, 3));
      d[7] = bounce<PREC>(P, d[7], 7, wall_dot(P, 7, 3));
      if constexpr (THERMAL) g[4] = heat_bounce<PREC>(P, g[4], 3);
    }
    if constexpr (XE) {
      const float inv = P.inv_scale;
      if (left && c == 0) {
        d[0] = bounce<PREC>(P, true_value<PREC>(e[0], inv), 0, dot[0]);
        if (!lo) d[4] = bounce<PREC>(P, true_value<PREC>(e[1], inv), 4, dot[1]);
        if (!hi) d[7] = bounce<PREC>(P, true_value<PREC>(e[2], inv), 7, dot[2]);
        if constexpr (THERMAL) g[1] = heat_bounce<PREC>(P, true_value<PREC>(eg, inv), 0);
      }
      if (right && c == cr) {
        d[2] = bounce<PREC>(P, true_value<PREC>(e[0], inv), 2, dot[0]);
        if (!lo) d[5] = bounce<PREC>(P, true_value<PREC>(e[1], inv), 5, dot[1]);
        if (!hi) d[6] = bounce<PREC>(P, true_value<PREC>(e[2], inv), 6, dot[2]);
        if constexpr (THERMAL) g[3] = heat_bounce<PREC>(P, true_value<PREC>(eg, inv), 1);
      }
    }
  }

  // The FP32 collision of the lane's cells of row y, in place, wall links first.
  __device__ __forceinline__ float collide_edge(int y, const float ph[], const float k[], const uint32_t e[3], uint32_t eg, V w[8],
                                                V gw[5]) const {
    float check = 0.0f;
#pragma unroll
      for (int h = 0; h < C / 2; ++h) {
        const int ca = 2 * h, cb = ca + 1;
        float da[8], db[8], ga[5], gb[5];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          da[i] = get_cell<PREC, C>(w[i], ca, P.inv_scale);
          db[i] = get_cell<PREC, C>(w[i], cb, P.inv_scale);
        }
        if constexpr (THERMAL) {
#pragma unroll
          for (int i = 0; i < 5; ++i) {
            ga[i] = get_cell<PREC, C>(gw[i], ca, P.inv_scale);
            gb[i] = get_cell<PREC, C>(gw[i], cb, P.inv_scale);
          }
        }
        patch_cell(ca, y, e, eg, da, ga);
        patch_cell(cb, y, e, eg, db, gb);
        PairMedium m;
        if constexpr (HET) {
          const float* sv = P.sv ? P.sv + (int64_t)y * P.pitch : nullptr;
          m = pair_medium(coef_of(P, ph[ca], k[ca], sv ? __ldg(sv + col(ca)) : P.s_v), coef_of(P, ph[cb], k[cb], sv ? __ldg(sv + col(cb)) : P.s_v));
        } else {
          m = pair_medium(coef_uniform(P), coef_uniform(P));
        }
        float2 d[8], g[5], n0, ay = f2(P.ay), ux, uy;
#pragma unroll
        for (int i = 0; i < 8; ++i) d[i] = make_float2(da[i], db[i]);
        if constexpr (THERMAL) {
#pragma unroll
          for (int i = 0; i < 5; ++i) g[i] = make_float2(ga[i], gb[i]);
          n0 = add2(add2(add2(add2(g[0], g[1]), g[2]), g[3]), g[4]);
          ay = fma2(f2(P.g_beta), n0, ay);  // a = g beta (T - T0) j
        }
        collide_d2q8_pair(d, m, P.ax, ay, P, ux, uy);
        check += (fabsf(ux.x) + fabsf(uy.x)) + (fabsf(ux.y) + fabsf(uy.y));
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          put_cell<PREC, C>(w[i], ca, d[i].x, P.scale);
          put_cell<PREC, C>(w[i], cb, d[i].y, P.scale);
        }
        if constexpr (THERMAL) {
          collide_d2q5_pair_fp32(g, n0, ux, uy, P);
#pragma unroll
          for (int i = 0; i < 5; ++i) {
            put_cell<PREC, C>(gw[i], ca, g[i].x, P.scale);
            put_cell<PREC, C>(gw[i], cb, g[i].y, P.scale);
          }
        }
      }
    return check;
  }

  // viscous rates of the lane's cells a, a + 1 of row y
  __device__ __forceinline__ float2 rates(int y, int a) const {
    const float* sv = P.sv + (int64_t)y * P.pitch;
    return make_float2(__ldg(sv + col(a)), __ldg(sv + col(a + 1)));
  }

  // Collision of the lane's cells of row y, in place; returns the sum of |u| over the cells.
  __device__ __forceinline__ float collide(int y, const float ph[], const float k[], V w[8], V gw[5]) const {
    float check = 0.0f;
    if constexpr (PREC == PREC_FP32) {
#pragma unroll
      for (int h = 0; h < C / 2; ++h) {
        const int a = 2 * h, b = a + 1;
        float2 d[8], ux, uy, ay = f2(P.ay);
#pragma unroll
        for (int i = 0; i < 8; ++i) d[i] = make_float2(__uint_as_float(w[i].v[a]), __uint_as_float(w[i].v[b]));
        PairMedium m;
        if constexpr (HET) {
          const float2 sv = P.sv ? rates(y, a) : f2(P.s_v);
          m = pair_medium(coef_of(P, ph[a], k[a], sv.x), coef_of(P, ph[b], k[b], sv.y));
        } else {
          m = pair_medium(coef_uniform(P), coef_uniform(P));
        }
        float2 g[5], n0;
        if constexpr (THERMAL) {
#pragma unroll
          for (int i = 0; i < 5; ++i) g[i] = make_float2(__uint_as_float(gw[i].v[a]), __uint_as_float(gw[i].v[b]));
          n0 = add2(add2(add2(add2(g[0], g[1]), g[2]), g[3]), g[4]);
          ay = fma2(f2(P.g_beta), n0, ay);  // a = g beta (T - T0) j
        }
        collide_d2q8_pair(d, m, P.ax, ay, P, ux, uy);
        check += (fabsf(ux.x) + fabsf(uy.x)) + (fabsf(ux.y) + fabsf(uy.y));
#pragma unroll
        for (int i = 0; i < 8; ++i) { w[i].v[a] = __float_as_uint(d[i].x); w[i].v[b] = __float_as_uint(d[i].y); }
        if constexpr (THERMAL) {
          collide_d2q5_pair_fp32(g, n0, ux, uy, P);
#pragma unroll
          for (int i = 0; i < 5; ++i) { gw[i].v[a] = __float_as_uint(g[i].x); gw[i].v[b] = __float_as_uint(g[i].y); }
        }
      }
    } else {
#pragma unroll
      for (int h = 0; h < C / 2; ++h) {
        float2 dp[8], ux, uy;
#pragma unroll
        for (int i = 0; i < 8; ++i) dp[i] = S::w2f(w[i].v[h]);
        if constexpr (HET) {
          float2 hx, hy;
          const float2 sv = P.sv ? rates(y, 2 * h) : f2(P.s_v);
          const PairCoef c = pair_coef_het(P, make_float2(ph[2 * h], ph[2 * h + 1]), make_float2(k[2 * h], k[2 * h + 1]), sv, hx, hy);
          collide_pair(dp, c, hx, hy, P.pc, ux, uy);
        } else if constexpr (THERMAL) {
          float2 gp[5];
#pragma unroll
          for (int i = 0; i < 5; ++i) gp[i] = S::w2f(gw[i].v[h]);
          const float2 sTd = add2(add2(add2(gp[0], gp[1]), add2(gp[2], gp[3])), gp[4]);  // s (T - T0)
          const float2 hy = mul2(f2(P.phi_u), fma2(f2(0.5f * P.g_beta * P.inv_scale), sTd, f2(P.pc.hay)));
          collide_pair(dp, pair_coef_uniform(P.pc), f2(P.pc.u_hx), hy, P.pc, ux, uy);
          collide_d2q5_pair(gp, ux, uy, P);
#pragma unroll
          for (int i = 0; i < 5; ++i) gw[i].v[h] = S::f2w(gp[i]);
        } else {
          collide_pair(dp, pair_coef_uniform(P.pc), f2(P.pc.u_hx), f2(P.pc.u_hy), P.pc, ux, uy);
        }
        check += (fabsf(ux.x) + fabsf(uy.x)) + (fabsf(ux.y) + fabsf(uy.y));
#pragma unroll
        for (int i = 0; i < 8; ++i) w[i].v[h] = S::f2w(dp[i]);
      }
    }
    return check;
  }

  __device__ __forceinline__ float collide_row(int y, const float ph[], const float k[], const uint32_t e[3], uint32_t eg, V w[8],
                                               V gw[5]) const {
    if constexpr (EDGE) {
      if (PREC == PREC_FP32 || frame || low(y) || high(y)) return collide_edge(y, ph, k, e, eg, w, gw);
    }
    return collide(y, ph, k, w, gw);
  }

  // bits of component cr
  __device__ __forceinline__ uint32_t pick(const V& v) const {
    uint32_t r = cell_bits<PREC, C>(v, 0);
#pragma unroll
    for (int c = 1; c < C; ++c) r = cr == c ? cell_bits<PREC, C>(v, c) : r;
    return r;
  }

  __device__ __forceinline__ void store(int y, V w[8], V gw[5]) const {
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
    lane = threadIdx.x & 31;
    xs = march_x0<PREC, C>(strip, M.wrap);
    x0 = xs + lane * C;
    const int halo = march_halo<PREC, C>(M.wrap);
    if constexpr (!XE) {
      out = lane >= halo && lane < 32 - halo;
    } else {
      const int nx = P.nx;
      const bool first = !M.wrap && strip == 0, last = !M.wrap && strip == M.strips - 1;
      out = (lane >= halo || first) && (lane < 32 - halo || last) && x0 < nx;
      slow = M.wrap && (xs < 0 || xs + 32 * C > nx);
      left = P.bc_x == BC_WALL && x0 == 0;
      right = P.bc_x == BC_WALL && x0 <= nx - 1 && x0 + C > nx - 1;
      cr = (nx - 1) & (C - 1);
      frame = PREC != PREC_FP32 && (x0 < 4 || x0 + C > (nx - 1) / 4 * 4);
      if (left || right) {
        const int w = left ? 0 : 1;
        dot[0] = left ? wall_dot(P, 0, w) : wall_dot(P, 2, w);
        dot[1] = left ? wall_dot(P, 4, w) : wall_dot(P, 5, w);
        dot[2] = left ? wall_dot(P, 7, w) : wall_dot(P, 6, w);
      }
    }
    if constexpr (EDGE && !XE) frame = false;
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

__device__ __forceinline__ void launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void wait_prerequisites() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// The warps at the sides: the bottom and top segments, then the strips with an x side in pieces of
// `rows` rows.  A kernel of its own, so that the rules at the sides cost the main one no registers;
// it lets the main kernel start at once (the two write different cells).
template <int PREC, bool HET, bool THERMAL, int C, int STAGES>
__global__ void __launch_bounds__(kMarchThreads) k_march_side(const __grid_constant__ StepParams P, const __grid_constant__ March M) {
  extern __shared__ __align__(16) char smem[];
  launch_dependents();
  constexpr int kBytes = STAGES * Marcher<PREC, HET, THERMAL, C, STAGES, false, false>::kStage;
  int item = (int)((blockIdx.x * kMarchThreads + threadIdx.x) >> 5);
  char* buf = smem + (threadIdx.x >> 5) * kBytes;
  const int ny = P.ny, sides = M.strips - (M.s1 - M.s0);
  if (item < 2 * M.strips) {
    const int top = item >= M.strips;
    Marcher<PREC, HET, THERMAL, C, STAGES, true, true> m(P, buf);
    m.run(M, top ? item - M.strips : item, top ? ny - kMarchSide : 0, top ? ny : kMarchSide);
    return;
  }
  item -= 2 * M.strips;
  if (item >= sides * M.side_segs) return;
  const int seg = item / sides;
  int strip = item - seg * sides;
  if (strip >= M.s0) strip += M.s1 - M.s0;
  const int ya = kMarchSide + seg * M.side_rows, yb = min(ya + M.side_rows, ny - kMarchSide);
  Marcher<PREC, HET, THERMAL, C, STAGES, true, false> m(P, buf);
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

// Which contexts take their steps in pairs.  Periodic and halfway-wall sides; with 16-bit storage and
// periodic x sides the halo must be whole groups of four cells (k_step's frame groups round
// differently).  Below the size of L2 (129 MB) single steps do not go to HBM and their many small
// warps win: 1024^2 FP32 8.6 us per step against 9.8 in pairs, 1536^2 24.6 against 17.0; with
// temperature 1024^2 (109 MB) 16.5 against 11.6.  16-bit storage is bound by the collisions rather
// than by HBM, and gains only where the state is several times L2.
bool march_takes(const StepParams& P, int prec, bool het, bool thermal) {
  const uint64_t bytes = 2 * (uint64_t)(thermal ? 13 : 8) * (uint64_t)P.nx * P.ny * (prec == PREC_FP32 ? 4 : 2);
  if (bytes < (prec == PREC_FP32 ? 100ull << 20 : 400ull << 20)) return false;
  if (prec != PREC_FP32 && (het || thermal)) return false;
  if (P.inplace || P.nx < 16 || P.ny < 16) return false;
  if (P.bc_x > BC_WALL || P.bc_y > BC_WALL) return false;
  if (P.bc_x == BC_PERIODIC && prec != PREC_FP32 && (P.nx & 3)) return false;
  if (het && thermal) return false;
  if (8 * (uint64_t)P.plane * (prec == PREC_FP32 ? 4 : 2) / 16 >= (1ull << 32)) return false;  // (fill's 32-bit offsets)
  return true;
}

static int sm_count() {
  int dev = 0, n = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n < 1) {
    cudaGetLastError();
    return 152;
  }
  return n;
}

template <int PREC, bool HET, bool THERMAL, int C, int STAGES, int CTAS>
static cudaError_t launch_march_t(const StepParams& P, cudaStream_t s) {
  March M;
  M.wrap = P.bc_x == BC_PERIODIC;
  M.strips = march_strips<PREC, C>(P.nx, M.wrap);
  // sides: short segments, whose warps are done before the main kernel's
  M.side_rows = 8;
  auto xs = [&](int k) { return march_x0<PREC, C>(k, M.wrap); };
  auto inner_strip = [&](int k) { return xs(k) >= 4 && xs(k) + 32 * C <= (P.nx - 1) / 4 * 4; };
  for (M.s0 = 0; M.s0 < M.strips && !inner_strip(M.s0);) ++M.s0;
  for (M.s1 = M.s0; M.s1 < M.strips && inner_strip(M.s1);) ++M.s1;
  // rows per segment: whole waves of resident warps, at most 24 rows (longer segments drift apart and
  // lose the halo columns from L2: 4096^2 FP32 93.5 us at 25 rows, 102 at 50), at least 12
  const int ny = P.ny - 2 * kMarchSide, strips = M.s1 - M.s0 > 0 ? M.s1 - M.s0 : 1;
  const int64_t resident = (int64_t)sm_count() * CTAS * (kMarchThreads / 32);
  M.rows = ny;
  for (int64_t wave = 1; M.rows > 24; ++wave) {
    const int64_t segs = wave * resident / strips;
    if (segs > 0) M.rows = (int)((ny + segs - 1) / segs);
  }
  if (M.rows < 12) M.rows = 12;
  M.segs = (ny + M.rows - 1) / M.rows;
  M.side_segs = (ny + M.side_rows - 1) / M.side_rows;
  const size_t bytes = (kMarchThreads / 32) * STAGES * Marcher<PREC, HET, THERMAL, C, STAGES, false, false>::kStage;
  auto side = k_march_side<PREC, HET, THERMAL, C, STAGES>;
  auto main = k_march<PREC, HET, THERMAL, C, STAGES, CTAS>;
  cudaError_t e = cudaFuncSetAttribute(side, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(main, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  if (e != cudaSuccess) return e;
  const int side_items = 2 * M.strips + (M.strips - (M.s1 - M.s0)) * M.side_segs;
  side<<<(side_items + 3) / 4, kMarchThreads, bytes, s>>>(P, M);
  const int items = (M.s1 - M.s0) * M.segs;
  if (items > 0) {
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t c = {};
    c.gridDim = dim3((items + 3) / 4);
    c.blockDim = dim3(kMarchThreads);
    c.dynamicSmemBytes = bytes;
    c.stream = s;
    c.attrs = &at;
    c.numAttrs = 1;
    e = cudaLaunchKernelEx(&c, main, P, M);
    if (e != cudaSuccess) return e;
  }
  return cudaGetLastError();
}

template <int PREC>
static cudaError_t launch_march_p(const StepParams& P, bool het, bool thermal, cudaStream_t s) {
  // cells per lane and CTAs per SM: the widest forms that hold their registers without a spill (any
  // spill costs more than a missing CTA: local memory shares the little L1 that the stages leave)
  if constexpr (PREC == PREC_FP32) {
    if (thermal) return launch_march_t<PREC, false, true, 2, 3, 4>(P, s);
    return het ? launch_march_t<PREC, true, false, 2, 3, 4>(P, s) : launch_march_t<PREC, false, false, 4, 3, 3>(P, s);
  } else {
    return launch_march_t<PREC, false, false, 4, 3, 3>(P, s);
  }
}

cudaError_t launch_march(const StepParams& P, int prec, bool het, bool thermal, cudaStream_t s) {
  switch (prec) {
    case PREC_FP32: return launch_march_p<PREC_FP32>(P, het, thermal, s);
    case PREC_FP16: return launch_march_p<PREC_FP16>(P, het, thermal, s);
    default: return launch_march_p<PREC_BF16>(P, het, thermal, s);
  }
}

}  // namespace lbm
