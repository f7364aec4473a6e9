// Rows of cells held by a warp, C per lane: loads, one-cell shifts, wall rules and collisions shared by
// the kernels that take several time steps in one pass (march.cu, tile.cu).
#pragma once

#include "lbm_device.cuh"
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

// The rules of one row for a warp whose lane holds the cells x0 .. x0 + C - 1.  XE: the warp's cells have
// an x side (or, with 16-bit storage, a frame group) within reach; YE: the rows a y side.  PRESS: the x
// sides may be pressure columns; without their rules the other lattices' side cells are faster (per step
// 64^2 1.34 -> 1.26 us, 400^2 2.89 -> 2.76, 2048^2 with a per-cell medium 36.0 -> 34.2).
template <int PREC, bool HET, bool THERMAL, int C, bool XE, bool YE, bool PRESS>
struct RowOps {
  using S = Store<PREC>;
  using E = typename S::T;
  using V = Cells<PREC, C>;
  static constexpr bool EDGE = XE || YE;
  static constexpr bool kPressure = PRESS && XE;

  const StepParams& P;
  int lane, x0;         // (unwrapped) column of the lane's first cell
  // XE only
  bool slow;            // (uniform) the warp's cells cross a periodic side
  bool left, right;     // the lane holds the first / last column, between walls
  bool any_left, any_right;  // (uniform) one of the warp's lanes does
  bool inlet, outlet;        // the lane holds a pressure column, x = 0 or nx - 1 (FP32 storage)
  bool frame;           // 16-bit storage: the lane's cells are a frame group of k_step, which takes the FP32 collision
  int cr;               // component of the last column
  float dot[3];         // e_i . u_w of the side wall of the lane's first / last column

  __device__ __forceinline__ explicit RowOps(const StepParams& p) : P(p) {}

  // cells: cells per warp; xs: column of the warp's first cell
  __device__ __forceinline__ void set_lane(int xs, bool wrap) {
    lane = threadIdx.x & 31;
    x0 = xs + lane * C;
    frame = false;
    if constexpr (XE) {
      const int nx = P.nx;
      slow = wrap && (xs < 0 || xs + 32 * C > nx);
      left = P.bc_x == BC_WALL && x0 == 0;
      right = P.bc_x == BC_WALL && x0 <= nx - 1 && x0 + C > nx - 1;
      any_left = P.bc_x == BC_WALL && xs <= 0;
      any_right = P.bc_x == BC_WALL && xs + 32 * C > nx - 1;
      inlet = kPressure && P.bc_x == BC_PRESSURE && x0 == 0;
      outlet = kPressure && P.bc_x == BC_PRESSURE && x0 <= nx - 1 && x0 + C > nx - 1;
      cr = (nx - 1) & (C - 1);
      frame = PREC != PREC_FP32 && frame_cells();
    }
  }

  // the side wall's velocity, after set_lane and once it may be read
  __device__ __forceinline__ void read_wall() {
    if constexpr (XE) {
      dot[0] = dot[1] = dot[2] = 0.0f;
      if (left || right) {
        const int w = left ? 0 : 1;
        dot[0] = left ? wall_dot(P, 0, w) : wall_dot(P, 2, w);
        dot[1] = left ? wall_dot(P, 4, w) : wall_dot(P, 5, w);
        dot[2] = left ? wall_dot(P, 7, w) : wall_dot(P, 6, w);
      }
    }
  }

  // the lane's cells (or their periodic images) belong to a group of four with the first or last column
  __device__ __forceinline__ bool frame_cells() const {
    const int last = (P.nx - 1) / 4 * 4, x = slow ? wrap_x(x0) : x0;
    return x < 4 || x + C > last;
  }

  __device__ __forceinline__ int wrap_x(int x) const { return x < 0 ? x + P.nx : (x >= P.nx ? x - P.nx : x); }
  __device__ __forceinline__ int wrap_y(int y) const { return !YE ? y : y < 0 ? y + P.ny : (y >= P.ny ? y - P.ny : y); }
  __device__ __forceinline__ bool low(int y) const { return YE && P.bc_y == BC_WALL && y == 0; }
  __device__ __forceinline__ bool high(int y) const { return YE && P.bc_y == BC_WALL && y == P.ny - 1; }
  // a row of the lattice; n columns, from a multiple of n on, of a row with its padding (debug builds check)
  __device__ __forceinline__ int in_rows(int y) const { return dbg_check(P, y >= 0 && y < P.ny) ? y : 0; }
  __device__ __forceinline__ int in_cols(int x, int n) const {
    return dbg_check(P, x >= 0 && x + n <= P.pitch && (x & (n - 1)) == 0) ? x : 0;
  }
  // column of the lane's cell c in memory; where the cell is never part of a stored result, some column
  // that keeps the alignment of the lane's first cell
  __device__ __forceinline__ int col(int c) const {
    if constexpr (!XE) return x0 + c;
    const int x = slow ? wrap_x(x0 + c) : x0 + c;
    return x < P.nx ? x : c;
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
    if constexpr (XE) {  // (selects rather than branches: only one lane holds the side column)
      const float inv = P.inv_scale;
      if (any_left && c == 0) {
        const float v0 = bounce<PREC>(P, true_value<PREC>(e[0], inv), 0, dot[0]);
        const float v4 = bounce<PREC>(P, true_value<PREC>(e[1], inv), 4, dot[1]), v7 = bounce<PREC>(P, true_value<PREC>(e[2], inv), 7, dot[2]);
        d[0] = left ? v0 : d[0];
        d[4] = left && !lo ? v4 : d[4];
        d[7] = left && !hi ? v7 : d[7];
        if constexpr (THERMAL) {
          const float t = heat_bounce<PREC>(P, true_value<PREC>(eg, inv), 0);
          g[1] = left ? t : g[1];
        }
      }
      if (any_right) {
        const bool at = right && c == cr;
        const float v2 = bounce<PREC>(P, true_value<PREC>(e[0], inv), 2, dot[0]);
        const float v5 = bounce<PREC>(P, true_value<PREC>(e[1], inv), 5, dot[1]), v6 = bounce<PREC>(P, true_value<PREC>(e[2], inv), 6, dot[2]);
        d[2] = at ? v2 : d[2];
        d[5] = at && !lo ? v5 : d[5];
        d[6] = at && !hi ? v6 : d[6];
        if constexpr (THERMAL) {
          const float t = heat_bounce<PREC>(P, true_value<PREC>(eg, inv), 1);
          g[3] = at ? t : g[3];
        }
      }
    }
  }

  // The FP32 collision of the lane's cells of row y, in place, wall links first.
  __device__ __forceinline__ float collide_edge(int y, const float ph[], const float k[], const uint32_t e[3], uint32_t eg, V w[8],
                                                V gw[5]) const {
    float check = 0.0f;
    // Pressure columns are extrapolated from the pulled state of their inner neighbour.  Where the last
    // column is the first cell of a pair, that neighbour is in the pair or the lane before.
    float inner[8], inner_ph = 0.0f, inner_k = 0.0f;
    if constexpr (kPressure) {
      if (P.bc_x == BC_PRESSURE && (cr & 1) == 0) {
        float unused[5];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const float before = __shfl_up_sync(kFull, get_cell<PREC, C>(w[i], C - 1, 1.0f), 1);
          inner[i] = C == 4 && cr == 2 ? get_cell<PREC, C>(w[i], 1, 1.0f) : before;
        }
        if constexpr (HET) {
          inner_ph = __shfl_up_sync(kFull, ph[C - 1], 1);
          inner_k = __shfl_up_sync(kFull, k[C - 1], 1);
          if (C == 4 && cr == 2) {
            inner_ph = ph[1];
            inner_k = k[1];
          }
        }
        patch_cell(-1, y, e, eg, inner, unused);
      }
    }
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
      Coef ma, mb;
      if constexpr (HET) {
        const float* sv = P.sv ? P.sv + (int64_t)in_rows(y) * P.pitch : nullptr;
        ma = coef_of(P, ph[ca], k[ca], sv ? __ldg(sv + in_cols(col(ca), 1)) : P.s_v);
        mb = coef_of(P, ph[cb], k[cb], sv ? __ldg(sv + in_cols(col(cb), 1)) : P.s_v);
      } else {
        ma = mb = coef_uniform(P);
      }
      if constexpr (kPressure) {
        if (inlet && h == 0) pressure_cell(P, db, mb, ma, P.p_in, da);
        if (outlet && cr == ca) pressure_cell(P, inner, HET ? coef_of(P, inner_ph, inner_k, P.s_v) : ma, ma, P.p_out, da);
        if (outlet && cr == cb) pressure_cell(P, da, ma, mb, P.p_out, db);
      }
      const PairMedium m = pair_medium(ma, mb);
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
    const float* sv = P.sv + (int64_t)in_rows(y) * P.pitch;
    return make_float2(__ldg(sv + in_cols(col(a), 1)), __ldg(sv + in_cols(col(a + 1), 1)));
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

};

}  // namespace lbm
