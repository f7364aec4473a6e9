// Device-side building blocks of the porous D2Q8 MRT-LB step (Liu & He, arXiv 1311.7239) and of
// the D2Q5 temperature step (its Appendix B), for sm_103a.
//
// Storage: structure-of-arrays planes [q][ny][pitch].  Every plane holds the deviation of a
// post-collision population from the rest equilibrium, d_i = f_i - f_rest,i with
// f_rest,i = 3 w_i p_rest (Eq. 22 at u = 0, phi p = p_rest) for the flow and T0 / 5 (Eq. B.6 at
// u = 0, T = T0) for the temperature; FP16/BF16 planes scale d by 2^k.  The collision below works
// in those deviation variables throughout, which keeps FP32 arithmetic (and FP16 storage) far
// from the cancellation of subtracting two O(1) populations.
//
// One time step per cell (pull form of Eq. 15 followed by Eq. 14):
//   gather d_i(x - e_i) (bounce-back/periodic/pressure rules at the edges)
//   m = M d (Eq. 10, expanded), v, u (Eqs. 18-19), phi p (Eq. 20), F (Eq. 3), S (Eq. 16),
//   m+ = m - Lambda (m - m_eq) + (I - Lambda/2) S (Eqs. 11-14), d+ = M^-1 m+ (Eq. 8, expanded).
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <stdint.h>

namespace lbm {

enum : int { PREC_FP32 = 0, PREC_FP16 = 1, PREC_BF16 = 2 };
enum : int { BC_PERIODIC = 0, BC_WALL = 1, BC_PRESSURE = 2, BC_NEE = 3 };

// Constants of the two-cell collision (collide_pair), derived on the host from the configuration.
// Moments there are taken of the stored (scaled) deviations s d, so every constant that turns a
// physical quantity into a moment increment carries the storage scale s (1 for FP32 and BF16).
struct PairConst {
  float inv_rho0s;             // 1 / (rho0 s)
  float nphip;                 // -(2/3) rho0 s                 (Eq. 20)
  float nse8, sq6, nsq12;      // -s_e / 8, s_q / 6, -s_q / 12   (Lambda times the diagonal of M^-1)
  float r3, r12;               // rho0 s / 3, rho0 s / 12        (rho0 F through M^-1)
  float hay;                   // a_y / 2
  float cq;                    // -s_v / 4
  // medium coefficients of the uniform medium (see PairCoef) and phi a / 2
  float u_inv_phi, u_l0, u_l0sq, u_l1, u_nclin, u_ncnl, u_c2, u_nR, u_cf7, u_cf8, u_hx, u_hy;
  // per-cell media (pair_coef_het): 0.1 (1 - s_e/2) rho0 s, rho0 s, a_x / 2
  float k_c2, k_rs, hax;
};

// Everything a step kernel needs, passed by value.
struct StepParams {
  const void* src;   // current post-collision planes (8)
  void* dst;         // next post-collision planes (8)
  const void* gsrc;  // temperature planes (5), thermal only
  void* gdst;
  const float* phi;  // per-cell porosity [ny][pitch], or nullptr for uniform
  const float* K;    // per-cell permeability [ny][pitch], or nullptr for uniform
  const float* sv;   // per-cell viscous rate s_v = 1/(1/2 + 3 J nu) [ny][pitch] (heterogeneous mode), or nullptr
  int nx, ny, pitch;
  int64_t plane;     // elements per plane = ny * pitch
  int bc_x, bc_y;
  int forch;
  int inplace;       // 1: one population buffer with in-place streaming (see ip_off), 0: A-B buffers
  int parity;        // in-place: parity of the next step (selects the slots it loads from)
  float rho0, inv_rho0, nu, s_e, s_q, s_v;
  float ax, ay;
  // uniform-medium coefficients
  float phi_u, inv_phi_u, c_lin_u, c_nl_u;
  const float* uw;    // wall velocities [4][2] in device memory: left, right, bottom, top
  float p_in, p_out;  // pressure columns
  float p_rest;       // phi p of the stored rest state
  float scale, inv_scale;  // storage scale 2^k (1 for FP32)
  // temperature
  float zeta1, zeta3, zeta4, inv_sigma, varpi, g_beta, T0;
  float Tw[4];
  int Tdir[4];        // 1 = wall temperature prescribed, 0 = adiabatic
  unsigned int* err;  // bit 0: non-finite velocity
  float* urec;        // in-place step: if set, the velocity of every cell's collision, dense [2][ny][nx]
  float* edge;        // in-place step with extrapolated sides: pre-collision states of the boundary nodes (see k_edge_ip)
  PairConst pc;
};

// Debug builds (-DLBM_DEBUG) check the index invariants of the kernels: a violation sets bit 2 of
// the error word, which the next synchronising call reports, and the access is skipped or clamped.
// Release builds compile the checks away.
__device__ __forceinline__ bool dbg_check(const StepParams& P, bool ok) {
#ifdef LBM_DEBUG
  if (!ok) atomicOr(P.err, 4u);
  return ok;
#else
  (void)P;
  (void)ok;
  return true;
#endif
}

// The same for shared memory: what ends at `end` lies within the CTA's dynamic shared memory, from smem on.
__device__ __forceinline__ bool dbg_shared(const StepParams& P, const char* smem, const void* end) {
#ifdef LBM_DEBUG
  uint32_t bytes;
  asm("mov.u32 %0, %%dynamic_smem_size;" : "=r"(bytes));
  return dbg_check(P, static_cast<const char*>(end) <= smem + bytes);
#else
  (void)P;
  (void)smem;
  (void)end;
  return true;
#endif
}

// Programmatic dependent launch: the kernels of a step sequence let the next one on the stream be
// launched while they still run, and touch memory only after the one before has ended, which hides
// the launch latency (launch_early on the host).
__device__ __forceinline__ void launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void wait_prerequisites() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// D2Q8 velocities of Eq. 7 and the weights w_i listed after Eq. 20 (w_1..4 = 1/9, w_5..8 = 1/36).
__device__ __forceinline__ int ex_of(int i) { return (i == 0 || i == 4 || i == 7) ? 1 : ((i == 2 || i == 5 || i == 6) ? -1 : 0); }
__device__ __forceinline__ int ey_of(int i) { return (i == 1 || i == 4 || i == 5) ? 1 : ((i == 3 || i == 6 || i == 7) ? -1 : 0); }
__device__ __forceinline__ int opp_of(int i) { return i < 4 ? (i + 2) & 3 : 4 + ((i - 4 + 2) & 3); }
__device__ __forceinline__ float w_of(int i) { return i < 4 ? (1.0f / 9.0f) : (1.0f / 36.0f); }

// ---------------------------------------------------------------------------------------------
// storage codecs
// ---------------------------------------------------------------------------------------------
template <int PREC> struct Store;
// dec/enc and load4/store4 convert between stored and true deviations (the FP16 scale); decr,
// load4r and store4r move the stored values unchanged.
template <> struct Store<PREC_FP32> {
  using T = float;
  __device__ static __forceinline__ float decr(T v) { return v; }
  __device__ static __forceinline__ void load4r(const T* p, float o[4]) { load4(p, o, 1.0f); }
  __device__ static __forceinline__ void store4r(T* p, const float o[4]) { store4(p, o, 1.0f); }
  __device__ static __forceinline__ void store2r(T* p, float2 v) { *reinterpret_cast<float2*>(p) = v; }
  __device__ static __forceinline__ void load2(const T* p, float o[2], float) {
    const float2 v = *reinterpret_cast<const float2*>(p);
    o[0] = v.x; o[1] = v.y;
  }
  __device__ static __forceinline__ float dec(T v, float) { return v; }
  __device__ static __forceinline__ T enc(float v, float) { return v; }
  __device__ static __forceinline__ void load4(const T* p, float o[4], float) {
    const float4 v = *reinterpret_cast<const float4*>(p);
    o[0] = v.x; o[1] = v.y; o[2] = v.z; o[3] = v.w;
  }
  __device__ static __forceinline__ void store4(T* p, const float o[4], float) {
    *reinterpret_cast<float4*>(p) = make_float4(o[0], o[1], o[2], o[3]);
  }
};
template <> struct Store<PREC_FP16> {
  using T = __half;
  __device__ static __forceinline__ float decr(T v) { return __half2float(v); }
  __device__ static __forceinline__ void load4r(const T* p, float o[4]) {
    const uint2 raw = *reinterpret_cast<const uint2*>(p);
    const float2 a = __half22float2(*reinterpret_cast<const __half2*>(&raw.x));
    const float2 b = __half22float2(*reinterpret_cast<const __half2*>(&raw.y));
    o[0] = a.x; o[1] = a.y; o[2] = b.x; o[3] = b.y;
  }
  __device__ static __forceinline__ void store4r(T* p, const float o[4]) {
    __half2 a = __floats2half2_rn(o[0], o[1]);
    __half2 b = __floats2half2_rn(o[2], o[3]);
    uint2 raw;
    raw.x = *reinterpret_cast<unsigned int*>(&a);
    raw.y = *reinterpret_cast<unsigned int*>(&b);
    *reinterpret_cast<uint2*>(p) = raw;
  }
  __device__ static __forceinline__ void store2r(T* p, float2 v) { *reinterpret_cast<__half2*>(p) = __float22half2_rn(v); }
  // a 32-bit word holding two stored values <-> the pair as float2 (no scale applied)
  __device__ static __forceinline__ float2 w2f(uint32_t w) { return __half22float2(*reinterpret_cast<const __half2*>(&w)); }
  __device__ static __forceinline__ uint32_t f2w(float2 v) {
    const __half2 h = __float22half2_rn(v);
    return *reinterpret_cast<const uint32_t*>(&h);
  }
  __device__ static __forceinline__ uint32_t bits(T v) { return *reinterpret_cast<const unsigned short*>(&v); }
  __device__ static __forceinline__ void load2(const T* p, float o[2], float inv) {
    const float2 a = __half22float2(*reinterpret_cast<const __half2*>(p));
    o[0] = a.x * inv; o[1] = a.y * inv;
  }
  __device__ static __forceinline__ float dec(T v, float inv) { return __half2float(v) * inv; }
  __device__ static __forceinline__ T enc(float v, float sc) { return __float2half_rn(v * sc); }
  __device__ static __forceinline__ void load4(const T* p, float o[4], float inv) {
    const uint2 raw = *reinterpret_cast<const uint2*>(p);
    const float2 a = __half22float2(*reinterpret_cast<const __half2*>(&raw.x));
    const float2 b = __half22float2(*reinterpret_cast<const __half2*>(&raw.y));
    o[0] = a.x * inv; o[1] = a.y * inv; o[2] = b.x * inv; o[3] = b.y * inv;
  }
  __device__ static __forceinline__ void store4(T* p, const float o[4], float sc) {
    __half2 a = __floats2half2_rn(o[0] * sc, o[1] * sc);
    __half2 b = __floats2half2_rn(o[2] * sc, o[3] * sc);
    uint2 raw;
    raw.x = *reinterpret_cast<unsigned int*>(&a);
    raw.y = *reinterpret_cast<unsigned int*>(&b);
    *reinterpret_cast<uint2*>(p) = raw;
  }
};
// BF16 keeps FP32's exponent range, so its deviations are stored unscaled (scale = 1).
template <> struct Store<PREC_BF16> {
  using T = __nv_bfloat16;
  __device__ static __forceinline__ float decr(T v) { return __bfloat162float(v); }
  __device__ static __forceinline__ void load4r(const T* p, float o[4]) { load4(p, o, 1.0f); }
  __device__ static __forceinline__ void store4r(T* p, const float o[4]) { store4(p, o, 1.0f); }
  __device__ static __forceinline__ void store2r(T* p, float2 v) { *reinterpret_cast<__nv_bfloat162*>(p) = __float22bfloat162_rn(v); }
  // a BF16 value is the high half of its FP32 value
  __device__ static __forceinline__ float2 w2f(uint32_t w) { return make_float2(__uint_as_float(w << 16), __uint_as_float(w & 0xffff0000u)); }
  __device__ static __forceinline__ uint32_t f2w(float2 v) {
    const __nv_bfloat162 h = __float22bfloat162_rn(v);
    return *reinterpret_cast<const uint32_t*>(&h);
  }
  __device__ static __forceinline__ uint32_t bits(T v) { return *reinterpret_cast<const unsigned short*>(&v); }
  __device__ static __forceinline__ void load2(const T* p, float o[2], float) {
    const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(p));
    o[0] = a.x; o[1] = a.y;
  }
  __device__ static __forceinline__ float dec(T v, float) { return __bfloat162float(v); }
  __device__ static __forceinline__ T enc(float v, float) { return __float2bfloat16_rn(v); }
  __device__ static __forceinline__ void load4(const T* p, float o[4], float) {
    const uint2 raw = *reinterpret_cast<const uint2*>(p);
    const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&raw.x));
    const float2 b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&raw.y));
    o[0] = a.x; o[1] = a.y; o[2] = b.x; o[3] = b.y;
  }
  __device__ static __forceinline__ void store4(T* p, const float o[4], float) {
    __nv_bfloat162 a = __floats2bfloat162_rn(o[0], o[1]);
    __nv_bfloat162 b = __floats2bfloat162_rn(o[2], o[3]);
    uint2 raw;
    raw.x = *reinterpret_cast<unsigned int*>(&a);
    raw.y = *reinterpret_cast<unsigned int*>(&b);
    *reinterpret_cast<uint2*>(p) = raw;
  }
};

// ---------------------------------------------------------------------------------------------
// medium coefficients of one cell
// ---------------------------------------------------------------------------------------------
struct Coef {
  float phi, inv_phi;
  float s_v;    // viscous relaxation rate s7 = s8 (Eq. 13, Eq. 21 with upsilon_e = J upsilon)
  float c_lin;  // phi nu / K          (linear Darcy drag of Eq. 3)
  float c_nl;   // phi F_phi / sqrt(K)  (Forchheimer drag of Eq. 3; = 1.75 / sqrt(150 phi K) by Eq. 4)
};

// Reciprocal and square root through the SFU approximations (a few ulp), which the FP32 error
// budget of the method tolerates; sqrt of 0 is 0.
__device__ __forceinline__ float fast_rcp(float x) { return __fdividef(1.0f, x); }
__device__ __forceinline__ float fast_sqrt(float x) { return x > 0.0f ? x * rsqrtf(x) : 0.0f; }

// The same for arguments known to be normal numbers (or inf, NaN): without the instructions that scale
// subnormal ones.
__device__ __forceinline__ float rcp_normal(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float rsqrt_normal(float x) {
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

__device__ __forceinline__ float f4_get(const float4& v, int c) { return c == 0 ? v.x : c == 1 ? v.y : c == 2 ? v.z : v.w; }

// Between the cells that a thread collides one after another: keeps the compiler from holding the
// parameters, or a second cell's intermediate results, in registers across cells, which made the kernels
// that are capped at 64 registers spill (bytes of spill stores: the in-place step that records u, FP32,
// 144-168 -> 0 and 4096^2 208 -> 184 us; the in-place batches 48-72 -> 24-28).
__device__ __forceinline__ void next_cell() { asm volatile("" ::: "memory"); }

// Coefficients of a cell with porosity ph, permeability k and viscous rate sv (Eqs. 3-4, 13).
__device__ __forceinline__ Coef coef_of(const StepParams& P, float ph, float k, float sv) {
  Coef c;
  c.phi = ph;
  c.inv_phi = fast_rcp(ph);
  c.c_lin = ph * P.nu * fast_rcp(k);
  c.c_nl = P.forch ? 1.75f * rsqrtf(150.0f * ph * k) : 0.0f;
  c.s_v = sv;
  return c;
}

__device__ __forceinline__ Coef coef_uniform(const StepParams& P) {
  Coef c;
  c.phi = P.phi_u; c.inv_phi = P.inv_phi_u; c.c_lin = P.c_lin_u; c.c_nl = P.c_nl_u; c.s_v = P.s_v;
  return c;
}

template <bool HET>
__device__ __forceinline__ Coef coef_at(const StepParams& P, int x, int y) {
  if (!HET) return coef_uniform(P);
  const int64_t o = (int64_t)y * P.pitch + x;
  return coef_of(P, __ldg(P.phi + o), __ldg(P.K + o), P.sv ? __ldg(P.sv + o) : P.s_v);
}

// ---------------------------------------------------------------------------------------------
// macroscopic velocity and pressure deviation of a pre-collision cell (Eqs. 17-20)
// ---------------------------------------------------------------------------------------------
struct Macro {
  float dm1;       // sum of deviations (first moment of M applied to d)
  float ux, uy;    // velocity, Eq. 18
  float phip_dev;  // phi p - p_rest, Eq. 20
};

// Eqs. 18-19; also returns |u| = |v| / (l0 + sqrt(l0^2 + l1 |v|)) for the Forchheimer drag.
__device__ __forceinline__ void velocity_from_j(float jx, float jy, const Coef& c, float ax, float ay,
                                                float inv_rho0, float& ux, float& uy, float& umag) {
  // v = sum e f / rho0 + phi a / 2 ; l0 = (1 + phi nu / (2K)) / 2 ; l1 = phi F_phi / (2 sqrt K)
  const float vx = jx * inv_rho0 + 0.5f * c.phi * ax;
  const float vy = jy * inv_rho0 + 0.5f * c.phi * ay;
  const float l0 = 0.5f + 0.25f * c.c_lin;
  const float l1 = 0.5f * c.c_nl;
  const float vmag = fast_sqrt(vx * vx + vy * vy);
  // Eq. 18, the cancellation-free root of l1 |u|^2 + 2 l0 |u| - |v| = 0
  const float inv = fast_rcp(l0 + fast_sqrt(l0 * l0 + l1 * vmag));
  ux = vx * inv;
  uy = vy * inv;
  umag = vmag * inv;
}

// ---------------------------------------------------------------------------------------------
// collision of one cell in deviation variables, d[8] in (pre-collision), out (post-collision)
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ void collide_d2q8(float d[8], const Coef& c, float ax, float ay, const StepParams& P,
                                             float& ux_out, float& uy_out, float& phip_out) {
  const float rho0 = P.rho0;
  // m = M d, Eq. 10 with shared partial sums
  const float a13 = d[0] + d[2], a24 = d[1] + d[3];
  const float d13 = d[0] - d[2], d24 = d[1] - d[3];
  const float s57 = d[4] + d[6], s68 = d[5] + d[7];
  const float t57 = d[4] - d[6], t68 = d[5] - d[7];
  const float diag = s57 + s68;
  const float m1 = a13 + a24 + diag;        // p      (deviation)
  const float m2 = -(a13 + a24) + diag;     // e      (deviation)
  const float dxs = t57 - t68;              // e_x-weighted diagonal sum
  const float dys = t57 + t68;              // e_y-weighted diagonal sum
  const float m3 = d13 + dxs;               // j_x  (q_x = -2 d13 + dxs enters k4 below)
  const float m5 = d24 + dys;               // j_y  (q_y = -2 d24 + dys enters k6 below)
  const float m7 = a13 - a24;               // p_xx
  const float m8 = s57 - s68;               // p_xy

  // (from here the multiply-adds are written out: the collision of two cells at once, and every kernel,
  // must round as this one does)
  const float h = 0.5f * c.phi;
  const float vx = __fmaf_rn(h, ax, __fmul_rn(m3, P.inv_rho0)), vy = __fmaf_rn(h, ay, __fmul_rn(m5, P.inv_rho0));
  const float l0 = __fmaf_rn(0.25f, c.c_lin, 0.5f), l1 = 0.5f * c.c_nl;
  const float vmag = fast_sqrt(__fmaf_rn(vx, vx, __fmul_rn(vy, vy)));
  // Eq. 18, the cancellation-free root of l1 |u|^2 + 2 l0 |u| - |v| = 0
  const float R = __fmaf_rn(l0, l0, __fmul_rn(l1, vmag));  // >= l0^2 >= 1/4
  const float inv = rcp_normal(__fadd_rn(l0, __fmul_rn(R, rsqrt_normal(R))));
  const float ux = vx * inv, uy = vy * inv, umag = vmag * inv;
  const float uy2 = uy * uy, usq = __fmaf_rn(ux, ux, uy2);
  // Eq. 20 with c_s^2 / (1 - w0) = 3/5 and s0 = -2|u|^2 / (3 phi): phi p = 3/5 Y, Y = sum f - 2/3 rho0 |u|^2 / phi
  const float Y = __fmaf_rn(-__fmul_rn((2.0f / 3.0f) * rho0, usq), c.inv_phi, m1);
  const float phip_dev = 0.6f * Y;
  // Eq. 3
  const float drag = __fmaf_rn(c.c_nl, umag, c.c_lin);
  const float Fx = __fmaf_rn(c.phi, ax, __fmul_rn(-drag, ux));
  const float Fy = __fmaf_rn(c.phi, ay, __fmul_rn(-drag, uy));

  // Eqs. 11-14 as increments k = m+ - m = -Lambda (m - m_eq) + (I - Lambda/2) S.  m1 is conserved
  // (m1_eq = m1, S1 = 0); m3, m5 gain rho0 F for any s3, s5.  The q moments relax towards
  // -rho0 u, and m4 + rho0 u_x = (m4 + m3) + rho0 F_x / 2 by Eq. 17: that form avoids subtracting
  // two O(u) numbers.  Adding the increments to the pulled populations (instead of rebuilding
  // them from m+) keeps FP32 rounding at about one unit of d per step.
  const float s_e = P.s_e, s_q = P.s_q, s_v = c.s_v;
  const float rFx = rho0 * Fx, rFy = rho0 * Fy;
  const float be = __fmaf_rn(-0.5f, s_e, 1.0f), bq = __fmaf_rn(-0.5f, s_q, 1.0f), hv = __fmaf_rn(-0.5f, s_v, 1.0f);
  const float S2 = __fmul_rn(__fmul_rn(rho0 * 0.8f, __fmaf_rn(ux, Fx, __fmul_rn(uy, Fy))), c.inv_phi);
  const float k2 = __fmaf_rn(be, S2, __fmul_rn(-s_e, __fmaf_rn(0.6f, Y, m2)));  // e_eq = -phi p
  const float gx = __fmaf_rn(0.5f, rFx, __fmaf_rn(2.0f, dxs, -d13)), gy = __fmaf_rn(0.5f, rFy, __fmaf_rn(2.0f, dys, -d24));
  const float k4 = __fmaf_rn(-s_q, gx, -__fmul_rn(bq, rFx)), k6 = __fmaf_rn(-s_q, gy, -__fmul_rn(bq, rFy));
  const float A7 = __fmaf_rn(-__fmul_rn(rho0, __fmaf_rn(ux, ux, -uy2)), c.inv_phi, m7);
  const float Z7 = __fmul_rn(__fmul_rn(hv * 2.0f, rho0), __fmaf_rn(ux, Fx, -__fmul_rn(uy, Fy)));
  const float k7 = __fmaf_rn(Z7, c.inv_phi, -__fmul_rn(s_v, A7));
  const float A8 = __fmaf_rn(-__fmul_rn(__fmul_rn(rho0, ux), uy), c.inv_phi, m8);
  const float Z8 = __fmul_rn(__fmul_rn(hv, rho0), __fmaf_rn(ux, Fy, __fmul_rn(uy, Fx)));
  const float k8 = __fmaf_rn(Z8, c.inv_phi, -__fmul_rn(s_v, A8));

  // d+ = d + M^-1 k, M^-1 = M^T diag(1/8, 1/8, 1/6, 1/12, 1/6, 1/12, 1/4, 1/4), k1 = 0, k3 = rFx, k5 = rFy
  const float q2 = k2 * 0.125f;
  const float q4 = __fmul_rn(k4, 1.0f / 12.0f), q6 = __fmul_rn(k6, 1.0f / 12.0f);
  const float q7 = k7 * 0.25f, q8 = k8 * 0.25f;
  const float X = __fmaf_rn(rFx, 1.0f / 6.0f, -2.0f * q4), Y3 = __fmaf_rn(rFy, 1.0f / 6.0f, -2.0f * q6);
  const float Px = __fmaf_rn(rFx, 1.0f / 6.0f, q4), Py = __fmaf_rn(rFy, 1.0f / 6.0f, q6);
  d[0] += (X + q7) - q2;
  d[1] += (Y3 - q7) - q2;
  d[2] += (q7 - X) - q2;
  d[3] += (-Y3 - q7) - q2;
  d[4] += (Px + Py + q8) + q2;
  d[5] += (Py - Px - q8) + q2;
  d[6] += (q8 - Px - Py) + q2;
  d[7] += (Px - Py - q8) + q2;
  ux_out = ux;
  uy_out = uy;
  phip_out = phip_dev;
}

// ---------------------------------------------------------------------------------------------
// The same collision for two cells at once, on the packed FP32 pairs of sm_100+ (FADD2, FMUL2,
// FFMA2: one instruction for both cells, each lane rounded as the scalar operation).  d holds the
// stored deviations s d of the two cells (s: storage scale), so the scale is folded into the
// constants instead of being applied on every load and store; u is returned in lattice units.
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ float2 f2(float v) { return make_float2(v, v); }
__device__ __forceinline__ float2 neg2(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __fadd2_rn(a, neg2(b)); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }

// Medium coefficients of a cell pair (Eqs. 3-4, 13, 18), scaled as PairConst says (uniform medium:
// the same for both cells, from the host).
struct PairCoef {
  float2 inv_phi;     // 1 / phi
  float2 l0, l0sq;    // l0 = 1/2 + c_lin / 4 and l0^2 (Eq. 18)
  float2 l1;          // l1 = c_nl / 2
  float2 nclin, ncnl; // -c_lin = -phi nu / K, -c_nl = -1.75 / sqrt(150 phi K)
  float2 c2;          // 0.1 (1 - s_e/2) rho0 s / phi     (S2 / 8 = c2 (u . F))
  float2 cq;          // -s_v / 4
  float2 nR;          // -rho0 s / phi
  float2 cf7, cf8;    // (1 - s_v/2) rho0 s / (2 phi), / (4 phi)
};

__device__ __forceinline__ PairCoef pair_coef_uniform(const PairConst& K) {
  PairCoef c;
  c.inv_phi = f2(K.u_inv_phi); c.l0 = f2(K.u_l0); c.l0sq = f2(K.u_l0sq); c.l1 = f2(K.u_l1);
  c.nclin = f2(K.u_nclin); c.ncnl = f2(K.u_ncnl); c.c2 = f2(K.u_c2); c.cq = f2(K.cq); c.nR = f2(K.u_nR);
  c.cf7 = f2(K.u_cf7); c.cf8 = f2(K.u_cf8);
  return c;
}

// The same for a pair of cells of a per-cell medium: porosity ph, permeability k and viscous rate
// sv of the two cells (Eqs. 3-4, 13, 18, as coef_of); hx, hy receive phi a / 2.
__device__ __forceinline__ PairCoef pair_coef_het(const StepParams& P, float2 ph, float2 k, float2 sv, float2& hx, float2& hy) {
  const PairConst& K = P.pc;
  PairCoef c;
  c.inv_phi = make_float2(fast_rcp(ph.x), fast_rcp(ph.y));
  const float2 clin = mul2(mul2(ph, f2(P.nu)), make_float2(fast_rcp(k.x), fast_rcp(k.y)));  // phi nu / K
  const float2 cnl = P.forch ? make_float2(1.75f * rsqrtf(150.0f * ph.x * k.x), 1.75f * rsqrtf(150.0f * ph.y * k.y)) : f2(0.0f);
  c.l0 = fma2(f2(0.25f), clin, f2(0.5f));
  c.l0sq = mul2(c.l0, c.l0);
  c.l1 = mul2(f2(0.5f), cnl);
  c.nclin = neg2(clin);
  c.ncnl = neg2(cnl);
  const float2 rs_phi = mul2(f2(K.k_rs), c.inv_phi);
  c.c2 = mul2(f2(K.k_c2), c.inv_phi);
  c.cq = mul2(f2(-0.25f), sv);
  c.nR = neg2(rs_phi);
  const float2 hvr = mul2(fma2(f2(-0.5f), sv, f2(1.0f)), rs_phi);  // (1 - s_v/2) rho0 s / phi
  c.cf7 = mul2(f2(0.5f), hvr);
  c.cf8 = mul2(f2(0.25f), hvr);
  hx = mul2(f2(K.hax), ph);
  hy = mul2(f2(K.hay), ph);
  return c;
}

// hx, hy: phi a / 2 of the two cells.  d: in, stored pre-collision deviations; out, post-collision.
// FTZ: the reciprocal and the root by rcp_normal and rsqrt_normal, which give the bits of fast_rcp and
// rsqrtf for normal arguments (every float in range compared).  Fewer instructions (k_march 4096^2 FP16
// 86 -> 81 us per step), but another schedule, in which k_step with a per-cell medium spills 60 bytes
// instead of 24 (4096^2 FP16 110.0 -> 112.0 us) and the in-place step slows down (100.1 -> 102.1 us).
template <bool FTZ = true>
__device__ __forceinline__ void collide_pair(float2 d[8], const PairCoef& c, float2 hx, float2 hy, const PairConst& K, float2& ux,
                                             float2& uy) {
  // m = M d, Eq. 10 (as collide_d2q8)
  const float2 a13 = add2(d[0], d[2]), a24 = add2(d[1], d[3]);
  const float2 d13 = sub2(d[0], d[2]), d24 = sub2(d[1], d[3]);
  const float2 s57 = add2(d[4], d[6]), s68 = add2(d[5], d[7]);
  const float2 t57 = sub2(d[4], d[6]), t68 = sub2(d[5], d[7]);
  const float2 diag = add2(s57, s68), A = add2(a13, a24);
  const float2 m1 = add2(A, diag), m2 = sub2(diag, A);
  const float2 dxs = sub2(t57, t68), dys = add2(t57, t68);
  const float2 m3 = add2(d13, dxs), m5 = add2(d24, dys);
  const float2 m7 = sub2(a13, a24), m8 = sub2(s57, s68);

  // Eqs. 18-19: v = j / rho0 + phi a / 2, |u| = |v| / (l0 + sqrt(l0^2 + l1 |v|))
  const float2 vx = fma2(m3, f2(K.inv_rho0s), hx), vy = fma2(m5, f2(K.inv_rho0s), hy);
  const float2 vsq = fma2(vx, vx, mul2(vy, vy));
  const float2 vmag = mul2(vsq, make_float2(vsq.x > 0.0f ? rsqrtf(vsq.x) : 0.0f, vsq.y > 0.0f ? rsqrtf(vsq.y) : 0.0f));
  const float2 t = fma2(c.l1, vmag, c.l0sq);  // >= l0^2 >= 1/4
  const float2 den = add2(c.l0, mul2(t, FTZ ? make_float2(rsqrt_normal(t.x), rsqrt_normal(t.y)) : make_float2(rsqrtf(t.x), rsqrtf(t.y))));
  const float2 inv = FTZ ? make_float2(rcp_normal(den.x), rcp_normal(den.y)) : make_float2(fast_rcp(den.x), fast_rcp(den.y));
  ux = mul2(vx, inv);
  uy = mul2(vy, inv);
  const float2 umag = mul2(vmag, inv);
  // Eq. 20: phi p - p_rest = 3/5 (m1 - 2/3 rho0 |u|^2 / phi)   (times s)
  const float2 phip = mul2(f2(0.6f), fma2(f2(K.nphip), mul2(fma2(ux, ux, mul2(uy, uy)), c.inv_phi), m1));
  // Eq. 3: F = -(c_lin + c_nl |u|) u + phi a
  const float2 nd = fma2(c.ncnl, umag, c.nclin);
  const float2 Fx = fma2(nd, ux, add2(hx, hx)), Fy = fma2(nd, uy, add2(hy, hy));

  // increments k = m+ - m (Eqs. 11-14, as collide_d2q8) times the diagonal of M^-1:
  //   q2 = k2/8, X = k3/6 - k4/6 = rho0 F_x / 3 + s_q (m4 + m3) / 6, P_x = k3/6 + k4/12 =
  //   rho0 F_x / 12 - s_q (m4 + m3) / 12 (k4 = -s_q (m4 + m3) - rho0 F_x), q7 = k7/4, q8 = k8/4
  const float2 pxF = mul2(ux, Fx), pyF = mul2(uy, Fy);
  const float2 q2 = fma2(f2(K.nse8), add2(m2, phip), mul2(c.c2, add2(pxF, pyF)));
  const float2 gx = fma2(f2(2.0f), dxs, neg2(d13)), gy = fma2(f2(2.0f), dys, neg2(d24));  // m4 + m3, m6 + m5
  const float2 X = fma2(f2(K.sq6), gx, mul2(f2(K.r3), Fx)), Y = fma2(f2(K.sq6), gy, mul2(f2(K.r3), Fy));
  const float2 Px = fma2(f2(K.nsq12), gx, mul2(f2(K.r12), Fx)), Py = fma2(f2(K.nsq12), gy, mul2(f2(K.r12), Fy));
  const float2 q7 = fma2(c.cq, fma2(c.nR, fma2(ux, ux, neg2(mul2(uy, uy))), m7), mul2(c.cf7, sub2(pxF, pyF)));
  const float2 q8 = fma2(c.cq, fma2(c.nR, mul2(ux, uy), m8), mul2(c.cf8, fma2(ux, Fy, mul2(uy, Fx))));

  // d+ = d + M^-1 k (as collide_d2q8, with shared partial sums)
  const float2 B = sub2(q7, q2), Cn = add2(q7, q2);
  d[0] = add2(d[0], add2(B, X));
  d[2] = add2(d[2], sub2(B, X));
  d[1] = add2(d[1], sub2(Y, Cn));
  d[3] = sub2(d[3], add2(Y, Cn));
  const float2 G = add2(q8, q2), H = sub2(q2, q8), PP = add2(Px, Py), PM = sub2(Px, Py);
  d[4] = add2(d[4], add2(PP, G));
  d[6] = add2(d[6], sub2(G, PP));
  d[5] = add2(d[5], sub2(H, PM));
  d[7] = add2(d[7], add2(H, PM));
}

// collide_d2q8 for two cells at once on the packed FP32 pairs, in true units and with the roundings
// of the scalar form operation by operation, so that both give the same bits: FP32 storage may take
// either.  Differences are multiply-adds by -1,
// since the packed instructions have no negated operands.
struct PairMedium {
  float2 phi, inv_phi, l0, l1, nclin, ncnl, s_v;  // l0 = 1/2 + c_lin / 4, l1 = c_nl / 2, -c_lin, -c_nl
};
__device__ __forceinline__ float2 less2(float2 a, float2 b) { return __ffma2_rn(b, f2(-1.0f), a); }  // a - b

__device__ __forceinline__ PairMedium pair_medium(const Coef& a, const Coef& b) {
  PairMedium m;
  m.phi = make_float2(a.phi, b.phi);
  m.inv_phi = make_float2(a.inv_phi, b.inv_phi);
  m.l0 = make_float2(__fmaf_rn(0.25f, a.c_lin, 0.5f), __fmaf_rn(0.25f, b.c_lin, 0.5f));
  m.l1 = make_float2(0.5f * a.c_nl, 0.5f * b.c_nl);
  m.nclin = make_float2(-a.c_lin, -b.c_lin);
  m.ncnl = make_float2(-a.c_nl, -b.c_nl);
  m.s_v = make_float2(a.s_v, b.s_v);
  return m;
}

__device__ __forceinline__ void collide_d2q8_pair(float2 d[8], const PairMedium& c, float ax, float2 ay, const StepParams& P, float2& ux,
                                                  float2& uy) {
  const float rho0 = P.rho0;
  // m = M d, Eq. 10 (n13, n24: -(d1 - d3), -(d2 - d4))
  const float2 a13 = add2(d[0], d[2]), a24 = add2(d[1], d[3]);
  const float2 n13 = less2(d[2], d[0]), n24 = less2(d[3], d[1]);
  const float2 s57 = add2(d[4], d[6]), s68 = add2(d[5], d[7]);
  const float2 t57 = less2(d[4], d[6]), t68 = less2(d[5], d[7]);
  const float2 diag = add2(s57, s68), A = add2(a13, a24);
  const float2 m1 = add2(A, diag), m2 = less2(diag, A);
  const float2 dxs = less2(t57, t68), dys = add2(t57, t68);
  const float2 m3 = less2(dxs, n13), m5 = less2(dys, n24);
  const float2 m7 = less2(a13, a24), m8 = less2(s57, s68);
  // Eqs. 17-19
  const float2 h = mul2(f2(0.5f), c.phi);
  const float2 vx = fma2(h, f2(ax), mul2(m3, f2(P.inv_rho0))), vy = fma2(h, ay, mul2(m5, f2(P.inv_rho0)));
  const float2 vsq = fma2(vx, vx, mul2(vy, vy));
  const float2 vmag = make_float2(fast_sqrt(vsq.x), fast_sqrt(vsq.y));
  const float2 R = fma2(c.l0, c.l0, mul2(c.l1, vmag));  // >= l0^2 >= 1/4
  // (scalar products: a packed product would be fused with the sum)
  const float2 den = add2(c.l0, make_float2(__fmul_rn(R.x, rsqrt_normal(R.x)), __fmul_rn(R.y, rsqrt_normal(R.y))));
  const float2 inv = make_float2(rcp_normal(den.x), rcp_normal(den.y));
  ux = mul2(vx, inv);
  uy = mul2(vy, inv);
  const float2 umag = mul2(vmag, inv), nuy = mul2(uy, f2(-1.0f));
  // Eq. 20 (phi p = 0.6 Y) and Eq. 3
  const float2 usq = fma2(ux, ux, mul2(uy, uy));
  const float2 Y = fma2(mul2(f2(-(2.0f / 3.0f) * rho0), usq), c.inv_phi, m1);
  const float2 nd = fma2(c.ncnl, umag, c.nclin);
  const float2 Fx = fma2(c.phi, f2(ax), mul2(nd, ux)), Fy = fma2(c.phi, ay, mul2(nd, uy));
  // Eqs. 11-14 as increments (collide_d2q8)
  const float2 rFx = mul2(f2(rho0), Fx), rFy = mul2(f2(rho0), Fy);
  const float be = __fmaf_rn(-0.5f, P.s_e, 1.0f), nbq = -__fmaf_rn(-0.5f, P.s_q, 1.0f);
  const float2 S2 = mul2(mul2(f2(rho0 * 0.8f), fma2(ux, Fx, mul2(uy, Fy))), c.inv_phi);
  const float2 k2 = fma2(f2(be), S2, mul2(f2(-P.s_e), fma2(f2(0.6f), Y, m2)));
  const float2 gx = fma2(f2(0.5f), rFx, fma2(f2(2.0f), dxs, n13)), gy = fma2(f2(0.5f), rFy, fma2(f2(2.0f), dys, n24));
  const float2 k4 = fma2(f2(-P.s_q), gx, mul2(f2(nbq), rFx)), k6 = fma2(f2(-P.s_q), gy, mul2(f2(nbq), rFy));
  const float2 hv = fma2(f2(-0.5f), c.s_v, f2(1.0f)), nsv = mul2(f2(-1.0f), c.s_v);
  const float2 A7 = fma2(mul2(f2(-rho0), fma2(ux, ux, mul2(nuy, uy))), c.inv_phi, m7);
  const float2 Z7 = mul2(mul2(mul2(hv, f2(2.0f)), f2(rho0)), fma2(ux, Fx, mul2(nuy, Fy)));
  const float2 k7 = fma2(Z7, c.inv_phi, mul2(nsv, A7));
  const float2 A8 = fma2(mul2(mul2(f2(-rho0), ux), uy), c.inv_phi, m8);
  const float2 Z8 = mul2(mul2(hv, f2(rho0)), fma2(ux, Fy, mul2(uy, Fx)));
  const float2 k8 = fma2(Z8, c.inv_phi, mul2(nsv, A8));
  // d+ = d + M^-1 k
  const float2 q2 = mul2(k2, f2(0.125f)), q7 = mul2(k7, f2(0.25f)), q8 = mul2(k8, f2(0.25f));
  const float2 q4 = mul2(k4, f2(1.0f / 12.0f)), q6 = mul2(k6, f2(1.0f / 12.0f));
  const float2 X = fma2(rFx, f2(1.0f / 6.0f), mul2(f2(-2.0f), q4)), Yy = fma2(rFy, f2(1.0f / 6.0f), mul2(f2(-2.0f), q6));
  const float2 Px = fma2(rFx, f2(1.0f / 6.0f), q4), Py = fma2(rFy, f2(1.0f / 6.0f), q6);
  d[0] = add2(d[0], less2(add2(X, q7), q2));
  d[1] = add2(d[1], less2(less2(Yy, q7), q2));
  d[2] = add2(d[2], less2(less2(q7, X), q2));
  d[3] = less2(d[3], add2(add2(Yy, q7), q2));
  d[4] = add2(d[4], add2(add2(add2(Px, Py), q8), q2));
  d[5] = add2(d[5], add2(less2(less2(Py, Px), q8), q2));
  d[6] = add2(d[6], add2(less2(less2(q8, Px), Py), q2));
  d[7] = add2(d[7], add2(less2(less2(Px, Py), q8), q2));
}

// macroscopic quantities only (no collision), for read-out kernels
__device__ __forceinline__ Macro macro_d2q8(const float d[8], const Coef& c, float ax, float ay, float rho0) {
  Macro r;
  const float m1 = d[0] + d[1] + d[2] + d[3] + d[4] + d[5] + d[6] + d[7];
  const float jx = (d[0] - d[2]) + (d[4] - d[5] - d[6] + d[7]);
  const float jy = (d[1] - d[3]) + (d[4] + d[5] - d[6] - d[7]);
  float umag;
  velocity_from_j(jx, jy, c, ax, ay, fast_rcp(rho0), r.ux, r.uy, umag);
  r.dm1 = m1;
  r.phip_dev = 0.6f * (m1 - (2.0f / 3.0f) * rho0 * (r.ux * r.ux + r.uy * r.uy) * c.inv_phi);
  return r;
}

// Equilibrium deviation f_eq,i(p, u; phi) - f_rest,i (Eq. 22 with rho0), phip_dev = phi p - p_rest.
__device__ __forceinline__ void feq_dev_d2q8(float phip_dev, float ux, float uy, float inv_phi, float rho0, float out[8]) {
  const float usq15 = 1.5f * (ux * ux + uy * uy) * inv_phi;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const float eu = (float)ex_of(i) * ux + (float)ey_of(i) * uy;
    out[i] = w_of(i) * (3.0f * phip_dev + rho0 * (3.0f * eu + 4.5f * eu * eu * inv_phi - usq15));
  }
}

// ---------------------------------------------------------------------------------------------
// D2Q5 temperature collision in deviation variables (Eq. B.2 with n_eq of Eq. B.6)
// g[5]: deviations from T0/5, in (pre-collision) and out (post-collision); returns T.
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ float collide_d2q5(float g[5], float ux, float uy, const StepParams& P) {
  // n = N g, Eq. B.4
  const float n0 = g[0] + g[1] + g[2] + g[3] + g[4];
  const float n1 = g[1] - g[3];
  const float n2 = g[2] - g[4];
  const float side = g[1] + g[2] + g[3] + g[4];
  const float n3 = side - 4.0f * g[0];
  const float n4 = g[1] - g[2] + g[3] - g[4];
  const float T = P.T0 + n0;
  // increments n+ - n (n0 conserved), then g+ = g + N^-1 (n+ - n) with
  // N^-1 = N^T diag(1/5, 1/2, 1/2, 1/20, 1/4); multiply-adds written out (see collide_d2q8)
  const float z1 = -0.5f * P.zeta1, z4 = -0.25f * P.zeta4;
  const float b1 = __fmaf_rn(-__fmul_rn(ux, T), P.inv_sigma, n1), b2 = __fmaf_rn(-__fmul_rn(uy, T), P.inv_sigma, n2);
  const float r3 = __fmul_rn(-0.05f * P.zeta3, __fmaf_rn(-P.varpi, T, n3));
  g[0] = __fmaf_rn(-4.0f, r3, g[0]);
  g[1] += __fmaf_rn(z4, n4, __fmaf_rn(z1, b1, r3));
  g[2] += __fmaf_rn(-z4, n4, __fmaf_rn(z1, b2, r3));
  g[3] += __fmaf_rn(z4, n4, __fmaf_rn(-z1, b1, r3));
  g[4] += __fmaf_rn(-z4, n4, __fmaf_rn(-z1, b2, r3));
  return T;
}

// The same for two cells at once on packed FP32 pairs; g holds the stored deviations s g (s: the
// storage scale), u is in lattice units.  T = T0 + n0 / s is carried as s T = s T0 + n0.
__device__ __forceinline__ void collide_d2q5_pair(float2 g[5], float2 ux, float2 uy, const StepParams& P) {
  const float2 n0 = add2(add2(add2(g[0], g[1]), add2(g[2], g[3])), g[4]);
  const float2 n1 = sub2(g[1], g[3]), n2 = sub2(g[2], g[4]);
  const float2 side = add2(add2(g[1], g[2]), add2(g[3], g[4]));
  const float2 n3 = fma2(f2(-4.0f), g[0], side);
  const float2 n4 = sub2(add2(g[1], g[3]), add2(g[2], g[4]));
  const float2 sT = add2(f2(P.scale * P.T0), n0);  // s T
  const float2 q = mul2(sT, f2(P.inv_sigma));
  // increments n+ - n (n0 conserved) times the diagonal of N^-1 (as collide_d2q5)
  const float2 r1 = mul2(f2(-0.5f * P.zeta1), fma2(neg2(ux), q, n1));
  const float2 r2 = mul2(f2(-0.5f * P.zeta1), fma2(neg2(uy), q, n2));
  const float2 r3 = mul2(f2(-0.05f * P.zeta3), fma2(f2(-P.varpi), sT, n3));
  const float2 r4 = mul2(f2(-0.25f * P.zeta4), n4);
  const float2 a = add2(r3, r4), b = sub2(r3, r4);
  g[0] = fma2(f2(-4.0f), r3, g[0]);
  g[1] = add2(g[1], add2(r1, a));
  g[2] = add2(g[2], add2(r2, b));
  g[3] = add2(g[3], sub2(a, r1));
  g[4] = add2(g[4], sub2(b, r2));
}

// collide_d2q5 for two cells at once, rounded as the scalar form (see collide_d2q8_pair); n0 = T - T0.
__device__ __forceinline__ void collide_d2q5_pair_fp32(float2 g[5], float2 n0, float2 ux, float2 uy, const StepParams& P) {
  const float2 n1 = less2(g[1], g[3]), n2 = less2(g[2], g[4]);
  const float2 n3 = fma2(f2(-4.0f), g[0], add2(add2(add2(g[1], g[2]), g[3]), g[4]));
  const float2 n4 = less2(add2(less2(g[1], g[2]), g[3]), g[4]);
  const float2 T = add2(f2(P.T0), n0), nT = mul2(T, f2(-1.0f));
  const float2 b1 = fma2(mul2(ux, nT), f2(P.inv_sigma), n1), b2 = fma2(mul2(uy, nT), f2(P.inv_sigma), n2);
  const float2 r3 = mul2(f2(-0.05f * P.zeta3), fma2(f2(-P.varpi), T, n3));
  const float2 z1 = f2(-0.5f * P.zeta1), nz1 = f2(0.5f * P.zeta1), z4 = f2(-0.25f * P.zeta4), nz4 = f2(0.25f * P.zeta4);
  g[0] = fma2(f2(-4.0f), r3, g[0]);
  g[1] = add2(g[1], fma2(z4, n4, fma2(z1, b1, r3)));
  g[2] = add2(g[2], fma2(nz4, n4, fma2(z1, b2, r3)));
  g[3] = add2(g[3], fma2(z4, n4, fma2(nz1, b1, r3)));
  g[4] = add2(g[4], fma2(nz4, n4, fma2(nz1, b2, r3)));
}

// D2Q5 velocities of Eq. B.3 (0 rest, 1..4 as D2Q8's first four)
__device__ __forceinline__ int ex5(int i) { return i == 1 ? 1 : (i == 3 ? -1 : 0); }
__device__ __forceinline__ int ey5(int i) { return i == 2 ? 1 : (i == 4 ? -1 : 0); }
__device__ __forceinline__ int opp5(int i) { return i == 0 ? 0 : 1 + ((i - 1 + 2) & 3); }

// ---------------------------------------------------------------------------------------------
// generic pull of one population with every edge rule (used on edge cells and read-outs)
// ---------------------------------------------------------------------------------------------
// Wall that owns a link whose source (sx, sy) lies outside: y sides first (corners included).
__device__ __forceinline__ int wall_of(int sx, int sy, int ny) {
  if (sy < 0) return 2;
  if (sy >= ny) return 3;
  return sx < 0 ? 0 : 1;
}

// ---------------------------------------------------------------------------------------------
// In-place streaming: one population buffer.  Of each pair of opposite velocities the member with
// e_x > 0, or e_x = 0 and e_y > 0 (e1, e2, e5, e8), is "positive".  At parity par a cell c reads
// population i from plane (par ? i : opp(i)) at c itself when i is positive and at c - e_i
// otherwise, and writes its post-collision population j where the cell c + e_j reads j at the
// next parity.  The slots a cell writes are then exactly the slots it read (each receives the
// population opposite to the one read from it), so the two halves of Eq. 15 share one buffer
// without races and the buffer alternates between two layouts.  Populations that leave through a
// wall are parked in ghost slots (rows -1 and ny, column nx; never updated as cells) until the
// same cell reads them back as its bounce-back (Eq. 15 at a wall).  Ghost rows -1 and ny are rows of
// the planes; the ghost column lives after the last plane, q columns of ny + 2 slots (so that a
// lattice width that is a multiple of the row pitch needs no wider rows).  Extrapolated sides (wall
// nodes, pressure columns) keep the slot rules of a halfway wall; their boundary nodes' states are
// computed before each step (k_edge_ip), since they read a neighbour that the step overwrites.
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ bool ip_positive(int i) { return i == 0 || i == 1 || i == 4 || i == 7; }

__device__ __forceinline__ int wrap_periodic(int v, int n, bool periodic) {
  return periodic ? (v < 0 ? v + n : (v >= n ? v - n : v)) : v;
}

// element offset (from row 0 of plane 0) of slot (plane, cx, cy) of a buffer of q planes
__device__ __forceinline__ int64_t ip_slot(const StepParams& P, int q, int plane, int cx, int cy) {
  if (cx >= P.nx) return (int64_t)q * P.plane - P.pitch + (int64_t)plane * (P.ny + 2) + (cy + 1);  // ghost column
  return (int64_t)plane * P.plane + (int64_t)cy * P.pitch + cx;
}

// element offset of the slot from which cell (cx, cy) (a lattice or ghost cell) reads population
// i at parity par
__device__ __forceinline__ int64_t ip_off(const StepParams& P, int cx, int cy, int i, int par) {
  if (!ip_positive(i)) {
    cx -= ex_of(i);
    cy -= ey_of(i);
  }
  cx = wrap_periodic(cx, P.nx, P.bc_x == BC_PERIODIC);
  cy = wrap_periodic(cy, P.ny, P.bc_y == BC_PERIODIC);
  dbg_check(P, cx >= 0 && cx <= P.nx && cy >= -1 && cy <= P.ny);
  return ip_slot(P, 8, par ? i : opp_of(i), cx, cy);
}

// the same for the D2Q5 temperature populations (positive: 1 and 2; the rest population stays)
__device__ __forceinline__ int64_t ip_off5(const StepParams& P, int cx, int cy, int i, int par) {
  if (i == 3 || i == 4) {
    cx -= ex5(i);
    cy -= ey5(i);
  }
  cx = wrap_periodic(cx, P.nx, P.bc_x == BC_PERIODIC);
  cy = wrap_periodic(cy, P.ny, P.bc_y == BC_PERIODIC);
  dbg_check(P, cx >= 0 && cx <= P.nx && cy >= -1 && cy <= P.ny);
  return ip_slot(P, 5, i == 0 ? 0 : (par ? i : opp5(i)), cx, cy);
}

// Source of the pull of population i into cell (x, y) at the current parity: the slot the cell
// reads (wall = -1), or, where x - e_i lies beyond a wall, the slot in which the cell parked its
// own post-collision population opp(i) (wall = the wall's index).
__device__ __forceinline__ int64_t ip_source(const StepParams& P, int x, int y, int i, int& wall) {
  int sx = x - ex_of(i), sy = y - ey_of(i);
  sx = wrap_periodic(sx, P.nx, P.bc_x == BC_PERIODIC);
  sy = wrap_periodic(sy, P.ny, P.bc_y == BC_PERIODIC);
  if (sx >= 0 && sx < P.nx && sy >= 0 && sy < P.ny) {
    wall = -1;
    return ip_off(P, x, y, i, P.parity);
  }
  wall = wall_of(sx, sy, P.ny);
  return ip_off(P, sx, sy, opp_of(i), P.parity);
}

__device__ __forceinline__ int64_t ip_source5(const StepParams& P, int x, int y, int i, int& wall) {
  int sx = x - ex5(i), sy = y - ey5(i);
  sx = wrap_periodic(sx, P.nx, P.bc_x == BC_PERIODIC);
  sy = wrap_periodic(sy, P.ny, P.bc_y == BC_PERIODIC);
  if (sx >= 0 && sx < P.nx && sy >= 0 && sy < P.ny) {
    wall = -1;
    return ip_off5(P, x, y, i, P.parity);
  }
  wall = wall_of(sx, sy, P.ny);
  return ip_off5(P, sx, sy, opp5(i), P.parity);
}

// Component c of the velocity of wall w.  lbm_set_walls may write it while a kernel that was launched
// early is already resident: an ordinary load that stays behind wait_prerequisites(), and not one
// through the read-only path, which takes memory that is constant for as long as the kernel lives.
// (Written as an instruction, so that it is not moved: as a plain load it let the compiler interleave
// several cells, 72 -> 128 registers in the residual's kernel; a C++ volatile one passes by L1, and
// steps bound by their frame cells slowed down, in place 1024^2 FP16 with a per-cell medium 12.3 -> 13.5 us.)
__device__ __forceinline__ float wall_velocity(const StepParams& P, int w, int c) {
  float v;
  asm volatile("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(P.uw + 2 * w + c));
  return v;
}

// momentum correction of the moving-wall bounce-back, 2 w_i rho0 (e_i . u_w) / c_s^2
__device__ __forceinline__ float wall_term(const StepParams& P, int i, int w) {
  return 6.0f * w_of(i) * P.rho0 * ((float)ex_of(i) * wall_velocity(P, w, 0) + (float)ey_of(i) * wall_velocity(P, w, 1));
}

// e_i . u_w of wall w
__device__ __forceinline__ float wall_dot(const StepParams& P, int i, int w) {
  return __fadd_rn((float)ex_of(i) * wall_velocity(P, w, 0), (float)ey_of(i) * wall_velocity(P, w, 1));
}

// Halfway bounce-back: f_i(x) = f+_opp(i)(x) + 2 w_i rho0 (e_i . u_w) / c_s^2 with own = f+_opp(i)(x),
// dot = e_i . u_w; and its counterpart for the temperature, anti-bounce-back at a wall with a prescribed
// temperature (deviation form of g_i = -g+_opp + 2 T_w / 5, reference T0 / 5), bounce-back at an adiabatic
// one.  The roundings are written out so that every kernel that applies a wall gives the same bits (with
// FP16 storage the scale's product is part of own, and the wall term is rounded before it is added).
template <int PREC>
__device__ __forceinline__ float bounce(const StepParams& P, float own, int i, float dot) {
  const float c = 6.0f * w_of(i) * P.rho0;
  return PREC == PREC_FP16 ? __fadd_rn(own, __fmul_rn(c, dot)) : __fmaf_rn(c, dot, own);
}
template <int PREC>
__device__ __forceinline__ float heat_bounce(const StepParams& P, float own, int w) {
  if (!P.Tdir[w]) return own;
  const float d = P.Tw[w] - P.T0;
  return PREC == PREC_FP16 ? __fadd_rn(-own, __fmul_rn(0.4f, d)) : __fmaf_rn(0.4f, d, -own);
}

template <int PREC>
__device__ __forceinline__ float pull_one(const StepParams& P, const typename Store<PREC>::T* src, int x, int y, int i) {
  using S = Store<PREC>;
  if (!dbg_check(P, x >= 0 && x < P.pitch && y >= 0 && y < P.ny)) return 0.0f;
  if (P.inplace) {
    int w;
    const float v = S::dec(src[ip_source(P, x, y, i, w)], P.inv_scale);
    return w < 0 ? v : v + wall_term(P, i, w);
  }
  int sx = x - ex_of(i), sy = y - ey_of(i);
  if (P.bc_x != BC_WALL) sx = (sx + P.nx) % P.nx;
  if (P.bc_y != BC_WALL) sy = (sy + P.ny) % P.ny;
  if (sx >= 0 && sx < P.nx && sy >= 0 && sy < P.ny)
    return S::dec(src[(int64_t)i * P.plane + (int64_t)sy * P.pitch + sx], P.inv_scale);
  const int w = wall_of(sx, sy, P.ny);
  return bounce<PREC>(P, S::dec(src[(int64_t)opp_of(i) * P.plane + (int64_t)y * P.pitch + x], P.inv_scale), i, wall_dot(P, i, w));
}

template <int PREC>
__device__ __forceinline__ void pull_cell(const StepParams& P, const typename Store<PREC>::T* src, int x, int y, float d[8]) {
#pragma unroll
  for (int i = 0; i < 8; ++i) d[i] = pull_one<PREC>(P, src, x, y, i);
}

// temperature: anti-bounce-back at walls with a prescribed temperature, bounce-back otherwise
template <int PREC>
__device__ __forceinline__ float pull_one_g(const StepParams& P, const typename Store<PREC>::T* src, int x, int y, int i) {
  using S = Store<PREC>;
  if (!dbg_check(P, x >= 0 && x < P.pitch && y >= 0 && y < P.ny)) return 0.0f;
  if (P.inplace) {
    int w;
    const float v = S::dec(src[ip_source5(P, x, y, i, w)], P.inv_scale);
    return (w < 0 || !P.Tdir[w]) ? v : (-v + 0.4f * (P.Tw[w] - P.T0));
  }
  if (i == 0) return S::dec(src[(int64_t)y * P.pitch + x], P.inv_scale);
  int sx = x - ex5(i), sy = y - ey5(i);
  if (P.bc_x != BC_WALL) sx = (sx + P.nx) % P.nx;
  if (P.bc_y != BC_WALL) sy = (sy + P.ny) % P.ny;
  if (sx >= 0 && sx < P.nx && sy >= 0 && sy < P.ny)
    return S::dec(src[(int64_t)i * P.plane + (int64_t)sy * P.pitch + sx], P.inv_scale);
  const int w = wall_of(sx, sy, P.ny);
  return heat_bounce<PREC>(P, S::dec(src[(int64_t)opp5(i) * P.plane + (int64_t)y * P.pitch + x], P.inv_scale), w);
}

template <int PREC>
__device__ __forceinline__ void pull_cell_g(const StepParams& P, const typename Store<PREC>::T* src, int x, int y, float g[5]) {
#pragma unroll
  for (int i = 0; i < 5; ++i) g[i] = pull_one_g<PREC>(P, src, x, y, i);
}

// Non-equilibrium extrapolation of a pressure column: replaces d of the cell (xb, y) by
// f_eq(p_b, u_nb; phi_b) + f_nb - f_eq(p_nb, u_nb; phi_nb) with nb = (xb +- 1, y), in deviations.
// (dn: the pulled state of nb)
// The multiply-adds are written out, so that every kernel extrapolates to the same bits (macro_d2q8
// and feq_dev_d2q8, which leave them to the compiler, serve the read-outs).
// (cn, cb: the medium of the inner neighbour and of the column's cell, pb its pressure)
__device__ __forceinline__ void pressure_cell(const StepParams& P, const float dn[8], const Coef& cn, const Coef& cb, float pb, float d[8]) {
  const float m1 = dn[0] + dn[1] + dn[2] + dn[3] + dn[4] + dn[5] + dn[6] + dn[7];
  const float jx = (dn[0] - dn[2]) + (dn[4] - dn[5] - dn[6] + dn[7]);
  const float jy = (dn[1] - dn[3]) + (dn[4] + dn[5] - dn[6] - dn[7]);
  const float h = 0.5f * cn.phi, inv_rho0 = fast_rcp(P.rho0);
  const float vx = __fmaf_rn(h, P.ax, __fmul_rn(jx, inv_rho0)), vy = __fmaf_rn(h, P.ay, __fmul_rn(jy, inv_rho0));
  const float l0 = __fmaf_rn(0.25f, cn.c_lin, 0.5f);
  const float R = __fmaf_rn(l0, l0, __fmul_rn(0.5f * cn.c_nl, fast_sqrt(__fmaf_rn(vx, vx, __fmul_rn(vy, vy)))));
  const float inv = rcp_normal(__fadd_rn(l0, __fmul_rn(R, rsqrt_normal(R))));
  const float ux = vx * inv, uy = vy * inv, usq = __fmaf_rn(ux, ux, __fmul_rn(uy, uy));
  const float pn = 0.6f * __fmaf_rn(-__fmul_rn((2.0f / 3.0f) * P.rho0, usq), cn.inv_phi, m1);  // phi p - p_rest, Eq. 20
  const float pd = __fmaf_rn(cb.phi, pb, -P.p_rest);
  const float ub = __fmul_rn(1.5f * usq, cb.inv_phi), un = __fmul_rn(1.5f * usq, cn.inv_phi);
#pragma unroll
  for (int i = 0; i < 8; ++i) {  // f_eq of Eq. 22 in deviations
    const float eu = __fadd_rn((float)ex_of(i) * ux, (float)ey_of(i) * uy), q = __fmul_rn(4.5f * eu, eu);
    const float eb = __fmul_rn(w_of(i), __fmaf_rn(3.0f, pd, __fmul_rn(P.rho0, __fmaf_rn(3.0f, eu, __fmaf_rn(q, cb.inv_phi, -ub)))));
    const float en = __fmul_rn(w_of(i), __fmaf_rn(3.0f, pn, __fmul_rn(P.rho0, __fmaf_rn(3.0f, eu, __fmaf_rn(q, cn.inv_phi, -un)))));
    d[i] = __fadd_rn(__fadd_rn(eb, dn[i]), -en);
  }
}

template <bool HET>
__device__ __forceinline__ void pressure_column_from(const StepParams& P, const float dn[8], int xb, int y, float d[8]) {
  pressure_cell(P, dn, coef_at<HET>(P, xb == 0 ? 1 : P.nx - 2, y), coef_at<HET>(P, xb, y), xb == 0 ? P.p_in : P.p_out, d);
}

template <int PREC, bool HET>
__device__ __forceinline__ void pressure_column(const StepParams& P, const typename Store<PREC>::T* src, int xb, int y, float d[8]) {
  float dn[8];
  pull_cell<PREC>(P, src, xb == 0 ? 1 : P.nx - 2, y, dn);
  pressure_column_from<HET>(P, dn, xb, y, d);
}

// Wall node of a side with non-equilibrium extrapolation (BC_NEE, the paper's wall treatment of
// Sec. 3): true for (x, y) on such a wall, with nb = (xn, yn) one step inward along the wall
// normal and w the wall (0 left, 1 right, 2 bottom, 3 top).  Bottom/top walls own the corners,
// whose nb is the diagonal node when the x sides are not periodic.
__device__ __forceinline__ bool nee_node(const StepParams& P, int x, int y, int& xn, int& yn, int& w) {
  if (P.bc_y == BC_NEE && (y == 0 || y == P.ny - 1)) {
    yn = y == 0 ? 1 : P.ny - 2;
    w = y == 0 ? 2 : 3;
    xn = (P.bc_x != BC_PERIODIC && (x == 0 || x == P.nx - 1)) ? (x == 0 ? 1 : P.nx - 2) : x;
    return true;
  }
  if (P.bc_x == BC_NEE && (x == 0 || x == P.nx - 1)) {
    xn = x == 0 ? 1 : P.nx - 2;
    yn = y;
    w = x == 0 ? 0 : 1;
    return true;
  }
  return false;
}

// d of a wall node: f_eq(p_nb, u_w; phi_b) + f_nb - f_eq(p_nb, u_nb; phi_nb) (pressure extrapolated
// with zero normal gradient), in deviations; ay_nb is a_y at nb (with its buoyancy in a thermal
// context), u_nb is returned; dn is the pulled state of nb.
template <bool HET>
__device__ __forceinline__ void wall_node_from(const StepParams& P, const float dn[8], int x, int y, int xn, int yn, int w, float ay_nb,
                                               float d[8], float& ux_nb, float& uy_nb) {
  const Coef cn = coef_at<HET>(P, xn, yn);
  const Coef cb = coef_at<HET>(P, x, y);
  const Macro mn = macro_d2q8(dn, cn, P.ax, ay_nb, P.rho0);
  ux_nb = mn.ux;
  uy_nb = mn.uy;
  // phi_b p_nb - p_rest = phi_nb p_nb - p_rest + (phi_b / phi_nb - 1) phi_nb p_nb, kept in deviations
  // (exact for phi_b = phi_nb; forming p_nb itself would add p_rest to a small deviation)
  const float dr = (cb.phi - cn.phi) * cn.inv_phi;
  const float phip_b = mn.phip_dev + dr * (mn.phip_dev + P.p_rest);
  float eb[8], en[8];
  feq_dev_d2q8(phip_b, wall_velocity(P, w, 0), wall_velocity(P, w, 1), cb.inv_phi, P.rho0, eb);
  feq_dev_d2q8(mn.phip_dev, mn.ux, mn.uy, cn.inv_phi, P.rho0, en);
#pragma unroll
  for (int i = 0; i < 8; ++i) d[i] = eb[i] + dn[i] - en[i];
}

template <int PREC, bool HET>
__device__ __forceinline__ void wall_node(const StepParams& P, const typename Store<PREC>::T* src, int x, int y, int xn, int yn,
                                          int w, float ay_nb, float d[8], float& ux_nb, float& uy_nb) {
  float dn[8];
  pull_cell<PREC>(P, src, xn, yn, dn);
  wall_node_from<HET>(P, dn, x, y, xn, yn, w, ay_nb, d, ux_nb, uy_nb);
}

// Pre-collision state of any cell: the pull of Eq. 15 with its wall rules, or the extrapolated
// state of a wall node or pressure column.
template <int PREC, bool HET>
__device__ __forceinline__ void gather_cell(const StepParams& P, const typename Store<PREC>::T* src, int x, int y, float d[8]) {
  int xn, yn, w;
  float uxn, uyn;
  if (nee_node(P, x, y, xn, yn, w))
    wall_node<PREC, HET>(P, src, x, y, xn, yn, w, P.ay, d, uxn, uyn);
  else if (P.bc_x == BC_PRESSURE && (x == 0 || x == P.nx - 1))
    pressure_column<PREC, HET>(P, src, x, y, d);
  else
    pull_cell<PREC>(P, src, x, y, d);
}

// thermal equilibrium (Eq. B.6) deviation from T0/5
__device__ __forceinline__ void geq_dev(const StepParams& P, float T, float ux, float uy, float out[5]) {
  const float a = 0.2f * T - 0.2f * P.T0;
  const float b = 0.05f * P.varpi * T;
  const float hx = 0.5f * ux * T * P.inv_sigma, hy = 0.5f * uy * T * P.inv_sigma;
  out[0] = a - 4.0f * b;
  out[1] = a + hx + b;
  out[2] = a + hy + b;
  out[3] = a - hx + b;
  out[4] = a - hy + b;
}

// Pre-collision temperature of a cell: on a wall node of an extrapolated side the wall temperature
// (isothermal wall) or that of its inner neighbour (adiabatic wall), which is what the node's
// extrapolated populations sum to.
template <int PREC>
__device__ __forceinline__ double temperature_at(const StepParams& P, const typename Store<PREC>::T* gsrc, int x, int y) {
  int xn = x, yn = y, w = 0;
  if (nee_node(P, x, y, xn, yn, w) && P.Tdir[w]) return (double)P.Tw[w];
  float g[5];
  pull_cell_g<PREC>(P, gsrc, xn, yn, g);
  return (double)P.T0 + ((double)g[0] + g[1] + g[2] + g[3] + g[4]);
}

// Flow and temperature state of a wall node of a thermal context from the pulled states dn, gn of
// its nb (see gather_cell_thermal).
template <bool HET>
__device__ __forceinline__ void thermal_wall_node_from(const StepParams& P, const float dn[8], const float gn[5], int x, int y, int xn,
                                                       int yn, int w, float d[8], float g[5]) {
  const float Tn = gn[0] + gn[1] + gn[2] + gn[3] + gn[4];  // T_nb - T0
  float uxn, uyn;
  wall_node_from<HET>(P, dn, x, y, xn, yn, w, P.ay + P.g_beta * Tn, d, uxn, uyn);
  const float Tb = P.Tdir[w] ? P.Tw[w] - P.T0 : Tn;
  float eb[5], en[5];
  geq_dev(P, P.T0 + Tb, wall_velocity(P, w, 0), wall_velocity(P, w, 1), eb);
  geq_dev(P, P.T0 + Tn, uxn, uyn, en);
#pragma unroll
  for (int i = 0; i < 5; ++i) g[i] = eb[i] + gn[i] - en[i];
}

// Pre-collision flow (d) and temperature (g, deviations from T0/5) state of a cell of a thermal
// context.  On a wall node of an extrapolated side, g = g_eq(T_b, u_w) + g_nb - g_eq(T_nb, u_nb)
// with T_b the wall temperature (isothermal wall) or T_nb (adiabatic wall), and the flow part
// uses the velocity of nb with the buoyancy of T_nb.
template <int PREC, bool HET>
__device__ __forceinline__ void gather_cell_thermal(const StepParams& P, const typename Store<PREC>::T* src,
                                                    const typename Store<PREC>::T* gsrc, int x, int y, float d[8], float g[5]) {
  int xn, yn, w;
  if (nee_node(P, x, y, xn, yn, w)) {
    float dn[8], gn[5];
    pull_cell<PREC>(P, src, xn, yn, dn);
    pull_cell_g<PREC>(P, gsrc, xn, yn, gn);
    thermal_wall_node_from<HET>(P, dn, gn, x, y, xn, yn, w, d, g);
  } else {
    gather_cell<PREC, HET>(P, src, x, y, d);
    pull_cell_g<PREC>(P, gsrc, x, y, g);
  }
}

}  // namespace lbm
