// kernels.cu -- sm_103a kernels of one forward-Euler stage of the hyperbolic
// (Euler) operator of arXiv:2106.02159 (Appendix B, Algorithm 1) and of the
// boundary post-processing of Sec. 4.
//
// Design: on GB300 an FP64 FMA issues at 1/72 of the FP32 rate, so this path
// is bound by FP64 instruction issue, not by HBM. Every edge loop therefore
// runs one thread per CSR row (no idle lanes in 7/9/27-entry rows), sums in
// the row's column order (bitwise reproducible), and trades bytes for FP64
// work: per-node quantities (primitives, a p^-z, Phi, eta, E + p; in the FP32
// record of mixed mode also the flux f(U)) are computed once per stage in
// k_prep and gathered; |c_ij|, 1/|c_ij|, m_ij/m_j and m_ji/m_i are static
// per-edge arrays; (f(U_j) - f(U_i)) c_ij is computed once per edge in k_visc
// and reused by k_low; the limiter directions P_ij are stored.
//
// Work that cannot change a result is skipped, exactly: an edge between two
// bit-identical states takes the closed form of its values; a node record made
// from the same state bits is kept, and an edge between two kept states that
// were equal at the previous stage keeps its stored values; a row none of whose
// neighbours differs has P_ij = 0 and every limiter 1; a limiter pass leaves
// its remainder (1 - l) P_ij as the factor 1 - l (nothing is read where it is
// 0); a row whose limiters are all 1 stores none and says so in a flag.
#include "integer_fp64.cuh"
#include "../../include/euler_hyp.h"
#include "kernels.cuh"

#include <cooperative_groups.h>
#include <cooperative_groups/scan.h>

#include <algorithm>
#include <cmath>
#include <type_traits>

namespace eh {

// threads (= rows) per block of the row kernels: chosen per kernel at run time
// (eh_create's defaults, eh_autotune, eh_set_launch_shape), at most TPB_MAX

__host__ __device__ inline unsigned nblocks(int64_t n, int tpb) { return (unsigned)((n + tpb - 1) / tpb); }

// ---------------------------------------------------------------------------
// comparisons and min/max of doubles of known sign, on the bit patterns: a
// non-negative double orders like its bit pattern read as a signed 64-bit
// integer, and every negative double reads as a negative integer. An FP64
// compare or min/max issues on the FP64 pipe (2 lanes per SM and clock on
// GB300); the integer form runs on the ALUs. No operand is NaN on these paths.
// ---------------------------------------------------------------------------
__device__ __forceinline__ long long dbits(double x) { return __double_as_longlong(x); }
// x > y and x < y for y > 0, x of either sign
__device__ __forceinline__ bool gt_pos(double x, double y) { return dbits(x) > dbits(y); }
__device__ __forceinline__ bool lt_pos(double x, double y) { return dbits(x) < dbits(y); }
// an integer key with the order of the doubles (either sign)
__device__ __forceinline__ long long order_key(double x) {
  const long long b = dbits(x);
  return b ^ ((b >> 63) & 0x7FFFFFFFFFFFFFFFLL);
}
// max(x, 0); a > b and max(a, b) for a, b >= 0 (FP32: the plain instructions)
__device__ __forceinline__ double pos_part(double x) { return dbits(x) > 0 ? x : 0.0; }
__device__ __forceinline__ float pos_part(float x) { return fmaxf(x, 0.0f); }
__device__ __forceinline__ bool gt_nonneg(double a, double b) { return dbits(a) > dbits(b); }
__device__ __forceinline__ bool gt_nonneg(float a, float b) { return a > b; }
__device__ __forceinline__ double max_nonneg(double a, double b) { return dbits(a) > dbits(b) ? a : b; }
__device__ __forceinline__ float max_nonneg(float a, float b) { return fmaxf(a, b); }
// x > 0 and x < 0 (strict: false for both zeros)
__device__ __forceinline__ bool pos_strict(double x) { return dbits(x) > 0; }
__device__ __forceinline__ bool neg_strict(double x) { return dbits(x) < 0 && (dbits(x) << 1) != 0; }
// min(max(x, 0), 1)
__device__ __forceinline__ double clamp01(double x) { return dbits(x) <= 0 ? 0.0 : (gt_pos(x, 1.0) ? 1.0 : x); }
// |x| by clearing the sign bit
__device__ __forceinline__ double abs_bits(double x) {
  return __longlong_as_double(dbits(x) & 0x7FFFFFFFFFFFFFFFLL);
}
__device__ __forceinline__ float abs_bits(float x) { return fabsf(x); }

// x rounded towards zero to FP32 on the integer units (relative error 2^-23;
// 0 below 2^-126, +-inf from 2^127 on and for NaN): an FP64 -> FP32 conversion
// instruction takes part of an FP64 issue slot, this takes none
__device__ __forceinline__ float trunc_f32(double x) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const unsigned e = (hi >> 20) & 0x7ffu, sg = hi & 0x80000000u;
  unsigned r = ((__funnelshift_l(lo, hi, 3) - (384u << 23)) & 0x7fffffffu) | sg;
  if (e < 897u) r = sg;
  if (e > 1149u) r = sg | 0x7f800000u;
  return __uint_as_float(r);
}

// 256-bit accesses (sm_100 on): a lane's 32-byte sector in one instruction.
// Lanes of a row kernel read sectors of different lines (rows are 64 to 288
// bytes apart), so L1 serves one lane's line at a time whatever the width:
// with 8-byte loads and stores the viscosity kernel ran its L1 at 74-81 % and
// wrote five times the sectors it had values for. The compiler may move a load
// across stores: each is of data that the kernel does not write, or (k_prep's
// old record) its values decide a branch that the stores lie behind.
__device__ __forceinline__ void ld4(const double *p, double &a, double &b, double &c, double &d) {
  asm("ld.global.v4.f64 {%0,%1,%2,%3}, [%4];" : "=d"(a), "=d"(b), "=d"(c), "=d"(d) : "l"(p));
}
__device__ __forceinline__ void ld4(const float *p, float &a, float &b, float &c, float &d) {
  const float4 v = *reinterpret_cast<const float4 *>(p);
  a = v.x;
  b = v.y;
  c = v.z;
  d = v.w;
}
__device__ __forceinline__ void st4(double *p, double a, double b, double c, double d) {
  asm volatile("st.global.v4.f64 [%0], {%1,%2,%3,%4};" ::"l"(p), "d"(a), "d"(b), "d"(c), "d"(d) : "memory");
}
__device__ __forceinline__ void ld8(const float *p, float *v) {
  asm("ld.global.v8.f32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
      : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7])
      : "l"(p));
}
__device__ __forceinline__ void st8(float *p, const float *v) {
  asm volatile("st.global.v8.f32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"l"(p), "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]),
               "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7])
               : "memory");
}
__device__ __forceinline__ void ld2(const double *p, double &a, double &b) {
  const double2 v = *reinterpret_cast<const double2 *>(p);
  a = v.x;
  b = v.y;
}
// a state vector of stride Layout::SP (2D: one sector; 3D: 48 bytes)
template <int DIM> __device__ __forceinline__ void load_vec(const double *p, double *v) {
  if constexpr (DIM == 2) {
    ld4(p, v[0], v[1], v[2], v[3]);
  } else {
    ld2(p, v[0], v[1]);
    ld2(p + 2, v[2], v[3]);
    v[4] = p[4];
  }
}
template <int DIM> __device__ __forceinline__ void store_vec(double *p, const double *v) {
  if constexpr (DIM == 2) {
    st4(p, v[0], v[1], v[2], v[3]);
  } else {
    reinterpret_cast<double2 *>(p)[0] = make_double2(v[0], v[1]);
    reinterpret_cast<double2 *>(p)[1] = make_double2(v[2], v[3]);
    p[4] = v[4];
  }
}
// the state of a node from its FP64 record
template <int DIM> __device__ __forceinline__ void load_rec_state(const double *R, double *u) {
  ld4(R, u[0], u[1], u[2], u[3]);
  if constexpr (DIM == 3) u[4] = R[4];
}

// the per-entry viscosity quantities (layout: EdgeLayout)
template <int DIM, typename T> __device__ __forceinline__ T *w_slot(const Work &w, int64_t k) {
  return (T *)w.vw + k * EdgeLayout<DIM, T>::SPW;
}
template <int DIM, typename T> __device__ __forceinline__ T *d_ptr(const Work &w, int64_t k) {
  return EdgeLayout<DIM, T>::packed ? w_slot<DIM, T>(w, k) + EdgeLayout<DIM, T>::D : (T *)w.vad + 2 * k + 1;
}
// w_ij (S values), a_ij and d_ij of entry k
template <int DIM, typename T>
__device__ __forceinline__ void store_edge(const Work &w, int64_t k, const T *wv, T a, T d) {
  constexpr int S = DIM + 2;
  if constexpr (sizeof(T) == 4) {
    float v[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int s = 0; s < S; ++s) v[s] = wv[s];
    v[S] = a;
    v[S + 1] = d;
    st8(w_slot<DIM, T>(w, k), v);
  } else if constexpr (DIM == 3) {
    st4(w_slot<DIM, T>(w, k), wv[0], wv[1], wv[2], wv[3]);
    st4(w_slot<DIM, T>(w, k) + 4, wv[S - 1], a, d, 0.0);
  } else {
    st4(w_slot<DIM, T>(w, k), wv[0], wv[1], wv[2], wv[3]);
    reinterpret_cast<double2 *>(w.vad)[k] = make_double2(a, d);
  }
}
template <int DIM, typename T>
__device__ __forceinline__ void load_edge(const Work &w, int64_t k, T *wv, T &a, T &d) {
  constexpr int S = DIM + 2;
  if constexpr (sizeof(T) == 4) {
    float v[8];
    ld8(w_slot<DIM, T>(w, k), v);
#pragma unroll
    for (int s = 0; s < S; ++s) wv[s] = v[s];
    a = v[S];
    d = v[S + 1];
  } else if constexpr (DIM == 3) {
    double z;
    ld4(w_slot<DIM, T>(w, k), wv[0], wv[1], wv[2], wv[3]);
    ld4(w_slot<DIM, T>(w, k) + 4, wv[S - 1], a, d, z);
  } else {
    ld4(w_slot<DIM, T>(w, k), wv[0], wv[1], wv[2], wv[3]);
    ld2((const double *)w.vad + 2 * k, a, d);
  }
}
// the entry k of an edge between equal states: w = 0, a = 0, and d
template <int DIM, typename T> __device__ __forceinline__ void store_zero_edge(const Work &w, int64_t k, T d) {
  T z[DIM + 2];
#pragma unroll
  for (int s = 0; s < DIM + 2; ++s) z[s] = T(0);
  store_edge<DIM, T>(w, k, z, T(0), d);
}
// c_ij, |c_ij| and 1/|c_ij| of entry k (MeshView::geo)
template <int DIM, typename T>
__device__ __forceinline__ void load_geo(const MeshView &m, int64_t k, T *c, T &cn, T &ci) {
  const T *g = (const T *)m.geo + 4 * k;
  if constexpr (DIM == 2) {
    ld4(g, c[0], c[1], cn, ci);
  } else {
    ld4(g, c[0], c[1], c[2], cn);
    ci = ((const T *)m.geo_inv)[k];
  }
}

// ---------------------------------------------------------------------------
// roots and powers for gamma = 7/5 (division-free Newton iterations from an
// FP32 seed; two steps take the ~2^-21 seed error below double rounding)
// ---------------------------------------------------------------------------

// x^(-1/5): Newton's method on r^-5 = x, r <- r (6 - x r^5) / 5.
__device__ __forceinline__ double rroot5(double x) {
  if (!(gt_pos(x, 1e-30) && lt_pos(x, 1e30))) return pow(x, -0.2);
  double r = (double)exp2f(-0.2f * log2f((float)x));
#pragma unroll
  for (int it = 0; it < 2; ++it) {
    double r2 = r * r;
    double r5 = r2 * r2 * r;
    r = r * (6.0 - x * r5) * 0.2;
  }
  return r;
}

// x^(-1/7): Newton's method on r^-7 = x, r <- r (8 - x r^7) / 7.
__device__ __forceinline__ double rroot7(double x) {
  if (!(gt_pos(x, 1e-30) && lt_pos(x, 1e30))) return pow(x, -1.0 / 7.0);
  double r = (double)exp2f((-1.0f / 7.0f) * log2f((float)x));
#pragma unroll
  for (int it = 0; it < 2; ++it) {
    double r2 = r * r;
    double r7 = r2 * r2 * r2 * r;
    r = r * (8.0 - x * r7) * (1.0 / 7.0);
  }
  return r;
}

// rho^gamma
__device__ __forceinline__ double pow_gamma(const Params &p, double rho) {
  if (p.gamma75) {
    double r = rroot5(rho);  // rho^(-1/5); rho^(7/5) = rho^2 r^3
    return rho * rho * (r * r * r);
  }
  return pow(rho, p.gamma);
}

// rho^(gamma - 1)
__device__ __forceinline__ double pow_gamma_m1(const Params &p, double rho) {
  if (p.gamma75) {
    double r = rroot5(rho);  // rho^(2/5) = rho r^3
    return rho * (r * r * r);
  }
  return pow(rho, p.gamma - 1.0);
}

// ---------------------------------------------------------------------------
// Sec. 3.1: guaranteed upper bound on the maximum wave speed
// ---------------------------------------------------------------------------
// Two-rarefaction pressure p_tr >= p* (1 < gamma <= 5/3), then the outer wave
// speeds of the 1- and 3-waves evaluated at p_tr. Inputs per side: normal
// velocity, p, a, a p^-z, 1/p.
template <typename T>
__device__ __forceinline__ T lambda_max(const Params &p, T unl, T pl, T al, T azl, T ipl, T unr, T pr, T ar, T azr,
                                        T ipr) {
  T num = al + ar - T(0.5) * T(p.gm1) * (unr - unl);
  num = pos_part(num);
  T x = num / (azl + azr);
  T ptr;
  if (p.gamma75) {
    T x2 = x * x;
    T x4 = x2 * x2;
    ptr = x4 * x2 * x;  // x^(2 gamma/(gamma-1)) = x^7
  } else {
    ptr = pow(x, T(p.inv_z));
  }
  const T ks = T(p.kshock);
  T sl = gt_nonneg(ptr, pl) ? sqrt(T(1) + ks * (ptr - pl) * ipl) : T(1);
  T sr = gt_nonneg(ptr, pr) ? sqrt(T(1) + ks * (ptr - pr) * ipr) : T(1);
  T lam1 = unl - al * sl;
  T lam3 = unr + ar * sr;
  return max_nonneg(pos_part(-lam1), pos_part(lam3));
}

// a + b, a - b, |a| + |b| on the integer units (ALU) or the FP64 pipe: the same values
template <bool ALU> __device__ __forceinline__ double add_on(double a, double b) {
  if constexpr (ALU) return add_alu(a, b); else return __dadd_rn(a, b);
}
template <bool ALU> __device__ __forceinline__ double sub_on(double a, double b) {
  if constexpr (ALU) return sub_alu(a, b); else return __dsub_rn(a, b);
}
template <bool ALU> __device__ __forceinline__ double add_abs_on(double a, double b) {
  if constexpr (ALU) return add_abs_alu(a, b); else return __dadd_rn(abs_bits(a), abs_bits(b));
}
// (FP32: the plain instructions)
template <bool ALU> __device__ __forceinline__ float add_on(float a, float b) { return a + b; }
template <bool ALU> __device__ __forceinline__ float sub_on(float a, float b) { return a - b; }
template <bool ALU> __device__ __forceinline__ float add_abs_on(float a, float b) { return fabsf(a) + fabsf(b); }

// a and p of a node as an FP32 pair in one FP64 slot of its record (Rec::F32),
// for lambda_max_sel; a = NaN when a, p or a p^-z could leave FP32's range
__device__ __forceinline__ double pack_f32(double a, double pr, double az) {
  const bool ok = gt_pos(a, 1e-15) && lt_pos(a, 1e15) && gt_pos(pr, 1e-25) && lt_pos(pr, 1e25) && gt_pos(az, 1e-25) &&
                  lt_pos(az, 1e25);
  const float af = ok ? __double2float_rn(a) : __int_as_float(0x7fffffff);
  return __hiloint2double(__float_as_int(__double2float_rn(pr)), __float_as_int(af));
}
__device__ __forceinline__ float2 unpack_f32(double x) {
  return make_float2(__int_as_float(__double2loint(x)), __int_as_float(__double2hiint(x)));
}

// lambda_max in FP64, evaluated only where it can matter; the value is that of
// lambda_max above, bit for bit. The result is the larger of two outer speeds
// (a_l s_l - u_l and u_r + a_r s_r), each with s = 1 unless p_tr exceeds that
// side's pressure. FP32 intervals around both decide, where they are clear,
// which speed is the larger (the other side's root is not evaluated) and
// whether p_tr stays below the pressure there (then neither p_tr -- a division
// and a power -- nor a root is). An FP64 instruction costs 76 FP32 ones on this
// part, and neighbouring rows agree on their decisions, so the intervals cost
// little against the ~25 of 64 FP64 issue slots an edge that they save.
// Errors, u = 2^-24: a and p are rounded (u), a p^-z, v.c and 1/|c| truncated
// (2u); normal velocities 5u; the numerator of p_tr 6u of its terms'
// magnitudes (gamma <= 5/3); the quotient 8u more; the seventh power (or exp2
// of inv_z log2) multiplies the relative error by 7 (inv_z). A v.c below 2^-126 is
// truncated to 0, which moves a normal velocity by up to 2^-126 / |c|: that has to
// stay below u of the speeds. Anything unclear, or out of FP32's range (a = NaN),
// takes the full evaluation.
template <bool ALU>
__device__ __forceinline__ double lambda_max_sel(const Params &p, double vcl, double vcr, double ci, double pl, double al,
                                                 double azl, double ipl, float2 fl, double pr, double ar, double azr,
                                                 double ipr, float2 fr) {
  constexpr float u = 5.9604645e-8f;  // 2^-24
  const float cif = trunc_f32(ci);
  const float ulf = trunc_f32(vcl) * cif, urf = trunc_f32(vcr) * cif;
  const float num_f = fl.x + fr.x - 0.5f * p.gm1_f * (urf - ulf);
  const float mag = fl.x + fr.x + fabsf(ulf) + fabsf(urf);
  const float en = __fdividef(6.0f * u * mag, num_f);  // relative error of the numerator
  const float xf = __fdividef(num_f, trunc_f32(azl) + trunc_f32(azr));
  float ptr_f, rel;
  if (p.gamma75) {
    const float x2 = xf * xf;
    ptr_f = x2 * x2 * x2 * xf;
    rel = 7.5f * en + 80.0f * u;
  } else {
    const float lg = log2f(xf);
    ptr_f = exp2f(p.inv_z_f * lg);
    rel = 1.2f * p.inv_z_f * (en + 12.0f * u + 4.0f * u * fabsf(lg)) + 24.0f * u;
  }
  bool left = false, two = true, need = true;
  if (num_f > 0.0f && en < 0.01f && rel < 0.05f && ptr_f > 1e-30f && ptr_f < 1e30f && mag < 1e18f &&
      4e-31f * cif < mag) {
    const float plo = ptr_f * (1.0f - rel), phi = ptr_f * (1.0f + rel);
    const float ql = __fdividef(1.0f, fl.y), qr = __fdividef(1.0f, fr.y);
    constexpr float r8 = 8.0f * u;
    const float kf = p.kshock_f;
    // brackets of s - 1's argument; 1 -/+ 8u covers p, 1/p and the products
    const float sl_lo = sqrtf(1.0f + kf * fmaxf(plo * ql * (1.0f - r8) - 1.0f - r8, 0.0f));
    const float sl_hi = sqrtf(1.0f + kf * fmaxf(phi * ql * (1.0f + r8) - 1.0f + r8, 0.0f));
    const float sr_lo = sqrtf(1.0f + kf * fmaxf(plo * qr * (1.0f - r8) - 1.0f - r8, 0.0f));
    const float sr_hi = sqrtf(1.0f + kf * fmaxf(phi * qr * (1.0f + r8) - 1.0f + r8, 0.0f));
    const float el = 12.0f * u * (fl.x * sl_hi + fabsf(ulf)), er = 12.0f * u * (fr.x * sr_hi + fabsf(urf));
    const bool L = fl.x * sl_lo - ulf - el > fr.x * sr_hi + urf + er;
    const bool R = fr.x * sr_lo + urf - er > fl.x * sl_hi - ulf + el;
    if (L || R) {
      left = L;
      two = false;
      need = !(phi < (L ? fl.y : fr.y) * (1.0f - r8));
    }
  }
  // the selected side (the right one first when both are evaluated)
  const double as = left ? al : ar;
  if (!need) {
    const double us = __dmul_rn(left ? -vcl : vcr, ci);
    return pos_part(add_on<ALU>(us, as));
  }
  const double unl = __dmul_rn(vcl, ci), unr = __dmul_rn(vcr, ci);
  double num = __fma_rn(-(0.5 * p.gm1), sub_on<ALU>(unr, unl), add_on<ALU>(al, ar));
  num = pos_part(num);
  const double x = div_alu(num, add_on<ALU>(azl, azr));
  double ptr;
  if (p.gamma75) {
    const double x2 = x * x;
    const double x4 = x2 * x2;
    ptr = x4 * x2 * x;  // x^(2 gamma/(gamma-1)) = x^7
  } else {
    ptr = pow(x, p.inv_z);
  }
  const double ks = p.kshock;
  const double ps = left ? pl : pr, ips = left ? ipl : ipr, us = left ? -unl : unr;
  const double ss = gt_nonneg(ptr, ps) ? sqrt_alu(1.0 + ks * sub_on<ALU>(ptr, ps) * ips) : 1.0;
  double lam = pos_part(us + as * ss);
  if (two) {
    const double so = gt_nonneg(ptr, pl) ? sqrt(1.0 + ks * (ptr - pl) * ipl) : 1.0;
    lam = max_nonneg(lam, pos_part(-(unl - al * so)));
  }
  return lam;
}

// ---------------------------------------------------------------------------
// Sec. 3.3: line search for the largest l in [0,1] within the local bounds
// ---------------------------------------------------------------------------
template <int DIM>
__device__ __forceinline__ double psi(const Params &p, const double *ub, const double *P, double l, double phimin) {
  constexpr int S = DIM + 2;
  double u[S];
#pragma unroll
  for (int s = 0; s < S; ++s) u[s] = ub[s] + l * P[s];
  double m2 = 0.0;
#pragma unroll
  for (int k = 0; k < DIM; ++k) m2 += u[1 + k] * u[1 + k];
  double eps = u[S - 1] - m2 / (2.0 * u[0]);
  return eps - phimin * pow_gamma(p, u[0]);
}

template <int DIM>
__device__ __forceinline__ double dpsi(const Params &p, const double *ub, const double *P, double l, double phimin) {
  constexpr int S = DIM + 2;
  double u[S];
#pragma unroll
  for (int s = 0; s < S; ++s) u[s] = ub[s] + l * P[s];
  double irho = 1.0 / u[0];
  double v2 = 0.0, vP = 0.0;
#pragma unroll
  for (int k = 0; k < DIM; ++k) {
    double v = u[1 + k] * irho;
    v2 += v * v;
    vP += v * P[1 + k];
  }
  double deps = P[S - 1] - vP + 0.5 * v2 * P[0];
  return deps - phimin * p.gamma * pow_gamma_m1(p, u[0]) * P[0];
}

constexpr int LINE_SEARCH_ITERATIONS = 6;

// gamma = 7/5: psi(l) as psi() above, also returning r = rho(l)^(-1/5), so
// that psi'(lR) reuses the root of the psi(lR) evaluation (rho^(2/5) = rho r^3);
// the values are those of psi()/dpsi() bit for bit.
template <int DIM>
__device__ __forceinline__ double psi_g75(const double *ub, const double *P, double l, double phimin, double *r_out) {
  constexpr int S = DIM + 2;
  double u[S];
#pragma unroll
  for (int s = 0; s < S; ++s) u[s] = ub[s] + l * P[s];
  double m2 = 0.0;
#pragma unroll
  for (int k = 0; k < DIM; ++k) m2 += u[1 + k] * u[1 + k];
  const double eps = u[S - 1] - div_alu(m2, 2.0 * u[0]);
  const double r = rroot5(u[0]);
  *r_out = r;
  return eps - phimin * (u[0] * u[0] * (r * r * r));
}

template <int DIM>
__device__ __forceinline__ double dpsi_g75(const double *ub, const double *P, double l, double r, double phimin) {
  constexpr int S = DIM + 2;
  double u[S];
#pragma unroll
  for (int s = 0; s < S; ++s) u[s] = ub[s] + l * P[s];
  const double irho = div_alu(1.0, u[0]);
  double v2 = 0.0, vP = 0.0;
#pragma unroll
  for (int k = 0; k < DIM; ++k) {
    const double v = u[1 + k] * irho;
    v2 += v * v;
    vP += v * P[1 + k];
  }
  const double deps = P[S - 1] - vP + 0.5 * v2 * P[0];
  return deps - phimin * 1.4 * (u[0] * (r * r * r)) * P[0];
}

// The line search in two parts. line_search_start takes every exit that needs
// no iteration (P = 0, the density limit, the entropy bound met at that limit,
// psi(0) <= 0) and otherwise returns the bracket [0, l] with psi at both ends;
// line_search_iterate runs the fixed number of secant (feasible side) / Newton
// (infeasible side) steps on that bracket and returns its feasible end. For
// gamma = 7/5 the root of rho is shared between psi(lR) and psi'(lR), and psi
// is evaluated once when the Newton and secant points coincide.
struct LsBracket {
  double l;   // the result when done; else the right end of the bracket
  double pl;  // psi(0) > 0
  double pr;  // psi(l) < 0
  double rR;  // rho(l)^(-1/5) (gamma = 7/5)
  bool done;
};

// the exits without psi: P = 0, the density limit l, (gamma = 7/5) the entropy
// bound met there; otherwise done = false and l is set. phimin5 = phimin^5 (used
// by the gamma = 7/5 fast check only).
template <int DIM>
__device__ __forceinline__ LsBracket line_search_bracket(const Params &p, const double *ub, const double *P, double rmin,
                                                         double rmax, double phimin5) {
  constexpr int S = DIM + 2;
  LsBracket b{1.0, 0.0, 0.0, 0.0, true};
  // P = 0 (every edge whose previous limiter was 1, uniform flow): every l gives
  // the same state; the largest, 1, is returned without any FP64 work
  bool zero = true;
#pragma unroll
  for (int s = 0; s < S; ++s) zero &= (__double_as_longlong(P[s]) << 1) == 0;
  if (zero) return b;
  // (compares on the bit patterns; the density bounds are positive)
  double l = 1.0;
  const double rb = ub[0], rp = P[0];
  // density: the division is needed only when l = 1 leaves [rho_min, rho_max]
  if (pos_strict(rp)) {
    if (gt_pos(rb + rp, rmax)) l = clamp01(div_alu(rmax - rb, rp));
  } else if (neg_strict(rp)) {
    if (lt_pos(rb + rp, rmin)) l = clamp01(div_alu(rmin - rb, rp));
  }
  b.l = l;
  if (p.gamma75) {
    // entropy at l: psi(l) >= 0 <=> (eps rho)^5 >= Phi_min^5 rho^12 when
    // eps rho > 0 -- no division and no root on the common path
    double u[S];
#pragma unroll
    for (int s = 0; s < S; ++s) u[s] = ub[s] + l * P[s];
    const double rho = u[0];
    if (gt_pos(rho, 1e-6) && lt_pos(rho, 1e6)) {
      double m2 = 0.0;
#pragma unroll
      for (int q = 0; q < DIM; ++q) m2 += u[1 + q] * u[1 + q];
      const double er = u[S - 1] * rho - 0.5 * m2;
      if (pos_strict(er)) {
        const double r2 = rho * rho, r4 = r2 * r2, r12 = r4 * r4 * r4;
        const double e2 = er * er;
        const double lhs = e2 * e2 * er, rhs = phimin5 * r12;  // lhs > 0, rhs >= 0
        if (lt_pos(rhs, 1e300) && dbits(lhs) >= dbits(rhs)) return b;
      }
    }
  }
  b.done = false;
  return b;
}

template <int DIM>
__device__ LsBracket line_search_start(const Params &p, const double *ub, const double *P, double rmin, double rmax,
                                       double phimin, double phimin5) {
  LsBracket b = line_search_bracket<DIM>(p, ub, P, rmin, rmax, phimin5);
  if (b.done) return b;
  b.done = true;
  if (p.gamma75) {
    double r0;
    b.pr = psi_g75<DIM>(ub, P, b.l, phimin, &b.rR);
    if (!neg_strict(b.pr)) return b;
    b.pl = psi_g75<DIM>(ub, P, 0.0, phimin, &r0);
  } else {
    b.pr = psi<DIM>(p, ub, P, b.l, phimin);
    if (!neg_strict(b.pr)) return b;
    b.pl = psi<DIM>(p, ub, P, 0.0, phimin);
  }
  if (!pos_strict(b.pl)) {
    b.l = 0.0;
    return b;
  }
  b.done = false;
  return b;
}

template <int DIM>
__device__ double line_search_iterate(const Params &p, const double *ub, const double *P, double phimin,
                                      const LsBracket &b) {
  double lL = 0.0, lR = b.l, pl = b.pl, pr = b.pr, rR = b.rR;
  for (int it = 0; it < LINE_SEARCH_ITERATIONS; ++it) {
    double ls = lL + div_alu(pl * (lR - lL), pl - pr);
    double dr = p.gamma75 ? dpsi_g75<DIM>(ub, P, lR, rR, phimin) : dpsi<DIM>(p, ub, P, lR, phimin);
    double ln = neg_strict(dr) ? lR - div_alu(pr, dr) : lR;
    if (order_key(ln) < order_key(ls)) ln = ls;
    double ps, pn, rs, rn;
    if (p.gamma75) {
      ps = psi_g75<DIM>(ub, P, ls, phimin, &rs);
      pn = ps;
      rn = rs;
      if (dbits(ln) != dbits(ls)) pn = psi_g75<DIM>(ub, P, ln, phimin, &rn);
    } else {
      ps = psi<DIM>(p, ub, P, ls, phimin);
      pn = psi<DIM>(p, ub, P, ln, phimin);
      rn = 0.0;
    }
    if (!neg_strict(ps)) {
      lL = ls;
      pl = ps;
    }
    if (neg_strict(pn)) {
      lR = ln;
      pr = pn;
      rR = rn;
    } else {
      lL = ln;
      pl = pn;
    }
  }
  return lL;
}

// The line search by pairs of neighbouring lanes that hold the same search, with
// line_search_start's and line_search_iterate's values bit for bit: psi(l) and
// psi(0), the secant's and Newton's divisions, and psi at their two points are
// evaluated side by side (52 instead of 85 FP64 instructions an iteration, at
// 63 cycles each). For queues that leave the chip idle; a full one is faster
// with a search per lane. gamma = 7/5 (with another gamma the powers are most of
// the time). All lanes of a warp call both.
template <int DIM>
__device__ __forceinline__ LsBracket line_search_start_pair(const Params &p, const double *ub, const double *P,
                                                            double rmin, double rmax, double phimin, double phimin5) {
  constexpr unsigned all = 0xffffffffu;
  const bool odd = threadIdx.x & 1;
  LsBracket b = line_search_bracket<DIM>(p, ub, P, rmin, rmax, phimin5);
  double r;
  const double mine = psi_g75<DIM>(ub, P, odd ? 0.0 : b.l, phimin, &r);
  const double other = __shfl_xor_sync(all, mine, 1), r_other = __shfl_xor_sync(all, r, 1);
  b.pr = odd ? other : mine;
  b.pl = odd ? mine : other;
  b.rR = odd ? r_other : r;
  if (!b.done && !neg_strict(b.pr)) b.done = true;
  if (!b.done && !pos_strict(b.pl)) {
    b.l = 0.0;
    b.done = true;
  }
  return b;
}

template <int DIM>
__device__ __forceinline__ double line_search_iterate_pair(const double *ub, const double *P, double phimin,
                                                           const LsBracket &b) {
  constexpr unsigned all = 0xffffffffu;
  const bool odd = threadIdx.x & 1;
  bool done = b.done;
  double lL = 0.0, lR = b.l, pl = b.pl, pr = b.pr, rR = b.rR, result = b.l;
  for (int it = 0; it < LINE_SEARCH_ITERATIONS; ++it) {
    if (__all_sync(all, done)) break;
    const double dr = dpsi_g75<DIM>(ub, P, lR, rR, phimin);
    // (a finished search divides 1 by 1: a zero would take the division's slow path)
    const double q = div_alu(done ? 1.0 : odd ? pr : pl * (lR - lL), done ? 1.0 : odd ? dr : pl - pr);
    const double mine = odd ? (neg_strict(dr) ? lR - q : lR) : lL + q;
    const double other = __shfl_xor_sync(all, mine, 1);
    const double ls = odd ? other : mine;
    double ln = odd ? mine : other;
    if (order_key(ln) < order_key(ls)) ln = ls;
    double r_mine;
    const double p_mine = psi_g75<DIM>(ub, P, odd ? ln : ls, phimin, &r_mine);
    const double p_other = __shfl_xor_sync(all, p_mine, 1), r_other = __shfl_xor_sync(all, r_mine, 1);
    const double ps = odd ? p_other : p_mine, pn = odd ? p_mine : p_other, rn = odd ? r_mine : r_other;
    if (!neg_strict(ps)) {
      lL = ls;
      pl = ps;
    }
    if (neg_strict(pn)) {
      lR = ln;
      pr = pn;
      rR = rn;
    } else {
      lL = ln;
      pl = pn;
    }
    if (!done) result = lL;
  }
  return result;
}

// ---------------------------------------------------------------------------
// Pre-decision of the entropy test at l = 1: with u = ub + P, does
// rho E - |m|^2/2 >= Phi_min rho^(gamma+1) hold (gamma = 7/5: fifth powers of
// both sides), for the FP64 inputs, in exact arithmetic? +1: it holds, -1: it
// fails, each with a margin far beyond the FP64 test's own rounding (~1e-15),
// so that it is the outcome the FP64 test reaches; 0: too close to call, or
// outside the range of the FP32 powers. Two levels, both on the FP32 units (76
// instructions for one FP64 issue slot), where the FP64 test takes 17 slots
// and a warp with one open lane pays for all:
//  - FP32 with error bounds built from the inputs' magnitudes (relative margin
//    ~1e-5 at Mach 3);
//  - gamma = 7/5: pairs of FP32 values (48 bits; margin ~1e-12), which leave
//    the FP64 test to states that agree to their last bits.
// ---------------------------------------------------------------------------
struct RowF32 {
  float u[5];  // ub truncated to FP32
  float phi;   // Phi_min^5 (gamma = 7/5) or Phi_min, truncated; 0: no pre-decision for the row
};
// The row's FP32 data. Rows whose density bounds, or whose smallest and largest
// Phi over the stencil, agree to 2^17 ulps (3e-11) skip the pre-decision: their
// states differ from their neighbours' by rounding (on the Mach-3 cylinder most
// such rows by a few ulps, psi(1) within 1e-13 of 0), or the flow is isentropic
// there and psi(1) is rounding (a vortex in a uniform stream).
template <int DIM>
__device__ __forceinline__ RowF32 row_f32(const Params &p, const double *ub, double rmin, double rmax, double phimin,
                                          double phimax, double phimin5) {
  RowF32 r;
#pragma unroll
  for (int s = 0; s < DIM + 2; ++s) r.u[s] = 0.0f;
  r.phi = 0.0f;
  // 2^-40 <= Phi_min^5 <= 2^40 (gamma != 7/5: Phi_min itself)
  const double ph = p.gamma75 ? phimin5 : phimin;
  if (!(dbits(rmax) - dbits(rmin) > 1 << 17 && dbits(phimax) - dbits(phimin) > 1 << 17 &&
        gt_pos(ph, 9.094947017729282e-13) && lt_pos(ph, 1.099511627776e12)))
    return r;
#pragma unroll
  for (int s = 0; s < DIM + 2; ++s) r.u[s] = trunc_f32(ub[s]);
  r.phi = trunc_f32(ph);
  return r;
}

// sums of two FP32 values: relative error of an addition or a product at most
// 2^-44 (of the magnitudes added, resp. of the product)
struct Pair {
  float h, l;
};
__device__ __forceinline__ Pair quick_pair(float h, float l) {  // |h| >= |l|
  const float s = __fadd_rn(h, l);
  return Pair{s, __fsub_rn(l, __fsub_rn(s, h))};
}
__device__ __forceinline__ Pair two_sum(float a, float b) {
  const float s = __fadd_rn(a, b), t = __fsub_rn(s, a);
  return Pair{s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, t)), __fsub_rn(b, t))};
}
__device__ __forceinline__ Pair operator+(const Pair &a, const Pair &b) {
  Pair s = two_sum(a.h, b.h), t = two_sum(a.l, b.l);
  s = quick_pair(s.h, __fadd_rn(s.l, t.h));
  return quick_pair(s.h, __fadd_rn(s.l, t.l));
}
__device__ __forceinline__ Pair operator*(const Pair &a, const Pair &b) {
  const float q = __fmul_rn(a.h, b.h);
  float e = __fmaf_rn(a.h, b.h, -q);
  e = __fmaf_rn(a.h, b.l, __fmaf_rn(a.l, b.h, e));
  return quick_pair(q, e);
}
// x as a pair: the upper 24 significant bits, and the other 29 as an integer
// scaled by x's exponent. Relative error 2^-47 down to |x| = 2^-74, 2^-23 below,
// where the low part is left out (at most 2^-97, beside tested magnitudes of 2^-12
// and bounds of 2^-44 of them: nothing) and x itself is 0 below 2^-126
__device__ __forceinline__ Pair split_f32(double x) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const float h = trunc_f32(x);
  const int e = (int)((hi >> 20) & 0x7ffu) - 1023 - 52 + 127;  // biased FP32 exponent of the last place
  float l = e > 0 && e < 254 ? (float)(lo & 0x1fffffffu) * __int_as_float(e << 23) : 0.0f;
  if (hi & 0x80000000u) l = -l;
  return Pair{h, l};
}

// the second level (gamma = 7/5)
template <int DIM>
__device__ __forceinline__ int entropy_at_one_pair(const double *ub, const double *P, double phimin5) {
  constexpr int S = DIM + 2;
  constexpr float u44 = 5.684342e-14f;  // 2^-44
  Pair u[S];
  float A[S];
#pragma unroll
  for (int s = 0; s < S; ++s) {
    const Pair a = split_f32(ub[s]), b = split_f32(P[s]);
    u[s] = a + b;
    A[s] = fabsf(a.h) + fabsf(b.h);  // |u - exact| <= 2^-45 A
  }
  Pair m2{0.0f, 0.0f};
  float Am = 0.0f;
#pragma unroll
  for (int q = 0; q < DIM; ++q) {
    m2 = m2 + u[1 + q] * u[1 + q];
    Am += A[1 + q] * A[1 + q];
  }
  const Pair er = u[S - 1] * u[0] + Pair{-0.5f * m2.h, -0.5f * m2.l};
  const float B = 2.0f * u44 * (A[0] * A[S - 1] + Am);  // inputs 2^-45 each, operations 2^-44
  // 2^-12 <= er <= 2^12: the low parts of the powers stay above FP32's range
  if (!(er.h > 2.4414063e-4f && er.h < 4096.0f && B < 0.01f * er.h)) return 0;
  const Pair e2 = er * er, lhs = e2 * e2 * er;
  const Pair r2 = u[0] * u[0], r4 = r2 * r2, rhs = split_f32(phimin5) * (r4 * r4 * r4);
  const float rel = 6.0f * __fdividef(B, er.h) + u44 * (40.0f + 16.0f * __fdividef(A[0], u[0].h));
  const Pair d = lhs + Pair{-rhs.h, -rhs.l};
  const float tol = 1.1f * rel * fmaxf(lhs.h, rhs.h);
  return d.h > tol ? 1 : d.h < -tol ? -1 : 0;
}

// the first level; 2: undecided, but within the second level's range
template <int DIM>
__device__ __forceinline__ int entropy_at_one_f32(const Params &p, const RowF32 &r, const double *P) {
  constexpr int S = DIM + 2;
  constexpr float u24 = 5.9604645e-8f;  // 2^-24
  if (r.phi == 0.0f) return 0;
  float u[S], e[S];
#pragma unroll
  for (int s = 0; s < S; ++s) {
    const float pf = trunc_f32(P[s]);
    u[s] = r.u[s] + pf;
    // |u_f - u| <= 2^-24 (2 |ub| + 2 |P| + |u_f|) (two truncations, one add)
    e[s] = 5.0f * u24 * (fabsf(r.u[s]) + fabsf(pf));
  }
  const float rho = u[0], E = u[S - 1];
  // 2^-6 <= rho <= 2^6 with its error: rho^12 stays within FP32's range
  if (!(rho - e[0] >= 0.015625f && rho + e[0] <= 64.0f)) return 0;
  float m2h = 0.0f, em = 0.0f;
#pragma unroll
  for (int q = 0; q < DIM; ++q) {
    m2h += u[1 + q] * u[1 + q];
    em += fabsf(u[1 + q]) * e[1 + q] + 0.5f * e[1 + q] * e[1 + q];
  }
  m2h *= 0.5f;
  const float rE = rho * E;
  const float er = rE - m2h;
  // |er_f - er| <= propagated input errors + 8 roundings of the magnitudes
  const float B = 1.01f * (rho * e[S - 1] + fabsf(E) * e[0] + e[0] * e[S - 1] + em +
                           8.0f * u24 * (fabsf(rE) + m2h));
  const float elo = er - B, ehi = er + B;
  // 2^-24 <= er <= 2^24 with its error: er^5 stays within FP32's range
  if (!(elo >= 5.9604645e-8f && ehi <= 16777216.0f)) return 0;
  const float rlo = rho - e[0], rhi = rho + e[0];
  if (!p.gamma75) {
    // Phi_min rho^(gamma+1), 2 < gamma + 1 <= 8/3: the power as exp2(g log2),
    // |log2 rho| <= 6 (log2f and exp2f are within 2 units: 2 (6 g + 1) 2^-23 at most)
    const float g = p.gamma_f + 1.0f;
    const float rhs_lo = r.phi * exp2f(g * log2f(rlo)) * (1.0f - 128.0f * u24);
    const float rhs_hi = r.phi * exp2f(g * log2f(rhi)) * (1.0f + 128.0f * u24);
    return elo > rhs_hi ? 1 : ehi < rhs_lo ? -1 : 0;
  }
  const float l2 = elo * elo, h2 = ehi * ehi;
  const float lhs_lo = l2 * l2 * elo * (1.0f - 8.0f * u24);
  const float lhs_hi = h2 * h2 * ehi * (1.0f + 8.0f * u24);
  const float a2 = rlo * rlo, a4 = a2 * a2, b2 = rhi * rhi, b4 = b2 * b2;
  const float rhs_lo = r.phi * (a4 * a4 * a4) * (1.0f - 18.0f * u24);
  const float rhs_hi = r.phi * (b4 * b4 * b4) * (1.0f + 18.0f * u24);
  if (lhs_lo > rhs_hi) return 1;
  if (lhs_hi < rhs_lo) return -1;
  return 2;
}

// The common outcome of the line search, decided with a short branch-free
// sequence: P = 0, or l = 1 inside the density bounds and (gamma = 7/5) inside
// the entropy bound. Returns true exactly where line_search returns 1 through
// one of these exits; false leaves the entry to the full search. (A warp whose
// lanes took the search's other exits -- density clipping, psi evaluations,
// the secant/Newton loop -- inline would issue each of them for all 32 lanes.)
// The entropy test is pre-decided on the FP32 units and evaluated in FP64 only
// where that is too close to call. For another gamma than 7/5 only the
// pre-decision settles an entry here (l = 1 certain); the rest is left open.
// Measured: 246k cylinder, gamma = 1.3 (every entry with P_ij != 0 was queued),
// the queued searches of a pass 280 -> 175 us; gamma = 7/5, second level and
// truncated inputs: k_lim1 500 -> 422 us on the 998k cylinder, 822 -> 679 us on
// 375k rows in 3D, 191 -> 120 us on the sweep of 256 small cylinders.
template <int DIM>
__device__ __forceinline__ bool line_search_at_one(const Params &p, const double *ub, const double *P, double rmin,
                                                   double rmax, double phimin5, const RowF32 &rf) {
  constexpr int S = DIM + 2;
  bool zero = true;
#pragma unroll
  for (int s = 0; s < S; ++s) zero &= (__double_as_longlong(P[s]) << 1) == 0;
  if (zero) return true;
  // the compares below run on the bit patterns (all thresholds are positive);
  // rp = -0 may take the density test, which can only send the entry to the
  // full search
  const double rb = ub[0], rp = P[0];
  if (dbits(rp) > 0) {
    if (gt_pos(rb + rp, rmax)) return false;
  } else if (dbits(rp) < 0) {
    if (lt_pos(rb + rp, rmin)) return false;
  }
  int pre = entropy_at_one_f32<DIM>(p, rf, P);
  if (!p.gamma75) return pre > 0;
  if (pre == 2) pre = entropy_at_one_pair<DIM>(ub, P, phimin5);
  if (pre != 0) return pre > 0;
  double u[S];
#pragma unroll
  for (int s = 0; s < S; ++s) u[s] = ub[s] + P[s];
  const double rho = u[0];
  if (!(gt_pos(rho, 1e-6) && lt_pos(rho, 1e6))) return false;
  double m2 = 0.0;
#pragma unroll
  for (int q = 0; q < DIM; ++q) m2 += u[1 + q] * u[1 + q];
  const double er = u[S - 1] * rho - 0.5 * m2;
  if (!(dbits(er) > 0)) return false;
  const double r2 = rho * rho, r4 = r2 * r2, r12 = r4 * r4 * r4;
  const double e2 = er * er;
  const double lhs = e2 * e2 * er, rhs = phimin5 * r12;  // lhs > 0, rhs >= 0
  return lt_pos(rhs, 1e300) && dbits(lhs) >= dbits(rhs);
}

// Queues the line searches of row i's entries k0 + b for every bit b of 'mask'
// for k_ls_deferred: one atomic per group of converged lanes (normally once
// per warp and kernel). The queue holds nnz entries and a pass queues each
// entry at most once, so it cannot fill; the bounds check only guards memory
// (an overflow would be reported as EH_ERR_STATE).
__device__ __forceinline__ void defer_line_searches(const Work &w, int slot, int i, int64_t k0, uint64_t mask) {
  namespace cg = cooperative_groups;
  cg::coalesced_group g = cg::coalesced_threads();
  const unsigned cnt = (unsigned)__popcll(mask);
  const unsigned off = cg::exclusive_scan(g, cnt);
  const unsigned total = g.shfl(off + cnt, g.size() - 1);
  if (total == 0) return;
  unsigned base = 0;
  if (g.thread_rank() == 0) base = atomicAdd(&w.lsq_count[slot], total);
  base = g.shfl(base, 0) + off;
  while (mask) {
    const int b = __ffsll((long long)mask) - 1;
    mask &= mask - 1;
    if (base < w.lsq_cap)
      w.lsq[base++] = make_int2(i, (int)(k0 + b));
    else
      atomicExch(&w.st->err, 7);  // EH_ERR_STATE
  }
}

// ---------------------------------------------------------------------------
// flux f(U) = (m, m v^T + p I, v (E + p)) of one node (Sec. 2.1), row s =
// component, from its momentum, velocity, pressure and E + p
// ---------------------------------------------------------------------------
template <int DIM, typename T>
__device__ __forceinline__ void node_flux(const T *mv, const T *v, T pr, T H, T f[DIM + 2][DIM]) {
#pragma unroll
  for (int q = 0; q < DIM; ++q) f[0][q] = mv[q];
#pragma unroll
  for (int a = 0; a < DIM; ++a)
#pragma unroll
    for (int b = 0; b < DIM; ++b) f[1 + a][b] = mv[a] * v[b] + (a == b ? pr : T(0));
#pragma unroll
  for (int q = 0; q < DIM; ++q) f[DIM + 1][q] = v[q] * H;
}

// ---------------------------------------------------------------------------
// k_prep: node records (primitives and derived quantities), once per stage
// ---------------------------------------------------------------------------
// Bound by FP64 issue: the logarithm and the two roots are 60 of ~70 instructions
// a node (102 with the divisions and the square root on that pipe: 998k-vertex
// cylinder 200 -> 160 us, mixed 250 -> 207).
template <int DIM, typename T>
__global__ void __launch_bounds__(TPB_MAX) k_prep(MeshView m, Params p, const double *__restrict__ U,
                                              double *__restrict__ rec, T *__restrict__ vrec,
                                              unsigned char *__restrict__ rough,
                                              unsigned char *__restrict__ steady, const DevStatus *st) {
  constexpr int S = DIM + 2;
  using R = Rec<DIM>;
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= m.n || st->err) return;
  const unsigned char was_rough = rough[i];  // as the previous k_visc left it
  rough[i] = 0;  // set by k_visc where a neighbour's state differs
  double u[S];
#pragma unroll
  for (int s = 0; s < S; ++s) u[s] = U[(int64_t)s * m.n + i];
  double *Rr = rec + (int64_t)i * R::SIZE;
  {
    // the record (both precisions) is a function of U_i and gamma alone, so
    // where the stored one was made from the same bits it stands as it is:
    // nodes of a uniform region keep their state exactly from stage to stage
    // (every P_ij and increment is 0). The records start as NaN bit patterns,
    // which no admissible state matches.
    bool same = true;
    double old[S];
    load_rec_state<DIM>(Rr, old);
#pragma unroll
    for (int s = 0; s < S; ++s) same &= dbits(old[s]) == dbits(u[s]);
    steady[i] = same ? (unsigned char)(was_rough ? 1 : 3) : (unsigned char)0;
    if (same) return;
  }
  double rho = u[0];
  double irho = div_alu(1.0, rho);
  double v[DIM], m2 = 0.0;
#pragma unroll
  for (int k = 0; k < DIM; ++k) {
    v[k] = u[1 + k] * irho;
    m2 += u[1 + k] * u[1 + k];
  }
  double eps = u[S - 1] - 0.5 * m2 * irho;
  double pr = p.gm1 * eps;
  double a = sqrt_alu(p.gamma * pr * irho);
  double az, phi;
  if (p.gamma75) {
    az = a * rroot7(pr);
    double r = rroot5(rho);  // rho^(-1/5); rho^(-7/5) = r^7
    double r2 = r * r;
    phi = eps * (r2 * r2 * r2 * r);
  } else {
    az = a * pow(pr, -p.z);
    phi = eps * pow(rho, -p.gamma);
  }
  double eta = -rho * (log(phi) * p.inv_gm1);
  double r[R::SIZE];
#pragma unroll
  for (int q = 0; q < R::SIZE; ++q) r[q] = 0.0;
#pragma unroll
  for (int s = 0; s < S; ++s) r[s] = u[s];
#pragma unroll
  for (int k = 0; k < DIM; ++k) r[R::V + k] = v[k];
  r[R::P] = pr;
  r[R::A] = a;
  r[R::AZ] = az;
  r[R::IP] = div_alu(1.0, pr);
  r[R::PHI] = phi;
  r[R::ETA] = eta;
  r[R::H] = u[S - 1] + pr;
  r[R::IRHO] = irho;
  r[R::IEPS] = div_alu(1.0, eps);
  r[R::F32] = pack_f32(a, pr, az);
#pragma unroll
  for (int q = 0; q <= R::IEPS; q += 4) st4(Rr + q, r[q], r[q + 1], r[q + 2], r[q + 3]);
  if constexpr (!std::is_same<T, double>::value) {
    // the same record in the viscosity precision (mixed mode), with the flux
    T *Rv = vrec + (int64_t)i * R::VSIZE;
#pragma unroll
    for (int q = 0; q <= R::IEPS; ++q)
      if (q != R::F32) Rv[q] = (T)r[q];
    double f[S][DIM];
    node_flux<DIM, double>(u + 1, v, pr, r[R::H], f);
#pragma unroll
    for (int s = 0; s < S; ++s)
#pragma unroll
      for (int q = 0; q < DIM; ++q) Rv[R::F + s * DIM + q] = (T)f[s][q];
  }
}

// ---------------------------------------------------------------------------
// k_visc: Algorithm 1 step 1 -- d_ij (j > i, mirrored through the transpose
// index), the flux differences w_ij and a_ij of the indicator
// ---------------------------------------------------------------------------
// node i of an edge, as the row loop keeps it
template <int DIM, typename T> struct ViscNode {
  T v[DIM], mo[DIM], p, a, az, ip, eta, H;
  T f[DIM + 2][DIM], q[DIM];  // FP32: the flux and the entropy flux
  long long bits[DIM + 2];  // the FP64 state (the identical-state test compares FP64 bits in either precision)
  float2 f32;               // FP64: the FP32 pair of the record
  unsigned char steady;
  // FP64: from the first 16 values of a record
  __device__ __forceinline__ void from_record(const double *r) {
    using R = Rec<DIM>;
#pragma unroll
    for (int k = 0; k < DIM; ++k) {
      v[k] = r[R::V + k];
      mo[k] = r[1 + k];
    }
    p = r[R::P];
    a = r[R::A];
    az = r[R::AZ];
    ip = r[R::IP];
    eta = r[R::ETA];
    H = r[R::H];
    f32 = unpack_f32(r[R::F32]);
  }
};

// the first 16 values of a node's FP64 record (everything k_visc reads)
template <int DIM> __device__ __forceinline__ void load_rec(const Work &w, int i, double *r) {
  static_assert(Rec<DIM>::H < 16 && Rec<DIM>::SIZE % 4 == 0, "record layout");
  const double *R = w.rec + (int64_t)i * Rec<DIM>::SIZE;
#pragma unroll
  for (int q = 0; q < 16; q += 4) ld4(R + q, r[q], r[q + 1], r[q + 2], r[q + 3]);
}

template <int DIM, typename T>
__device__ __forceinline__ ViscNode<DIM, T> visc_node(const Work &w, int i) {
  constexpr int S = DIM + 2;
  using R = Rec<DIM>;
  ViscNode<DIM, T> n;
  if constexpr (sizeof(T) == 4) {
    const T *Ri = (const T *)w.vrec + (int64_t)i * vrec_stride<DIM, T>();
#pragma unroll
    for (int k = 0; k < DIM; ++k) {
      n.v[k] = Ri[R::V + k];
      n.mo[k] = Ri[1 + k];
    }
    n.p = Ri[R::P];
    n.a = Ri[R::A];
    n.az = Ri[R::AZ];
    n.ip = Ri[R::IP];
    n.eta = Ri[R::ETA];
    n.H = Ri[R::H];
#pragma unroll
    for (int s = 0; s < S; ++s)
#pragma unroll
      for (int q = 0; q < DIM; ++q) n.f[s][q] = Ri[R::F + s * DIM + q];
#pragma unroll
    for (int q = 0; q < DIM; ++q) n.q[q] = n.v[q] * n.eta;
    double u[S];
    load_rec_state<DIM>(w.rec + (int64_t)i * R::SIZE, u);
#pragma unroll
    for (int s = 0; s < S; ++s) n.bits[s] = dbits(u[s]);
  } else {
    double r[16];
    load_rec<DIM>(w, i, r);
    n.from_record(r);
#pragma unroll
    for (int s = 0; s < S; ++s) n.bits[s] = dbits(r[s]);
  }
  n.steady = w.steady[i];
  return n;
}

// the edge values of entry k = (i, j), j > i, and its mirror. BOTH: i and j
// are boundary nodes (c_ji != -c_ij, Sec. 3.1: both directions evaluated).
// FP64: w_ij from v.c_ij of both nodes (fewest FP64 operations). FP32: as
// differences of the two nodes' fluxes (rounded from FP64 by k_prep), then
// dotted with c_ij -- products taken per entry in FP32 (m_i (v_i.c_ij), or
// the flux formed in FP32) carry rounding errors that the difference of
// rounded fluxes does not: they left ~20x more of the limiter's l = 1
// checks failing on the Mach-3 cylinder and raised the error against FP64
template <int DIM, typename T, bool BOTH, bool ALU>
__device__ __forceinline__ void visc_edge(const MeshView &m, const Params &p, const Work &w, const ViscNode<DIM, T> &n,
                                          int i, int j, int64_t k) {
  constexpr int S = DIM + 2;
  using R = Rec<DIM>;
  constexpr bool flux_diff = sizeof(T) == 4;
  if (n.steady & 1) {
    // both states unchanged since the previous k_visc, which stored this
    // edge's values from the same bits; they were equal then (one of the
    // two nodes had no differing neighbour), so they are now: nothing to
    // store and no rough mark to set
    const unsigned char stj = w.steady[j];
    if ((stj & 1) && ((n.steady | stj) & 2)) return;
  }
  const int32_t kt = m.tr[k];
  T c[DIM], cn, ci, ct[DIM], cnt = T(0), cit = T(0);  // c_ij, and (BOTH) c_ji
  load_geo<DIM, T>(m, k, c, cn, ci);
  if constexpr (BOTH) load_geo<DIM, T>(m, kt, ct, cnt, cit);
  double r[16];
  bool same = true;
  if constexpr (flux_diff) {
    load_rec_state<DIM>(w.rec + (int64_t)j * R::SIZE, r);
  } else {
    load_rec<DIM>(w, j, r);
  }
#pragma unroll
  for (int s = 0; s < S; ++s) same &= dbits(r[s]) == n.bits[s];
  if (same) {
    // U_j = U_i bit for bit: the flux and entropy-flux differences vanish,
    // w_ij = a_ij = 0 exactly, and the two-rarefaction bound of Sec. 3.1
    // reduces to lambda_max = |v.n_ij| + a (p_tr = p, both outer waves
    // rarefactions), so d_ij = |v.c_ij| + a |c_ij| with no division, power
    // or root. Any other edge marks both of its nodes rough.
    T vc = T(0);
#pragma unroll
    for (int q = 0; q < DIM; ++q) vc += n.v[q] * c[q];
    T dij = abs_bits(vc) + n.a * cn;
    if constexpr (BOTH) {  // the max over both directions
      T vct = T(0);
#pragma unroll
      for (int q = 0; q < DIM; ++q) vct += n.v[q] * ct[q];
      dij = max_nonneg(dij, abs_bits(vct) + n.a * cnt);
    }
    store_zero_edge<DIM, T>(w, k, dij);
    store_zero_edge<DIM, T>(w, kt, dij);
    return;
  }
  w.rough[i] = 1;
  w.rough[j] = 1;
  const T *Rj = (const T *)w.vrec + (int64_t)j * vrec_stride<DIM, T>();  // FP32 only
  T vj[DIM], mj[DIM], pj, etaj, Hj, aj, azj, ipj;
  float2 fj;
  if constexpr (flux_diff) {
    pj = Rj[R::P];
    etaj = Rj[R::ETA];
    Hj = Rj[R::H];
    aj = Rj[R::A];
    azj = Rj[R::AZ];
    ipj = Rj[R::IP];
#pragma unroll
    for (int q = 0; q < DIM; ++q) {
      vj[q] = Rj[R::V + q];
      mj[q] = Rj[1 + q];
    }
  } else {
    ViscNode<DIM, T> nj;
    nj.from_record(r);
    pj = nj.p;
    etaj = nj.eta;
    Hj = nj.H;
    aj = nj.a;
    azj = nj.az;
    ipj = nj.ip;
    fj = nj.f32;
#pragma unroll
    for (int q = 0; q < DIM; ++q) {
      vj[q] = nj.v[q];
      mj[q] = nj.mo[q];
    }
  }
  // w_ij = (f(U_j) - f(U_i)) c_ij with f = (m, m v^T + p I, v (E + p));
  // a_ij = (q_j - q_i) . c_ij with q = eta v
  T vjc = T(0), vic = T(0);
#pragma unroll
  for (int q = 0; q < DIM; ++q) {
    vjc += vj[q] * c[q];
    vic += n.v[q] * c[q];
  }
  const T dp = sub_on<ALU>(pj, n.p);
  T wv[S], a_ = T(0), dm[DIM], dH, de;
  if constexpr (flux_diff) {
#pragma unroll
    for (int s = 0; s < S; ++s) {
      T acc = T(0);
#pragma unroll
      for (int q = 0; q < DIM; ++q) acc += (Rj[R::F + s * DIM + q] - n.f[s][q]) * c[q];
      wv[s] = acc;
    }
#pragma unroll
    for (int q = 0; q < DIM; ++q) a_ += __fsub_rn(__fmul_rn(vj[q], etaj), n.q[q]) * c[q];
  } else {
    // X_j (v_j.c) - X_i (v_i.c) as (X_j - X_i) (v_j.c) + X_i (v_j.c - v_i.c):
    // exactly 0 when the two states are equal (a contracted X_j v_j.c -
    // X_i v_i.c leaves the rounding error of one product), so that uniform
    // regions keep P_ij = 0 and the limiter's cheapest exit
    T w0 = T(0);
#pragma unroll
    for (int q = 0; q < DIM; ++q) {
      dm[q] = sub_on<ALU>(mj[q], n.mo[q]);
      w0 += dm[q] * c[q];
    }
    const T dv = sub_on<ALU>(vjc, vic);
    wv[0] = w0;
#pragma unroll
    for (int a = 0; a < DIM; ++a) wv[1 + a] = dm[a] * vjc + n.mo[a] * dv + dp * c[a];
    dH = sub_on<ALU>(Hj, n.H);
    de = sub_on<ALU>(etaj, n.eta);
    wv[S - 1] = __fma_rn(dH, vjc, __dmul_rn(n.H, dv));
    a_ = __fma_rn(de, vjc, __dmul_rn(n.eta, dv));
  }
  // the transposed entry: c_ji = -c_ij unless both nodes lie on the boundary
  // (Sec. 3.1), so w_ji = w_ij and a_ji = a_ij; otherwise evaluate with c_ji
  T wt[S], at = a_, vjct = T(0), vict = T(0);
  if constexpr (!BOTH) {
#pragma unroll
    for (int s = 0; s < S; ++s) wt[s] = wv[s];
  } else {
#pragma unroll
    for (int q = 0; q < DIM; ++q) {
      vjct += vj[q] * ct[q];
      vict += n.v[q] * ct[q];
    }
    if constexpr (flux_diff) {
      at = T(0);
#pragma unroll
      for (int s = 0; s < S; ++s) {
        T acc = T(0);
#pragma unroll
        for (int q = 0; q < DIM; ++q) acc += (n.f[s][q] - Rj[R::F + s * DIM + q]) * ct[q];
        wt[s] = acc;
      }
#pragma unroll
      for (int q = 0; q < DIM; ++q) at += __fsub_rn(n.q[q], __fmul_rn(vj[q], etaj)) * ct[q];
    } else {
      // (f_i - f_j) . c_ji = -[(f_j . c_ji) - (f_i . c_ji)], in the form above
      T w0t = T(0);
#pragma unroll
      for (int q = 0; q < DIM; ++q) w0t += dm[q] * ct[q];
      const T dvt = vjct - vict;
      wt[0] = -w0t;
#pragma unroll
      for (int a = 0; a < DIM; ++a) wt[1 + a] = -(dm[a] * vjct + n.mo[a] * dvt + dp * ct[a]);
      wt[S - 1] = -__fma_rn(dH, vjct, __dmul_rn(n.H, dvt));
      at = -__fma_rn(de, vjct, __dmul_rn(n.eta, dvt));
    }
  }
  // d_ij (Sec. 3.1), mirrored; normal velocities v . c_ij / |c_ij| (FP32:
  // v . (c_ij / |c_ij|))
  T dij;
  if constexpr (flux_diff) {
    T unl = T(0), unr = T(0);
#pragma unroll
    for (int q = 0; q < DIM; ++q) {
      unl += n.v[q] * (c[q] * ci);
      unr += vj[q] * (c[q] * ci);
    }
    dij = lambda_max<T>(p, unl, n.p, n.a, n.az, n.ip, unr, pj, aj, azj, ipj) * cn;
    if constexpr (BOTH) {
      T unj = T(0), uni = T(0);
#pragma unroll
      for (int q = 0; q < DIM; ++q) {
        T nq = ct[q] * cit;
        unj += vj[q] * nq;
        uni += n.v[q] * nq;
      }
      T dji = lambda_max<T>(p, unj, pj, aj, azj, ipj, uni, n.p, n.a, n.az, n.ip) * cnt;
      dij = max_nonneg(dij, dji);
    }
  } else {
    dij = lambda_max_sel<ALU>(p, vic, vjc, ci, n.p, n.a, n.az, n.ip, n.f32, pj, aj, azj, ipj, fj) * cn;
    if constexpr (BOTH) {
      const T dji = lambda_max_sel<ALU>(p, vjct, vict, cit, pj, aj, azj, ipj, fj, n.p, n.a, n.az, n.ip, n.f32) * cnt;
      dij = max_nonneg(dij, dji);
    }
  }
  store_edge<DIM, T>(w, k, wv, a_, dij);
  store_edge<DIM, T>(w, kt, wt, at, dij);
}

// Blocks [0, row_blocks): chunks of 32 rows, one row per lane, the entries of a
// chunk dealt out to 2^lparts warps (entry q of a row to warp q mod 2^lparts),
// so that on small meshes a row's edges run side by side: an FP64 instruction
// occupies its warp for 63 cycles whatever else it could issue, and a few
// thousand rows make too few warps with one thread per row. Every unique edge
// is taken from the row of min(i, j); lanes of a warp work on the same entry
// position, whose decisions agree between neighbouring rows. The remaining
// blocks take the edges between two boundary nodes, one per thread, from a
// list: in the row blocks a single such lane (a wall every few rows on small
// meshes) would make its warp evaluate both directions (sweep of 256 small
// cylinders: 238 -> 179 us with k_alpha).
// Bound by FP64 issue beside integer issue: on a 998k-vertex cylinder, every edge
// general, 254 us and 3.21M FP64 warp instructions (FP64 pipe 67 % of the 84 % that
// it sustains, integer units 59 %; 375k in 3D 403 us), 493 us and 7.4M before. Of
// these, the choice of the outer wave took 7.4M to 5.4M (442 us), 32-byte accesses
// the L1 from 74 % of its throughput (358 us), the differences on the integer units
// (ALU) 4.35M (299 us), the division and the root there the rest. 80 registers a
// thread, so that 768 rows run on an SM (64-thread blocks, 12 of them).
template <int DIM, typename T, bool ALU>
__global__ void __launch_bounds__(TPB_MAX, 3) k_visc(MeshView m, Params p, Work w, unsigned row_blocks, int lparts) {
  if (w.st->err) return;
  if (blockIdx.x >= row_blocks) {
    const int q = (blockIdx.x - row_blocks) * blockDim.x + threadIdx.x;
    if (q >= m.n_bp) return;
    const int i = m.bp_row[q], k = m.bp_pos[q];
    const ViscNode<DIM, T> n = visc_node<DIM, T>(w, i);
    visc_edge<DIM, T, true, ALU>(m, p, w, n, i, m.col[k], k);
    return;
  }
  const unsigned warp = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int i = (warp >> lparts) * 32 + (threadIdx.x & 31);
  if (i >= m.n) return;
  const ViscNode<DIM, T> n = visc_node<DIM, T>(w, i);
  const bool bi = m.isb[i] != 0;
  const int64_t k1 = m.row_ptr[i + 1];
  for (int64_t k = m.row_ptr[i] + (warp & ((1 << lparts) - 1)); k < k1; k += 1 << lparts) {
    const int j = m.col[k];
    if (j <= i || (bi && m.isb[j])) continue;
    visc_edge<DIM, T, false, ALU>(m, p, w, n, i, j, k);
  }
}

// ---------------------------------------------------------------------------
// k_alpha: the indicator alpha_i (Sec. 3.2) from the row's w_ij and a_ij
// ---------------------------------------------------------------------------
// eta'(U_i) from node i's record
template <int DIM, typename T> __device__ __forceinline__ void entropy_gradient(const Params &p, const T *Ri, T *deta) {
  using R = Rec<DIM>;
  // eta' = (-s - rho/(gamma-1) (|v|^2/(2 eps) - gamma/rho), g1 v, -g1), g1 = rho/((gamma-1) eps)
  const T igm1 = T(p.inv_gm1);
  const T rho = Ri[0], irho = Ri[R::IRHO], ieps = Ri[R::IEPS];
  T s_i = -Ri[R::ETA] * irho;
  T g1 = rho * igm1 * ieps;
  T v2 = T(0);
#pragma unroll
  for (int k = 0; k < DIM; ++k) v2 += Ri[R::V + k] * Ri[R::V + k];
  deta[0] = -s_i - rho * igm1 * (T(0.5) * v2 * ieps - T(p.gamma) * irho);
#pragma unroll
  for (int k = 0; k < DIM; ++k) deta[1 + k] = g1 * Ri[R::V + k];
  deta[DIM + 1] = -g1;
}
// entry k's terms of N_i and D_i
template <int DIM, typename T, bool ALU>
__device__ __forceinline__ void indicator_terms(const Work &w, int64_t k, const T *deta, T &n, T &d) {
  constexpr int S = DIM + 2;
  T wk[S], a_, d_;
  load_edge<DIM, T>(w, k, wk, a_, d_);
  T b_ = T(0);
#pragma unroll
  for (int s = 0; s < S; ++s) b_ += deta[s] * wk[s];
  n = sub_on<ALU>(a_, b_);
  d = add_abs_on<ALU>(a_, b_);
}
// alpha_i / 2 (exact): d^H_ij = (a_i/2 + a_j/2) d_ij
template <typename T> __device__ __forceinline__ double half_alpha(T N, T D) {
  if constexpr (sizeof(T) == 8)
    return D > T(0) ? 0.5 * div_alu(abs_bits(N), D) : 0.0;
  else
    return D > T(0) ? 0.5 * (double)(fabs(N) / D) : 0.0;
}

// Three of an entry's four additions on the integer units: 998k cylinder 168 -> 134
// us with all four there, 132 with the quotient too (integer units 73 % busy, FP64
// pipe 58 %), and with the sum of D back on the FP64 pipe k_visc and k_alpha 399 ->
// 392 us (375k in 3D 578 -> 560). 643 MB are read, 95 us at the memory's rate.
template <int DIM, typename T>
__global__ void __launch_bounds__(TPB_MAX) k_alpha(MeshView m, Params p, Work w) {
  constexpr int S = DIM + 2;
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= m.n || w.st->err) return;
  if (!w.rough[i]) {  // every w_ij and a_ij of the row is 0: N_i = D_i = 0
    w.alpha[i] = 0.0;
    return;
  }
  T deta[S];
  entropy_gradient<DIM, T>(p, (const T *)w.vrec + (int64_t)i * vrec_stride<DIM, T>(), deta);
  T N = T(0), D = T(0);
  const int64_t k0 = m.row_ptr[i], k1 = m.row_ptr[i + 1];
  for (int64_t k = k0; k < k1; ++k) {
    if (m.col[k] == i) continue;
    T n, d;
    indicator_terms<DIM, T, true>(w, k, deta, n, d);
    N = add_on<true>(N, n);
    D = add_on<false>(D, d);
  }
  w.alpha[i] = half_alpha(N, D);
}

// ---------------------------------------------------------------------------
// Small meshes. One thread per row leaves most of the chip's 608 FP64 units
// without a warp below ~20k rows, and an FP64 instruction holds its warp for 63
// cycles: a row's serial chain (9 entries of 8 to 27 of them) is what a kernel
// then takes. The *_split kernels give a chunk of 32 rows (a lane each) to a
// block of several warps: the entries are dealt out (entry q to warp q mod
// PARTS) where they are independent, the components of a sum where the order of
// its terms matters (every sum keeps its row's column order, so the results
// are the row kernels' bit for bit). The instruction count grows by what the
// warps repeat, so large meshes keep one thread per row (SPLIT_ROWS).
// ---------------------------------------------------------------------------
constexpr int PARTS = 4;

template <int DIM, typename T>
__global__ void __launch_bounds__(32 * PARTS) k_alpha_split(MeshView m, Params p, Work w) {
  constexpr int S = DIM + 2;
  __shared__ T sn[2][PARTS][32], sd[2][PARTS][32], sD[32];
  const int lane = threadIdx.x & 31, part = threadIdx.x >> 5, i = blockIdx.x * 32 + lane;
  const bool in = i < m.n && !w.st->err;
  const bool act = in && w.rough[i];
  T deta[S];
  int64_t k0 = 0, k1 = 0;
  if (act) {
    entropy_gradient<DIM, T>(p, (const T *)w.vrec + (int64_t)i * vrec_stride<DIM, T>(), deta);
    k0 = m.row_ptr[i];
    k1 = m.row_ptr[i + 1];
  }
  // rounds of PARTS entries: every warp its entry's terms, then warp 0 adds the
  // round's N terms and warp 1 its D terms in column order (an absent or
  // diagonal entry adds 0, exactly)
  T sum = T(0);
  for (int r = 0;; ++r) {
    const int64_t k = k0 + r * PARTS + part;
    T n = T(0), d = T(0);
    if (k < k1 && m.col[k] != i) indicator_terms<DIM, T, false>(w, k, deta, n, d);
    sn[r & 1][part][lane] = n;
    sd[r & 1][part][lane] = d;
    const int more = __syncthreads_or(k0 + (r + 1) * PARTS < k1);
    if (part < 2) {
#pragma unroll
      for (int q = 0; q < PARTS; ++q) sum += part == 0 ? sn[r & 1][q][lane] : sd[r & 1][q][lane];
    }
    if (!more) break;  // (the next round writes the other half of the buffers)
  }
  if (part == 1) sD[lane] = sum;
  __syncthreads();
  if (part == 0 && in) w.alpha[i] = act ? half_alpha(sum, sD[lane]) : 0.0;
}

// The running minimum and maximum of a row's bar-state densities rho_bar = num /
// den, den = 2 d_ij > 0, kept as fractions. Against both, a new fraction is
// first compared in FP32 (8 units of 2^-24 a quotient; margin 2e-6, 32 units):
// most lie clearly between, or clearly outside; only near ties are compared as
// the FP64 cross products decide (4 FP64 instructions an entry otherwise).
struct DensityBounds {
  double nmin, dmin, nmax, dmax;
  float fmin, fmax;  // the fractions in FP32
  __device__ __forceinline__ explicit DensityBounds(double rho)
      : nmin(rho), dmin(1.0), nmax(rho), dmax(1.0), fmin(trunc_f32(rho)), fmax(fmin) {}
  __device__ __forceinline__ void add(double num, double dk) {  // dk = d_ij > 0
    const float nf = trunc_f32(num), df = 2.0f * trunc_f32(dk);
    const float q = __fdividef(nf, df);
    constexpr float lo = 1.0f - 2e-6f, hi = 1.0f + 2e-6f;
    const bool fine = nf > 1e-30f && nf < 1e30f && df > 1e-30f && df < 1e30f && fmin > 1e-30f && fmax < 1e30f;
    if (fine && q > fmin * hi && q < fmax * lo) return;
    const double den = 2.0 * dk;
    if (fine && q < fmin * lo) {
      nmin = num;
      dmin = den;
      fmin = q;
    } else if (fine && q > fmax * hi) {
      nmax = num;
      dmax = den;
      fmax = q;
    } else {
      if (order_key(num * dmin) < order_key(nmin * den)) {
        nmin = num;
        dmin = den;
        fmin = q;
      }
      if (order_key(num * dmax) > order_key(nmax * den)) {
        nmax = num;
        dmax = den;
        fmax = q;
      }
    }
  }
  __device__ __forceinline__ double rho_min() const { return dmin == 1.0 ? nmin : div_alu(nmin, dmin); }
  __device__ __forceinline__ double rho_max() const { return dmax == 1.0 ? nmax : div_alu(nmax, dmax); }
};

// c_cfl m_i / (2 sum_j d_ij), or +inf where FP32 shows it to be above the
// instance's minimum so far (which only ever falls): the division is then left
// out. Numerator and minimum well within FP32's normal range: a minimum below it
// would be truncated to 0, above which every row's estimate lies.
__device__ __forceinline__ double row_cfl_bound(const Params &p, double m, double dsum, unsigned long long so_far) {
  const float num = 0.5f * p.cfl_f * trunc_f32(m), est = __fdividef(num, trunc_f32(dsum));
  const float low = trunc_f32(__longlong_as_double((long long)so_far));
  if (num > 1e-30f && low > 1e-30f && est > low * (1.0f + 4e-6f) && est < 1e30f) return INFINITY;
  return p.cfl * m / (2.0 * dsum);
}

// the local bounds, relaxed by (1 -/+ r_i) where the context asks for it
__device__ __forceinline__ void store_bounds(const MeshView &m, const Params &p, const Work &w, int i, double rmin,
                                             double rmax, double phimin, double phimax) {
  if (p.relaxed) {
    const double r = m.relax[i];
    rmin = (1.0 - r) * rmin;
    rmax = (1.0 + r) * rmax;
    phimin = (1.0 - r) * phimin;
  }
  st4(w.bounds + (int64_t)i * 4, rmin, rmax, phimin, phimax);
}

// Algorithm 1 steps 2-3 for one row; returns the row's CFL bound
// c_cfl m_i / (2 sum_{j != i} d_ij), or +inf (row_cfl_bound)
template <int DIM, typename T, bool ALU>
__device__ __forceinline__ double low_row(const MeshView &m, const Params &p, const Work &w, int i,
                                          unsigned long long so_far) {
  constexpr int S = DIM + 2;
  constexpr int SP = Layout<DIM>::SP;
  using R = Rec<DIM>;
  const double *Ri = w.rec + (int64_t)i * R::SIZE;
  double ui[S];
  load_rec_state<DIM>(Ri, ui);
  const double alphai = w.alpha[i];

  // U^L increment and the bounds in FP64; F^H in the viscosity precision T
  // U^L increment in FP64 (also in mixed mode); the sum of the w_ij in their
  // own precision T (FP32 values summed in FP32 in mixed mode, converted once)
  double inc[S];
  T wsum[S];
  T fh[S];
#pragma unroll
  for (int s = 0; s < S; ++s) {
    inc[s] = 0.0;
    wsum[s] = T(0);
    fh[s] = T(0);
  }
  DensityBounds rb(ui[0]);
  double phimin = Ri[R::PHI], phimax = phimin, dsum = 0.0;
  int64_t kd = -1;
  const int64_t k0 = m.row_ptr[i], k1 = m.row_ptr[i + 1];
  for (int64_t k = k0; k < k1; ++k) {
    const int j = m.col[k];
    if (j == i) {
      kd = k;
      continue;
    }
    const double *Rj64 = w.rec + (int64_t)j * R::SIZE;
    double Rj[S];
    load_rec_state<DIM>(Rj64, Rj);
    T wk[S], ak, dkT;
    load_edge<DIM, T>(w, k, wk, ak, dkT);
    const double dk = (double)dkT;
    const T dH = T(sizeof(T) == 4 ? add_on<ALU>(alphai, w.alpha[j]) : alphai + w.alpha[j]) * dkT;  // w.alpha holds alpha / 2
    const double w0 = (double)wk[0];
#pragma unroll
    for (int s = 0; s < S; ++s) {
      const double du = s == 0 || s == 1 || s == S - 1 ? sub_near(Rj[s], ui[s]) : sub_on<ALU>(Rj[s], ui[s]);
      inc[s] += dk * du;  // sum_j d_ij (U_j - U_i); the sum of w_ij is subtracted once
      fh[s] += dH * (T)du;
      wsum[s] = add_on<ALU>(wsum[s], wk[s]);
    }
    if (dbits(dk) > 0) rb.add(dk * (sizeof(T) == 4 ? add_on<ALU>(ui[0], Rj[0]) : ui[0] + Rj[0]) - w0, dk);  // dk >= 0
    // Phi > 0: the integer order of the bit patterns is the numeric order
    const double pj = Rj64[R::PHI];
    phimin = dbits(pj) < dbits(phimin) ? pj : phimin;
    phimax = dbits(pj) > dbits(phimax) ? pj : phimax;
    dsum = add_on<ALU && sizeof(T) == 4>(dsum, dk);
  }
#pragma unroll
  for (int s = 0; s < S; ++s) {
    inc[s] -= (double)wsum[s];
    fh[s] -= wsum[s];
  }
  *d_ptr<DIM, T>(w, kd) = (T)(-dsum);
  double *inci = w.inc + (int64_t)i * SP;
  T *fhi = (T *)w.vFH + (int64_t)i * SP;  // stored as F^H_i / m_i
  const T imi = T(m.inv_mi[i]);
#pragma unroll
  for (int s = 0; s < S; ++s) {
    inci[s] = inc[s];
    fhi[s] = fh[s] * imi;
    if constexpr (sizeof(T) == 4) w.G64[(int64_t)i * SP + s] = (double)fhi[s];
  }
  store_bounds(m, p, w, i, rb.rho_min(), rb.rho_max(), phimin, phimax);
  w.rough2[i] = 1;
  return row_cfl_bound(p, m.mi[i], dsum, so_far);
}

// The same for a row whose neighbours all carry U_i bit for bit (rough[i] =
// 0): every w_ij is 0 and U_j - U_i = 0, so the increment and F^H vanish,
// every bar state is U_i (rho_min = rho_max = rho_i) and Phi_min = Phi_i --
// the values the general row gives, bit for bit. Only sum_j d_ij remains
// (same order). rough2[i] records whether a neighbour is rough.
template <int DIM, typename T>
__device__ __forceinline__ double low_row_smooth(const MeshView &m, const Params &p, const Work &w, int i,
                                                 unsigned long long so_far) {
  constexpr int S = DIM + 2;
  constexpr int SP = Layout<DIM>::SP;
  using R = Rec<DIM>;
  double dsum = 0.0;
  int64_t kd = -1;
  unsigned char r2 = 0;
  const int64_t k0 = m.row_ptr[i], k1 = m.row_ptr[i + 1];
  for (int64_t k = k0; k < k1; ++k) {
    const int j = m.col[k];
    if (j == i) {
      kd = k;
      continue;
    }
    dsum += (double)*d_ptr<DIM, T>(w, k);
    r2 |= w.rough[j];
  }
  *d_ptr<DIM, T>(w, kd) = (T)(-dsum);
  double *inci = w.inc + (int64_t)i * SP;
  T *fhi = (T *)w.vFH + (int64_t)i * SP;
#pragma unroll
  for (int s = 0; s < S; ++s) {
    inci[s] = 0.0;
    fhi[s] = T(0);
    if constexpr (sizeof(T) == 4) w.G64[(int64_t)i * SP + s] = 0.0;
  }
  const double *Ri = w.rec + (int64_t)i * R::SIZE;
  const double rho = Ri[0];
  const double phi = Ri[R::PHI];
  store_bounds(m, p, w, i, rho, rho, phi, phi);
  w.rough2[i] = r2;
  return row_cfl_bound(p, m.mi[i], dsum, so_far);
}

// ---------------------------------------------------------------------------
// k_low: Algorithm 1 steps 2-3 -- d_ii, CFL bound, low-order increment, local
// bounds and high-order fluxes
// ---------------------------------------------------------------------------
// the smallest of a warp's bit patterns
__device__ __forceinline__ unsigned long long warp_min_bits(unsigned long long b) {
  const unsigned hi = __reduce_min_sync(0xffffffffu, (unsigned)(b >> 32));
  const unsigned lo = __reduce_min_sync(0xffffffffu, (unsigned)(b >> 32) == hi ? (unsigned)b : 0xffffffffu);
  return (unsigned long long)hi << 32 | lo;
}

// Folds the rows' CFL bounds into their instances' minima (exact and order
// independent: the bit patterns of positive doubles order like their values,
// and NaN patterns like values above every bound). A warp whose rows lie in one
// instance reduces first; an atomic is issued only below the minimum so far.
__device__ __forceinline__ void fold_bound(const Work &w, double bound, int inst, unsigned long long so_far) {
  const unsigned long long b = (unsigned long long)dbits(bound), inf = 0x7FF0000000000000ull;
  if (__reduce_min_sync(0xffffffffu, (unsigned)inst) == __reduce_max_sync(0xffffffffu, (unsigned)inst)) {
    const unsigned long long m = warp_min_bits(b);
    if ((threadIdx.x & 31) == 0 && m < inf && m < so_far) atomicMin(&w.bound_bits[inst], m);
  } else if (b < inf && b < so_far) {
    atomicMin(&w.bound_bits[inst], b);
  }
}

// Bound by FP64 issue. Of the 32.6 FP64 instructions an entry that a row took
// (998k cylinder: 8.1M warp instructions, 486 us), the sums need 21; the bar
// states' cross products, the relaxation of strict bounds, most rows' division
// for the CFL bound and the minima's FP64 compares are gone (26.7, 397 us), and the
// sum of w_ij, du, the bounds' two divisions and (mixed) the sums around d_ij are on
// the integer units: 4.19M, 323 us, mixed 285 (FP64 pipe 68 %, integer units 55 %).
// ALU: 80 registers a thread, 768 rows an SM (512 rows 350 us, 1024 with spills 392,
// when 768 took 336).
template <int DIM, typename T, bool ALU>
__global__ void __launch_bounds__(TPB_MAX, ALU && DIM == 2 ? 3 : 2) k_low(MeshView m, Params p, Work w) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  double bound = INFINITY;
  const int inst = m.inst ? m.inst[min(i, m.n - 1)] : 0;
  const unsigned long long so_far = __ldcg(&w.bound_bits[inst]);
  if (i < m.n && !w.st->err)
    bound = w.rough[i] ? low_row<DIM, T, ALU>(m, p, w, i, so_far) : low_row_smooth<DIM, T>(m, p, w, i, so_far);
  __syncwarp();
  fold_bound(w, bound, inst, so_far);
}

// The split form: warp s < S the sums of component s, warp S the bar-state and
// Phi bounds, sum_j d_ij and the CFL bound.
template <int DIM, typename T>
__global__ void __launch_bounds__(32 * (DIM + 3)) k_low_split(MeshView m, Params p, Work w) {
  constexpr int S = DIM + 2, SP = Layout<DIM>::SP;
  using R = Rec<DIM>;
  const int lane = threadIdx.x & 31, part = threadIdx.x >> 5, i = blockIdx.x * 32 + lane;
  const bool in = i < m.n && !w.st->err;
  const bool rough = in && w.rough[i];
  const int64_t k0 = in ? m.row_ptr[i] : 0, k1 = in ? m.row_ptr[i + 1] : 0;
  if (part < S) {
    if (!rough) return;  // (warp S writes a smooth row's zeros)
    const int c = part;
    const double ui = w.rec[(int64_t)i * R::SIZE + c], alphai = w.alpha[i];
    double inc = 0.0;
    T wsum = T(0), fh = T(0);
    for (int64_t k = k0; k < k1; ++k) {
      const int j = m.col[k];
      if (j == i) continue;
      const T dkT = *d_ptr<DIM, T>(w, k);
      const T dH = T(alphai + w.alpha[j]) * dkT;
      const double du = w.rec[(int64_t)j * R::SIZE + c] - ui;
      inc += (double)dkT * du;
      fh += dH * (T)du;
      wsum += w_slot<DIM, T>(w, k)[c];
    }
    inc -= (double)wsum;
    fh -= wsum;
    const T g = fh * T(m.inv_mi[i]);
    w.inc[(int64_t)i * SP + c] = inc;
    ((T *)w.vFH)[(int64_t)i * SP + c] = g;
    if constexpr (sizeof(T) == 4) w.G64[(int64_t)i * SP + c] = (double)g;
    return;
  }
  const int inst = m.inst ? m.inst[min(i, m.n - 1)] : 0;
  const unsigned long long so_far = __ldcg(&w.bound_bits[inst]);
  double bound = INFINITY;
  if (rough) {
    const double *Ri = w.rec + (int64_t)i * R::SIZE;
    const double rho = Ri[0];
    DensityBounds rb(rho);
    double phimin = Ri[R::PHI], phimax = phimin, dsum = 0.0;
    int64_t kd = -1;
    for (int64_t k = k0; k < k1; ++k) {
      const int j = m.col[k];
      if (j == i) {
        kd = k;
        continue;
      }
      const double *Rj = w.rec + (int64_t)j * R::SIZE;
      const double dk = (double)*d_ptr<DIM, T>(w, k);
      if (dbits(dk) > 0) rb.add(dk * (rho + Rj[0]) - (double)w_slot<DIM, T>(w, k)[0], dk);
      const double pj = Rj[R::PHI];
      phimin = dbits(pj) < dbits(phimin) ? pj : phimin;
      phimax = dbits(pj) > dbits(phimax) ? pj : phimax;
      dsum += dk;
    }
    *d_ptr<DIM, T>(w, kd) = (T)(-dsum);
    store_bounds(m, p, w, i, rb.rho_min(), rb.rho_max(), phimin, phimax);
    w.rough2[i] = 1;
    bound = row_cfl_bound(p, m.mi[i], dsum, so_far);
  } else if (in) {
    bound = low_row_smooth<DIM, T>(m, p, w, i, so_far);
  }
  __syncwarp();
  fold_bound(w, bound, inst, so_far);
}

// ---------------------------------------------------------------------------
// k_tau: each instance's CFL bound (the minimum gathered by k_low); fixes the
// instance's tau at the first stage (Sec. 3.1) and resets the minimum
// ---------------------------------------------------------------------------
constexpr unsigned long long kInfBits = 0x7FF0000000000000ull;

__global__ void __launch_bounds__(256) k_tau(MeshView m, Work w, int stage, double dt_given, double cfl,
                                             int advance_time) {
  DevStatus *st = w.st;
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k < LSQ_SLOTS) {  // the stage's queued line searches start empty
    w.lsq_count[k] = 0;
    w.lsq2_count[k] = 0;
  }
  if (k >= m.ninst || st->err) return;
  const double bound = __longlong_as_double((long long)w.bound_bits[k]);
  w.bound_bits[k] = kInfBits;
  w.bound_inst[stage * m.ninst + k] = bound;
  if (k == 0) st->stage_bound[stage] = bound;
  const double limit = bound / cfl;  // invariant-domain limit, c_cfl = 1
  if (stage == 0) {
    double tau;
    if (dt_given > 0.0) {
      if (dt_given > limit) {
        atomicExch(&st->err, 5);  // EH_ERR_CFL
        return;
      }
      tau = dt_given;
    } else {
      tau = bound;
    }
    const double left = w.tfinal_inst[k] - w.t_inst[k];
    if (tau > left) tau = left > 0.0 ? left : 0.0;  // land on t_final; finished instances stay frozen
    w.tau_inst[k] = tau;
    if (k == 0) st->tau = tau;
  } else {
    if (w.tau_inst[k] > limit) atomicAdd(&st->cfl_violations, 1ull);
    if (advance_time && stage == 2) {
      w.t_inst[k] += w.tau_inst[k];
      if (w.tau_inst[k] > 0.0) w.steps_inst[k] += 1ull;
    }
  }
}

// ---------------------------------------------------------------------------
// k_lim1: Algorithm 1 step 4 -- U^L, P_ij and the first line search
// ---------------------------------------------------------------------------
// U^L and the entries q = part, part + STEP, ... of row i; returns the mask of
// entries left to the queued searches (of the first 64 of a row; later ones are
// queued at once and set long_deferred)
template <int DIM, typename T, int STEP, bool ALU>
__device__ __forceinline__ uint64_t lim1_entries(const MeshView &m, const Params &p, const Work &w, double *P_trace,
                                                 int i, int part, bool &long_deferred) {
  constexpr int S = DIM + 2;
  constexpr int SP = Layout<DIM>::SP;
  using R = Rec<DIM>;
  if (!w.rough2[i]) {
    // row and neighbours without a differing neighbour state: the increment
    // is 0 (U^L = U_i) and every P_ij = (tc m_ij/m_i)(0 - 0) + (.)(U_j - U_i)
    // is 0, so every search returns 1 (reading R5b) -- as the general row
    if (part == 0) {
      double u[S];
      load_rec_state<DIM>(w.rec + (int64_t)i * R::SIZE, u);
      store_vec<DIM>(w.UL + (int64_t)i * SP, u);
      if (P_trace) {
        for (int64_t k = m.row_ptr[i]; k < m.row_ptr[i + 1]; ++k) {
#pragma unroll
          for (int s = 0; s < S; ++s) P_trace[k * SP + s] = 0.0;
        }
      }
    }
    return 0;  // every limiter is 1; la is not written (readers check lone first)
  }
  const double tau = w.tau_inst[m.inst ? m.inst[i] : 0];
  const double *Ri = w.rec + (int64_t)i * R::SIZE;
  double ui[S], ul[S], gi[S];
  const double *inci = w.inc + (int64_t)i * SP;
  const double *Garr = w.G64;  // G = F^H / m per node, in FP64 (widened once per node in mixed mode)

  const double *Gi = Garr + (int64_t)i * SP;
  const double tm = tau * m.inv_mi[i];
#pragma unroll
  for (int s = 0; s < S; ++s) {
    ui[s] = Ri[s];
    ul[s] = ui[s] + tm * inci[s];
    gi[s] = Gi[s];
  }
  if (part == 0) {
    store_vec<DIM>(w.UL + (int64_t)i * SP, ul);
    // U^L admissible: rho > 0 and rho E - |M|^2/2 > 0 (no division); with
    // c_cfl <= 1 it always is (invariant-domain property), above 1 the
    // adaptive step restarts on it
    double m2 = 0.0;
#pragma unroll
    for (int q = 0; q < DIM; ++q) m2 += ul[1 + q] * ul[1 + q];
    if (!(pos_strict(ul[0]) && pos_strict(ul[S - 1] * ul[0] - 0.5 * m2)))
      atomicAdd(&w.st->low_not_admissible, 1ull);
  }
  double rmin, rmax, phimin, phimax;
  ld4(w.bounds + (int64_t)i * 4, rmin, rmax, phimin, phimax);
  const double phimin2 = phimin * phimin, phimin5 = phimin2 * phimin2 * phimin;
  const RowF32 rf = row_f32<DIM>(p, ul, rmin, rmax, phimin, phimax, phimin5);
  const double alphai = w.alpha[i];
  const int64_t k0 = m.row_ptr[i], k1 = m.row_ptr[i + 1];
  // P_ij = tau/(m_i lambda_i) (b_ij F^H_j - b_ji F^H_i + (d^H_ij - d_ij)(U_j - U_i))
  // with b_ij = -m_ij/m_j, b_ji = -m_ji/m_i and m_ij = m_ji:
  //      = (tc m_ij/m_i) (G_i - G_j) + (tc/m_i) (d^H_ij - d_ij)(U_j - U_i),
  // G = F^H/m, tc = tau (card I(i) - 1)
  const double tc = tau * (double)(k1 - k0 - 1);
  const double coef = tc * m.inv_mi[i];
  uint64_t defer = 0;  // entries whose line search goes to k_ls_deferred
  const bool longrow = k1 - k0 > 64;  // limiters stored as they are known
  for (int64_t k = k0 + part; k < k1; k += STEP) {
    const int j = m.col[k];
    double *Pk = w.P + k * SP;
    if (j == i) {
#pragma unroll
      for (int s = 0; s < S; ++s) Pk[s] = 0.0;
      if (P_trace) {
#pragma unroll
        for (int s = 0; s < S; ++s) P_trace[k * SP + s] = 0.0;
      }
      if (longrow) w.la[k] = 1.0;
      continue;
    }
    double Rj[S], Gj[S];
    load_rec_state<DIM>(w.rec + (int64_t)j * R::SIZE, Rj);
    load_vec<DIM>(Garr + (int64_t)j * SP, Gj);
    const double dk = (double)*d_ptr<DIM, T>(w, k);
    const double dH = (alphai + w.alpha[j]) * dk;  // w.alpha holds alpha / 2
    const double cm = tc * m.betat[k], cd = coef * (dH - dk);
    double P[S];
#pragma unroll
    for (int s = 0; s < S; ++s) {
      const double du = s == 0 || s == 1 || s == S - 1 ? sub_near(Rj[s], ui[s]) : sub_on<ALU>(Rj[s], ui[s]);
      P[s] = __fma_rn(cm, sub_on<ALU>(gi[s], Gj[s]), __dmul_rn(cd, du));
    }
    store_vec<DIM>(Pk, P);
    if (P_trace) {
#pragma unroll
      for (int s = 0; s < S; ++s) P_trace[k * SP + s] = P[s];
    }
    if (line_search_at_one<DIM>(p, ul, P, rmin, rmax, phimin5, rf)) {
      if (longrow) w.la[k] = 1.0;
    } else if (k - k0 < 64) {
      defer |= 1ull << (k - k0);
    } else {
      defer_line_searches(w, 0, i, k, 1ull);  // rows longer than 64 entries
      long_deferred = true;
    }
  }
  return defer;
}

// the row's all-ones flag, the limiters it stores and its queued searches: a row
// with a queued search stores its other limiters (1); a row without one stores
// none (every limiter of it is 1, and its lone flag says so)
template <int STEP>
__device__ __forceinline__ void lim_finish(const MeshView &m, const Work &w, unsigned char *lone_out, double *lout,
                                           int slot, int i, int part, uint64_t defer, bool lone) {
  const int64_t k0 = m.row_ptr[i], k1 = m.row_ptr[i + 1];
  if (part == 0) lone_out[i] = lone ? 1 : 0;
  if (!lone && k1 - k0 <= 64)
    for (int64_t k = k0 + part; k < k1; k += STEP)
      if (!((defer >> (k - k0)) & 1ull)) lout[k] = 1.0;
  defer_line_searches(w, slot, i, k0, defer);
}

// rows i, i + grid size, ... (the grid may be capped to limit the rows in
// flight; one row per thread otherwise). The differences of P_ij on the integer
// units where ALU: 998k cylinder 386 -> 328 us (FP64 pipe 77 %, integer 58 %),
// mixed 415 -> 349.
template <int DIM, typename T, bool ALU>
__global__ void __launch_bounds__(TPB_MAX, ALU && DIM == 2 ? 3 : 2) k_lim1(MeshView m, Params p, Work w, double *P_trace) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < m.n; i += gridDim.x * blockDim.x) {
    if (w.st->err) return;
    bool long_deferred = false;
    const uint64_t defer = lim1_entries<DIM, T, 1, ALU>(m, p, w, P_trace, i, 0, long_deferred);
    lim_finish<1>(m, w, w.lone, w.la, 0, i, 0, defer, defer == 0 && !long_deferred);
  }
}

// the split form: the entries dealt out to PARTS warps
template <int DIM, typename T>
__global__ void __launch_bounds__(32 * PARTS) k_lim1_split(MeshView m, Params p, Work w, double *P_trace) {
  __shared__ int queued[32];
  const int lane = threadIdx.x & 31, part = threadIdx.x >> 5, i = blockIdx.x * 32 + lane;
  if (part == 0) queued[lane] = 0;
  __syncthreads();
  const bool in = i < m.n && !w.st->err;
  bool long_deferred = false;
  uint64_t defer = 0;
  if (in) defer = lim1_entries<DIM, T, PARTS, false>(m, p, w, P_trace, i, part, long_deferred);
  if (defer != 0 || long_deferred) queued[lane] = 1;
  __syncthreads();
  if (in) lim_finish<PARTS>(m, w, w.lone, w.la, 0, i, part, defer, queued[lane] == 0);
}


// min of two limiters in [0, 1]: non-negative doubles order like their bit
// patterns, so an integer min (no FP64 instruction) gives the same value
__device__ __forceinline__ double lmin(double a, double b) {
  const long long x = __double_as_longlong(a), y = __double_as_longlong(b);
  return __longlong_as_double(x < y ? x : y);
}

// The symmetrised limiters l_ij = min(l_k, l_tr[k]) of the cnt <= LCHUNK
// entries kb, kb + 1, ... of row i (diag[q]: the entry is the diagonal); a
// row whose lone flag is set has every limiter 1 (and none stored). Every
// load of the chunk is issued before the first use: the transposed value is a
// dependent gather (tr[k], then l at tr[k]), and issuing a chunk's gathers
// together overlaps their latencies instead of paying them one entry at a time.
constexpr int LCHUNK = 3;  // measured on the 4.0M cylinder: 3 shortens k_final by 7%; 4 and 9 lengthen it
                           // (one limiter pass; after two or more k_final gathers only where rem != 0)
__device__ __forceinline__ void sym_limiters(const MeshView &m, const double *__restrict__ lin,
                                             const unsigned char *__restrict__ lone, int64_t kb, int cnt, int i,
                                             double *ls, bool *diag) {
  int32_t t[LCHUNK], c[LCHUNK];
#pragma unroll
  for (int q = 0; q < LCHUNK; ++q)
    if (q < cnt) {
      t[q] = m.tr[kb + q];
      c[q] = m.col[kb + q];
    }
  const bool one_i = lone[i] != 0;
  double a[LCHUNK], b[LCHUNK];
#pragma unroll
  for (int q = 0; q < LCHUNK; ++q)
    if (q < cnt) {
      a[q] = one_i ? 1.0 : lin[kb + q];
      b[q] = lone[c[q]] ? 1.0 : lin[t[q]];
    }
#pragma unroll
  for (int q = 0; q < LCHUNK; ++q)
    if (q < cnt) {
      ls[q] = lmin(a[q], b[q]);
      diag[q] = c[q] == i;
    }
}

// ---------------------------------------------------------------------------
// k_pass: symmetrise the limiter, update, shrink P and search again
// ---------------------------------------------------------------------------
// the next search from the updated state u on the entries q = part, part + STEP,
// ... of row i (as lim1_entries)
template <int DIM, int STEP>
__device__ __forceinline__ uint64_t pass_search(const MeshView &m, const Params &p, const Work &w, const double *u,
                                                double *__restrict__ lout, int slot, int i, int part,
                                                bool &long_deferred) {
  constexpr int S = DIM + 2;
  constexpr int SP = Layout<DIM>::SP;
  const int64_t k0 = m.row_ptr[i], k1 = m.row_ptr[i + 1];
  double rmin, rmax, phimin, phimax;
  ld4(w.bounds + (int64_t)i * 4, rmin, rmax, phimin, phimax);
  const double phimin2 = phimin * phimin, phimin5 = phimin2 * phimin2 * phimin;
  const RowF32 rf = row_f32<DIM>(p, u, rmin, rmax, phimin, phimax, phimin5);
  uint64_t defer = 0;
  const bool longrow = k1 - k0 > 64;  // limiters stored as they are known
  for (int64_t k = k0 + part; k < k1; k += STEP) {
    if (m.col[k] == i) {
      if (longrow) lout[k] = 1.0;
      continue;
    }
    const double r = w.rem[k];
    if (dbits(r) == 0) {  // the remainder is 0: every l gives the same state, the largest is 1
      if (longrow) lout[k] = 1.0;
      continue;
    }
    const double *Pk = w.P + k * SP;
    double P[S];
#pragma unroll
    for (int s = 0; s < S; ++s) P[s] = r * Pk[s];
    if (line_search_at_one<DIM>(p, u, P, rmin, rmax, phimin5, rf)) {
      if (longrow) lout[k] = 1.0;
    } else if (k - k0 < 64) {
      defer |= 1ull << (k - k0);
    } else {
      defer_line_searches(w, slot, i, k, 1ull);
      long_deferred = true;
    }
  }
  return defer;
}

template <int DIM>
__device__ __forceinline__ void pass_row(const MeshView &m, const Params &p, const Work &w, const double *__restrict__ Uin,
                                         double *__restrict__ Uout, const double *__restrict__ lin,
                                         double *__restrict__ lout, double *lsym_trace, int slot, int i) {
  constexpr int S = DIM + 2;
  constexpr int SP = Layout<DIM>::SP;
  const int64_t k0 = m.row_ptr[i], k1 = m.row_ptr[i + 1];
  const double lambda_i = m.lam[i];
  double u[S];
  load_vec<DIM>(Uin + (int64_t)i * SP, u);
  const unsigned char *lone_in = w.lone + (int64_t)((slot - 1) & 1) * m.n;
  unsigned char *lone_out = w.lone + (int64_t)(slot & 1) * m.n;
  if (!w.rough2[i]) {  // every P_ij is 0 (see lim1_row): the state stays, every next search returns 1
    double *Uo = Uout + (int64_t)i * SP;
#pragma unroll
    for (int s = 0; s < S; ++s) Uo[s] = u[s];
    if (lsym_trace) {
      for (int64_t k = k0; k < k1; ++k) {
        const int j = m.col[k];
        lsym_trace[k] = j == i ? 1.0 : lmin(lone_in[i] ? 1.0 : lin[k], lone_in[j] ? 1.0 : lin[m.tr[k]]);
      }
    }
    lone_out[i] = 1;  // every next limiter is 1; lout is not written
    return;
  }
  const bool one_i = lone_in[i] != 0;
  if (one_i && !lsym_trace) {
    // a row whose limiters, and whose neighbours' limiters, are all 1 (most
    // rows): no limiter is gathered, and nothing is left of P_ij -- the row is
    // marked spent, its rem entries are neither written nor read again
    bool all = true;
    for (int64_t k = k0; k < k1; ++k) all &= lone_in[m.col[k]] != 0;
    if (all) {
      const bool before = slot > 1 && w.spent[i];
      for (int64_t k = k0; k < k1 && !before; ++k) {
        if (m.col[k] == i) continue;
        double P[S];
        load_vec<DIM>(w.P + k * SP, P);
        if (slot > 1) {
          const double r = w.rem[k];
          if (dbits(r) == 0) continue;
#pragma unroll
          for (int s = 0; s < S; ++s) P[s] = r * P[s];
        }
#pragma unroll
        for (int s = 0; s < S; ++s) u[s] += lambda_i * P[s];  // l = 1
      }
      store_vec<DIM>(Uout + (int64_t)i * SP, u);
      lone_out[i] = 1;
      w.spent[i] = 1;
      return;
    }
  }
  const bool spent = slot > 1 && w.spent[i];  // nothing is left already: rem is not there to be read
  // slot = the pass (1, 2, ...): pass 1 starts from k_lim1's P_ij, a later
  // pass from the remainder rem[k] P[k] that the previous one left
  for (int64_t k = k0; k < k1; ++k) {
    const int j = m.col[k];
    if (j == i) {
      if (lsym_trace) lsym_trace[k] = 1.0;
      continue;
    }
    // a row whose limiters are all 1 has none stored: its side is 1, and an
    // entry between two such rows needs no gather of the transposed limiter
    const double l = lmin(one_i ? 1.0 : lin[k], lone_in[j] ? 1.0 : lin[m.tr[k]]);
    if (lsym_trace) lsym_trace[k] = l;
    double *Pk = w.P + k * SP;
    double P[S];
    if (slot > 1) {
      const double r = spent ? 0.0 : w.rem[k];
      if (dbits(r) == 0) continue;  // nothing left of P_ij (rem stays 0)
#pragma unroll
      for (int s = 0; s < S; ++s) P[s] = r * Pk[s];
      store_vec<DIM>(Pk, P);  // this pass's P_ij, for the remainder it leaves
    } else {
      load_vec<DIM>(Pk, P);
    }
    // the update with l P; the remainder (1 - l) P is left as rem[k] (a
    // store of (1 - l) P here costs more than forming it where it is read,
    // and for l = 1 -- most entries -- nothing is read at all)
#pragma unroll
    for (int s = 0; s < S; ++s) u[s] += lambda_i * l * P[s];
    w.rem[k] = 1.0 - l;
  }
  store_vec<DIM>(Uout + (int64_t)i * SP, u);
  if (spent) {
    lone_out[i] = 1;
    return;
  }
  w.spent[i] = 0;
  bool long_deferred = false;
  const uint64_t defer = pass_search<DIM, 1>(m, p, w, u, lout, slot, i, 0, long_deferred);
  lim_finish<1>(m, w, lone_out, lout, slot, i, 0, defer, defer == 0 && !long_deferred);
}

// Bound by the latency of the limiters' gathers and by its reads of P: at most 64
// registers, so that 1024 rows are in flight per SM (the pre-decision's second
// level alone would take 92, with 142 -> 174 us on the 998k cylinder); 142 -> 107
// us with the spent rows. Listing the rows that need a limiter, so that the
// others run beside the queued searches on a second stream, measured the same
// step time (5.17 against 5.19 ms) and slowed meshes below 0.4M rows.
template <int DIM>
__global__ void __launch_bounds__(TPB_MAX, 4) k_pass(MeshView m, Params p, Work w, const double *__restrict__ Uin,
                                              double *__restrict__ Uout, const double *__restrict__ lin,
                                              double *__restrict__ lout, double *lsym_trace, int slot) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < m.n; i += gridDim.x * blockDim.x) {
    if (w.st->err) return;
    pass_row<DIM>(m, p, w, Uin, Uout, lin, lout, lsym_trace, slot, i);
  }
}

// The split form, of the first pass after k_lim1 only (a later pass also
// rewrites P in place): warp s adds up component s of the update (3D: warp 0
// also the fifth), the last warp stores the remainder factors, then the
// entries of the next search are dealt out.
template <int DIM>
__global__ void __launch_bounds__(32 * PARTS) k_pass_split(MeshView m, Params p, Work w, const double *__restrict__ Uin,
                                                           double *__restrict__ Uout, const double *__restrict__ lin,
                                                           double *__restrict__ lout, double *lsym_trace) {
  constexpr int S = DIM + 2;
  constexpr int SP = Layout<DIM>::SP;
  __shared__ double su[S][32];
  __shared__ int queued[32];
  const int lane = threadIdx.x & 31, part = threadIdx.x >> 5, i = blockIdx.x * 32 + lane;
  if (part == 0) queued[lane] = 0;
  const bool in = i < m.n && !w.st->err;
  const unsigned char *lone_in = w.lone;
  unsigned char *lone_out = w.lone + (int64_t)m.n;
  const bool rough = in && w.rough2[i];
  const int64_t k0 = in ? m.row_ptr[i] : 0, k1 = in ? m.row_ptr[i + 1] : 0;
  if (in) {
    const bool one_i = lone_in[i] != 0;
    const double lambda_i = m.lam[i];
    double u = Uin[(int64_t)i * SP + part], u4 = 0.0;
    if constexpr (S > PARTS) u4 = Uin[(int64_t)i * SP + PARTS];
    if (rough || (lsym_trace && part == PARTS - 1)) {
      for (int64_t k = k0; k < k1; ++k) {
        const int j = m.col[k];
        if (j == i) {
          if (lsym_trace && part == PARTS - 1) lsym_trace[k] = 1.0;
          continue;
        }
        const double l = lmin(one_i ? 1.0 : lin[k], lone_in[j] ? 1.0 : lin[m.tr[k]]);
        if (part == PARTS - 1) {
          if (lsym_trace) lsym_trace[k] = l;
          if (rough) w.rem[k] = 1.0 - l;
        }
        if (!rough) continue;
        const double *Pk = w.P + k * SP;
        u += lambda_i * l * Pk[part];
        if constexpr (S > PARTS) {
          if (part == 0) u4 += lambda_i * l * Pk[PARTS];
        }
      }
    }
    su[part][lane] = u;
    if constexpr (S > PARTS) {
      if (part == 0) su[PARTS][lane] = u4;
    }
  }
  __syncthreads();
  double u[S];
#pragma unroll
  for (int c = 0; c < S; ++c) u[c] = su[c][lane];
  if (in && part == 0) store_vec<DIM>(Uout + (int64_t)i * SP, u);
  bool long_deferred = false;
  uint64_t defer = 0;
  if (rough && part == 0) w.spent[i] = 0;
  if (rough) defer = pass_search<DIM, PARTS>(m, p, w, u, lout, 1, i, part, long_deferred);
  if (defer != 0 || long_deferred) queued[lane] = 1;
  __syncthreads();
  if (in) lim_finish<PARTS>(m, w, lone_out, lout, 1, i, part, defer, queued[lane] == 0);
}

// ---------------------------------------------------------------------------
// k_ls_deferred / k_ls_iterate: the queued line searches of one pass, one per
// thread, from the pass's start state ub, the stored P_ij and the row's
// bounds. The first kernel takes every exit without iteration and queues the
// rest for the second, whose threads then all run the same iteration count.
// ---------------------------------------------------------------------------
__device__ __forceinline__ bool queue_iteration(const Work &w, int slot, const LsItem &it) {
  namespace cg = cooperative_groups;
  cg::coalesced_group g = cg::coalesced_threads();
  unsigned base = 0;
  if (g.thread_rank() == 0) base = atomicAdd(&w.lsq2_count[slot], g.size());
  base = g.shfl(base, 0) + g.thread_rank();
  if (base >= w.lsq2_cap) return false;  // full: the caller iterates itself
  w.lsq2[base] = it;
  return true;
}

// queues of at most this many searches are run by lane pairs: two lanes for each
// still leave every FP64 unit at most one warp (608 units, 32 lanes)
constexpr unsigned LS_PAIRS = 608 * 32 / 2;

// the start state and direction of search (i, k) of pass 'slot'
template <int DIM>
__device__ __forceinline__ void ls_load(const Work &w, const double *__restrict__ ub, int slot, int i, int k, double *u,
                                        double *P) {
  constexpr int S = DIM + 2;
  constexpr int SP = Layout<DIM>::SP;
  const double r = slot > 0 ? w.rem[k] : 1.0;  // a later pass: the remainder rem P
#pragma unroll
  for (int s = 0; s < S; ++s) {
    u[s] = ub[(int64_t)i * SP + s];
    P[s] = slot > 0 ? r * w.P[(int64_t)k * SP + s] : w.P[(int64_t)k * SP + s];
  }
}
// the lane pair's place in a queue run by pairs: one warp (16 searches) a block,
// and so an SM, before a second one anywhere
__device__ __forceinline__ unsigned pair_warp() { return (threadIdx.x >> 5) * gridDim.x + blockIdx.x; }

template <int DIM>
__global__ void __launch_bounds__(256) k_ls_deferred(MeshView m, Params p, Work w, const double *__restrict__ ub,
                                                     int slot, double *__restrict__ lout) {
  constexpr int S = DIM + 2;
  if (w.st->err) return;
  const unsigned cnt = min(w.lsq_count[slot], w.lsq_cap);
  if (blockIdx.x == 0 && threadIdx.x == 0) atomicAdd(&w.st->line_searches_deferred, (unsigned long long)cnt);
  if (cnt == 0) return;
  if (p.gamma75 && cnt <= LS_PAIRS) {
    // few searches: to their end here, by lane pairs, one warp (16 searches) a
    // block and SM before a second one anywhere
    const unsigned first = pair_warp() * 16, q = first + ((threadIdx.x & 31) >> 1);
    if (first >= cnt) return;
    const int2 it = w.lsq[min(q, cnt - 1)];
    const double *bi = w.bounds + (int64_t)it.x * 4;
    const double phimin = bi[2], phimin2 = phimin * phimin, phimin5 = phimin2 * phimin2 * phimin;
    double u[S], P[S];
    ls_load<DIM>(w, ub, slot, it.x, it.y, u, P);
    LsBracket b = line_search_start_pair<DIM>(p, u, P, bi[0], bi[1], phimin, phimin5);
    if (q >= cnt) b.done = true;
    const unsigned open = __ballot_sync(0xffffffffu, !b.done);
    if (open && (threadIdx.x & 31) == 0)
      atomicAdd(&w.st->line_searches_iterated, (unsigned long long)(__popc(open) / 2));
    const double l = line_search_iterate_pair<DIM>(u, P, phimin, b);
    if (q < cnt && !(threadIdx.x & 1)) lout[it.y] = l;
    return;
  }
  for (unsigned q = blockIdx.x * blockDim.x + threadIdx.x; q < cnt; q += gridDim.x * blockDim.x) {
    const int2 it = w.lsq[q];
    const double *bi = w.bounds + (int64_t)it.x * 4;
    const double phimin = bi[2], phimin2 = phimin * phimin, phimin5 = phimin2 * phimin2 * phimin;
    double u[S], P[S];
    ls_load<DIM>(w, ub, slot, it.x, it.y, u, P);
    const LsBracket b = line_search_start<DIM>(p, u, P, bi[0], bi[1], phimin, phimin5);
    if (b.done)
      lout[it.y] = b.l;
    else if (!queue_iteration(w, slot, LsItem{it.x, it.y, b.l, b.pl, b.pr, b.rR}))
      lout[it.y] = line_search_iterate<DIM>(p, u, P, phimin, b);
  }
}

template <int DIM>
__global__ void __launch_bounds__(256) k_ls_iterate(MeshView m, Params p, Work w, const double *__restrict__ ub,
                                                    int slot, double *__restrict__ lout) {
  constexpr int S = DIM + 2;
  if (w.st->err) return;
  const unsigned cnt = min(w.lsq2_count[slot], w.lsq2_cap);
  if (blockIdx.x == 0 && threadIdx.x == 0) atomicAdd(&w.st->line_searches_iterated, (unsigned long long)cnt);
  if (cnt == 0) return;
  if (p.gamma75 && cnt <= LS_PAIRS) {
    const unsigned first = pair_warp() * 16, q = first + ((threadIdx.x & 31) >> 1);
    if (first >= cnt) return;
    const LsItem it = w.lsq2[min(q, cnt - 1)];
    double u[S], P[S];
    ls_load<DIM>(w, ub, slot, it.i, it.k, u, P);
    const double l = line_search_iterate_pair<DIM>(u, P, w.bounds[(int64_t)it.i * 4 + 2],
                                                   LsBracket{it.l, it.pl, it.pr, it.rR, q >= cnt});
    if (q < cnt && !(threadIdx.x & 1)) lout[it.k] = l;
    return;
  }
  for (unsigned q = blockIdx.x * blockDim.x + threadIdx.x; q < cnt; q += gridDim.x * blockDim.x) {
    const LsItem it = w.lsq2[q];
    const double phimin = w.bounds[(int64_t)it.i * 4 + 2];
    double u[S], P[S];
    ls_load<DIM>(w, ub, slot, it.i, it.k, u, P);
    const LsBracket b{it.l, it.pl, it.pr, it.rR, false};
    lout[it.k] = line_search_iterate<DIM>(p, u, P, phimin, b);
  }
}

// ---------------------------------------------------------------------------
// k_final: last limited update, boundary post-processing (Sec. 4), SSP
// combination (Sec. 4.1) and admissibility check
// ---------------------------------------------------------------------------
// ---------------------------------------------------------------------------
// Sec. 4.2: non-reflecting post-processing of one state along the unit
// outward normal nv with the far-field (Dirichlet) state ud
// ---------------------------------------------------------------------------
template <int DIM> struct NormalState {
  double rho, un, ut[DIM], p, c;  // density, normal and tangential velocity, pressure, sound speed
};

template <int DIM>
__device__ NormalState<DIM> split_normal(const double *u, const double *nv, double gamma) {
  NormalState<DIM> w;
  w.rho = u[0];
  const double ir = 1.0 / u[0];
  double un = 0.0, v2 = 0.0;
#pragma unroll
  for (int q = 0; q < DIM; ++q) {
    const double v = u[1 + q] * ir;
    un += v * nv[q];
    v2 += v * v;
  }
  w.un = un;
#pragma unroll
  for (int q = 0; q < DIM; ++q) w.ut[q] = u[1 + q] * ir - un * nv[q];
  w.p = (gamma - 1.0) * (u[DIM + 1] - 0.5 * u[0] * v2);
  w.c = sqrt(gamma * w.p * ir);
  return w;
}

template <int DIM>
__device__ void join_normal(double rho, double un, const double *ut, double pr, const double *nv, double gamma,
                            double *u) {
  u[0] = rho;
  double v2 = 0.0;
#pragma unroll
  for (int q = 0; q < DIM; ++q) {
    const double v = ut[q] + un * nv[q];
    u[1 + q] = rho * v;
    v2 += v * v;
  }
  u[DIM + 1] = pr / (gamma - 1.0) + 0.5 * rho * v2;
}

// Sec. 4.2.2: incoming characteristics (C_1 = u_n - 2c/(gamma-1) at speed
// u_n - c; entropy p rho^-gamma and tangential velocity at u_n; C_3 = u_n +
// 2c/(gamma-1) at u_n + c) take the far-field values, outgoing ones keep the
// node's: eqs. Supersonic_inflow, Subsonic_inflow, Subsonic_outflow,
// Supersonic_outflow.
template <int DIM>
__device__ void bc_characteristic(double *u, const double *nv, const double *ud, double gamma) {
  const NormalState<DIM> in = split_normal<DIM>(u, nv, gamma);
  if (in.un < 0.0 && -in.un > in.c) {  // every wave enters
#pragma unroll
    for (int s = 0; s < DIM + 2; ++s) u[s] = ud[s];
    return;
  }
  if (in.un >= 0.0 && in.un >= in.c) return;  // every wave leaves
  const NormalState<DIM> far = split_normal<DIM>(ud, nv, gamma);
  const double k = 2.0 / (gamma - 1.0);
  const double c3 = in.un + k * in.c, c1 = far.un - k * far.c;
  const NormalState<DIM> &up = in.un < 0.0 ? far : in;  // source of entropy and tangential velocity
  const double ent = up.p * pow(up.rho, -gamma);
  const double cp = 0.25 * (gamma - 1.0) * (c3 - c1);
  const double rho = pow(cp * cp / (gamma * ent), 1.0 / (gamma - 1.0));
  join_normal<DIM>(rho, 0.5 * (c1 + c3), up.ut, ent * pow(rho, gamma), nv, gamma, u);
}

// wave curve of side w through its state: the jump in normal velocity across
// a 1- or 3-wave that leads to pressure p, and its derivative in p
template <int DIM>
__device__ void wave_curve(double p, const NormalState<DIM> &w, double gamma, double *f, double *df) {
  if (p > w.p) {  // shock (Rankine-Hugoniot)
    const double A = 2.0 / ((gamma + 1.0) * w.rho), B = w.p * (gamma - 1.0) / (gamma + 1.0);
    const double r = sqrt(A / (B + p));
    *f = (p - w.p) * r;
    *df = r * (1.0 - 0.5 * (p - w.p) / (B + p));
  } else {  // rarefaction (isentropic)
    const double e = 0.5 * (gamma - 1.0) / gamma;
    const double q = pow(p / w.p, e);
    *f = 2.0 * w.c / (gamma - 1.0) * (q - 1.0);
    *df = q * w.c / (gamma * p);
  }
}

// Sec. 4.2.1, eq. Godunov_bc: the exact solution at x/t = 0 of the Riemann
// problem along nv with the node's state on the inside (left) and the far
// field outside (right)
template <int DIM>
__device__ void bc_godunov(double *u, const double *nv, const double *ud, double gamma) {
  const NormalState<DIM> L = split_normal<DIM>(u, nv, gamma), R = split_normal<DIM>(ud, nv, gamma);
  const double gm = gamma - 1.0, gp = gamma + 1.0, e = 0.5 * gm / gamma;
  const double jump = R.un - L.un;
  double rho, un, pr;
  const double *ut;
  if (2.0 * (L.c + R.c) / gm <= jump) {  // vacuum between two rarefactions
    const double head_l = L.un - L.c, edge_l = L.un + 2.0 * L.c / gm;
    const double edge_r = R.un - 2.0 * R.c / gm, head_r = R.un + R.c;
    if (head_l >= 0.0) {
      rho = L.rho; un = L.un; pr = L.p; ut = L.ut;
    } else if (edge_l > 0.0) {
      const double c = 2.0 / gp * (L.c + 0.5 * gm * L.un);
      rho = L.rho * pow(c / L.c, 2.0 / gm); un = c; pr = L.p * pow(c / L.c, 1.0 / e); ut = L.ut;
    } else if (edge_r >= 0.0) {
      rho = 0.0; un = 0.0; pr = 0.0; ut = L.ut;
    } else if (head_r > 0.0) {
      const double c = 2.0 / gp * (R.c - 0.5 * gm * R.un);
      rho = R.rho * pow(c / R.c, 2.0 / gm); un = -c; pr = R.p * pow(c / R.c, 1.0 / e); ut = R.ut;
    } else {
      rho = R.rho; un = R.un; pr = R.p; ut = R.ut;
    }
    join_normal<DIM>(rho, un, ut, pr, nv, gamma, u);
    if (rho == 0.0) {
#pragma unroll
      for (int s = 0; s < DIM + 2; ++s) u[s] = 0.0;
    }
    return;
  }
  // star pressure: Newton from the two-rarefaction value to a relative change of 1e-15
  double ps = pow((L.c + R.c - 0.5 * gm * jump) / (L.c * pow(L.p, -e) + R.c * pow(R.p, -e)), 1.0 / e);
  for (int it = 0; it < 100; ++it) {
    double fl, dl, fr, dr;
    wave_curve<DIM>(ps, L, gamma, &fl, &dl);
    wave_curve<DIM>(ps, R, gamma, &fr, &dr);
    double pn = ps - (fl + fr + jump) / (dl + dr);
    if (!(pn > 0.0)) pn = 0.5 * ps;
    const double rel = fabs(pn - ps) / (0.5 * (pn + ps));
    ps = pn;
    if (rel < 1e-15) break;
  }
  double fl, dl, fr, dr;
  wave_curve<DIM>(ps, L, gamma, &fl, &dl);
  wave_curve<DIM>(ps, R, gamma, &fr, &dr);
  const double us = 0.5 * (L.un + R.un + fr - fl);  // contact speed
  const bool left = us >= 0.0;
  const NormalState<DIM> &K = left ? L : R;
  const double sgn = left ? 1.0 : -1.0;  // mirror the right side onto the left
  ut = K.ut;
  const double uk = sgn * K.un, ustar = sgn * us;
  if (ps > K.p) {  // shock moving away from the contact
    const double speed = uk - K.c * sqrt(0.5 * gp / gamma * ps / K.p + e);
    if (speed >= 0.0) {
      rho = K.rho; un = K.un; pr = K.p;
    } else {
      const double r = ps / K.p, g6 = gm / gp;
      rho = K.rho * (r + g6) / (g6 * r + 1.0); un = us; pr = ps;
    }
  } else if (uk - K.c >= 0.0) {  // rarefaction entirely on the far side of x = 0
    rho = K.rho; un = K.un; pr = K.p;
  } else if (ustar - K.c * pow(ps / K.p, e) < 0.0) {  // x = 0 in the star region
    rho = K.rho * pow(ps / K.p, 1.0 / gamma); un = us; pr = ps;
  } else {  // x = 0 inside the rarefaction fan
    const double c = 2.0 / gp * (K.c + 0.5 * gm * uk);
    rho = K.rho * pow(c / K.c, 2.0 / gm); un = sgn * c; pr = K.p * pow(c / K.c, 1.0 / e);
  }
  join_normal<DIM>(rho, un, ut, pr, nv, gamma, u);
}

// Sec. 4 without the non-reflecting kinds: slip and Dirichlet applied, the
// return value tells whether the node is a non-reflecting one (its
// post-processing then runs in k_final_nonreflecting, out of the row kernel,
// whose register budget it would otherwise set)
template <int DIM>
__device__ __forceinline__ bool apply_bc_node_local(const MeshView &m, int i, double *u) {
  const int b = m.bnd_index[i];
  if (b < 0) return false;
  const int kind = m.bnd_kind[b];
  if (kind == 1) {  // slip: M <- M - (M . n^s) n^s
    double mn = 0.0;
#pragma unroll
    for (int q = 0; q < DIM; ++q) mn += u[1 + q] * m.bnd_normal[(int64_t)q * m.n_bnd + b];
#pragma unroll
    for (int q = 0; q < DIM; ++q) u[1 + q] -= mn * m.bnd_normal[(int64_t)q * m.n_bnd + b];
  } else if (kind == 2) {  // supersonic inflow: U <- U^D
#pragma unroll
    for (int s = 0; s < DIM + 2; ++s) u[s] = m.bnd_state[(int64_t)s * m.n_bnd + b];
  }
  return kind == 4 || kind == 5;
}

// Sec. 4: slip (M <- M - (M . n^s) n^s), Dirichlet / supersonic inflow
// (U <- U^D), do nothing, and the two non-reflecting post-processings
template <int DIM>
__device__ __forceinline__ void apply_bc_node(const MeshView &m, const Params &p, int i, double *u) {
  const int b = m.bnd_index[i];
  if (b < 0) return;
  const int kind = m.bnd_kind[b];
  if (kind == 1) {  // slip: M <- M - (M . n^s) n^s
    double mn = 0.0;
#pragma unroll
    for (int q = 0; q < DIM; ++q) mn += u[1 + q] * m.bnd_normal[(int64_t)q * m.n_bnd + b];
#pragma unroll
    for (int q = 0; q < DIM; ++q) u[1 + q] -= mn * m.bnd_normal[(int64_t)q * m.n_bnd + b];
  } else if (kind == 2) {  // supersonic inflow: U <- U^D
#pragma unroll
    for (int s = 0; s < DIM + 2; ++s) u[s] = m.bnd_state[(int64_t)s * m.n_bnd + b];
  } else if (kind == 4 || kind == 5) {
    double nv[DIM], ud[DIM + 2];
#pragma unroll
    for (int q = 0; q < DIM; ++q) nv[q] = m.bnd_normal[(int64_t)q * m.n_bnd + b];
#pragma unroll
    for (int s = 0; s < DIM + 2; ++s) ud[s] = m.bnd_state[(int64_t)s * m.n_bnd + b];
    if (kind == 4)
      bc_characteristic<DIM>(u, nv, ud, p.gamma);
    else
      bc_godunov<DIM>(u, nv, ud, p.gamma);
  }
}

// rho > 0 and E - |m|^2/(2 rho) > 0; the division only where FP32 does not show
// rho E - |m|^2/2 to be positive with a margin of 1e-5 rho E (its roundings: 12 x 2^-23)
template <int DIM>
__device__ __forceinline__ bool admissible(const double *u) {
  {
    const float r = trunc_f32(u[0]), e = trunc_f32(u[DIM + 1]);
    float m2 = 0.0f;
#pragma unroll
    for (int q = 0; q < DIM; ++q) {
      const float mq = trunc_f32(u[1 + q]);
      m2 += mq * mq;
    }
    const float re = r * e;
    if (r > 1e-15f && r < 1e15f && e > 1e-15f && e < 1e15f && re - 0.5f * m2 > 1e-5f * re) return true;
  }
  double m2 = 0.0;
#pragma unroll
  for (int q = 0; q < DIM; ++q) m2 += u[1 + q] * u[1 + q];
  return u[0] > 0.0 && (u[DIM + 1] - m2 / (2.0 * u[0])) > 0.0;
}

template <int DIM>
__device__ __forceinline__ void final_row(const MeshView &m, const Params &p, const Work &w, const double *__restrict__ Uin,
                                          const double *__restrict__ lin, const double *U0, double coef, double *out,
                                          double *Upre_trace, double *lsym_trace, int i) {
  constexpr int S = DIM + 2;
  constexpr int SP = Layout<DIM>::SP;
  const int64_t k0 = m.row_ptr[i], k1 = m.row_ptr[i + 1];
  const double lambda_i = m.lam[i];
  double u[S];
  load_vec<DIM>(Uin + (int64_t)i * SP, u);
  const unsigned char *lone = w.lone + (int64_t)((p.limiter_passes - 1) & 1) * m.n;  // of the last pass
  if (w.rough2[i] && p.limiter_passes >= 2 && w.spent[i] && !lsym_trace) {
    // nothing is left of P_ij
  } else if (w.rough2[i] && p.limiter_passes >= 2) {
    // the remainder rem P that the last k_pass left: where rem = 0 (most
    // entries) the update adds nothing, and the symmetrised limiter -- a
    // dependent gather of the transposed one -- is not needed. Four entries at a
    // time, so that their loads overlap (with the admissibility test's division
    // left out and the spent rows, k_final 71 -> 47 us on the 998k cylinder, 257 ->
    // 194 us at 4.0M vertices).
    const bool one_i = lone[i] != 0, spent = w.spent[i] != 0;
    for (int64_t kb = k0; kb < k1; kb += 4) {
      double r[4], l[4];
      int c[4], t[4];
      bool need[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        c[q] = kb + q < k1 ? m.col[kb + q] : i;
        r[q] = kb + q < k1 && !spent ? w.rem[kb + q] : 0.0;
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        need[q] = c[q] != i && (lsym_trace || dbits(r[q]) != 0);
        t[q] = need[q] ? m.tr[kb + q] : 0;
      }
#pragma unroll
      for (int q = 0; q < 4; ++q)
        l[q] = need[q] ? lmin(one_i ? 1.0 : lin[kb + q], lone[c[q]] ? 1.0 : lin[t[q]]) : 1.0;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        if (kb + q >= k1) break;
        if (lsym_trace) lsym_trace[kb + q] = l[q];
        if (!need[q] || dbits(r[q]) == 0) continue;
        double P[S];
        load_vec<DIM>(w.P + (kb + q) * SP, P);
#pragma unroll
        for (int s = 0; s < S; ++s) u[s] += lambda_i * l[q] * (r[q] * P[s]);
      }
    }
  } else if (w.rough2[i]) {  // else every P_ij is 0 (see lim1_row) and the update adds nothing
    for (int64_t kb = k0; kb < k1; kb += LCHUNK) {
      const int cnt = (int)min((int64_t)LCHUNK, k1 - kb);
      double ls[LCHUNK];
      bool dg[LCHUNK];
      sym_limiters(m, lin, lone, kb, cnt, i, ls, dg);
#pragma unroll
      for (int q = 0; q < LCHUNK; ++q) {
        if (q >= cnt) break;
        const int64_t k = kb + q;
        if (dg[q]) {
          if (lsym_trace) lsym_trace[k] = 1.0;
          continue;
        }
        if (lsym_trace) lsym_trace[k] = ls[q];
        const double *Pk = w.P + k * SP;
#pragma unroll
        for (int s = 0; s < S; ++s) u[s] += lambda_i * ls[q] * Pk[s];
      }
    }
  } else if (lsym_trace) {
    for (int64_t k = k0; k < k1; ++k) {
      const int j = m.col[k];
      lsym_trace[k] = j == i ? 1.0 : lmin(lone[i] ? 1.0 : lin[k], lone[j] ? 1.0 : lin[m.tr[k]]);
    }
  }
  if (Upre_trace) {
#pragma unroll
    for (int s = 0; s < S; ++s) Upre_trace[(int64_t)i * SP + s] = u[s];
  }
  // a finished instance (tau = 0) keeps its state bit for bit: the stage is
  // the identity there, and re-applying the post-processing would not be
  if (w.tau_inst[m.inst ? m.inst[i] : 0] != 0.0 && apply_bc_node_local<DIM>(m, i, u)) {
    // non-reflecting node: hand the state to k_final_nonreflecting (the
    // low-order increment rows are free at this point of the stage)
    double *h = w.inc + (int64_t)i * SP;
#pragma unroll
    for (int s = 0; s < S; ++s) h[s] = u[s];
    return;
  }
  if (coef >= 0.0) {
#pragma unroll
    for (int s = 0; s < S; ++s) {
      const double u0 = U0[(int64_t)s * m.n + i];
      u[s] = u0 + coef * (u[s] - u0);
    }
  }
  if (!admissible<DIM>(u)) {
    atomicAdd(&w.st->not_admissible, 1ull);
    atomicExch(&w.st->err, 4);  // EH_ERR_NOT_ADMISSIBLE
  }
#pragma unroll
  for (int s = 0; s < S; ++s) out[(int64_t)s * m.n + i] = u[s];
}

template <int DIM>
__global__ void __launch_bounds__(TPB_MAX) k_final(MeshView m, Params p, Work w, const double *__restrict__ Uin,
                                               const double *__restrict__ lin, const double *U0, double coef,
                                               double *out, double *Upre_trace, double *lsym_trace) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < m.n; i += gridDim.x * blockDim.x) {
    if (w.st->err) return;
    final_row<DIM>(m, p, w, Uin, lin, U0, coef, out, Upre_trace, lsym_trace, i);
  }
}

// the non-reflecting boundary nodes of a stage: post-processing (Sec. 4.2),
// SSP combination and admissibility, as k_final does for the other nodes
template <int DIM>
__global__ void __launch_bounds__(32) k_final_nonreflecting(MeshView m, Params p, Work w, const double *U0,
                                                             double coef, double *out) {
  constexpr int S = DIM + 2;
  constexpr int SP = Layout<DIM>::SP;
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= m.n_bnd || w.st->err) return;
  const int kind = m.bnd_kind[b];
  if (kind != 4 && kind != 5) return;
  const int i = m.bnd_node[b];
  if (w.tau_inst[m.inst ? m.inst[i] : 0] == 0.0) return;  // frozen instance: k_final wrote it
  double u[S], nv[DIM], ud[S];
#pragma unroll
  for (int s = 0; s < S; ++s) {
    u[s] = w.inc[(int64_t)i * SP + s];
    ud[s] = m.bnd_state[(int64_t)s * m.n_bnd + b];
  }
#pragma unroll
  for (int q = 0; q < DIM; ++q) nv[q] = m.bnd_normal[(int64_t)q * m.n_bnd + b];
  if (kind == 4)
    bc_characteristic<DIM>(u, nv, ud, p.gamma);
  else
    bc_godunov<DIM>(u, nv, ud, p.gamma);
  if (coef >= 0.0) {
#pragma unroll
    for (int s = 0; s < S; ++s) {
      const double u0 = U0[(int64_t)s * m.n + i];
      u[s] = u0 + coef * (u[s] - u0);
    }
  }
  if (!admissible<DIM>(u)) {
    atomicAdd(&w.st->not_admissible, 1ull);
    atomicExch(&w.st->err, 4);  // EH_ERR_NOT_ADMISSIBLE
  }
#pragma unroll
  for (int s = 0; s < S; ++s) out[(int64_t)s * m.n + i] = u[s];
}

template <int DIM> __global__ void k_apply_bc(MeshView m, Params p, double *U) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= m.n || m.bnd_index[i] < 0) return;
  double u[DIM + 2];
#pragma unroll
  for (int s = 0; s < DIM + 2; ++s) u[s] = U[(int64_t)s * m.n + i];
  apply_bc_node<DIM>(m, p, i, u);
#pragma unroll
  for (int s = 0; s < DIM + 2; ++s) U[(int64_t)s * m.n + i] = u[s];
}

template <int DIM> __global__ void k_count_not_admissible(int n, const double *U, DevStatus *st) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  double u[DIM + 2];
#pragma unroll
  for (int s = 0; s < DIM + 2; ++s) u[s] = U[(int64_t)s * n + i];
  if (!admissible<DIM>(u)) atomicAdd(&st->not_admissible, 1ull);
}

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
// rows below which the split forms run. Microseconds a launch, row form / split
// form, FP64, flow behind a shock (perturbed flow):
//   2D rows           8k          24k          40k          62k          77k
//   k_visc + k_alpha  27/21       33/29        38/38 (40/41) 46/48        50/53
//   k_low             26/20       27/27 (23/27) 29/35       35/43        40/48
//   k_lim1            40/20       41/29        44/39        51/49 (41/46) 56/54 (44/52)
//   k_pass            39/22       39/24        40/28        42/38 (27/27) 43/44 (28/32)
//   3D rows           5k          16k          29k          35k          62k          76k
//   k_visc + k_alpha  57/35       73/53        95/75        107/88       140/130      147/141
//   k_low             74/33       79/54        87/78 (73/64) 90/95 (76/79) 115/136     123/158
//   k_lim1            127/40      135/60       150/95       157/107      190/153 (128/128) 215/183 (142/146)
//   k_pass            124/57      139/64       153/78       155/112      174/156 (104/122) 193/190 (110/147)
// In 3D the lines are where k_low and k_lim1 cross; in 2D k_low crosses earlier,
// between 16k and 24k rows, and k_alpha later. (The launch shape of
// eh_set_launch_shape applies to the row forms.)
constexpr int SPLIT_SUMS = 32 * 1024;     // k_alpha, k_low: the warps repeat loads and half of the products
constexpr int SPLIT_ENTRIES = 64 * 1024;  // k_lim1, k_pass: the entries are independent
// Additions on the integer units (add_on<true>) in 2D k_low and k_lim1 from here
// on. Below, one wave of the form with FP64 additions holds all rows (92 to 106
// registers, 152 SMs x 576 rows = 88k) and finishes sooner: 40 against 47 us for
// k_low at 78k rows behind a shock; at 103k it takes a second wave: k_low 61
// against 50 us, k_lim1 61 against 51 (developed flow; behind a shock 45 against
// 54 and 58 against 59), at 998k 391 against 336 and 386 against 328. 3D k_low has
// them from SPLIT_SUMS on (95k rows 175 -> 172 us), 3D k_lim1 nowhere (625 -> 642 us).
constexpr int ALU_ROWS = 96 * 1024;
bool launch_shape_used(int kernel, int64_t n, int limiter_passes) {
  switch (kernel) {
    case EH_KERNEL_LOW: return n >= SPLIT_SUMS;
    case EH_KERNEL_LIM1: return n >= SPLIT_ENTRIES;
    case EH_KERNEL_PASS: return n >= SPLIT_ENTRIES || limiter_passes > 2;  // the first of the passes is split
    default: return true;
  }
}
template <int DIM, typename T>
void launch_prep(const MeshView &m, const Params &p, const double *U, const Work &w, int tpb, cudaStream_t s) {
  k_prep<DIM, T><<<nblocks(m.n, tpb), tpb, 0, s>>>(m, p, U, w.rec, (T *)w.vrec, w.rough, w.steady, w.st);
}
template <int DIM, typename T>
void launch_visc(const MeshView &m, const Params &p, const Work &w, int tpb, cudaStream_t s) {
  // warps a 32-row chunk, by the rows there are for the chip's 608 FP64 units:
  // small meshes split the rows' chains (4k-vertex P1 vortex, k_visc + k_alpha
  // 30.4 / 24.6 / 21.7 us with 1 / 2 / 4 warps; 62k cylinder 59.2 / 59.3 /
  // 53.5), large ones read node i once (998k cylinder 552 / 565 / 642; between,
  // 246k cylinder behind a shock 252 / 208 / 209, 375k in 3D 830 / 824 / 834)
  const int lparts = m.n < 160 * 1024 ? 2 : m.n < 640 * 1024 ? 1 : 0;
  const unsigned rows = nblocks((int64_t)nblocks(m.n, 32) << lparts, tpb / 32);
  // differences on the integer units where the FP64 pipe is full (FP64 form 358 ->
  // 299 us at 998k rows, 78k 54.7 -> 53.2, 3D 95k 238 -> 216); small meshes wait on
  // latencies instead (4k vortex: 17.9 us on the FP64 pipe, 19.1 on the integer
  // units). The mixed form's differences are FP32 ones already.
  const unsigned grid = rows + nblocks(m.n_bp, tpb);
  if (sizeof(T) == 8 && m.n >= SPLIT_ENTRIES)
    k_visc<DIM, T, sizeof(T) == 8><<<grid, tpb, 0, s>>>(m, p, w, rows, lparts);
  else
    k_visc<DIM, T, false><<<grid, tpb, 0, s>>>(m, p, w, rows, lparts);
}
template <int DIM, typename T>
void launch_alpha(const MeshView &m, const Params &p, const Work &w, int tpb, cudaStream_t s) {
  if (m.n < SPLIT_SUMS)
    k_alpha_split<DIM, T><<<nblocks(m.n, 32), 32 * PARTS, 0, s>>>(m, p, w);
  else
    k_alpha<DIM, T><<<nblocks(m.n, tpb), tpb, 0, s>>>(m, p, w);
}
template <int DIM, typename T>
void launch_low(const MeshView &m, const Params &p, const Work &w, int tpb, cudaStream_t s) {
  if (m.n < SPLIT_SUMS)
    k_low_split<DIM, T><<<nblocks(m.n, 32), 32 * (DIM + 3), 0, s>>>(m, p, w);
  else if (DIM == 2 && m.n < ALU_ROWS)
    k_low<DIM, T, DIM == 3><<<nblocks(m.n, tpb), tpb, 0, s>>>(m, p, w);
  else
    k_low<DIM, T, true><<<nblocks(m.n, tpb), tpb, 0, s>>>(m, p, w);
}
void launch_tau(const MeshView &m, const Work &w, int stage, double dt_given, double cfl, bool advance_time,
                cudaStream_t s) {
  k_tau<<<nblocks(m.ninst, 256), 256, 0, s>>>(m, w, stage, dt_given, cfl, advance_time ? 1 : 0);
}
// grid of the grid-stride row kernels: one thread per row, or at most
// max_blocks blocks (max_blocks > 0)
inline unsigned capped_grid(int64_t n, int tpb, int max_blocks) {
  const unsigned g = nblocks(n, tpb);
  return (max_blocks > 0 && g > (unsigned)max_blocks) ? (unsigned)max_blocks : g;
}
template <int DIM, typename T>
void launch_lim1(const MeshView &m, const Params &p, const Work &w, double *P_trace, int tpb, int max_blocks,
                 cudaStream_t s) {
  if (m.n < SPLIT_ENTRIES)
    k_lim1_split<DIM, T><<<nblocks(m.n, 32), 32 * PARTS, 0, s>>>(m, p, w, P_trace);
  else if (DIM == 3 || m.n < ALU_ROWS)
    k_lim1<DIM, T, false><<<capped_grid(m.n, tpb, max_blocks), tpb, 0, s>>>(m, p, w, P_trace);
  else
    k_lim1<DIM, T, DIM == 2><<<capped_grid(m.n, tpb, max_blocks), tpb, 0, s>>>(m, p, w, P_trace);
}
template <int DIM>
void launch_pass(const MeshView &m, const Params &p, const Work &w, const double *Uin, double *Uout, const double *lin,
                 double *lout, double *lsym_trace, int slot, int tpb, int max_blocks, cudaStream_t s) {
  if (slot == 1 && m.n < SPLIT_ENTRIES)
    k_pass_split<DIM><<<nblocks(m.n, 32), 32 * PARTS, 0, s>>>(m, p, w, Uin, Uout, lin, lout, lsym_trace);
  else
    k_pass<DIM><<<capped_grid(m.n, tpb, max_blocks), tpb, 0, s>>>(m, p, w, Uin, Uout, lin, lout, lsym_trace, slot);
}
template <int DIM>
void launch_ls_deferred(const MeshView &m, const Params &p, const Work &w, const double *ub, int slot, double *lout,
                        int tpb, cudaStream_t s) {
  // a fixed grid (1024 threads per SM of a 152-SM GB300) that strides over
  // however many searches were queued; the count stays on the device
  k_ls_deferred<DIM><<<152 * 1024 / tpb, tpb, 0, s>>>(m, p, w, ub, slot, lout);
  k_ls_iterate<DIM><<<152 * 1024 / tpb, tpb, 0, s>>>(m, p, w, ub, slot, lout);
}
template <int DIM>
void launch_final(const MeshView &m, const Params &p, const Work &w, const double *Uin, const double *lin,
                  const double *U0, double coef, double *out, double *Upre_trace, double *lsym_trace, int tpb,
                  int max_blocks, cudaStream_t s) {
  k_final<DIM><<<capped_grid(m.n, tpb, max_blocks), tpb, 0, s>>>(m, p, w, Uin, lin, U0, coef, out, Upre_trace,
                                                                 lsym_trace);
  if (m.n_nonreflecting > 0)
    // a warp a block: the few hundred nodes of a boundary run chains of ~400 FP64
    // instructions (three powers); eight warps on one SM share its FP64 rate
    // (80 x 80 box: 49 -> 35 us with k_final)
    k_final_nonreflecting<DIM><<<nblocks(m.n_bnd, 32), 32, 0, s>>>(m, p, w, U0, coef, out);
}
template <int DIM> void launch_apply_bc(const MeshView &m, const Params &p, double *U, cudaStream_t s) {
  k_apply_bc<DIM><<<nblocks(m.n, 256), 256, 0, s>>>(m, p, U);
}
// min_i rho_i, min_i e_i (e = E/rho - |m|^2/(2 rho^2)) and sum_i m_i U_i over
// the whole state: a fixed grid of STAT_BLOCKS blocks with a grid stride,
// fixed shuffle and shared-memory trees per block, then one block summing the
// partials in a fixed order -- the same bits on every run
template <int DIM> __global__ void __launch_bounds__(256) k_state_partial(int n, const double *__restrict__ U,
                                                                        const double *__restrict__ mi,
                                                                        double *__restrict__ part) {
  constexpr int S = DIM + 2, NV = S + 2;
  double v[NV];
  v[0] = INFINITY;
  v[1] = INFINITY;
#pragma unroll
  for (int s = 0; s < S; ++s) v[2 + s] = 0.0;
  for (int i = blockIdx.x * 256 + threadIdx.x; i < n; i += STAT_BLOCKS * 256) {
    double u[S];
#pragma unroll
    for (int s = 0; s < S; ++s) u[s] = U[(int64_t)s * n + i];
    const double irho = 1.0 / u[0];
    double m2 = 0.0;
#pragma unroll
    for (int q = 0; q < DIM; ++q) m2 += u[1 + q] * u[1 + q];
    v[0] = fmin(v[0], u[0]);
    v[1] = fmin(v[1], u[S - 1] * irho - 0.5 * m2 * irho * irho);
    const double m = mi[i];
#pragma unroll
    for (int s = 0; s < S; ++s) v[2 + s] += m * u[s];
  }
  __shared__ double sh[NV][8];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int q = 0; q < NV; ++q) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const double x = __shfl_down_sync(0xffffffffu, v[q], o);
      v[q] = q < 2 ? fmin(v[q], x) : v[q] + x;
    }
    if (lane == 0) sh[q][warp] = v[q];
  }
  __syncthreads();
  if (threadIdx.x < NV) {
    const int q = threadIdx.x;
    double acc = sh[q][0];
    for (int w = 1; w < 8; ++w) acc = q < 2 ? fmin(acc, sh[q][w]) : acc + sh[q][w];
    part[q * STAT_BLOCKS + blockIdx.x] = acc;
  }
}

__global__ void k_state_final(int nv, const double *__restrict__ part, double *__restrict__ out) {
  const int q = threadIdx.x;
  if (q >= nv) return;
  double acc = part[q * STAT_BLOCKS];
  for (int b = 1; b < STAT_BLOCKS; ++b) acc = q < 2 ? fmin(acc, part[q * STAT_BLOCKS + b]) : acc + part[q * STAT_BLOCKS + b];
  out[q] = acc;
}

template <int DIM>
void launch_state_stats(int n, const double *U, const double *mi, double *part, double *out, cudaStream_t s) {
  k_state_partial<DIM><<<STAT_BLOCKS, 256, 0, s>>>(n, U, mi, part);
  k_state_final<<<1, 32, 0, s>>>(DIM + 4, part, out);
}
template <int DIM> void launch_count_not_admissible(int n, const double *U, DevStatus *st, cudaStream_t s) {
  k_count_not_admissible<DIM><<<nblocks(n, 256), 256, 0, s>>>(n, U, st);
}

// ---------------------------------------------------------------------------
// the mesh's checks and static arrays (eh_upload_mesh), one thread per row; on
// the host, one pass each over the entries for the checks, the transpose (a
// binary search an entry) and the norms took most of an upload (998k vertices,
// 9.0M entries: 104 ms; here 8.5 ms, bound by the copies of the caller's arrays)
// ---------------------------------------------------------------------------
__device__ __forceinline__ void mesh_error(unsigned long long *err, int phase, int row) {
  atomicMin(err, (unsigned long long)phase << 32 | (unsigned)row);
}
// an error of an earlier phase (one of the same phase leaves the other rows
// running: the smallest row counts, not the first thread)
__device__ __forceinline__ bool mesh_failed(const unsigned long long *err, int phase) {
  return (*(const volatile unsigned long long *)err >> 32) < (unsigned)phase;
}

__global__ void k_mesh_rows(MeshView m, double *inv_mi, double *lam, unsigned long long *err) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= m.n) return;
  const int64_t k0 = m.row_ptr[i], k1 = m.row_ptr[i + 1];
  bool diag = false, ok = m.mi[i] > 0.0;
  int prev = -1;
  for (int64_t k = k0; k < k1; ++k) {
    const int c = m.col[k];
    ok &= c > prev && c < m.n;
    diag |= c == i;
    prev = c;
  }
  if (!ok || !diag) mesh_error(err, 0, i);
  inv_mi[i] = 1.0 / m.mi[i];
  lam[i] = 1.0 / (double)(k1 - k0 - 1);
}

__global__ void k_mesh_transpose(MeshView m, int32_t *tr, unsigned long long *err) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= m.n || mesh_failed(err, 1)) return;
  for (int64_t k = m.row_ptr[i]; k < m.row_ptr[i + 1]; ++k) {
    const int j = m.col[k];
    int64_t lo = m.row_ptr[j], hi = m.row_ptr[j + 1];
    const int64_t end = hi;
    while (lo < hi) {  // the first entry of row j that is >= i
      const int64_t mid = lo + (hi - lo) / 2;
      if (m.col[mid] < i) lo = mid + 1; else hi = mid;
    }
    if (lo == end || m.col[lo] != i) {
      mesh_error(err, 1, i);
      return;
    }
    tr[k] = (int32_t)lo;
  }
}

template <int DIM, typename T>
__global__ void k_mesh_entries(MeshView m, const double *cij, const double *mij, T *geo, T *geo_inv, double *betat,
                               unsigned long long *err) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= m.n || mesh_failed(err, 2)) return;
  for (int64_t k = m.row_ptr[i]; k < m.row_ptr[i + 1]; ++k) {
    double c[DIM], s2 = 0.0;
#pragma unroll
    for (int q = 0; q < DIM; ++q) {
      c[q] = cij[(int64_t)q * m.nnz + k];
      s2 = __fma_rn(c[q], c[q], s2);
    }
    const double cn = sqrt(s2), ci = cn > 0.0 ? 1.0 / cn : 0.0;
    if (m.col[k] != i && !(cn > 0.0)) {
      mesh_error(err, 2, i);
      return;
    }
#pragma unroll
    for (int q = 0; q < DIM; ++q) geo[4 * k + q] = (T)c[q];
    geo[4 * k + DIM] = (T)cn;
    if constexpr (DIM == 2) geo[4 * k + 3] = (T)ci; else geo_inv[k] = (T)ci;
    // the consistent mass matrix is symmetric (m_ij = int phi_i phi_j);
    // k_lim1 relies on it, with the mean of the two entries
    const double a = mij[k], b = mij[m.tr[k]];
    if (fabs(a - b) > 1e-12 * fmax(fabs(a), fabs(b))) {
      mesh_error(err, 2, i);
      return;
    }
    betat[k] = 0.5 * (a + b) / m.mi[i];
  }
}

__global__ void k_mesh_boundary(MeshView m, int32_t *bnd_index, unsigned char *isb) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= m.n_bnd) return;
  bnd_index[m.bnd_node[b]] = b;
  isb[m.bnd_node[b]] = 1;
}

void launch_mesh_rows(const MeshView &m, double *inv_mi, double *lam, unsigned long long *err, cudaStream_t s) {
  k_mesh_rows<<<nblocks(m.n, 128), 128, 0, s>>>(m, inv_mi, lam, err);
}
void launch_mesh_transpose(const MeshView &m, int32_t *tr, unsigned long long *err, cudaStream_t s) {
  k_mesh_transpose<<<nblocks(m.n, 128), 128, 0, s>>>(m, tr, err);
}
template <int DIM, typename T>
void launch_mesh_entries(const MeshView &m, const double *cij, const double *mij, T *geo, T *geo_inv, double *betat,
                         unsigned long long *err, cudaStream_t s) {
  k_mesh_entries<DIM, T><<<nblocks(m.n, 128), 128, 0, s>>>(m, cij, mij, geo, geo_inv, betat, err);
}
void launch_mesh_boundary(const MeshView &m, int32_t *bnd_index, unsigned char *isb, cudaStream_t s) {
  if (m.n_bnd > 0) k_mesh_boundary<<<nblocks(m.n_bnd, 256), 256, 0, s>>>(m, bnd_index, isb);
}

__global__ void k_gather_second(double *dst, const double *pairs, int64_t count) {
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k < count) dst[k] = pairs[2 * k + 1];
}
void launch_gather_second(double *dst, const double *pairs, int64_t count, cudaStream_t s) {
  k_gather_second<<<nblocks(count, 256), 256, 0, s>>>(dst, pairs, count);
}

// dst[i] = src[i] + add (nonneg_only: only where src[i] >= 0; -1 entries
// stay): the index arrays of one instance placed into a block-diagonal union
template <typename I> __global__ void k_offset_copy(I *dst, const I *src, int64_t count, I add, int nonneg_only) {
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < count; q += (int64_t)gridDim.x * blockDim.x) {
    const I v = src[q];
    dst[q] = (nonneg_only && v < 0) ? v : v + add;
  }
}
template <typename I>
void launch_offset_copy(I *dst, const I *src, int64_t count, I add, bool nonneg_only, cudaStream_t s) {
  if (count <= 0) return;
  const unsigned grid = (unsigned)std::min<int64_t>((count + 255) / 256, 152 * 16);
  k_offset_copy<I><<<grid, 256, 0, s>>>(dst, src, count, add, nonneg_only ? 1 : 0);
}
template void launch_offset_copy<int32_t>(int32_t *, const int32_t *, int64_t, int32_t, bool, cudaStream_t);
template void launch_offset_copy<int64_t>(int64_t *, const int64_t *, int64_t, int64_t, bool, cudaStream_t);

#define EH_INSTANTIATE_T(DIM, T)                                                                                     \
  template void launch_mesh_entries<DIM, T>(const MeshView &, const double *, const double *, T *, T *, double *,      \
                                            unsigned long long *, cudaStream_t);                                     \
  template void launch_prep<DIM, T>(const MeshView &, const Params &, const double *, const Work &, int, cudaStream_t); \
  template void launch_visc<DIM, T>(const MeshView &, const Params &, const Work &, int, cudaStream_t);               \
  template void launch_alpha<DIM, T>(const MeshView &, const Params &, const Work &, int, cudaStream_t);              \
  template void launch_low<DIM, T>(const MeshView &, const Params &, const Work &, int, cudaStream_t);                \
  template void launch_lim1<DIM, T>(const MeshView &, const Params &, const Work &, double *, int, int, cudaStream_t);

EH_INSTANTIATE_T(2, double)
EH_INSTANTIATE_T(3, double)
EH_INSTANTIATE_T(2, float)
EH_INSTANTIATE_T(3, float)

#define EH_INSTANTIATE(DIM)                                                                                          \
  template void launch_pass<DIM>(const MeshView &, const Params &, const Work &, const double *, double *,            \
                                 const double *, double *, double *, int, int, int, cudaStream_t);                    \
  template void launch_ls_deferred<DIM>(const MeshView &, const Params &, const Work &, const double *, int, double *, \
                                        int, cudaStream_t);                                                          \
  template void launch_final<DIM>(const MeshView &, const Params &, const Work &, const double *, const double *,     \
                                  const double *, double, double *, double *, double *, int, int, cudaStream_t);      \
  template void launch_apply_bc<DIM>(const MeshView &, const Params &, double *, cudaStream_t);                       \
  template void launch_count_not_admissible<DIM>(int, const double *, DevStatus *, cudaStream_t);            \
  template void launch_state_stats<DIM>(int, const double *, const double *, double *, double *, cudaStream_t);

EH_INSTANTIATE(2)
EH_INSTANTIATE(3)

}  // namespace eh
