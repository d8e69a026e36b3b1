// noalloc.cu -- eh_cfl_dt_noalloc: the CFL time step computed from caller-owned
// device arrays without allocating anything.
//
// Why it exists: some callers cannot call cudaMalloc at the point where they
// need a time step -- a host framework that owns every byte of device memory
// through its own pool and forbids allocation from plug-in libraries, or a
// real-time loop where an allocation (which may synchronise the device and
// take milliseconds) is not allowed. They cannot create an eh_ctx either,
// since eh_upload_mesh allocates. This entry point needs only their own device
// arrays: its one piece of scratch memory, the per-block minima of the
// reduction, is the file-scope array below, sized for EH_CFL_NOALLOC_MAX_ROWS
// rows and kept by every GPU that loads the library until the process exits.
#include <cuda.h>
#include <cuda_runtime.h>

#include <cmath>
#include <mutex>

#include "../../include/euler_hyp.h"

namespace {

constexpr int kThreads = 128;
constexpr int kMaxBlocks = EH_CFL_NOALLOC_MAX_ROWS / kThreads;
constexpr int kMaxDevices = 64;

// The scratch: one 8-byte slot per block of kThreads rows (512 KiB; the lower end
// of the block's FP32 bracket) and two more: the smallest upper end over all
// blocks, and the order key of the smallest exact bound.
static __device__ __align__(256) double g_cfl_block_min[kMaxBlocks + 2];

// Device address of g_cfl_block_min, looked up once per device and context:
// the address belongs to the module loaded into one CUDA context, so the cache
// is keyed on that context's process-unique id (a device reset or a new
// primary context gets a new id, and the address is looked up again).
struct ScratchEntry {
  unsigned long long ctx_id;
  double *addr;
};
ScratchEntry g_scratch[kMaxDevices] = {};
std::mutex g_scratch_mutex;

// ---------------------------------------------------------------------------
// The exact bound of a row, in FP64
// ---------------------------------------------------------------------------
// state, pressure, sound speed, a p^-z and 1/p of node i
template <int DIM> struct Node {
  double rho, m[DIM], E, p, a, az, ip;
};

template <int DIM> __device__ inline Node<DIM> load_state(const double *U, int n, int i) {
  Node<DIM> w;
  w.rho = U[i];
#pragma unroll
  for (int q = 0; q < DIM; ++q) w.m[q] = U[(int64_t)(1 + q) * n + i];
  w.E = U[(int64_t)(DIM + 1) * n + i];
  return w;
}

// x^(-1/7): Newton's method on r^-7 = x, r <- r (8 - x r^7) / 7, from an FP32 seed
// (gamma = 7/5: p^-z with a tenth of pow's FP64 instructions; the same accuracy)
__device__ inline double inverse_root7(double x) {
  if (!(x > 1e-30 && x < 1e30)) return pow(x, -1.0 / 7.0);
  double r = (double)exp2f((-1.0f / 7.0f) * log2f((float)x));
#pragma unroll
  for (int it = 0; it < 2; ++it) {
    const double r2 = r * r, r7 = r2 * r2 * r2 * r;
    r = r * (8.0 - x * r7) * (1.0 / 7.0);
  }
  return r;
}

template <int DIM> __device__ inline void derive(Node<DIM> &w, double gamma) {
  double m2 = 0.0;
#pragma unroll
  for (int q = 0; q < DIM; ++q) m2 += w.m[q] * w.m[q];
  double eps = w.E - m2 / (2.0 * w.rho);
  w.p = (gamma - 1.0) * eps;
  w.a = sqrt(gamma * w.p / w.rho);
  w.az = w.a * (gamma == 1.4 ? inverse_root7(w.p) : pow(w.p, -(gamma - 1.0) / (2.0 * gamma)));
  w.ip = 1.0 / w.p;
}

// normal velocity of node w along the unit vector c * cinv
template <int DIM> __device__ inline double normal_velocity(const Node<DIM> &w, const double *c, double cinv) {
  double mn = 0.0;
#pragma unroll
  for (int q = 0; q < DIM; ++q) mn += w.m[q] * (c[q] * cinv);
  return mn / w.rho;
}

// Upper bound on the maximum wave speed (two-rarefaction pressure, then the
// outer shock speeds evaluated there).
template <int DIM>
__device__ inline double wave_bound(const Node<DIM> &l, double ul, const Node<DIM> &r, double ur, double gamma) {
  double num = fmax(l.a + r.a - 0.5 * (gamma - 1.0) * (ur - ul), 0.0);
  const double x = num / (l.az + r.az), x2 = x * x, x4 = x2 * x2;
  double ptr = gamma == 1.4 ? x4 * x2 * x : pow(x, 2.0 * gamma / (gamma - 1.0));
  double k = (gamma + 1.0) / (2.0 * gamma);
  double sl = ptr > l.p ? sqrt(1.0 + k * (ptr - l.p) * l.ip) : 1.0;
  double sr = ptr > r.p ? sqrt(1.0 + k * (ptr - r.p) * r.ip) : 1.0;
  return fmax(fmax(-(ul - l.a * sl), 0.0), fmax(ur + r.a * sr, 0.0));
}

// the position of entry (j, i) in the sorted row j, -1 if it is missing
// (unreachable for a symmetric pattern). 'guess' is tried first: rows of a
// structured mesh mirror each other.
__device__ inline int64_t transposed(const int64_t *row_ptr, const int32_t *col, int i, int j, int64_t from_start) {
  int64_t lo = row_ptr[j], hi = row_ptr[j + 1] - 1;
  const int64_t guess = hi - from_start;
  if (guess >= lo && col[guess] == i) return guess;
  while (lo <= hi) {
    const int64_t mid = lo + (hi - lo) / 2;
    const int cm = col[mid];
    if (cm == i) return mid;
    if (cm < i) lo = mid + 1; else hi = mid - 1;
  }
  return -1;
}

// the caller's arrays
struct Arrays {
  int n;
  int64_t nnz;
  const int64_t *row_ptr;
  const int32_t *col;
  const double *cij, *mi;
  const unsigned char *isb;
  const double *U;
  double gamma, cfl;
};

// d_ij of entry k of row i (column j != i), evaluated in its canonical
// orientation (from the row of min(i, j)), with the maximum over both
// directions when both nodes are boundary nodes; 'own' is node i, derived. For
// two states equal bit for bit the two-rarefaction pressure is the common
// pressure, both outer waves are rarefactions and the bound is max(a - v.n, v.n + a): no
// root, power or division (a uniform flow, where every row ties for the
// minimum and is evaluated here, then costs a few operations an entry).
template <int DIM>
__device__ inline double graph_viscosity(const Arrays &g, int i, int j, int64_t k, const Node<DIM> &own) {
  const int64_t kt = transposed(g.row_ptr, g.col, i, j, k - g.row_ptr[i]);
  if (kt < 0) return 0.0;
  Node<DIM> w = load_state<DIM>(g.U, g.n, j);
  bool same = __double_as_longlong(w.rho) == __double_as_longlong(own.rho) &&
              __double_as_longlong(w.E) == __double_as_longlong(own.E);
#pragma unroll
  for (int q = 0; q < DIM; ++q) same &= __double_as_longlong(w.m[q]) == __double_as_longlong(own.m[q]);
  if (!same) derive(w, g.gamma);
  const bool up = j > i;  // i is the left state of the canonical orientation
  const Node<DIM> l = up ? own : w, r = up ? w : own;
  double d = 0.0;
  const int directions = g.isb && g.isb[i] && g.isb[j] ? 2 : 1;
  for (int b = 0; b < directions; ++b) {
    // b = 0: from min(i, j) to max(i, j); b = 1: the other way round
    const int64_t pos = (up != (b == 1)) ? k : kt;
    double c[DIM], s2 = 0.0;
#pragma unroll
    for (int q = 0; q < DIM; ++q) {
      c[q] = g.cij[(int64_t)q * g.nnz + pos];
      s2 += c[q] * c[q];
    }
    const double cn = sqrt(s2);
    double lam;
    if (same) {
      // (as wave_bound: fmax drops the NaN of an entry with c = 0, whose d_ij is 0)
      const double ci = 1.0 / cn, un = normal_velocity(own, c, ci);
      lam = fmax(fmax(own.a - un, 0.0), fmax(un + own.a, 0.0));
    } else {
      const double ci = 1.0 / cn;
      const double ul = normal_velocity(l, c, ci), ur = normal_velocity(r, c, ci);
      lam = b == 0 ? wave_bound(l, ul, r, ur, g.gamma) : wave_bound(r, ur, l, ul, g.gamma);
    }
    d = b == 0 ? lam * cn : fmax(d, lam * cn);
  }
  return d;
}

// An integer key with the order of the doubles, a NaN below everything: a row
// whose state is not admissible (rho <= 0 or internal energy <= 0) gives a NaN
// bound, which must reach dt_out instead of being dropped by the reduction.
__device__ __forceinline__ long long bound_key(double x) {
  if (x != x) return (long long)0x8000000000000000ull;
  const long long b = __double_as_longlong(x);
  return b ^ ((b >> 63) & 0x7FFFFFFFFFFFFFFFLL);
}
__device__ __forceinline__ double key_bound(long long k) {
  if (k == (long long)0x8000000000000000ull) return NAN;
  return __longlong_as_double(k ^ ((k >> 63) & 0x7FFFFFFFFFFFFFFFLL));
}

// the row's own state must be admissible: otherwise the wave speeds are
// undefined and the step is NaN
template <int DIM> __device__ inline bool admissible(const Node<DIM> &w) {
  double m2 = 0.0;
#pragma unroll
  for (int q = 0; q < DIM; ++q) m2 += w.m[q] * w.m[q];
  return w.rho > 0.0 && w.E - m2 / (2.0 * w.rho) > 0.0;
}

// c_cfl m_i / (2 sum_j d_ij) of row i by one thread
template <int DIM> __device__ inline double row_bound(const Arrays &g, int i) {
  Node<DIM> own = load_state<DIM>(g.U, g.n, i);
  derive(own, g.gamma);
  double dsum = 0.0;
  for (int64_t k = g.row_ptr[i]; k < g.row_ptr[i + 1]; ++k) {
    const int j = g.col[k];
    if (j != i) dsum += graph_viscosity<DIM>(g, i, j, k, own);
  }
  return admissible(own) ? g.cfl * g.mi[i] / (2.0 * dsum) : NAN;
}

// the same by one warp, an entry per lane, summed in the same order
template <int DIM> __device__ inline double row_bound_warp(const Arrays &g, int i) {
  const int lane = threadIdx.x & 31;
  Node<DIM> own = load_state<DIM>(g.U, g.n, i);
  derive(own, g.gamma);
  double dsum = 0.0;
  const int64_t k0 = g.row_ptr[i], k1 = g.row_ptr[i + 1];
  for (int64_t kb = k0; kb < k1; kb += 32) {
    const int64_t k = kb + lane;
    const int j = k < k1 ? g.col[k] : i;
    const double d = j != i ? graph_viscosity<DIM>(g, i, j, k, own) : 0.0;
    __syncwarp();
    const int cnt = (int)(k1 - kb < 32 ? k1 - kb : 32);
    for (int q = 0; q < cnt; ++q) {
      const double dq = __shfl_sync(0xffffffffu, d, q);
      if (g.col[kb + q] != i) dsum += dq;
    }
  }
  return admissible(own) ? g.cfl * g.mi[i] / (2.0 * dsum) : NAN;
}

// ---------------------------------------------------------------------------
// The FP32 bracket of a row's bound. Only the smallest bound is wanted, and
// FP64 issues at 1/76 of the FP32 rate on this part: every row's bound is
// bracketed in FP32, and only rows whose lower end does not exceed the smallest
// upper end are evaluated in FP64. 998k-vertex Q1 cylinder, perturbed flow:
// 6757 us with every entry in FP64 (3 powers, 2 roots and 6 divisions an entry),
// 275 us with FP32 interval arithmetic (both ends of every quantity, 520
// instructions an entry), 179 us with a value and an error bound for each: bound by
// instruction issue in k_cfl_bracket. The bounds carry every rounding (u = 2^-23
// per conversion or operation is twice what either does; log2f and exp2f are
// within 2 units); a row with anything out of FP32's range, or not clearly
// admissible, gets (-inf, inf) and is evaluated in FP64.
// ---------------------------------------------------------------------------
struct Bracket {
  float lo, hi;
};

constexpr float kU = 1.1920929e-7f;  // 2^-23

// x rounded towards zero to FP32 on the integer units (an FP64 -> FP32
// conversion instruction costs a large part of an FP64 issue slot): 0 below
// 2^-126, +-inf from 2^127 on and for NaN
__device__ __forceinline__ float trunc_f32(double x) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const unsigned e = (hi >> 20) & 0x7ffu;
  const unsigned mag = __funnelshift_l(lo, hi, 3) - (384u << 23);
  unsigned r = (mag & 0x7fffffffu) | (hi & 0x80000000u);
  if (e < 897u) r = hi & 0x80000000u;
  if (e > 1149u) r = (hi & 0x80000000u) | 0x7f800000u;
  return __uint_as_float(r);
}

struct Gas {
  float gamma, gm1, g, z, iz, k;  // gamma, gamma-1, (gamma-1)/2, z, 1/z, (gamma+1)/(2 gamma)
  int gamma75;
};

// a node in FP32: velocity, its 1-norm, p, 1/p, a and a p^-z, and a bound on the
// relative error of those four (velocity: 5 u)
template <int DIM> struct NodeF {
  float v[DIM], V, p, ip, a, az, err;
};

// false: out of range, or not clearly admissible
template <int DIM> __device__ inline bool node_f32(const Arrays &g, const Gas &G, int i, NodeF<DIM> &w) {
  const float rho = trunc_f32(g.U[i]), E = trunc_f32(g.U[(int64_t)(DIM + 1) * g.n + i]);
  const float ir = __fdividef(1.0f, rho);
  float ke = 0.0f;  // as m v: the squares of small momenta would leave FP32's range
  w.V = 0.0f;
#pragma unroll
  for (int q = 0; q < DIM; ++q) {
    const float m = trunc_f32(g.U[(int64_t)(1 + q) * g.n + i]);
    w.v[q] = m * ir;
    ke += 0.5f * m * w.v[q];
    w.V += fabsf(w.v[q]);
  }
  const float eps = E - ke;
  const float ee = __fdividef(10.0f * kU * (E + ke), eps);  // relative error of eps
  w.p = G.gm1 * eps;
  w.ip = __fdividef(1.0f, w.p);
  w.a = sqrtf(G.gamma * w.p * ir);
  const float lp = __log2f(w.p);  // absolute error 2^-21.5 in [0.5, 2], else 3 ulps: within 4 u (1 + |lp|)
  w.az = w.a * exp2f(-G.z * lp);
  w.err = ee + 20.0f * kU + 6.0f * kU * G.z * (1.0f + fabsf(lp));
  return rho > 1e-30f && rho < 1e30f && eps > 1e-30f && ee < 0.01f && w.err < 0.02f && E < 1e30f && w.p > 1e-30f &&
         w.a > 1e-18f && w.a < 1e18f && w.V < 1e18f && w.az > 1e-30f && w.az < 1e30f;
}

// lambda_max |c| from l to r along c, as a value and a bound on its absolute
// error; false: out of range. An error of the numerator of p_tr is carried to
// x = num / den, to p_tr (iz times) and to s = sqrt(1 + k (p_tr/p - 1)_+): with
// s >= 1 and s^2 >= k p_tr/p + (1 - k), an error e of p_tr/p changes s by at most
// 0.5 k (p_tr/p) e / s <= 0.5 s e / (1 - ...) <= s e (taken twice over).
template <int DIM>
__device__ inline bool wave_f32(const Gas &G, const NodeF<DIM> &l, const NodeF<DIM> &r, const float *c, float *d,
                                float *err) {
  float s2 = 0.0f, vl = 0.0f, vr = 0.0f;
#pragma unroll
  for (int q = 0; q < DIM; ++q) {
    s2 += c[q] * c[q];
    vl += l.v[q] * c[q];
    vr += r.v[q] * c[q];
  }
  const float ci = rsqrtf(s2), cn = s2 * ci, ul = vl * ci, ur = vr * ci;
  const float num = l.a + r.a - G.g * (ur - ul);
  const float en = l.err * l.a + r.err * r.a + 10.0f * kU * (l.a + r.a + l.V + r.V);  // absolute
  const float ed = l.err + r.err + 8.0f * kU;
  float ptr = 0.0f, ep = 0.0f;  // p_tr and its relative error
  bool ok = s2 > 1e-30f && s2 < 1e30f;
  if (num > -en) {
    const float x = __fdividef(fmaxf(num, en), l.az + r.az);
    const float ex = __fdividef(en, fmaxf(num, en)) + ed + 4.0f * kU;
    if (G.gamma75) {
      const float x2 = x * x;
      ptr = x2 * x2 * x2 * x;
      ep = 7.0f * ex + 8.0f * kU;
    } else {
      const float lx = log2f(x);
      ptr = exp2f(G.iz * lx);
      ep = G.iz * (ex + 3.0f * kU * fabsf(lx) + 2.0f * kU) + 8.0f * kU;
    }
    // (a numerator within its error of 0: p_tr <= p on both sides only if the
    // upper end is; the bound below then covers it or the row is undecided)
    ep *= 1.1f;
    ok = ok && ep < 0.05f && ptr < 1e30f;
  }
  const float ql = ptr * l.ip, qr = ptr * r.ip;
  const float fl = ep + l.err + 4.0f * kU, fr = ep + r.err + 4.0f * kU;
  const float sl = sqrtf(1.0f + G.k * fmaxf(ql - 1.0f, 0.0f)), sr = sqrtf(1.0f + G.k * fmaxf(qr - 1.0f, 0.0f));
  // q (1 +- f) below 1 leaves s = 1 exactly
  const float dl = ql * (1.0f + 2.0f * fl) > 1.0f ? fl : 0.0f, dr = qr * (1.0f + 2.0f * fr) > 1.0f ? fr : 0.0f;
  const float wl = l.a * sl, wr = r.a * sr;
  const float L = wl - ul, R = wr + ur;
  const float eL = wl * (2.0f * dl + l.err + 16.0f * kU) + 16.0f * kU * l.V;
  const float eR = wr * (2.0f * dr + r.err + 16.0f * kU) + 16.0f * kU * r.V;
  const float lam = fmaxf(fmaxf(L, R), 0.0f);
  *d = lam * cn;
  *err = (fmaxf(eL, eR) + 8.0f * kU * lam) * cn * 1.01f;
  return ok && lam < 1e18f;
}

template <int DIM> __device__ inline Bracket row_bracket(const Arrays &g, const Gas &G, int i) {
  const Bracket unknown{-INFINITY, INFINITY};
  NodeF<DIM> own, w;
  bool ok = node_f32<DIM>(g, G, i, own);
  float sum = 0.0f, err = 0.0f;
  const int64_t k0 = g.row_ptr[i], k1 = g.row_ptr[i + 1];
  const bool bi = g.isb && g.isb[i];
  for (int64_t k = k0; k < k1; ++k) {
    const int j = g.col[k];
    if (j == i) continue;
    const bool both = bi && g.isb[j];
    const bool up = j > i;
    ok &= node_f32<DIM>(g, G, j, w);
    int64_t kt = k;
    if (!up || both) kt = transposed(g.row_ptr, g.col, i, j, k - k0);
    if (kt < 0) continue;
    float c[DIM], d, e;
    // from min(i, j) to max(i, j) with the entry of row min(i, j); a pair of
    // boundary nodes also the other way round
#pragma unroll
    for (int q = 0; q < DIM; ++q) c[q] = trunc_f32(g.cij[(int64_t)q * g.nnz + (up ? k : kt)]);
    if (up) ok &= wave_f32<DIM>(G, own, w, c, &d, &e);
    else ok &= wave_f32<DIM>(G, w, own, c, &d, &e);
    if (both) {
      float d2, e2;
#pragma unroll
      for (int q = 0; q < DIM; ++q) c[q] = trunc_f32(g.cij[(int64_t)q * g.nnz + (up ? kt : k)]);
      if (up) ok &= wave_f32<DIM>(G, w, own, c, &d2, &e2);
      else ok &= wave_f32<DIM>(G, own, w, c, &d2, &e2);
      d = fmaxf(d, d2);
      e = fmaxf(e, e2);
    }
    sum += d;
    err += e;
  }
  const float m = trunc_f32(g.mi[i]), e = ((float)(k1 - k0) + 16.0f) * kU;
  const float t = 0.5f * (float)g.cfl * m;
  if (!ok || !(t > 1e-30f && m < 1e30f && sum > 1e-30f && sum < 1e30f && e < 0.1f && err < 0.5f * sum)) return unknown;
  const float lo = t / (sum + err) * (1.0f - e), hi = t / (sum - err) * (1.0f + e);
  if (!(lo > 1e-30f && hi < 1e30f)) return unknown;
  return Bracket{lo, hi};
}

// the block's smallest lower end; the smallest upper end of all (positive
// floats order like their bit patterns; the caller fills the slot with 0x7f)
template <int DIM>
__global__ void __launch_bounds__(kThreads) k_cfl_bracket(Arrays g, Gas G, double *slots) {
  __shared__ float slo[kThreads / 32], shi[kThreads / 32];
  const int i = blockIdx.x * kThreads + threadIdx.x;
  Bracket b{INFINITY, INFINITY};
  if (i < g.n) b = row_bracket<DIM>(g, G, i);
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    b.lo = fminf(b.lo, __shfl_xor_sync(0xffffffffu, b.lo, off));
    b.hi = fminf(b.hi, __shfl_xor_sync(0xffffffffu, b.hi, off));
  }
  if ((threadIdx.x & 31) == 0) {
    slo[threadIdx.x >> 5] = b.lo;
    shi[threadIdx.x >> 5] = b.hi;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
#pragma unroll
    for (int q = 1; q < kThreads / 32; ++q) {
      b.lo = fminf(b.lo, slo[q]);
      b.hi = fminf(b.hi, shi[q]);
    }
    *reinterpret_cast<float *>(slots + blockIdx.x) = b.lo;
    unsigned *limit = reinterpret_cast<unsigned *>(slots + kMaxBlocks);
    if (b.hi < INFINITY && __float_as_uint(b.hi) < *(volatile unsigned *)limit) atomicMin(limit, __float_as_uint(b.hi));
    if (blockIdx.x == 0) *reinterpret_cast<long long *>(slots + kMaxBlocks + 1) = bound_key(INFINITY);
  }
}

// the exact bounds of the block's rows that can be the smallest. Few such rows:
// a warp each, an entry per lane (a thread would run the serial chain of a whole
// row, 9 entries of ~100 to 400 FP64 instructions at 63 cycles each); many: a
// thread each, which leaves no lane idle.
template <int DIM>
__global__ void __launch_bounds__(kThreads) k_cfl_exact(Arrays g, Gas G, double *slots) {
  __shared__ int list[kThreads], count;
  const float limit = *reinterpret_cast<const float *>(slots + kMaxBlocks);
  if (*reinterpret_cast<const float *>(slots + blockIdx.x) > limit) return;
  if (threadIdx.x == 0) count = 0;
  __syncthreads();
  const int i = blockIdx.x * kThreads + threadIdx.x;
  if (i < g.n && row_bracket<DIM>(g, G, i).lo <= limit) list[atomicAdd(&count, 1)] = i;
  __syncthreads();
  const int rows = count;
  long long key = bound_key(INFINITY);
  if (rows <= kThreads / 8) {
    for (int q = threadIdx.x >> 5; q < rows; q += kThreads / 32) {
      const long long b = bound_key(row_bound_warp<DIM>(g, list[q]));
      key = b < key ? b : key;
    }
  } else if ((int)threadIdx.x < rows) {
    key = bound_key(row_bound<DIM>(g, list[threadIdx.x]));
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    const long long o = __shfl_xor_sync(0xffffffffu, key, off);
    key = o < key ? o : key;
  }
  if ((threadIdx.x & 31) == 0) atomicMin(reinterpret_cast<long long *>(slots + kMaxBlocks + 1), key);
}

__global__ void k_cfl_store(const double *slots, double *dt_out) {
  *dt_out = key_bound(*reinterpret_cast<const long long *>(slots + kMaxBlocks + 1));
}

template <int DIM> cudaError_t launch_cfl(const Arrays &g, const Gas &G, double *slots, double *dt_out, cudaStream_t s) {
  const int nb = (g.n + kThreads - 1) / kThreads;
  cudaError_t e;
  // 0x7f7f7f7f: an FP32 value above every finite upper end
  if ((e = cudaMemsetAsync(slots + kMaxBlocks, 0x7f, sizeof(double), s)) != cudaSuccess) return e;
  k_cfl_bracket<DIM><<<nb, kThreads, 0, s>>>(g, G, slots);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  k_cfl_exact<DIM><<<nb, kThreads, 0, s>>>(g, G, slots);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  k_cfl_store<<<1, 1, 0, s>>>(slots, dt_out);
  return cudaGetLastError();
}

// The id of the CUDA context current on the calling thread, through driver
// entry points fetched by the runtime (the library does not link libcuda).
// Called with g_scratch_mutex held.
using CtxGetCurrentFn = CUresult (*)(CUcontext *);
using CtxGetIdFn = CUresult (*)(CUcontext, unsigned long long *);

eh_status current_context_id(unsigned long long *id) {
  static CtxGetCurrentFn get_current = nullptr;
  static CtxGetIdFn get_id = nullptr;
  if (!get_current || !get_id) {
    void *f1 = nullptr, *f2 = nullptr;
    cudaDriverEntryPointQueryResult q1, q2;
    if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &f1, 12000, cudaEnableDefault, &q1) != cudaSuccess ||
        cudaGetDriverEntryPointByVersion("cuCtxGetId", &f2, 12000, cudaEnableDefault, &q2) != cudaSuccess ||
        q1 != cudaDriverEntryPointSuccess || q2 != cudaDriverEntryPointSuccess || !f1 || !f2) {
      cudaGetLastError();
      return EH_ERR_CUDA;
    }
    get_current = (CtxGetCurrentFn)f1;
    get_id = (CtxGetIdFn)f2;
  }
  CUcontext ctx = nullptr;
  if (get_current(&ctx) != CUDA_SUCCESS || !ctx || get_id(ctx, id) != CUDA_SUCCESS) return EH_ERR_CUDA;
  return EH_OK;
}

// The scratch's device address in the current device's current context. The
// lookup (cudaGetSymbolAddress, which allocates nothing) runs on the first
// call in each context and is cached for the later ones.
eh_status scratch_for_current_device(double **out) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) {
    cudaGetLastError();
    return EH_ERR_CUDA;
  }
  // makes the device's primary context current if no context is yet
  if (cudaSetDevice(dev) != cudaSuccess) {
    cudaGetLastError();
    return EH_ERR_CUDA;
  }
  std::lock_guard<std::mutex> lock(g_scratch_mutex);  // also guards the entry points cached below
  unsigned long long ctx_id = 0;
  if (current_context_id(&ctx_id) != EH_OK) return EH_ERR_CUDA;
  ScratchEntry &e = g_scratch[dev];
  if (!e.addr || e.ctx_id != ctx_id) {
    void *p = nullptr;
    cudaError_t err = cudaGetSymbolAddress(&p, g_cfl_block_min);
    if (err != cudaSuccess || !p) {
      cudaGetLastError();
      return EH_ERR_CUDA;
    }
    e.addr = (double *)p;
    e.ctx_id = ctx_id;
  }
  *out = e.addr;
  return EH_OK;
}

}  // namespace

extern "C" eh_status eh_cfl_dt_noalloc(int32_t dim, double gamma, double cfl, int32_t n, int64_t nnz,
                                       const int64_t *row_ptr, const int32_t *col, const double *cij, const double *mi,
                                       const unsigned char *is_boundary, const double *U, double *dt_out,
                                       void *stream) {
  if ((dim != 2 && dim != 3) || !(gamma > 1.0 && gamma <= 5.0 / 3.0) || !(cfl > 0.0 && cfl <= 1.0))
    return EH_ERR_INVALID_ARG;
  if (n <= 0 || n > EH_CFL_NOALLOC_MAX_ROWS || nnz <= 0 || !row_ptr || !col || !cij || !mi || !U || !dt_out)
    return EH_ERR_INVALID_ARG;
  // an error left by earlier work of the caller is reported, not consumed:
  // the caller still finds it with its own cudaGetLastError
  if (cudaPeekAtLastError() != cudaSuccess) return EH_ERR_CUDA;
  double *scratch = nullptr;
  eh_status st = scratch_for_current_device(&scratch);
  if (st != EH_OK) return st;
  const Arrays g{n, nnz, row_ptr, col, cij, mi, is_boundary, U, gamma, cfl};
  const Gas G{(float)gamma, (float)(gamma - 1.0), (float)(0.5 * (gamma - 1.0)), (float)((gamma - 1.0) / (2.0 * gamma)),
              (float)(2.0 * gamma / (gamma - 1.0)), (float)((gamma + 1.0) / (2.0 * gamma)), gamma == 1.4};
  // (an error here is this call's only: none was pending)
  const cudaError_t e = dim == 2 ? launch_cfl<2>(g, G, scratch, dt_out, (cudaStream_t)stream)
                                 : launch_cfl<3>(g, G, scratch, dt_out, (cudaStream_t)stream);
  return e == cudaSuccess ? EH_OK : EH_ERR_CUDA;
}
