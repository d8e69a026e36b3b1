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

// The scratch: one 8-byte slot per block of kThreads rows (512 KiB; first the
// block's FP32 bracket of its smallest bound, then its exact minimum) and one
// more for the smallest upper end over all blocks.
static __device__ __align__(256) double g_cfl_block_min[kMaxBlocks + 1];

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

template <int DIM> __device__ inline void derive(Node<DIM> &w, double gamma) {
  double m2 = 0.0;
#pragma unroll
  for (int q = 0; q < DIM; ++q) m2 += w.m[q] * w.m[q];
  double eps = w.E - m2 / (2.0 * w.rho);
  w.p = (gamma - 1.0) * eps;
  w.a = sqrt(gamma * w.p / w.rho);
  w.az = w.a * pow(w.p, -(gamma - 1.0) / (2.0 * gamma));
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
  double ptr = pow(num / (l.az + r.az), 2.0 * gamma / (gamma - 1.0));
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
// pressure, both outer waves are rarefactions and the bound is |v.n| + a: no
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
      const double ci = 1.0 / cn;
      lam = fabs(normal_velocity(own, c, ci)) + own.a;
    } else {
      const double ci = 1.0 / cn;
      const double ul = normal_velocity(l, c, ci), ur = normal_velocity(r, c, ci);
      lam = b == 0 ? wave_bound(l, ul, r, ur, g.gamma) : wave_bound(r, ur, l, ul, g.gamma);
    }
    d = b == 0 ? lam * cn : fmax(d, lam * cn);
  }
  return d;
}

// min(a, b) that keeps a NaN: a row whose state is not admissible (rho <= 0 or
// internal energy <= 0) gives a NaN bound, which must reach dt_out instead of
// being dropped by the reduction
__device__ __forceinline__ double nan_min(double a, double b) { return (a < b || a != a) ? a : b; }

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
// bracketed in FP32 interval arithmetic, and only rows whose lower end does
// not exceed the smallest upper end are evaluated in FP64 (998k-vertex Q1
// cylinder, perturbed flow: 6757 -> 275 us for the step, the same bits; before,
// every entry took 3 powers, 2 roots and 6 divisions in FP64, twice per edge;
// what remains is the gather of the neighbours' states). The brackets below
// carry every rounding (u = 2^-23 per conversion or operation is twice what
// either does; log2f and exp2f are within 2 units); a row with anything out
// of FP32's range, or not clearly admissible, gets (-inf, inf) and is
// evaluated in FP64.
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

// a node in FP32: velocity, its 1-norm, p, a and a p^-z, and a bound on the
// relative error of those three (velocity: 5 u)
template <int DIM> struct NodeF {
  float v[DIM], V, p, a, az, err;
  bool ok;
};

template <int DIM> __device__ inline NodeF<DIM> node_f32(const Arrays &g, float gamma, float z, int i) {
  NodeF<DIM> w;
  const float rho = trunc_f32(g.U[i]), E = trunc_f32(g.U[(int64_t)(DIM + 1) * g.n + i]);
  const float ir = 1.0f / rho;
  float m2 = 0.0f;
  w.V = 0.0f;
#pragma unroll
  for (int q = 0; q < DIM; ++q) {
    const float m = trunc_f32(g.U[(int64_t)(1 + q) * g.n + i]);
    m2 += m * m;
    w.v[q] = m * ir;
    w.V += fabsf(w.v[q]);
  }
  const float ke = 0.5f * m2 * ir, eps = E - ke;
  const float ee = 10.0f * kU * (E + ke) / eps;  // relative error of eps
  w.p = (gamma - 1.0f) * eps;
  w.a = sqrtf(gamma * w.p * ir);
  const float lp = log2f(w.p);
  w.az = w.a * exp2f(-z * lp);
  w.err = ee + 16.0f * kU + 4.0f * kU * z * fabsf(lp);
  w.ok = rho > 1e-30f && eps > 1e-30f && ee < 0.01f && w.err < 0.02f && E < 1e30f && w.p > 1e-30f && w.a < 1e18f &&
         w.V < 1e18f && w.az > 1e-30f && w.az < 1e30f;
  return w;
}

struct Gas {
  float gamma, g, z, iz, k;  // gamma, (gamma-1)/2, z, 1/z, (gamma+1)/(2 gamma)
};

// bracket of lambda_max |c| from l to r along c; false: out of range
template <int DIM>
__device__ inline bool wave_f32(const Gas &G, const NodeF<DIM> &l, const NodeF<DIM> &r, const float *c, float sgn,
                                float *dlo, float *dhi) {
  float s2 = 0.0f, ul = 0.0f, ur = 0.0f;
#pragma unroll
  for (int q = 0; q < DIM; ++q) s2 += c[q] * c[q];
  const float cn = sqrtf(s2), ci = sgn / cn;
#pragma unroll
  for (int q = 0; q < DIM; ++q) {
    ul += l.v[q] * (c[q] * ci);
    ur += r.v[q] * (c[q] * ci);
  }
  const float du_l = 12.0f * kU * l.V, du_r = 12.0f * kU * r.V;  // absolute errors of ul, ur
  const float num = l.a + r.a - G.g * (ur - ul);
  const float en = l.err * l.a + r.err * r.a + 10.0f * kU * (l.a + r.a + l.V + r.V);
  const float iden = 1.0f / (l.az + r.az), ed = l.err + r.err + 8.0f * kU;
  const float xlo = fmaxf(num - en, 0.0f) * iden * (1.0f - ed), xhi = fmaxf(num + en, 0.0f) * iden * (1.0f + ed);
  const float Llo = log2f(xlo), Lhi = log2f(xhi);
  const float elo = G.iz * (3.0f * kU * fabsf(Llo) + 2.0f * kU) + 8.0f * kU;
  const float ehi = G.iz * (3.0f * kU * fabsf(Lhi) + 2.0f * kU) + 8.0f * kU;
  const float plo = xlo > 0.0f ? exp2f(G.iz * Llo) * (1.0f - fminf(elo, 1.0f)) : 0.0f;
  const float phi = xhi > 0.0f ? exp2f(G.iz * Lhi) * (1.0f + ehi) : 0.0f;
  const float fl = l.err + 4.0f * kU, fr = r.err + 4.0f * kU;
  const float ipl = 1.0f / l.p, ipr = 1.0f / r.p;
  // s = sqrt(1 + k (p_tr / p - 1)_+), a s, and the two outer speeds
  const float sll = sqrtf(1.0f + G.k * fmaxf(plo * ipl * (1.0f - fl) - 1.0f - 4.0f * kU, 0.0f));
  const float slh = sqrtf(1.0f + G.k * fmaxf(phi * ipl * (1.0f + fl) - 1.0f + 4.0f * kU, 0.0f));
  const float srl = sqrtf(1.0f + G.k * fmaxf(plo * ipr * (1.0f - fr) - 1.0f - 4.0f * kU, 0.0f));
  const float srh = sqrtf(1.0f + G.k * fmaxf(phi * ipr * (1.0f + fr) - 1.0f + 4.0f * kU, 0.0f));
  const float el = l.err + 12.0f * kU, er = r.err + 12.0f * kU;
  const float alo = l.a * sll * (1.0f - el), ahi = l.a * slh * (1.0f + el);
  const float blo = r.a * srl * (1.0f - er), bhi = r.a * srh * (1.0f + er);
  const float lo = fmaxf(fmaxf(alo - ul - du_l - 4.0f * kU * alo, blo + ur - du_r - 4.0f * kU * blo), 0.0f);
  const float hi = fmaxf(fmaxf(ahi - ul + du_l + 4.0f * kU * ahi, bhi + ur + du_r + 4.0f * kU * bhi), 0.0f);
  *dlo = lo * cn * (1.0f - 8.0f * kU);
  *dhi = hi * cn * (1.0f + 8.0f * kU);
  return s2 > 1e-30f && s2 < 1e30f && phi < 1e30f && ehi < 0.1f && hi < 1e18f;
}

template <int DIM> __device__ inline Bracket row_bracket(const Arrays &g, const Gas &G, int i) {
  const Bracket unknown{-INFINITY, INFINITY};
  const NodeF<DIM> own = node_f32<DIM>(g, G.gamma, G.z, i);
  bool ok = own.ok;
  float slo = 0.0f, shi = 0.0f;
  const int64_t k0 = g.row_ptr[i], k1 = g.row_ptr[i + 1];
  const bool bi = g.isb && g.isb[i];
  for (int64_t k = k0; k < k1; ++k) {
    const int j = g.col[k];
    if (j == i) continue;
    const bool both = bi && g.isb[j];
    const bool up = j > i;
    const NodeF<DIM> w = node_f32<DIM>(g, G.gamma, G.z, j);
    int64_t kt = k;
    if (!up || both) kt = transposed(g.row_ptr, g.col, i, j, k - k0);
    if (kt < 0) continue;
    float c[DIM], lo, hi;
    // from min(i, j) to max(i, j) with the entry of row min(i, j); a pair of
    // boundary nodes also the other way round
#pragma unroll
    for (int q = 0; q < DIM; ++q) c[q] = trunc_f32(g.cij[(int64_t)q * g.nnz + (up ? k : kt)]);
    // (along +c from the left state; seen from node i of a lower entry the
    // two sides swap)
    ok &= w.ok && wave_f32<DIM>(G, up ? own : w, up ? w : own, c, 1.0f, &lo, &hi);
    if (both) {
      float lo2, hi2;
#pragma unroll
      for (int q = 0; q < DIM; ++q) c[q] = trunc_f32(g.cij[(int64_t)q * g.nnz + (up ? kt : k)]);
      ok &= wave_f32<DIM>(G, up ? w : own, up ? own : w, c, 1.0f, &lo2, &hi2);
      lo = fmaxf(lo, lo2);
      hi = fmaxf(hi, hi2);
    }
    slo += lo;
    shi += hi;
  }
  const float m = trunc_f32(g.mi[i]), e = ((float)(k1 - k0) + 16.0f) * kU;
  if (!ok || !(m > 1e-30f && m < 1e30f && slo > 1e-30f && shi < 1e30f && e < 0.1f)) return unknown;
  const float t = 0.5f * (float)g.cfl * m;
  const float lo = t / shi * (1.0f - e), hi = t / slo * (1.0f + e);
  if (!(lo > 1e-30f && hi < 1e30f)) return unknown;
  return Bracket{lo, hi};
}

// the block's smallest lower and upper ends
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
    reinterpret_cast<float2 *>(slots)[blockIdx.x] = make_float2(b.lo, b.hi);
  }
}

// the smallest upper end over all blocks, into the last slot
__global__ void __launch_bounds__(1024) k_cfl_upper(double *slots, int nb) {
  __shared__ float sm[32];
  float b = INFINITY;
  const float2 *s = reinterpret_cast<const float2 *>(slots);
  for (int q = threadIdx.x; q < nb; q += blockDim.x) b = fminf(b, s[q].y);
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) b = fminf(b, __shfl_xor_sync(0xffffffffu, b, off));
  if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = b;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int q = 1; q < (int)(blockDim.x >> 5); ++q) b = fminf(b, sm[q]);
    *reinterpret_cast<float *>(slots + kMaxBlocks) = b;
  }
}

// the exact minimum over the block's rows that can hold the smallest bound (a
// NaN for a row that is not admissible); +inf for a block without one. Few
// such rows: a warp each, an entry per lane (a thread would run the serial
// chain of a whole row, 9 entries of ~400 FP64 instructions at 63 cycles each);
// many: a thread each, which leaves no lane idle.
template <int DIM>
__global__ void __launch_bounds__(kThreads) k_cfl_exact(Arrays g, Gas G, double *slots) {
  __shared__ double smin[kThreads / 32];
  __shared__ int list[kThreads], count;
  const float limit = *reinterpret_cast<const float *>(slots + kMaxBlocks);
  const float block_lo = reinterpret_cast<const float2 *>(slots)[blockIdx.x].x;
  __syncthreads();  // the slot is read by every thread before it is rewritten
  if (block_lo > limit) {
    if (threadIdx.x == 0) slots[blockIdx.x] = INFINITY;
    return;
  }
  if (threadIdx.x == 0) count = 0;
  __syncthreads();
  const int i = blockIdx.x * kThreads + threadIdx.x;
  if (i < g.n && row_bracket<DIM>(g, G, i).lo <= limit) list[atomicAdd(&count, 1)] = i;
  __syncthreads();
  const int rows = count;
  double bound = INFINITY;
  if (rows <= kThreads / 8) {
    for (int q = threadIdx.x >> 5; q < rows; q += kThreads / 32) bound = nan_min(bound, row_bound_warp<DIM>(g, list[q]));
  } else if ((int)threadIdx.x < rows) {
    bound = row_bound<DIM>(g, list[threadIdx.x]);
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) bound = nan_min(bound, __shfl_xor_sync(0xffffffffu, bound, off));
  if ((threadIdx.x & 31) == 0) smin[threadIdx.x >> 5] = bound;
  __syncthreads();
  if (threadIdx.x == 0) {
    double b = smin[0];
#pragma unroll
    for (int q = 1; q < kThreads / 32; ++q) b = nan_min(b, smin[q]);
    slots[blockIdx.x] = b;
  }
}

__global__ void __launch_bounds__(1024) k_cfl_reduce(const double *block_min, int nb, double *dt_out) {
  __shared__ double sm[32];
  double b = INFINITY;
  for (int q = threadIdx.x; q < nb; q += blockDim.x) b = nan_min(b, block_min[q]);
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) b = nan_min(b, __shfl_xor_sync(0xffffffffu, b, off));
  if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = b;
  __syncthreads();
  if (threadIdx.x == 0) {
    double m = sm[0];
    for (int q = 1; q < (int)(blockDim.x >> 5); ++q) m = nan_min(m, sm[q]);
    *dt_out = m;
  }
}

template <int DIM> cudaError_t launch_cfl(const Arrays &g, const Gas &G, double *slots, double *dt_out, cudaStream_t s) {
  const int nb = (g.n + kThreads - 1) / kThreads;
  cudaError_t e;
  k_cfl_bracket<DIM><<<nb, kThreads, 0, s>>>(g, G, slots);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  k_cfl_upper<<<1, 1024, 0, s>>>(slots, nb);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  k_cfl_exact<DIM><<<nb, kThreads, 0, s>>>(g, G, slots);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  k_cfl_reduce<<<1, 1024, 0, s>>>(slots, nb, dt_out);
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
  const Gas G{(float)gamma, (float)(0.5 * (gamma - 1.0)), (float)((gamma - 1.0) / (2.0 * gamma)),
              (float)(2.0 * gamma / (gamma - 1.0)), (float)((gamma + 1.0) / (2.0 * gamma))};
  // (an error here is this call's only: none was pending)
  const cudaError_t e = dim == 2 ? launch_cfl<2>(g, G, scratch, dt_out, (cudaStream_t)stream)
                                 : launch_cfl<3>(g, G, scratch, dt_out, (cudaStream_t)stream);
  return e == cudaSuccess ? EH_OK : EH_ERR_CUDA;
}
