// Particle and mesh kernels of the PM hot path (besides the FFT passes), templated on the
// real type.  Included once per precision.
//
//  k_scatter        CIC mass (and adjoint pi) assignment, Sec. 2.2 Eq. 10, int64 fixed point
//                   with global atomics (the allocation-free density entry point, deposits
//                   of few particles and interpolated densities; otherwise the engine
//                   assigns by mesh tiles, bin_kernels.cuh)
//  k_gather_fwd     CIC force gather + kick / kick / drift of Eq. 16 (one launch per step);
//                   counts the deposit bins of the new positions for the next step
//  k_gather_adj     CIC gather of a and alpha (Eq. 49 F line) + reverse kicks and drift of
//                   Eq. 49, FP64 partials of the theta terms of Eq. 51; bin counts as above
//  k_adjoint_init   xi_n = dJ/dx_n (density cotangent through the CIC weight gradient), pi_n
//  k_obs_cotangent  the same cotangent of an observed intermediate state, added to xi_j
//  k_density_out, k_mse, k_za_mul, k_za_adj_mul, k_ic_state, k_ic_adj_prep, k_final_theta,
//  k_lpt_hess, k_lpt_source, k_lpt_source_adj, k_lpt_hess_adj, k_ic_state2
#pragma once
#include <cuda_fp16.h>
#include "bin_geo.h"
#include "common.cuh"
#include "pm_internal.h"

namespace pmgb {

constexpr int kPtclThreads = 256;
constexpr int kMaxRedBlocks = 1024;

// Lattice and mesh geometry of one instance.
template <typename T> struct Geo {
  int lg_np;      // log2 n_ptcl
  int np, nm;     // particles / mesh nodes per side
  int ratio;      // nm / np
  T inv_l;        // 1 / cell size
  long long N;    // particles per instance
  long long M;    // mesh cells per instance
};

// correctly rounded products and fused multiply-adds, never re-associated or contracted
// differently by the compiler: the forward and reverse passes gather the same force on a
// particle bit for bit
template <typename T> __device__ __forceinline__ T mul_rn(T a, T b);
template <> __device__ __forceinline__ float mul_rn<float>(float a, float b) { return __fmul_rn(a, b); }
template <> __device__ __forceinline__ double mul_rn<double>(double a, double b) { return __dmul_rn(a, b); }
template <typename T> __device__ __forceinline__ T fma_rn(T a, T b, T c);
template <> __device__ __forceinline__ float fma_rn<float>(float a, float b, float c) { return __fmaf_rn(a, b, c); }
template <> __device__ __forceinline__ double fma_rn<double>(double a, double b, double c) { return __fma_rn(a, b, c); }


// Cell index and fraction along each axis for particle i at displacement s (floor
// convention: u = q/l + s/l with q/l = j*ratio + 1/2; the integer part of q/l is added
// separately so that the fraction keeps the precision of s, not of x).
template <typename T>
__device__ __forceinline__ void cic_cell(const Geo<T>& g, long long i, const T s[3], int cell[3], T t[3]) {
  const int j[3] = {(int)(i >> (2 * g.lg_np)), (int)((i >> g.lg_np) & (g.np - 1)), (int)(i & (g.np - 1))};
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const T v = fma_rn<T>(s[c], g.inv_l, (T)0.5);
    const T f = floor(v);
    t[c] = v - f;
    cell[c] = (j[c] * g.ratio + (int)f) & (g.nm - 1);
  }
}

// Work index -> lattice particle index: 8^3 Lagrangian blocks (x fastest inside a block,
// so a warp reads 8 x 4 particles in full 32-byte segments) visited in Morton order of the
// block coordinates, so that the particles in flight at any moment -- and the mesh cells
// they scatter to or gather from -- form a compact region that stays in L2.
__device__ __forceinline__ unsigned long long morton_compact3(unsigned long long x) {
  x &= 0x1249249249249249ull;
  x = (x ^ (x >> 2)) & 0x10c30c30c30c30c3ull;
  x = (x ^ (x >> 4)) & 0x100f00f00f00f00full;
  x = (x ^ (x >> 8)) & 0x1f0000ff0000ffull;
  x = (x ^ (x >> 16)) & 0x1f00000000ffffull;
  x = (x ^ (x >> 32)) & 0x1fffffull;
  return x;
}
template <typename T>
__device__ __forceinline__ long long particle_of(const Geo<T>& g, long long w) {
  const int tb = g.lg_np < 3 ? g.lg_np : 3;                 // block side 2^tb
  const long long inner = w & ((1LL << (3 * tb)) - 1);
  const unsigned long long blk = (unsigned long long)(w >> (3 * tb));
  const int mask = (1 << tb) - 1;
  const long long x = ((long long)morton_compact3(blk) << tb) | (inner & mask);
  const long long y = ((long long)morton_compact3(blk >> 1) << tb) | ((inner >> tb) & mask);
  const long long z = ((long long)morton_compact3(blk >> 2) << tb) | (inner >> (2 * tb));
  return (z << (2 * g.lg_np)) | (y << g.lg_np) | x;
}

template <typename T>
__device__ __forceinline__ long long corner_index(const Geo<T>& g, const int cell[3], int d) {
  const int m = g.nm - 1;
  const int i0 = (cell[0] + ((d >> 2) & 1)) & m;
  const int i1 = (cell[1] + ((d >> 1) & 1)) & m;
  const int i2 = (cell[2] + (d & 1)) & m;
  return ((long long)i0 * g.nm + i1) * g.nm + i2;
}

// The eight CIC corners of the [cell][4] force mesh: FP32 V4 per cell, or (H, FP32 path
// only) the FP16 mesh of k_fft_x_c2r4<..., true>: four halves per cell, each field of a row
// (fixed z, y) scaled by 2^-e with e an int8 of the row's packed quadruple in fexp.
template <typename T, bool H>
__device__ __forceinline__ void load_corners(const Geo<T>& g, const void* __restrict__ fvec,
                                             const int* __restrict__ fexp, int b, const int cell[3], V4<T> fv[8]) {
  if constexpr (!H) {
    const V4<T>* F = reinterpret_cast<const V4<T>*>(fvec) + (long long)b * g.M;
#pragma unroll
    for (int d = 0; d < 8; ++d) fv[d] = F[corner_index(g, cell, d)];
  } else {
    static_assert(sizeof(T) == 4, "the FP16 force mesh is an FP32-path form");
    const uint2* F = reinterpret_cast<const uint2*>(fvec) + (long long)b * g.M;
    const int* E = fexp + (long long)b * g.nm * g.nm;
    const int m = g.nm - 1;
    int ew[4];   // exponent quadruples of the rows (z0 + dz, y0 + dy), index 2 dz + dy
#pragma unroll
    for (int k = 0; k < 4; ++k) ew[k] = __ldg(E + ((cell[0] + (k >> 1)) & m) * g.nm + ((cell[1] + (k & 1)) & m));
#pragma unroll
    for (int d = 0; d < 8; ++d) {
      const uint2 u = __ldg(F + corner_index(g, cell, d));
      const int w = ew[(d >> 1) & 3];
      const float2 lo = __half22float2(*reinterpret_cast<const __half2*>(&u.x));
      const float2 hi = __half22float2(*reinterpret_cast<const __half2*>(&u.y));
      fv[d] = V4<T>{lo.x * __int_as_float(((int)(signed char)(w & 0xFF) + 127) << 23),
                    lo.y * __int_as_float(((int)(signed char)((w >> 8) & 0xFF) + 127) << 23),
                    hi.x * __int_as_float(((int)(signed char)((w >> 16) & 0xFF) + 127) << 23),
                    hi.y * __int_as_float(((int)(signed char)((w >> 24) & 0xFF) + 127) << 23)};
    }
  }
}

template <typename T> __device__ __forceinline__ long long to_fixed(T v);
template <> __device__ __forceinline__ long long to_fixed<float>(float v) { return f2ll_rn(v); }
template <> __device__ __forceinline__ long long to_fixed<double>(double v) { return __double2ll_rn(v); }

// Exactly reversible particle state (pm_config.fixed_state): displacement and momentum held
// as 64-bit integers, U = s / l in units of 2^-kFixES cells and W = p / l in units of
// 2^-kFixEP cells per unit of drift factor.  A kick adds round(a K / l 2^kFixEP), a drift
// round(w D 2^kFixES) with w the working-precision value of W; the reverse pass subtracts
// the same rounded increments (the same forces at the same positions), so it recovers the
// forward states bit for bit.  The kernels that read positions and momenta see working-
// precision shadows s = U l 2^-kFixES, p = W l 2^-kFixEP.
constexpr int kFixES = 40, kFixEP = 36;
template <typename T> struct FixState {
  long long* u;   // [batch][3][N] or null: floating-point state
  long long* w;
  T to_w;         // 2^kFixEP / l: momentum increment -> W units
  T from_u;       // l 2^-kFixES: U -> displacement
  T from_w;       // l 2^-kFixEP: W -> momentum
  T w_cells;      // 2^-kFixEP: W -> cells per unit of drift factor
  T du;           // 2^kFixES: cells -> U units
};
template <typename T> __device__ __forceinline__ T fix_to_real(long long v);
template <> __device__ __forceinline__ float fix_to_real<float>(long long v) { return ll2f_rn(v); }
template <> __device__ __forceinline__ double fix_to_real<double>(long long v) { return (double)v; }

// Deterministic sum of v over a block of whole warps (at most 256 threads), valid in thread 0.
// One warp adds: its lane l takes the values of threads l, l + 32, ... in turn, then come five
// shuffles, 13 warp-wide FP64 additions in all.  Shuffles in each of the eight warps took 40, on
// a pipe of two lanes per clock and SM, and weighed as much as several particles or cells of
// every thread: with 8 instances of 64^3 particles on 128^3 k_za_adj_mul 93 -> 57 us, k_mse 126
// -> 109, the gradient of 4 steps 6056 -> 5946.
__device__ __forceinline__ double block_sum(double v) {
  __shared__ double sh[256];
  __syncthreads();
  sh[threadIdx.x] = v;
  __syncthreads();
  double r = 0.0;
  if (threadIdx.x < 32) {
    for (unsigned i = threadIdx.x; i < blockDim.x; i += 32) r += sh[i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) r += __shfl_down_sync(0xffffffffu, r, o);
  }
  return r;
}

__device__ __forceinline__ float block_max(float v, float* sh) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_down_sync(0xffffffffu, v, o));
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  __syncthreads();
  if (l == 0) sh[w] = v;
  __syncthreads();
  float r = 0.f;
  if (threadIdx.x == 0)
    for (int i = 0; i < (int)(blockDim.x >> 5); ++i) r = fmaxf(r, sh[i]);
  return r;
}

// Per-thread partial sums of the theta terms: compensated (Kahan) summation in the working
// precision, handed to the FP64 block reduction; FP64 arithmetic is slow on this part.
template <typename T> struct KahanAcc {
  T s = 0, c = 0;
  __device__ __forceinline__ void add(T v) {
    const T y = v - c;
    const T t = s + y;
    c = (t - s) - y;
    s = t;
  }
  __device__ __forceinline__ double value() const { return (double)s - (double)c; }
};

template <typename T> __device__ __forceinline__ float abs_up(T v);
template <> __device__ __forceinline__ float abs_up<float>(float v) { return fabsf(v); }
template <> __device__ __forceinline__ float abs_up<double>(double v) { return __double2float_ru(fabs(v)); }

// ------------------------------------------------------------------------- scatter
// NQ = 1: acc[cell] += W * 2^e_d (weights).  NQ = 4: acc is [cell][4] and receives the
// weight and pi_c * W * 2^e_c (c = 0..2) in one 32-byte sector per cell.
// (terms rounded as in the tile deposit; FP32 ones are at most 2^30 in magnitude, fixed_top)
__device__ __forceinline__ unsigned long long term_fixed(float v) { return (unsigned long long)(long long)__float2int_rn(v); }
__device__ __forceinline__ unsigned long long term_fixed(double v) { return (unsigned long long)__double2ll_rn(v); }
template <typename T, int NQ>
__global__ void __launch_bounds__(kPtclThreads)
k_scatter(Geo<T> g, const T* __restrict__ s, const T* __restrict__ pi, unsigned long long* acc, int e_d,
          const int* __restrict__ e_pi) {
  const int b = blockIdx.y;
  const T* sb = s + (long long)b * 3 * g.N;
  const long long mo = (long long)b * g.M;
  const T sd = pow2i<T>(e_d);
  T sp[3] = {0, 0, 0};
  const T* pb = nullptr;
  if constexpr (NQ == 4) {
    pb = pi + (long long)b * 3 * g.N;
#pragma unroll
    for (int c = 0; c < 3; ++c) sp[c] = pow2i<T>(e_pi[c * gridDim.y + b]);
  }
  for (long long w = blockIdx.x * (long long)blockDim.x + threadIdx.x; w < g.N;
       w += (long long)gridDim.x * blockDim.x) {
    const long long i = particle_of(g, w);
    const T sv[3] = {sb[i], sb[g.N + i], sb[2 * g.N + i]};
    int cell[3];
    T t[3];
    cic_cell(g, i, sv, cell, t);
    T pv[3] = {0, 0, 0};
    if constexpr (NQ == 4) {
      pv[0] = pb[i] * sp[0];
      pv[1] = pb[g.N + i] * sp[1];
      pv[2] = pb[2 * g.N + i] * sp[2];
    }
#pragma unroll
    for (int d = 0; d < 8; ++d) {
      const T w = ((d & 4) ? t[0] : (T)1 - t[0]) * ((d & 2) ? t[1] : (T)1 - t[1]) * ((d & 1) ? t[2] : (T)1 - t[2]);
      const long long idx = mo + corner_index(g, cell, d);
      if constexpr (NQ == 1) {
        atomicAdd(acc + idx, term_fixed(w * sd));
      } else {
        unsigned long long* q = acc + 4 * idx;
        atomicAdd(q, term_fixed(w * sd));
        atomicAdd(q + 1, term_fixed(pv[0] * w));
        atomicAdd(q + 2, term_fixed(pv[1] * w));
        atomicAdd(q + 3, term_fixed(pv[2] * w));
      }
    }
  }
}

// fixed-point exponents of the pi scatters from max|pi_c| (layout [c][batch]): one
// contribution |pi| W 2^e is below 2^(E + e) and the sum over one cell below N 2^(E + e),
// with max|pi| < 2^E; e = top - E keeps them below 2^top and 2^(lg N + top) (top: see
// fixed_top).
static __global__ void k_pi_exponents(const unsigned* __restrict__ pimax, int* __restrict__ e_pi, int nq, int top) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= nq) return;
  const float mx = __uint_as_float(pimax[i]);
  int e = 0;
  if (mx > 0.f && isfinite(mx)) {
    const int E = ilogbf(mx) + 1;   // mx < 2^E
    e = top - E;
    if (e > 100) e = 100;
  }
  e_pi[i] = e;
}

// Bits of one fixed-point contribution of the assignment.  FP32: 2^30, so that a
// contribution is an int32 (its 24-bit significand loses nothing there) and the sum over a
// cell of N contributions stays below 2^61 for N <= 2^31; FP64: 61 - lg N, the widest
// quantum the int64 cell sums allow.
template <typename T> inline int fixed_top(int lgN);
template <> inline int fixed_top<float>(int lgN) { return 61 - lgN < 30 ? 61 - lgN : 30; }
template <> inline int fixed_top<double>(int lgN) { return 61 - lgN; }

// ------------------------------------------------------------------ deposit bins
// (tiles and bins: bin_geo.h)
// class bits of a cell: on the last layer of its tile along x (bit 0), y (bit 1), z (bit 2)
__device__ __forceinline__ unsigned bin_class(const BinGeo& bg, const int c[3]) {
  const unsigned mx = (1u << bg.lx) - 1, my = (1u << bg.ly) - 1, mz = (1u << bg.lz) - 1;
  return (unsigned)(((unsigned)c[2] & mx) == mx) | ((unsigned)(((unsigned)c[1] & my) == my) << 1) |
         ((unsigned)(((unsigned)c[0] & mz) == mz) << 2);
}
__device__ __forceinline__ unsigned bin_key(const BinGeo& bg, const int c[3]) {
  const unsigned tile = (((unsigned)c[0] >> bg.lz) * bg.nty + ((unsigned)c[1] >> bg.ly)) * bg.ntx + ((unsigned)c[2] >> bg.lx);
  return tile * 8u + bin_class(bg, c);
}

// Count a particle's bin for the next deposit (its key, and a warp-aggregated increment of
// the bin count).  Every lane of the warp calls this together.
template <typename T>
__device__ __forceinline__ void count_bin(const Geo<T>& g, const BinGeo& bg, long long i, const T sv[3], int b,
                                          unsigned* __restrict__ count, unsigned* __restrict__ keys) {
  int cell[3];
  T t[3];
  cic_cell(g, i, sv, cell, t);
  const unsigned key = bin_key(bg, cell);
  keys[(long long)b * g.N + i] = key;
  const unsigned peers = __match_any_sync(0xFFFFFFFFu, key);
  if ((int)(threadIdx.x & 31) == __ffs(peers) - 1) atomicAdd(count + (long long)b * bg.nkeys + key, (unsigned)__popc(peers));
}

// ---------------------------------------------------------------------- gathers
template <typename T>
struct StepCoef {  // per-instance coefficient tables [batch][n+1], indexed at step j
  const T* kA;
  const T* kB;
  const T* dr;
};

// a = sum_g W f(g);  p += a kA;  (store p_j);  p += a kB;  (store s_j);  s += p dr
// OP (the operator entry point): a into a_out and nothing else; reads the caller's s.
template <typename T, bool H = false, bool OP = false>
__global__ void __launch_bounds__(kPtclThreads)
k_gather_fwd(Geo<T> g, T* __restrict__ s, T* __restrict__ p, T* __restrict__ a_out,
             const void* __restrict__ fvec, const int* __restrict__ fexp, StepCoef<T> sc, int j, int nstep1,
             T* __restrict__ ck_s,
             T* __restrict__ ck_p, BinGeo bg, unsigned* __restrict__ bcount, unsigned* __restrict__ bkeys,
             T* __restrict__ snap_p = nullptr, FixState<T> fx = FixState<T>{}) {
  const int b = blockIdx.y;
  T kA = 0, kB = 0, dr = 0;
  if constexpr (!OP) kA = sc.kA[b * nstep1 + j], kB = sc.kB[b * nstep1 + j], dr = sc.dr[b * nstep1 + j];
  T* sb = s + (long long)b * 3 * g.N;
  T* pb = p + (long long)b * 3 * g.N;
  // the displacement of the thread's next particle is read one iteration ahead, so that
  // its latency overlaps this particle's corner loads (each particle has one thread: the
  // value is not written before it is used)
  const long long stride = (long long)gridDim.x * blockDim.x;
  long long w = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  T sn[3] = {0, 0, 0};
  if (w < g.N) {
    const long long i0 = particle_of(g, w);
    sn[0] = sb[i0], sn[1] = sb[g.N + i0], sn[2] = sb[2 * g.N + i0];
  }
  for (; w < g.N; w += stride) {
    const long long i = particle_of(g, w);
    T sv[3] = {sn[0], sn[1], sn[2]};
    T pv[3] = {0, 0, 0};
    if constexpr (!OP) pv[0] = pb[i], pv[1] = pb[g.N + i], pv[2] = pb[2 * g.N + i];   // in flight with the corner loads
    int cell[3];
    T t[3];
    cic_cell(g, i, sv, cell, t);
    V4<T> fv[8];
    load_corners<T, H>(g, fvec, fexp, b, cell, fv);
    if (w + stride < g.N) {
      const long long in = particle_of(g, w + stride);
      sn[0] = sb[in], sn[1] = sb[g.N + in], sn[2] = sb[2 * g.N + in];
    }
    T a[3] = {0, 0, 0};
#pragma unroll
    for (int d = 0; d < 8; ++d) {
      const T w0 = (d & 4) ? t[0] : (T)1 - t[0];
      const T w1 = (d & 2) ? t[1] : (T)1 - t[1];
      const T w2 = (d & 1) ? t[2] : (T)1 - t[2];
      const T w = mul_rn<T>(mul_rn<T>(w0, w1), w2);
      a[0] = fma_rn<T>(w, fv[d].x, a[0]);
      a[1] = fma_rn<T>(w, fv[d].y, a[1]);
      a[2] = fma_rn<T>(w, fv[d].z, a[2]);
    }
    if constexpr (OP) {
#pragma unroll
      for (int c = 0; c < 3; ++c) a_out[(long long)b * 3 * g.N + c * g.N + i] = a[c];
      continue;
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const long long o = (long long)b * 3 * g.N + c * g.N + i;
      if (fx.u) {
        // fixed-point state: exact integer kicks and drift, shadows for the other kernels
        long long W = fx.w[o], U = fx.u[o];
        W += to_fixed<T>(mul_rn<T>(mul_rn<T>(a[c], kA), fx.to_w));
        if (ck_p || snap_p) pv[c] = mul_rn<T>(fix_to_real<T>(W), fx.from_w);
        if (ck_p) ck_p[o] = pv[c];
        if (snap_p) snap_p[o] = pv[c];
        W += to_fixed<T>(mul_rn<T>(mul_rn<T>(a[c], kB), fx.to_w));
        if (ck_s) ck_s[o] = sv[c];
        U += to_fixed<T>(mul_rn<T>(mul_rn<T>(mul_rn<T>(fix_to_real<T>(W), fx.w_cells), dr), fx.du));
        fx.w[o] = W;
        fx.u[o] = U;
        pv[c] = mul_rn<T>(fix_to_real<T>(W), fx.from_w);
        sv[c] = mul_rn<T>(fix_to_real<T>(U), fx.from_u);
      } else {
        pv[c] += a[c] * kA;
        if (ck_p) ck_p[o] = pv[c];
        if (snap_p) snap_p[o] = pv[c];   // p_j of an observed state
        pv[c] += a[c] * kB;
        if (ck_s) ck_s[o] = sv[c];
        sv[c] += pv[c] * dr;
      }
      pb[c * g.N + i] = pv[c];
      sb[c * g.N + i] = sv[c];
      if (a_out) a_out[o] = a[c];
    }
    // bin of the new position for the next step's deposit (the loop is warp-uniform: N is
    // a multiple of 32 and so is the grid stride)
    if (bcount) count_bin(g, bg, i, sv, b, bcount, bkeys);
  }
}

// Reverse step at force step j (Eq. 49): a_j = sum W f, alpha_j = sum grad W [pi.f + m psi];
// p -= a K1_{j+1}; xi += alpha K1_{j+1}; (p := stored p_j); p -= a K2_j; xi += alpha K2_j;
// s -= p D_j; pi += xi D_j; (s := stored s_{j-1}).  FP64 partials of pi.a and xi.p.
// OP (the operator entry point): a and alpha into a_out and alpha_out and nothing else.
template <typename T, bool H = false, bool OP = false>
__global__ void __launch_bounds__(kPtclThreads)
k_gather_adj(Geo<T> g, T mass, T* __restrict__ s, T* __restrict__ p, T* __restrict__ xi, T* __restrict__ pi,
             T* __restrict__ a_out, T* __restrict__ alpha_out, const void* __restrict__ fvec,
             const int* __restrict__ fexp, StepCoef<T> sc, int j, int nstep1,
             const T* __restrict__ ck_p, const T* __restrict__ ck_s, double* __restrict__ part_pa,
             double* __restrict__ part_xp, unsigned* __restrict__ pimax, BinGeo bg, unsigned* __restrict__ bcount,
             unsigned* __restrict__ bkeys, FixState<T> fx = FixState<T>{}) {
  __shared__ float shf[kPtclThreads / 32];
  const int b = blockIdx.y;
  T cA = 0, cB = 0, dr = 0;
  if constexpr (!OP) cA = sc.kA[b * nstep1 + j], cB = sc.kB[b * nstep1 + j], dr = sc.dr[b * nstep1 + j];
  const long long po = (long long)b * 3 * g.N;
  const T il = g.inv_l;
  KahanAcc<T> acc_pa, acc_xp;
  float mx[3] = {0.f, 0.f, 0.f};
  for (long long w = blockIdx.x * (long long)blockDim.x + threadIdx.x; w < g.N;
       w += (long long)gridDim.x * blockDim.x) {
    const long long i = particle_of(g, w);
    T sv[3], pv[3], xv[3], qv[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      sv[c] = s[po + c * g.N + i];
      if constexpr (!OP) {
        pv[c] = p[po + c * g.N + i];
        xv[c] = xi[po + c * g.N + i];
      }
      qv[c] = pi[po + c * g.N + i];
    }
    int cell[3];
    T t[3];
    cic_cell(g, i, sv, cell, t);
    V4<T> fv[8];
    load_corners<T, H>(g, fvec, fexp, b, cell, fv);
    T a[3] = {0, 0, 0}, al[3] = {0, 0, 0};
#pragma unroll
    for (int d = 0; d < 8; ++d) {
      const T w0 = (d & 4) ? t[0] : (T)1 - t[0];
      const T w1 = (d & 2) ? t[1] : (T)1 - t[1];
      const T w2 = (d & 1) ? t[2] : (T)1 - t[2];
      const T g0 = (d & 4) ? il : -il, g1 = (d & 2) ? il : -il, g2 = (d & 1) ? il : -il;
      const T h = qv[0] * fv[d].x + qv[1] * fv[d].y + qv[2] * fv[d].z + mass * fv[d].w;
      const T w = mul_rn<T>(mul_rn<T>(w0, w1), w2);
      a[0] = fma_rn<T>(w, fv[d].x, a[0]);
      a[1] = fma_rn<T>(w, fv[d].y, a[1]);
      a[2] = fma_rn<T>(w, fv[d].z, a[2]);
      al[0] += g0 * w1 * w2 * h;
      al[1] += w0 * g1 * w2 * h;
      al[2] += w0 * w1 * g2 * h;
    }
    if constexpr (OP) {
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        a_out[po + c * g.N + i] = a[c];
        alpha_out[po + c * g.N + i] = al[c];
      }
      continue;
    }
    acc_pa.add(qv[0] * a[0] + qv[1] * a[1] + qv[2] * a[2]);
    long long W[3] = {0, 0, 0};
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      if (fx.u) {
        // the forward's rounded increments, subtracted in reverse order (checkpoints are
        // never combined with the fixed-point state)
        W[c] = fx.w[po + c * g.N + i];
        W[c] -= to_fixed<T>(mul_rn<T>(mul_rn<T>(a[c], cA), fx.to_w));
        W[c] -= to_fixed<T>(mul_rn<T>(mul_rn<T>(a[c], cB), fx.to_w));
        pv[c] = mul_rn<T>(fix_to_real<T>(W[c]), fx.from_w);
      } else {
        pv[c] -= a[c] * cA;
        if (ck_p) pv[c] = ck_p[po + c * g.N + i];
        pv[c] -= a[c] * cB;
      }
      xv[c] += al[c] * cA;
      xv[c] += al[c] * cB;
    }
    acc_xp.add(xv[0] * pv[0] + xv[1] * pv[1] + xv[2] * pv[2]);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      if (fx.u) {
        long long U = fx.u[po + c * g.N + i];
        U -= to_fixed<T>(mul_rn<T>(mul_rn<T>(mul_rn<T>(fix_to_real<T>(W[c]), fx.w_cells), dr), fx.du));
        fx.u[po + c * g.N + i] = U;
        fx.w[po + c * g.N + i] = W[c];
        sv[c] = mul_rn<T>(fix_to_real<T>(U), fx.from_u);
      } else {
        sv[c] -= pv[c] * dr;
      }
      qv[c] += xv[c] * dr;
      if (ck_s) sv[c] = ck_s[po + c * g.N + i];
      s[po + c * g.N + i] = sv[c];
      p[po + c * g.N + i] = pv[c];
      xi[po + c * g.N + i] = xv[c];
      pi[po + c * g.N + i] = qv[c];
      mx[c] = fmaxf(mx[c], abs_up<T>(qv[c]));
      if (a_out) a_out[po + c * g.N + i] = a[c];
      if (alpha_out) alpha_out[po + c * g.N + i] = al[c];
    }
    if (bcount) count_bin(g, bg, i, sv, b, bcount, bkeys);   // bin for the previous step's deposit
  }
  if constexpr (OP) return;
  const double spa = block_sum(acc_pa.value());
  const double sxp = block_sum(acc_xp.value());
  if (threadIdx.x == 0 && part_pa) {
    part_pa[(long long)b * gridDim.x + blockIdx.x] = spa;
    part_xp[(long long)b * gridDim.x + blockIdx.x] = sxp;
  }
  if (pimax) {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const float m = block_max(mx[c], shf);
      if (threadIdx.x == 0) atomicMax(pimax + c * gridDim.y + b, __float_as_uint(m));
    }
  }
}

// max |pi_c| of every instance (layout [c][batch]), for the fixed-point exponents
template <typename T>
__global__ void __launch_bounds__(kPtclThreads)
k_pi_max(const T* __restrict__ pi, long long N, unsigned* __restrict__ pimax) {
  __shared__ float shf[kPtclThreads / 32];
  const int b = blockIdx.y;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const T* q = pi + ((long long)b * 3 + c) * N;
    float mx = 0.f;
    for (long long i = blockIdx.x * (long long)kPtclThreads + threadIdx.x; i < N; i += (long long)gridDim.x * kPtclThreads)
      mx = fmaxf(mx, abs_up<T>(q[i]));
    const float m = block_max(mx, shf);
    if (threadIdx.x == 0) atomicMax(pimax + c * gridDim.y + b, __float_as_uint(m));
  }
}

// xv += m sum_g grad_x W(g - x_i) D(g) over the 8 CIC corners of particle i at
// displacement sv: a density cotangent D carried to the particle position through the
// weight gradient (floor convention, -1/l and +1/l per axis).
template <typename T>
__device__ __forceinline__ void cic_grad_gather(const Geo<T>& g, long long i, const T sv[3], const T* D, T mass,
                                                T xv[3]) {
  const T il = g.inv_l;
  int cell[3];
  T t[3];
  cic_cell(g, i, sv, cell, t);
#pragma unroll
  for (int d = 0; d < 8; ++d) {
    const T w0 = (d & 4) ? t[0] : (T)1 - t[0];
    const T w1 = (d & 2) ? t[1] : (T)1 - t[1];
    const T w2 = (d & 1) ? t[2] : (T)1 - t[2];
    const T g0 = (d & 4) ? il : -il, g1 = (d & 2) ? il : -il, g2 = (d & 1) ? il : -il;
    const T h = mass * __ldg(D + corner_index(g, cell, d));
    xv[0] += g0 * w1 * w2 * h;
    xv[1] += w0 * g1 * w2 * h;
    xv[2] += w0 * w1 * g2 * h;
  }
}

// xi = m sum_g grad W(g - x) dJ/ddelta(g) (+ dJ/dx);  pi = dJ/dp (or 0)
template <typename T>
__global__ void __launch_bounds__(kPtclThreads)
k_adjoint_init(Geo<T> g, T mass, const T* __restrict__ s, const T* __restrict__ djdd, const T* __restrict__ djdx,
               const T* __restrict__ djdp, T* __restrict__ xi, T* __restrict__ pi, unsigned* __restrict__ pimax) {
  __shared__ float shf[kPtclThreads / 32];
  const int b = blockIdx.y;
  const long long po = (long long)b * 3 * g.N;
  float mx[3] = {0.f, 0.f, 0.f};
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < g.N;
       i += (long long)gridDim.x * blockDim.x) {
    T xv[3] = {0, 0, 0};
    if (djdd) {
      const T sv[3] = {s[po + i], s[po + g.N + i], s[po + 2 * g.N + i]};
      cic_grad_gather(g, i, sv, djdd + (long long)b * g.M, mass, xv);
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      if (djdx) xv[c] += djdx[po + c * g.N + i];
      xi[po + c * g.N + i] = xv[c];
      const T q = djdp ? djdp[po + c * g.N + i] : (T)0;
      pi[po + c * g.N + i] = q;
      mx[c] = fmaxf(mx[c], abs_up<T>(q));
    }
  }
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const float m = block_max(mx[c], shf);
    if (threadIdx.x == 0) atomicMax(pimax + c * gridDim.y + b, __float_as_uint(m));
  }
}

// Cotangent of an observed intermediate state (Sec. 2.4, objectives on z_0..z_n), added
// when the reverse pass holds its positions x_j:  xi += m sum_g grad W dJ/d delta_j(g)
// + dJ/dx_j.  xi enters nothing before the reverse drift of step j, so the sum is exact
// whatever the kicks between add.
template <typename T>
__global__ void __launch_bounds__(kPtclThreads)
k_obs_cotangent(Geo<T> g, T mass, const T* __restrict__ s, const T* __restrict__ djdd, const T* __restrict__ djdx,
                T* __restrict__ xi) {
  const int b = blockIdx.y;
  const long long po = (long long)b * 3 * g.N;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < g.N;
       i += (long long)gridDim.x * blockDim.x) {
    T xv[3] = {0, 0, 0};
    if (djdd) {
      const T sv[3] = {s[po + i], s[po + g.N + i], s[po + 2 * g.N + i]};
      cic_grad_gather(g, i, sv, djdd + (long long)b * g.M, mass, xv);
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      if (djdx) xv[c] += djdx[po + c * g.N + i];
      xi[po + c * g.N + i] += xv[c];
    }
  }
}

// Cotangent v = dJ/dp_j of an observed momentum (Sec. 2.4), added to pi in two parts
// around the reverse step at force step j: the reverse kick K1_{j+1} uses pi, the
// reverse kick K2_j (the one that made p_j) pi + v.  The force VJP is linear in pi, so one
// VJP of pi + c v with c = K2_j / (K1_{j+1} + K2_j) gives both kicks' alpha terms:
//   mode 0 (before the force chain): pi += c v
//   mode 1 (after the reverse step):  pi += (1 - c) v, and the FP64 block sums of v . a_j
//   (the theta term of the K2_j kick that pi + c v does not carry).
// The fixed-point exponent of the next pi deposit is kept valid: max |pi| is folded into
// pimax.
template <typename T>
__global__ void __launch_bounds__(kPtclThreads)
k_obs_momentum(Geo<T> g, T* __restrict__ pi, const T* __restrict__ v, const T* __restrict__ ctab, int j, int nstep1,
               int mode, const T* __restrict__ a, double* __restrict__ part, unsigned* __restrict__ pimax) {
  __shared__ float shf[kPtclThreads / 32];
  const int b = blockIdx.y;
  const long long po = (long long)b * 3 * g.N;
  const T c = ctab[b * nstep1 + j];
  const T w = mode == 0 ? c : (T)1 - c;
  double acc = 0.0;
  float mx[3] = {0.f, 0.f, 0.f};
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < g.N; i += (long long)gridDim.x * blockDim.x) {
    T va = 0;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const long long o = po + k * g.N + i;
      const T q = pi[o] + w * v[o];
      pi[o] = q;
      mx[k] = fmaxf(mx[k], abs_up<T>(q));
      if (mode == 1) va += v[o] * a[o];
    }
    acc += (double)va;
  }
  if (mode == 1) {
    const double r = block_sum(acc);
    if (threadIdx.x == 0) part[(long long)b * gridDim.x + blockIdx.x] = r;
  }
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const float m = block_max(mx[k], shf);
    if (threadIdx.x == 0) atomicMax(pimax + k * gridDim.y + b, __float_as_uint(m));
  }
}

// Cotangent of positions observed at a scale factor a between steps j and j + 1 (Sec. 2.4):
// x(a) = q + s_j + Dp_j(a) p_{j+1/2} with the partial drift factor fac = Dp_j(a), taken
// while the reverse pass holds (s_j, p_{j+1/2}) before the force VJP at x_j:
//   u = m sum_g grad W(g - x(a)) dJ/d delta(a)(g) + dJ/dx(a);  xi += u;  pi += fac u;
// and the FP64 block sums of u . p_{j+1/2} (the theta term of Dp_j).
template <typename T>
__global__ void __launch_bounds__(kPtclThreads)
k_obs_interp(Geo<T> g, T mass, const T* __restrict__ s, const T* __restrict__ p, const T* __restrict__ fac_tab,
             const T* __restrict__ djdd, const T* __restrict__ djdx, T* __restrict__ xi, T* __restrict__ pi,
             double* __restrict__ part, unsigned* __restrict__ pimax) {
  __shared__ float shf[kPtclThreads / 32];
  const int b = blockIdx.y;
  const long long po = (long long)b * 3 * g.N;
  const T fac = fac_tab[b];
  double acc = 0.0;
  float mx[3] = {0.f, 0.f, 0.f};
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < g.N; i += (long long)gridDim.x * blockDim.x) {
    T u[3] = {0, 0, 0};
    const T pv[3] = {p[po + i], p[po + g.N + i], p[po + 2 * g.N + i]};
    if (djdd) {
      const T sa[3] = {s[po + i] + fac * pv[0], s[po + g.N + i] + fac * pv[1], s[po + 2 * g.N + i] + fac * pv[2]};
      cic_grad_gather(g, i, sa, djdd + (long long)b * g.M, mass, u);
    }
    T up = 0;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const long long o = po + k * g.N + i;
      if (djdx) u[k] += djdx[o];
      xi[o] += u[k];
      const T q = pi[o] + fac * u[k];
      pi[o] = q;
      mx[k] = fmaxf(mx[k], abs_up<T>(q));
      up += u[k] * pv[k];
    }
    acc += (double)up;
  }
  const double r = block_sum(acc);
  if (threadIdx.x == 0) part[(long long)b * gridDim.x + blockIdx.x] = r;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const float m = block_max(mx[k], shf);
    if (threadIdx.x == 0) atomicMax(pimax + k * gridDim.y + b, __float_as_uint(m));
  }
}

// Forward: the displacement at an observed scale factor a between steps j and j + 1 from
// the state right after the step's gather, s(a) = s_{j+1} + (Dp_j(a) - D_{j+1}) p_{j+1/2}.
template <typename T>
__global__ void k_interp_state(const T* __restrict__ s, const T* __restrict__ p, const T* __restrict__ cf_tab,
                               T* __restrict__ out, long long n3) {
  const int b = blockIdx.y;
  const T cf = cf_tab[b];
  const long long o = (long long)b * n3;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n3; i += (long long)gridDim.x * blockDim.x)
    out[o + i] = s[o + i] + cf * p[o + i];
}

// theta[b][2] (Omega_m) += sum_k w[k][b] sums[k][b]: the theta terms of the observations
static __global__ void k_obs_theta(const double* __restrict__ sums, const double* __restrict__ w, int nk, int batch,
                                   double* __restrict__ theta) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= batch) return;
  double acc = 0.0;
  for (int k = 0; k < nk; ++k) acc += w[(long long)k * batch + b] * sums[(long long)k * batch + b];
  theta[5 * b + 2] += acc;
}

// Real meshes from the sums of k_scatter<T, NQ>, the conversion of the tile deposit
// (k_pull_scatter): delta = m acc 2^-e_d - 1 into dout (instance stride dis), pi_c = acc 2^-e_c
// into p0..p2 (instance stride pis).  Leaves the sums zero for the next call.
__device__ __forceinline__ float sum_to_real(long long v, float) { return ll2f_rn(v); }
__device__ __forceinline__ double sum_to_real(long long v, double) { return (double)v; }
template <typename T, int NQ>
__global__ void __launch_bounds__(kPtclThreads)
k_mesh_out(long long* __restrict__ acc, long long M, int e_d, const int* __restrict__ e_pi, T mass, T* __restrict__ dout,
           long long dis, T* __restrict__ p0, T* __restrict__ p1, T* __restrict__ p2, long long pis) {
  const int b = blockIdx.y;
  const T md = mass * pow2i<T>(-e_d);
  T mp[3] = {0, 0, 0};
  if constexpr (NQ == 4) {
#pragma unroll
    for (int c = 0; c < 3; ++c) mp[c] = pow2i<T>(-e_pi[c * gridDim.y + b]);
  }
  for (long long i = blockIdx.x * (long long)kPtclThreads + threadIdx.x; i < M; i += (long long)gridDim.x * kPtclThreads) {
    long long* a = acc + NQ * (b * M + i);
    if constexpr (NQ == 1) {
      dout[b * dis + i] = sum_to_real(a[0], (T)0) * md + (T)-1;
      a[0] = 0;
    } else {
      longlong2* a2 = reinterpret_cast<longlong2*>(a);
      const longlong2 v0 = a2[0], v1 = a2[1];
      a2[0] = a2[1] = make_longlong2(0, 0);
      dout[b * dis + i] = sum_to_real(v0.x, (T)0) * md + (T)-1;
      p0[b * pis + i] = sum_to_real(v0.y, (T)0) * mp[0];
      p1[b * pis + i] = sum_to_real(v1.x, (T)0) * mp[1];
      p2[b * pis + i] = sum_to_real(v1.y, (T)0) * mp[2];
    }
  }
}

// delta = m acc 2^-e - 1 (no zeroing)
template <typename T>
__global__ void k_density_out(const long long* __restrict__ acc, T* __restrict__ out, long long total, T mul) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total; i += (long long)gridDim.x * blockDim.x)
    out[i] = (T)acc[i] * mul - (T)1;
}

// J partials sum (delta - target)^2 and dJ/ddelta = 2 (delta - target) / M
template <typename T>
__global__ void __launch_bounds__(kPtclThreads)
k_mse(const T* __restrict__ dens, const T* __restrict__ tgt, T* __restrict__ grad, long long M, double* part) {
  const int b = blockIdx.y;
  const T* d = dens + (long long)b * M;
  const T* q = tgt + (long long)b * M;
  T* gr = grad + (long long)b * M;
  const T two_over_m = (T)(2.0 / (double)M);
  double acc = 0.0;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < M; i += (long long)gridDim.x * blockDim.x) {
    const T diff = d[i] - q[i];
    acc += (double)diff * diff;
    gr[i] = two_over_m * diff;
  }
  const double r = block_sum(acc);
  if (threadIdx.x == 0) part[(long long)b * gridDim.x + blockIdx.x] = r;
}

// ------------------------------------------------------------------ lattice spectra
// Mode (i0, i1, kx) of an n^3 half spectrum from a flat index over main + side (n a power of
// two: shifts; 64-bit divisions took longer than the rest of the lattice kernels).
struct Mode { int f0, f1, f2; };
__device__ __forceinline__ Mode mode_of(long long u, int n) {
  const int lg = 31 - __clz(n);
  const long long main = (long long)n * n * (n / 2);
  const bool in = u < main;
  const long long t = in ? u >> (lg - 1) : u - main;
  Mode m;
  m.f1 = freq_of((int)t & (n - 1), n);
  m.f0 = freq_of((int)(t >> lg), n);
  m.f2 = in ? (int)u & (n / 2 - 1) : n / 2;
  return m;
}
__device__ __forceinline__ int nyq_zero(int f, int n, bool last) { return last ? (f == n / 2 ? 0 : f) : (f == -n / 2 ? 0 : f); }

// s1^_c = B_c Omega, B_c = i k_c / k^2 sqrt(P / l_p^3) / n^3 (Sec. 2.1, Eqs. 3-6).  With
// amp = null the amplitude is the constant `unit` (the 2LPT s2 from the source spectrum).
template <typename T>
__global__ void k_za_mul(const cx_t<T>* __restrict__ om, cx_t<T>* o0, cx_t<T>* o1, cx_t<T>* o2, int n,
                         const T* __restrict__ amp, int maxn2, T inv_kf, long long is, T unit) {
  using C = cx_t<T>;
  const int b = blockIdx.y;
  const long long tot = spec_len_cx(n);
  for (long long u = blockIdx.x * (long long)blockDim.x + threadIdx.x; u < tot; u += (long long)gridDim.x * blockDim.x) {
    const Mode m = mode_of(u, n);
    const int n2 = m.f0 * m.f0 + m.f1 * m.f1 + m.f2 * m.f2;
    const C v = om[b * is + u];
    const T base = n2 ? (amp ? amp[(long long)b * (maxn2 + 1) + n2] : unit) * inv_kf / (T)n2 : (T)0;
    const int fc[3] = {nyq_zero(m.f0, n, false), nyq_zero(m.f1, n, false), nyq_zero(m.f2, n, true)};
    C* outs[3] = {o0, o1, o2};
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const T sc = (T)fc[c] * base;
      outs[c][b * is + u] = cmake<C>(-v.y * sc, v.x * sc);  // i v sc
    }
  }
}

// Omega_bar = sum_c conj(B_c) S_c (+ acc, the 2LPT part, when given);  theta partials
// sum_k w Re[conj(Omega_bar) Omega] dlnP_j / 2.  With amp = null the amplitude is the
// constant `unit` and no partials are taken (hdlnp = null): the transpose of the 2LPT
// source -> s2 map.
template <typename T>
__global__ void __launch_bounds__(kPtclThreads)
k_za_adj_mul(const cx_t<T>* s0, const cx_t<T>* s1, const cx_t<T>* s2, const cx_t<T>* __restrict__ om,
             const cx_t<T>* acc_in, cx_t<T>* out, int n, const T* __restrict__ amp, T unit,
             const double* __restrict__ hdlnp, int maxn2, T inv_kf, long long is,
             double* part /* [5][batch][grid] */) {
  using C = cx_t<T>;
  const int b = blockIdx.y;
  const long long tot = spec_len_cx(n);
  double acc[5] = {0, 0, 0, 0, 0};
  const C* ins[3] = {s0, s1, s2};
  for (long long u = blockIdx.x * (long long)blockDim.x + threadIdx.x; u < tot; u += (long long)gridDim.x * blockDim.x) {
    const Mode m = mode_of(u, n);
    const int n2 = m.f0 * m.f0 + m.f1 * m.f1 + m.f2 * m.f2;
    const T base = n2 ? (amp ? amp[(long long)b * (maxn2 + 1) + n2] : unit) * inv_kf / (T)n2 : (T)0;
    const int fc[3] = {nyq_zero(m.f0, n, false), nyq_zero(m.f1, n, false), nyq_zero(m.f2, n, true)};
    C r = acc_in ? acc_in[b * is + u] : cmake<C>(0, 0);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const C v = ins[c][b * is + u];
      const T sc = (T)fc[c] * base;
      r = cadd(r, cmake<C>(v.y * sc, -v.x * sc));  // -i v sc
    }
    out[b * is + u] = r;
    if (!hdlnp) continue;
    const C w = om[b * is + u];
    const double re = (double)r.x * w.x + (double)r.y * w.y;
    const double wt = (m.f2 == 0 || m.f2 == n / 2) ? 1.0 : 2.0;
#pragma unroll
    for (int j = 0; j < 5; ++j) acc[j] += wt * re * hdlnp[((long long)b * 5 + j) * (maxn2 + 1) + n2];
  }
  if (!hdlnp) return;
#pragma unroll
  for (int j = 0; j < 5; ++j) {
    const double r = block_sum(acc[j]);
    if (threadIdx.x == 0) part[((long long)j * gridDim.y + b) * gridDim.x + blockIdx.x] = r;
  }
}

// ------------------------------------------------------------ 2LPT (Sec. 2.1, Eqs. 2-4)
// The Hessian pairs (i, j) of the first-order potential: group 0 the diagonal ones
// (00, 11, 22), group 1 the mixed ones (01, 02, 12).
__device__ __forceinline__ void lpt_pair(int group, int q, int& i, int& j) {
  i = group ? (q == 2 ? 1 : 0) : q;
  j = group ? (q == 0 ? 1 : 2) : q;
}

// Hessian spectra phi_ij^ = (i k_i)(i k_j)(-1/k^2) delta1^ = k_i k_j / k^2 amp Omega
// (laplacian phi = delta1, Eq. 4), each i k_c zeroed on the Nyquist plane of axis c, for
// the three pairs of `group`; amp = sqrt(P / l_p^3) / n^3 per |n|^2.
template <typename T>
__global__ void k_lpt_hess(const cx_t<T>* __restrict__ om, cx_t<T>* o0, cx_t<T>* o1, cx_t<T>* o2, int n,
                           const T* __restrict__ amp, int maxn2, long long is, int group) {
  using C = cx_t<T>;
  const int b = blockIdx.y;
  const long long tot = spec_len_cx(n);
  C* outs[3] = {o0, o1, o2};
  for (long long u = blockIdx.x * (long long)blockDim.x + threadIdx.x; u < tot; u += (long long)gridDim.x * blockDim.x) {
    const Mode m = mode_of(u, n);
    const int n2 = m.f0 * m.f0 + m.f1 * m.f1 + m.f2 * m.f2;
    const C v = om[b * is + u];
    const T base = n2 ? amp[(long long)b * (maxn2 + 1) + n2] / (T)n2 : (T)0;
    const int fc[3] = {nyq_zero(m.f0, n, false), nyq_zero(m.f1, n, false), nyq_zero(m.f2, n, true)};
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      int i, j;
      lpt_pair(group, q, i, j);
      const T sc = (T)(fc[i] * fc[j]) * base;
      outs[q][b * is + u] = cmake<C>(v.x * sc, v.y * sc);
    }
  }
}

// The 2LPT source S = sum_{i<j} (phi_ii phi_jj - phi_ij^2) (Eq. 4) from the real Hessian
// components r0..r2 of `group`: group 0 writes phi_00 phi_11 + phi_00 phi_22 +
// phi_11 phi_22, group 1 subtracts phi_01^2 + phi_02^2 + phi_12^2.
template <typename T>
__global__ void k_lpt_source(const T* __restrict__ r0, const T* __restrict__ r1, const T* __restrict__ r2,
                             long long ris, long long N, T* src, long long sis, int group) {
  const int b = blockIdx.y;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < N; i += (long long)gridDim.x * blockDim.x) {
    const T h0 = r0[b * ris + i], h1 = r1[b * ris + i], h2 = r2[b * ris + i];
    T* o = src + b * sis + i;
    if (group == 0)
      *o = h0 * h1 + h0 * h2 + h1 * h2;
    else
      *o = *o - (h0 * h0 + h1 * h1 + h2 * h2);
  }
}

// Transpose of the source at each point, in place over the Hessian components of
// `group`: phi_bar = dS/dphi S_bar, i.e. phi_bar_ii = S_bar sum_{j != i} phi_jj (group 0)
// and phi_bar_ij = -2 phi_ij S_bar (group 1).
template <typename T>
__global__ void k_lpt_source_adj(T* r0, T* r1, T* r2, long long ris, long long N, const T* __restrict__ sbar,
                                 long long sis, int group) {
  const int b = blockIdx.y;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < N; i += (long long)gridDim.x * blockDim.x) {
    const T h0 = r0[b * ris + i], h1 = r1[b * ris + i], h2 = r2[b * ris + i];
    const T sb = sbar[b * sis + i];
    if (group == 0) {
      r0[b * ris + i] = (h1 + h2) * sb;
      r1[b * ris + i] = (h0 + h2) * sb;
      r2[b * ris + i] = (h0 + h1) * sb;
    } else {
      r0[b * ris + i] = (T)-2 * h0 * sb;
      r1[b * ris + i] = (T)-2 * h1 * sb;
      r2[b * ris + i] = (T)-2 * h2 * sb;
    }
  }
}

// Transpose of Omega -> phi_ij (real even multipliers k_i k_j / k^2 amp): the spectra
// i0..i2 of the Hessian adjoints of `group` summed into acc (group 0 overwrites acc).
template <typename T>
__global__ void k_lpt_hess_adj(const cx_t<T>* __restrict__ i0, const cx_t<T>* __restrict__ i1,
                               const cx_t<T>* __restrict__ i2, cx_t<T>* acc, int n, const T* __restrict__ amp,
                               int maxn2, long long is, int group) {
  using C = cx_t<T>;
  const int b = blockIdx.y;
  const long long tot = spec_len_cx(n);
  const C* ins[3] = {i0, i1, i2};
  for (long long u = blockIdx.x * (long long)blockDim.x + threadIdx.x; u < tot; u += (long long)gridDim.x * blockDim.x) {
    const Mode m = mode_of(u, n);
    const int n2 = m.f0 * m.f0 + m.f1 * m.f1 + m.f2 * m.f2;
    const T base = n2 ? amp[(long long)b * (maxn2 + 1) + n2] / (T)n2 : (T)0;
    const int fc[3] = {nyq_zero(m.f0, n, false), nyq_zero(m.f1, n, false), nyq_zero(m.f2, n, true)};
    C r = group ? acc[b * is + u] : cmake<C>(0, 0);
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      int i, j;
      lpt_pair(group, q, i, j);
      const T sc = (T)(fc[i] * fc[j]) * base;
      const C v = ins[q][b * is + u];
      r = cadd(r, cmake<C>(v.x * sc, v.y * sc));
    }
    acc[b * is + u] = r;
  }
}

// Second-order terms of the initial state: s += D2 s2, p += G_D2 s2, s2 kept for the
// adjoint's Omega_m terms (Sec. 2.1, Eq. 2).
template <typename T>
__global__ void k_ic_state2(const T* __restrict__ r0, const T* __restrict__ r1, const T* __restrict__ r2,
                            long long ris, long long N, const T* __restrict__ d2, const T* __restrict__ gd2, T* s2,
                            T* s, T* p) {
  const int b = blockIdx.y;
  const T* rs[3] = {r0 + b * ris, r1 + b * ris, r2 + b * ris};
  const T d = d2[b], gd = gd2[b];
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < N; i += (long long)gridDim.x * blockDim.x) {
    const long long o = (long long)b * 3 * N + i;
    T v[3], sv[3], pv[3];   // every load before the first store
#pragma unroll
    for (int c = 0; c < 3; ++c) v[c] = rs[c][i], sv[c] = s[o + c * N], pv[c] = p[o + c * N];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      s2[o + c * N] = v[c];
      s[o + c * N] = sv[c] + d * v[c];
      p[o + c * N] = pv[c] + gd * v[c];
    }
  }
}

// s1 from the lattice C2R outputs; s = D1 s1, p = G_D s1
template <typename T>
__global__ void k_ic_state(const T* __restrict__ r0, const T* __restrict__ r1, const T* __restrict__ r2, long long ris,
                           long long N, const T* __restrict__ d1, const T* __restrict__ gd, T* s1, T* s, T* p) {
  const int b = blockIdx.y;
  const T* rs[3] = {r0 + b * ris, r1 + b * ris, r2 + b * ris};
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < N; i += (long long)gridDim.x * blockDim.x) {
    const T v[3] = {rs[0][i], rs[1][i], rs[2][i]};
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const long long o = (long long)b * 3 * N + c * N + i;
      if (s1) s1[o] = v[c];
      if (s) s[o] = d1[b] * v[c];
      if (p) p[o] = gd[b] * v[c];
    }
  }
}

// Fixed-point state from the initial state: U = round(s / l 2^kFixES), W = round(p / l
// 2^kFixEP), and s, p replaced by their shadows
template <typename T>
__global__ void k_fix_init(T* __restrict__ s, T* __restrict__ p, FixState<T> fx, T to_u, long long n3) {
  const int b = blockIdx.y;
  const long long o0 = (long long)b * n3;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n3; i += (long long)gridDim.x * blockDim.x) {
    const long long o = o0 + i;
    const long long U = to_fixed<T>(mul_rn<T>(s[o], to_u));
    const long long W = to_fixed<T>(mul_rn<T>(p[o], fx.to_w));
    fx.u[o] = U;
    fx.w[o] = W;
    s[o] = mul_rn<T>(fix_to_real<T>(U), fx.from_u);
    p[o] = mul_rn<T>(fix_to_real<T>(W), fx.from_w);
  }
}

// sbar = D1 xi + G_D pi into the lattice FFT inputs; partials of xi.s1 and pi.s1
template <typename T>
__global__ void __launch_bounds__(kPtclThreads)
k_ic_adj_prep(const T* __restrict__ xi, const T* __restrict__ pi, const T* __restrict__ s1, long long N,
              const T* __restrict__ d1, const T* __restrict__ gd, T* w0, T* w1, T* w2, long long wis,
              double* part_xs, double* part_ps) {
  const int b = blockIdx.y;
  T* ws[3] = {w0 + b * wis, w1 + b * wis, w2 + b * wis};
  double axs = 0, aps = 0;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < N; i += (long long)gridDim.x * blockDim.x) {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const long long o = (long long)b * 3 * N + c * N + i;
      const T x = xi[o], q = pi[o], u = s1[o];
      ws[c][i] = d1[b] * x + gd[b] * q;
      axs += (double)x * u;
      aps += (double)q * u;
    }
  }
  const double r1 = block_sum(axs);
  const double r2 = block_sum(aps);
  if (threadIdx.x == 0) {
    part_xs[(long long)b * gridDim.x + blockIdx.x] = r1;
    part_ps[(long long)b * gridDim.x + blockIdx.x] = r2;
  }
}

// Fixed-order sum of `count` partials for each instance: out[b] = sum_i part[b][i]
static __global__ void k_sum_partials(const double* __restrict__ part, int count, double* out, double scale) {
  const int b = blockIdx.x;
  double acc = 0.0;
  for (int i = threadIdx.x; i < count; i += blockDim.x) acc += part[(long long)b * count + i];
  const double r = block_sum(acc);
  if (threadIdx.x == 0) out[b] = r * scale;
}

// dJ/dtheta (Eq. 51): time-stepping terms (Omega_m only), initial-condition growth terms
// and the P_lin derivative terms.  sums: per instance the already reduced scalars.
struct ThetaIn {
  const double* step_pa;   // pi.a at step j, instance b: step_pa[j * step_stride + b]
  const double* step_xp;   // xi.p at step j: step_xp[j * step_stride + b]
  const double* w_pa;      // weight of pi.a: w_pa[j * batch + b]
  const double* w_xp;      // weight of xi.p
  const double* xs;        // [batch]   xi_0 . s1
  const double* ps;        // [batch]   pi_0 . s1
  const double* dlp;       // [5][batch]
  const double* dd1;       // [batch]   dD1(a0)/dOm
  const double* dgd;       // [batch]   dG_D(a0)/dOm
  const double* xs2;       // [batch]   xi_0 . s2   (2LPT; null at first order)
  const double* ps2;       // [batch]   pi_0 . s2
  const double* dd2;       // [batch]   dD2(a0)/dOm
  const double* dgd2;      // [batch]   dG_D2(a0)/dOm
  int nstep1, batch, step_stride;
};
static __global__ void k_final_theta(ThetaIn in, double* out) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= in.batch) return;
  double g = 0.0;
  for (int j = 0; j < in.nstep1; ++j) {
    const long long o = (long long)j * in.step_stride + b;
    const long long w = (long long)j * in.batch + b;
    g += in.step_pa[o] * in.w_pa[w] + in.step_xp[o] * in.w_xp[w];
  }
  g += in.xs[b] * in.dd1[b] + in.ps[b] * in.dgd[b];
  if (in.xs2) g += in.xs2[b] * in.dd2[b] + in.ps2[b] * in.dgd2[b];
  for (int j = 0; j < 5; ++j) out[5 * b + j] = in.dlp[j * in.batch + b] + (j == 2 ? g : 0.0);
}

// ------------------------------------------------------------- power spectrum
// Shell-averaged power of a half spectrum (summary statistic of Sec. 2.4): bin b < nb = n/2
// holds the modes with b <= |n| < b + 1; off-plane modes count twice (for their
// conjugates).  The side plane kx = n/2 and the Nyquist rows lie outside every bin.  The
// sums are exact int64 fixed point with a per-bin scale from a first max pass, so the
// result does not depend on the order of the additions.
//
// A thread takes runs of consecutive kx of one row.  |n| grows along a run, so its modes
// fall into few bins: they are summed in registers and added to the block's bins in shared
// memory where the bin changes, and a block adds its bins to the global ones once.  FP32
// spectra are squared and rounded to fixed point in error-free FP32 pairs, not on the slow
// FP64 pipe.  Measured at 256^3 (67 MB spectrum): one global atomic per mode and FP64
// arithmetic took 667 + 800 us for the two passes, these 19 + 29 us; the cotangent 60, now 25 us.
constexpr int kPowerMaxBins = 512;
constexpr int kPowerThreads = 256;

__device__ __forceinline__ int isqrt_floor(int v) {
  int r = (int)sqrtf((float)v);
  while (r * r > v) --r;
  while ((r + 1) * (r + 1) <= v) ++r;
  return r;
}

// Runs of `len` = min(8, n/2) consecutive kx of the main rows (z-blocked by 2^lzb, spec_row):
// run u -> first element and the row's part of |n|^2.
struct PowerRuns {
  int lgn, lzb, lglen;
  long long count;     // runs per instance
  __device__ __forceinline__ long long at(long long u, int& kx, int& n01) const {
    const int lgs = lgn - 1 - lglen, n = 1 << lgn;      // log2 runs per row
    const int row = (int)(u >> lgs);
    kx = ((int)u & ((1 << lgs) - 1)) << lglen;
    const int t = row >> lzb;
    const int f1 = freq_of(t & (n - 1), n), f0 = freq_of(((t >> lgn) << lzb) | (row & ((1 << lzb) - 1)), n);
    n01 = f0 * f0 + f1 * f1;
    return ((long long)row << (lgn - 1)) + kx;
  }
};
inline PowerRuns power_runs(int n, int lzb) {
  PowerRuns r{};
  while ((1 << r.lgn) < n) ++r.lgn;
  r.lzb = lzb;
  r.lglen = r.lgn - 1 < 3 ? r.lgn - 1 : 3;
  r.count = ((long long)n * n * (n / 2)) >> r.lglen;
  return r;
}

// a run of 4 or 8 modes, in pairs (16-byte loads for FP32: a lane's run is 64 bytes)
template <typename C> struct alignas(2 * sizeof(C)) ModePair { C a, b; };
template <typename C> __device__ __forceinline__ void load_run(const C* p, int lglen, C (&v)[8]) {
  const ModePair<C>* q = reinterpret_cast<const ModePair<C>*>(p);
#pragma unroll
  for (int k = 0; k < 4; ++k)
    if (2 * k < (1 << lglen)) {
      const ModePair<C> m = q[k];
      v[2 * k] = m.a, v[2 * k + 1] = m.b;
    }
}

// an upper bound of w |v|^2 as a float, w = 2^lw
__device__ __forceinline__ float power_up(float2 v, int lw) { return __fmaf_ru(v.x, v.x, __fmul_ru(v.y, v.y)) * (float)(1 << lw); }
__device__ __forceinline__ float power_up(double2 v, int lw) {
  return __double2float_ru((double)(1 << lw) * (v.x * v.x + v.y * v.y));
}

// Exponent of bin `bin`: w |v|^2 < 2^E of every mode, and a shell of unit thickness holds
// fewer than 64 (b + 1)^2 lattice points (its volume widened by half a cell diagonal on both
// sides), so the sum of the values times 2^e stays below 2^62.  FP32 values are kept below
// 2^48, so that the parts of power_fixed fit their conversions.
template <typename T> __device__ __forceinline__ int power_exponent(unsigned pmax, int bin, int lgM) {
  const float mx = __uint_as_float(pmax);
  if (!(mx > 0.f) || !isfinite(mx)) return 0;
  int lgc = min(lgM, 6 + 2 * (32 - __clz(bin)));         // bin + 1 <= 2^(32 - clz(bin))
  if (sizeof(T) == 4) lgc = max(lgc, 14);
  return min(62 - lgc - (ilogbf(mx) + 1), 1000);
}

// w |v|^2 2^e in fixed point, w = 2^lw
__device__ __forceinline__ long long power_fixed(double2 v, int lw, int e) {
  return __double2ll_rn(ldexp((double)(1 << lw) * (v.x * v.x + v.y * v.y), e));
}
// |v| < 2^48 rounded, by one int32 conversion for the multiple of 2^26 and one for the
// remainder (which is exact)
__device__ __forceinline__ long long f2ll_split(float v) {
  const int hi = __float2int_rn(v * 0x1p-26f);
  return (long long)hi * (1 << 26) + __float2int_rn(fmaf(-(float)hi, 0x1p26f, v));
}
// the squares as error-free pairs: their high parts below 2^48, the sum of the low ones
// below 2^25
__device__ __forceinline__ long long power_fixed(float2 v, int lw, int e) {
  const int et = e + lw;
  const float sc = pow2i<float>(et >> 1), r = (float)(1 << (et & 1));   // 2^et = sc^2 r
  const float x = v.x * sc, y = v.y * sc;
  const float hx = x * x, hy = y * y;
  const float lo = fmaf(x, x, -hx) + fmaf(y, y, -hy);
  return f2ll_split(hx * r) + f2ll_split(hy * r) + __float2int_rn(lo * r);
}

template <typename T>
__global__ void __launch_bounds__(kPowerThreads)
k_power_max(const cx_t<T>* __restrict__ spec, PowerRuns pr, long long is, int nb, unsigned* pmax) {
  __shared__ unsigned smax[kPowerMaxBins];
  const int b = blockIdx.y;
  for (int i = threadIdx.x; i < nb; i += kPowerThreads) smax[i] = 0u;
  __syncthreads();
  for (long long u = blockIdx.x * (long long)kPowerThreads + threadIdx.x; u < pr.count;
       u += (long long)gridDim.x * kPowerThreads) {
    int kx, n01;
    const cx_t<T>* p = spec + b * is + pr.at(u, kx, n01);
    int bin = isqrt_floor(n01 + kx * kx);
    if (bin >= nb) continue;                             // |n| only grows along the run
    cx_t<T> v[8];
    load_run(p, pr.lglen, v);
    // the powers are non-negative: their bit patterns order like the values, NaN above infinity
    // (its sign cleared), so that a NaN stays the maximum
    unsigned m = 0u;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      if (k >= (1 << pr.lglen)) break;
      const int n2 = n01 + (kx + k) * (kx + k);
      if (n2 >= (bin + 1) * (bin + 1)) {
        atomicMax(&smax[bin], m);
        m = 0u;
        while (n2 >= (bin + 1) * (bin + 1)) ++bin;
        if (bin >= nb) break;
      }
      m = max(m, __float_as_uint(power_up(v[k], kx + k == 0 ? 0 : 1)) & 0x7FFFFFFFu);
    }
    if (bin < nb) atomicMax(&smax[bin], m);
  }
  __syncthreads();
  for (int i = threadIdx.x; i < nb; i += kPowerThreads)
    if (smax[i]) atomicMax(pmax + b * nb + i, smax[i]);
}

template <typename T>
__global__ void __launch_bounds__(kPowerThreads)
k_power_acc(const cx_t<T>* __restrict__ spec, PowerRuns pr, long long is, int nb, int lgM,
            const unsigned* __restrict__ pmax, unsigned long long* acc) {
  __shared__ unsigned lo[kPowerMaxBins], hi[kPowerMaxBins];
  __shared__ int se[kPowerMaxBins];
  const int b = blockIdx.y;
  for (int i = threadIdx.x; i < nb; i += kPowerThreads) {
    lo[i] = hi[i] = 0u;
    se[i] = power_exponent<T>(pmax[b * nb + i], i, lgM);
  }
  __syncthreads();
  auto flush = [&](int bin, long long a) {
    smem_add64(&lo[bin], &hi[bin], (unsigned)a, (unsigned)((unsigned long long)a >> 32));
  };
  for (long long u = blockIdx.x * (long long)kPowerThreads + threadIdx.x; u < pr.count;
       u += (long long)gridDim.x * kPowerThreads) {
    int kx, n01;
    const cx_t<T>* p = spec + b * is + pr.at(u, kx, n01);
    int bin = isqrt_floor(n01 + kx * kx);
    if (bin >= nb) continue;
    cx_t<T> v[8];
    load_run(p, pr.lglen, v);
    long long a = 0;
    int e = se[bin];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      if (k >= (1 << pr.lglen)) break;
      const int n2 = n01 + (kx + k) * (kx + k);
      if (n2 >= (bin + 1) * (bin + 1)) {
        flush(bin, a);
        a = 0;
        while (n2 >= (bin + 1) * (bin + 1)) ++bin;
        if (bin >= nb) break;
        e = se[bin];
      }
      a += power_fixed(v[k], kx + k == 0 ? 0 : 1, e);
    }
    if (bin < nb) flush(bin, a);
  }
  __syncthreads();
  for (int i = threadIdx.x; i < nb; i += kPowerThreads) {
    const unsigned long long a = ((unsigned long long)hi[i] << 32) | lo[i];
    if (a) atomicAdd(acc + b * nb + i, a);
  }
}

// Modes per bin and the sum of |n| (units of 2^-20) per bin, which depend on the mesh side
// alone: a thread per pair |f0| >= |f1| of the sphere |n| < nb, each mode with the
// multiplicity of its signs and of the exchange.
static __global__ void __launch_bounds__(kPowerThreads)
k_power_modes(int nb, unsigned long long* __restrict__ cnt, unsigned long long* __restrict__ ksum) {
  __shared__ unsigned c_lo[kPowerMaxBins], c_hi[kPowerMaxBins], s_lo[kPowerMaxBins], s_hi[kPowerMaxBins];
  for (int i = threadIdx.x; i < nb; i += kPowerThreads) c_lo[i] = c_hi[i] = s_lo[i] = s_hi[i] = 0u;
  __syncthreads();
  for (int q = blockIdx.x * kPowerThreads + threadIdx.x; q < nb * nb; q += gridDim.x * kPowerThreads) {
    const int i = q / nb, j = q % nb;
    const int n01 = i * i + j * j;
    if (j > i || n01 >= nb * nb) continue;
    const unsigned long long mult = (i ? 2 : 1) * (j ? 2 : 1) * (i != j ? 2 : 1);
    int bin = isqrt_floor(n01);
    unsigned long long c = 0, s = 0;
    auto flush = [&]() {
      smem_add64(&c_lo[bin], &c_hi[bin], (unsigned)c, (unsigned)(c >> 32));
      smem_add64(&s_lo[bin], &s_hi[bin], (unsigned)s, (unsigned)(s >> 32));
      c = s = 0;
    };
    for (int k = 0; k < nb; ++k) {
      const int n2 = n01 + k * k;
      if (n2 >= (bin + 1) * (bin + 1)) {
        flush();
        while (n2 >= (bin + 1) * (bin + 1)) ++bin;
        if (bin >= nb) break;
      }
      const int w = k == 0 ? 1 : 2;
      c += w * mult;
      s += (unsigned long long)__double2ll_rn(w * sqrt((double)n2) * 1048576.0) * mult;
    }
    if (bin < nb) flush();
  }
  __syncthreads();
  for (int i = threadIdx.x; i < nb; i += kPowerThreads) {
    if (c_lo[i] | c_hi[i]) atomicAdd(cnt + i, ((unsigned long long)c_hi[i] << 32) | c_lo[i]);
    if (s_lo[i] | s_hi[i]) atomicAdd(ksum + i, ((unsigned long long)s_hi[i] << 32) | s_lo[i]);
  }
}

// (a bin whose largest power is not finite gets NaN)
template <typename T>
__global__ void k_power_final(const unsigned long long* acc, const unsigned long long* cnt,
                                     const unsigned long long* ksum, const unsigned* pmax, int lgM, int nb, int batch,
                                     double vol_m2, double kf, double* pk, double* kmean, double* nmodes) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= nb * batch) return;
  const int bin = i % nb;
  const double c = (double)cnt[bin];
  const float mx = __uint_as_float(pmax[i]);
  pk[i] = !isfinite(mx) ? (double)(mx - mx)
                        : (c > 0 ? vol_m2 * ldexp((double)(long long)acc[i], -power_exponent<T>(pmax[i], bin, lgM)) / c : 0.0);
  if (i < nb) {
    if (kmean) kmean[bin] = c > 0 ? kf * ldexp((double)(long long)ksum[bin], -20) / c : 0.0;
    if (nmodes) nmodes[bin] = c;
  }
}

// Objective on the shell power (summary statistic of Sec. 2.4), one block per instance:
// J = sum_b w_b (P_b - T_b)^2 in a fixed order, and the per-bin factor of its density
// cotangent g_b = 2 w_b (P_b - T_b) 2 V / (M^2 C_b) (0 for empty bins).
static __global__ void __launch_bounds__(kPowerThreads)
k_power_loss(const double* __restrict__ pk, const double* __restrict__ nmodes, const double* __restrict__ tgt,
             const double* __restrict__ w, int nb, double two_v_m2, double* loss, double* g) {
  const int b = blockIdx.x;
  double j = 0.0;
  for (int i = threadIdx.x; i < nb; i += kPowerThreads) {
    const long long o = (long long)b * nb + i;
    const double d = pk[o] - tgt[o];
    j += w[o] * d * d;
    const double c = nmodes[i];
    g[o] = c > 0 ? 2.0 * w[o] * d * two_v_m2 / c : 0.0;
  }
  const double r = block_sum(j);
  if (threadIdx.x == 0) loss[b] = r;
}

// Cotangent spectrum g_b(|n|) delta^ in place over the half spectrum (bins b < nb, 0 beyond,
// the side plane among it); its unnormalised inverse transform is dJ/d delta (d P_b / d
// delta(x) is 2V / (M^2 C_b) times the inverse transform of delta^ restricted to shell b).
template <typename T>
__global__ void __launch_bounds__(kPowerThreads)
k_power_grad(cx_t<T>* spec, PowerRuns pr, long long is, int nb, const double* __restrict__ g) {
  __shared__ T sg[kPowerMaxBins];
  const int b = blockIdx.y, n = 1 << pr.lgn;
  for (int i = threadIdx.x; i < nb; i += kPowerThreads) sg[i] = (T)g[(long long)b * nb + i];
  __syncthreads();
  cx_t<T>* sp = spec + b * is;
  for (long long u = blockIdx.x * (long long)kPowerThreads + threadIdx.x; u < pr.count;
       u += (long long)gridDim.x * kPowerThreads) {
    int kx, n01;
    cx_t<T>* p = sp + pr.at(u, kx, n01);
    int bin = isqrt_floor(n01 + kx * kx);
    cx_t<T> v[8];
    load_run(p, pr.lglen, v);
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      if (k >= (1 << pr.lglen)) break;
      const int n2 = n01 + (kx + k) * (kx + k);
      while (n2 >= (bin + 1) * (bin + 1)) ++bin;
      const T f = bin < nb ? sg[bin] : (T)0;
      v[k].x *= f;
      v[k].y *= f;
    }
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (2 * k < (1 << pr.lglen)) reinterpret_cast<ModePair<cx_t<T>>*>(p)[k] = ModePair<cx_t<T>>{v[2 * k], v[2 * k + 1]};
  }
  const long long side = (long long)n * n * (n / 2);
  for (int i = blockIdx.x * kPowerThreads + threadIdx.x; i < n * n; i += gridDim.x * kPowerThreads) {
    cx_t<T>* q = sp + side + i;
    *q = cmake<cx_t<T>>(q->x * (T)0, q->y * (T)0);
  }
}

// numpy rfftn layout <-> main + side spectrum layout (for the FFT operator entry point), a warp per
// row of the mesh: the odd row length n/2 + 1 of the numpy layout then needs no division.
template <typename T, bool TO_STD>
__global__ void __launch_bounds__(256)
k_spec_std(const cx_t<T>* __restrict__ in, cx_t<T>* __restrict__ out, int n, long long rows) {
  using C = cx_t<T>;
  const int lgn = 31 - __clz(n), half = n / 2, lane = threadIdx.x & 31;
  for (long long row = blockIdx.x * 8LL + (threadIdx.x >> 5); row < rows; row += gridDim.x * 8LL) {
    const long long b = row >> (2 * lgn), r = row & ((1LL << (2 * lgn)) - 1);
    const long long main = b * spec_len_cx(n) + spec_row(n, spec_lzb(n), (int)(r >> lgn), (int)r & (n - 1)) * half;
    const long long side = b * spec_len_cx(n) + spec_main_len(n) + r, std = row * (half + 1);
    const C* src = in + (TO_STD ? main : std);
    C* dst = out + (TO_STD ? std : main);
    const C last = lane == 0 ? in[TO_STD ? side : std + half] : cmake<C>(0, 0);
#pragma unroll 8
    for (int k = lane; k < half; k += 32) dst[k] = src[k];
    if (lane == 0) out[TO_STD ? std + half : side] = last;
  }
}

}  // namespace pmgb
