// FP32 x passes of the 3-D real FFT for rows of n = 128..1024 reals, one row per group of
// lanes of a warp.
//
// A row of L = n/2 complex values lives in the registers of 8, 16 or 32 lanes, lane j holding
// the elements j + LANES r.  That layout is both what coalesced global loads and stores
// deliver and what the first and the last radix stage want, so a row passes through shared
// memory once per stage boundary only, inside its own warp (no block barrier), at addresses
// padded to be free of bank conflicts.  The element L - k that the even/odd split pairs with k
// sits in lane LANES - j and comes by shuffle.  Blocks stay resident and loop over rows, with
// the twiddles of the stages and of the split in shared memory.
//
// What bounds these passes is HBM; the tile form they replace (fft_impl.cuh, still used for
// FP64 and for shorter rows) moved each row through shared memory three times, with two of
// five wavefronts lost to bank conflicts in the three-component C2R.  The R2C takes this form
// at L = 512 only (four buffers of 1024^3: 7.5 -> 5.3 ms, where the tile form has two 64 KB
// tiles per SM); below, the tile form splits and stores with fewer instructions (512^3, four
// buffers: 750 us, this form 867).
#pragma once
#include <cuda_fp16.h>

#include "fft.cuh"
#include "pm_internal.h"

namespace pmgb {

// Radix stages of a row: LANES lanes hold P = L / LANES elements each.
template <int L> struct WarpRow;
template <> struct WarpRow<64>  { static constexpr int LANES = 8,  R0 = 8,  R1 = 8,  R2 = 1, BUF = 72; };
template <> struct WarpRow<128> { static constexpr int LANES = 8,  R0 = 16, R1 = 8,  R2 = 1, BUF = 136; };
template <> struct WarpRow<256> { static constexpr int LANES = 16, R0 = 16, R1 = 16, R2 = 1, BUF = 272; };
template <> struct WarpRow<512> { static constexpr int LANES = 32, R0 = 8,  R1 = 8,  R2 = 8, BUF = 576; };

constexpr bool has_warp_rows(int L) { return L >= 64 && L <= 512; }
constexpr bool has_warp_rows_r2c(int L) { return L == 512; }

template <int L> struct RowShape : WarpRow<L> {
  using W = WarpRow<L>;
  static constexpr int P = L / W::LANES;
  static constexpr int NT = 128;
  static constexpr int RPW = 32 / W::LANES;         // rows per warp
  static constexpr int RPB = RPW * NT / 32;         // rows per block and iteration
  static constexpr int TW = W::R2 == 1 ? L : 64 + L;   // stage twiddles
  static constexpr int SMEM = (RPB * W::BUF + TW + L) * (int)sizeof(float2);
};

// Twiddle tables of a block: t[r R0 + i] = w_L^(r i) for the last stage (before it, for three
// stages, t2[8 r + i] = w_64^(r i)), and wn[k] = exp(-2 pi i k / N).
template <int L>
__device__ __forceinline__ void row_tables(float2* t, float2* wn, const float2* __restrict__ twL,
                                           const float2* __restrict__ twN) {
  using S = RowShape<L>;
  constexpr int LAST = S::R2 == 1 ? S::R0 : S::R0 * S::R1;   // items of the last stage
  for (int i = threadIdx.x; i < L; i += S::NT) {
    t[i] = __ldg(twL + (i / LAST) * (i % LAST));
    wn[i] = __ldg(twN + i);
  }
  if constexpr (S::R2 != 1)
    for (int i = threadIdx.x; i < 64; i += S::NT) t[L + i] = __ldg(twL + (i / 8) * (i % 8) * (L / 64));
  __syncthreads();
}

// Products with their roundings written out (which of the two terms is rounded on its own), so
// that they do not depend on what the compiler contracts around them: the row forms round like
// the tile forms.
__device__ __forceinline__ float2 cmul_fwd(float2 a, float2 b) {
  return cmake<float2>(__fmaf_rn(a.x, b.x, -__fmul_rn(a.y, b.y)), __fmaf_rn(a.x, b.y, __fmul_rn(a.y, b.x)));
}
__device__ __forceinline__ float2 cmul_inv(float2 a, float2 b) {
  return cmake<float2>(__fmaf_rn(a.x, b.x, -__fmul_rn(a.y, b.y)), __fmaf_rn(a.y, b.x, __fmul_rn(a.x, b.y)));
}
__device__ __forceinline__ float2 cadd_rn(float2 a, float2 b) {
  return cmake<float2>(__fadd_rn(a.x, b.x), __fadd_rn(a.y, b.y));
}

// v exp(DIR 2 pi i m / L) from the table's exp(-2 pi i m / L)
template <int DIR> __device__ __forceinline__ float2 tw_mul(float2 v, float2 w) {
  if constexpr (DIR > 0) return cmul_inv(v, cconj(w));
  return cmul_fwd(v, w);
}

// Length-L DFT of the row held as z[r] = element j + LANES r, in and out, through the row's
// buffer.  The stages are those of fft_tile's plans (L <= 256); every lane of the warp calls it.
template <int L, int DIR>
__device__ __forceinline__ void row_fft(float2 (&z)[RowShape<L>::P], float2* buf, int j, const float2* t) {
  using S = RowShape<L>;
  constexpr int LN = S::LANES;
  if constexpr (L == 512) {
    // 8 x 8 x 8, two items i = j + 32 s per lane; item i holds z[2 r + s]
    float2 v[2][8];
#pragma unroll
    for (int s = 0; s < 2; ++s) {
#pragma unroll
      for (int r = 0; r < 8; ++r) v[s][r] = z[2 * r + s];
      dft<8, DIR>(v[s]);
    }
#pragma unroll
    for (int s = 0; s < 2; ++s) {
      const int i = j + 32 * s;
#pragma unroll
      for (int r = 0; r < 8; ++r) buf[i * 8 + (i >> 1) + r] = v[s][r];     // element 8 i + r at e + e / 16
    }
    __syncwarp();
#pragma unroll
    for (int s = 0; s < 2; ++s) {
      const int i = j + 32 * s;
#pragma unroll
      for (int r = 0; r < 8; ++r) v[s][r] = buf[i + (i >> 4) + 68 * r];
#pragma unroll
      for (int r = 1; r < 8; ++r) v[s][r] = tw_mul<DIR>(v[s][r], t[L + 8 * r + (j & 7)]);
      dft<8, DIR>(v[s]);
    }
    __syncwarp();
#pragma unroll
    for (int s = 0; s < 2; ++s) {
      const int i = j + 32 * s;
#pragma unroll
      for (int r = 0; r < 8; ++r) buf[(i >> 3) * 72 + (i & 7) + 8 * r] = v[s][r];   // element e at e + 8 (e / 64)
    }
    __syncwarp();
#pragma unroll
    for (int s = 0; s < 2; ++s) {
      const int i = j + 32 * s;
#pragma unroll
      for (int r = 0; r < 8; ++r) v[s][r] = buf[i + 72 * r];
#pragma unroll
      for (int r = 1; r < 8; ++r) v[s][r] = tw_mul<DIR>(v[s][r], t[64 * r + i]);
      dft<8, DIR>(v[s]);
#pragma unroll
      for (int r = 0; r < 8; ++r) z[2 * r + s] = v[s][r];
    }
    __syncwarp();
  } else {
    // R0 x R1: one item of the first stage per lane, R0 / LANES of the second
    constexpr int R0 = S::R0, R1 = S::R1, K = R0 / LN;
    dft<R0, DIR>(z);
#pragma unroll
    for (int r = 0; r < R0; ++r) buf[j * (R0 + 1) + r] = z[r];               // element e at e + e / R0
    __syncwarp();
#pragma unroll
    for (int s = 0; s < K; ++s) {
      const int i = j + LN * s;
      float2 v[R1];
#pragma unroll
      for (int r = 0; r < R1; ++r) v[r] = buf[i + (R0 + 1) * r];
#pragma unroll
      for (int r = 1; r < R1; ++r) v[r] = tw_mul<DIR>(v[r], t[R0 * r + i]);
      dft<R1, DIR>(v);
#pragma unroll
      for (int r = 0; r < R1; ++r) z[K * r + s] = v[r];
    }
    __syncwarp();
  }
}

// element L - k of a row, k = j + LANES r, given z; `at0` is the partner of k = 0
template <int L>
__device__ __forceinline__ float2 row_partner(const float2 (&z)[RowShape<L>::P], int r, int j, float2 at0) {
  using S = RowShape<L>;
  const int src = (S::LANES - j) & (S::LANES - 1);
  const float2 s = cmake<float2>(__shfl_sync(0xFFFFFFFFu, z[S::P - 1 - r].x, src, S::LANES),
                                 __shfl_sync(0xFFFFFFFFu, z[S::P - 1 - r].y, src, S::LANES));
  const float2 own = r == 0 ? at0 : z[(S::P - r) & (S::P - 1)];
  return j == 0 ? own : s;
}

// where row `row` of the launch lies: instance, row of the instance, main row and side element
template <int L> struct RowPlace {
  long long inst, rr, main, side;
  __device__ __forceinline__ RowPlace(int row, int lzb) {
    constexpr int N = 2 * L;
    inst = row / (N * N);
    rr = row % (N * N);
    const long long base = inst * spec_len_cx(N);
    main = base + spec_row(N, lzb, (int)(rr / N), (int)(rr % N)) * L;
    side = base + spec_main_len(N) + rr;
  }
};

// R2C: rows of n = 2L reals, the pairs (2j, 2j+1) read as one complex number, to L complex
// (main) + 1 (side).  The output may alias the input when the rows keep their order.
template <int L>
__global__ void __launch_bounds__(RowShape<L>::NT)
k_rows_r2c(RowJob<float> job, int nrows, int nbuf, const float2* __restrict__ twL, const float2* __restrict__ twN) {
  using S = RowShape<L>;
  constexpr int N = 2 * L, P = S::P, LN = S::LANES;
  extern __shared__ __align__(16) float2 rsm[];
  float2* t = rsm + S::RPB * S::BUF;
  float2* wn = t + S::TW;
  row_tables<L>(t, wn, twL, twN);
  const int lane = threadIdx.x & 31, j = lane & (LN - 1);
  const int lrow = threadIdx.x / LN;                       // row of the block
  float2* buf = rsm + lrow * S::BUF;
  const int groups = nrows / S::RPB;                       // N^2 rows per instance: whole groups
  for (int g = blockIdx.x; g < groups * nbuf; g += gridDim.x) {
    const RowBuf<float> rb = pick(job.b, g % nbuf);
    const RowPlace<L> pl((g / nbuf) * S::RPB + lrow, job.lzb);
    const float2* in = reinterpret_cast<const float2*>(reinterpret_cast<const float*>(rb.real) + pl.inst * rb.real_is +
                                                       pl.rr * N);
    float2* out = rb.spec + pl.main;
    float2 z[P];
#pragma unroll
    for (int r = 0; r < P; ++r) z[r] = in[j + LN * r];
    row_fft<L, -1>(z, buf, j, t);
    // even/odd split of the pairs k, L - k with k < L/2: X[k] = E + W^k O, X[L-k] = conj(E - W^k O),
    // E = (Z[k] + conj Z[L-k]) / 2, O = -i (Z[k] - conj Z[L-k]) / 2; lane 0 has the middle k = L/2
    // (its own partner) besides
#pragma unroll
    for (int r = 0; r <= P / 2; ++r) {
      if (r == P / 2 && j != 0) break;
      const int k = j + LN * r;
      const float2 zk = z[r], zm = r < P / 2 ? row_partner<L>(z, r, j, z[0]) : zk;
      const float2 e = cscale(cadd(zk, cconj(zm)), 0.5f);
      const float2 d = cscale(csub(zk, cconj(zm)), 0.5f);
      const float2 wo = cmul_fwd(wn[k], cmake<float2>(d.y, -d.x));
      float2 x = cadd_rn(e, wo);
      if (r == 0 && j == 0) {
        x = cmake<float2>(zk.x + zk.y, 0.f);
        rb.spec[pl.side] = cmake<float2>(zk.x - zk.y, 0.f);
      } else if (r < P / 2) {
        out[L - k] = cmake<float2>(__fsub_rn(e.x, wo.x), -__fsub_rn(e.y, wo.y));
      }
      out[k] = x;
    }
  }
}

// C2R untangling: Z[k] = E' + i O', E' = X[k] + conj X[L-k], O' = (X[k] - conj X[L-k]) conj(W^k);
// x[r] = X[j + LANES r], xl = X[L] (real parts of X[0] and X[L] only).  With `deriv` the
// spectrum is -i k_x X (0 at kx = L).
template <int L>
__device__ __forceinline__ void row_untangle(float2 (&x)[RowShape<L>::P], float2 xl, int j, bool deriv, const float2* wn) {
  using S = RowShape<L>;
  constexpr int P = S::P, LN = S::LANES;
  if (deriv) {
#pragma unroll
    for (int r = 0; r < P; ++r) {
      const float sk = (float)(j + LN * r);
      x[r] = cmake<float2>(x[r].y * sk, -x[r].x * sk);
    }
    xl = cmake<float2>(xl.y * 0.f, -xl.x * 0.f);
  }
  float2 z[P];
#pragma unroll
  for (int r = 0; r < P; ++r) {
    const int k = j + LN * r;
    const float2 xk = x[r], xm = row_partner<L>(x, r, j, xl);
    const float2 e = cadd(xk, cconj(xm));
    const float2 o = cmul_inv(csub(xk, cconj(xm)), cconj(wn[k]));
    z[r] = cadd_rn(e, cmul_i(o));
    if (r == 0 && j == 0) z[r] = cmake<float2>(xk.x + xm.x, xk.x - xm.x);
  }
#pragma unroll
  for (int r = 0; r < P; ++r) x[r] = z[r];
}

// C2R of one component: L complex (main) + side -> n = 2L reals (unnormalised).  The output
// may alias the input.
template <int L>
__global__ void __launch_bounds__(RowShape<L>::NT)
k_rows_c2r(RowJob<float> job, int nrows, int nbuf, const float2* __restrict__ twL, const float2* __restrict__ twN) {
  using S = RowShape<L>;
  constexpr int N = 2 * L, P = S::P, LN = S::LANES;
  extern __shared__ __align__(16) float2 rsm[];
  float2* t = rsm + S::RPB * S::BUF;
  float2* wn = t + S::TW;
  row_tables<L>(t, wn, twL, twN);
  const int lane = threadIdx.x & 31, j = lane & (LN - 1);
  const int lrow = threadIdx.x / LN;
  float2* buf = rsm + lrow * S::BUF;
  const int groups = nrows / S::RPB;
  for (int g = blockIdx.x; g < groups * nbuf; g += gridDim.x) {
    const RowBuf<float> rb = pick(job.b, g % nbuf);
    const RowPlace<L> pl((g / nbuf) * S::RPB + lrow, job.lzb);
    const float2* in = rb.spec + pl.main;
    float2 z[P];
#pragma unroll
    for (int r = 0; r < P; ++r) z[r] = in[j + LN * r];
    row_untangle<L>(z, rb.spec[pl.side], j, false, wn);
    row_fft<L, +1>(z, buf, j, t);
    float2* out = reinterpret_cast<float2*>(reinterpret_cast<float*>(rb.real) + pl.inst * rb.real_is + pl.rr * N);
#pragma unroll
    for (int r = 0; r < P; ++r) out[j + LN * r] = z[r];
  }
}

// asynchronous copies into shared memory (the calling thread's groups)
__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}
__device__ __forceinline__ void cp_async8(void* dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int K> __device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(K) : "memory"); }

// 32-byte store (both cells of one complex value of the row)
__device__ __forceinline__ void store_cells(V4<float>* p, V4<float> a, V4<float> b) {
  asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "f"(a.x), "f"(a.y), "f"(a.z),
               "f"(a.w), "f"(b.x), "f"(b.y), "f"(b.z), "f"(b.w)
               : "memory");
}

// C2R of Q = 3 or 4 components of a row, written as one V4 per cell ([cell](c0, c1, c2, c3),
// c3 = 0 for Q = 3) straight from the registers that hold them all: component after component
// runs through a buffer of its own, then every lane stores whole 32-byte pairs of cells.
// Component dq (none if dq < 0) is multiplied by -i k_x on the way in.
//
// Q = 4 leaves registers for two blocks of 128 threads per SM, too few warps to hide the loads
// behind the transforms, so its loads are asynchronous copies: once a component's buffer has
// served its exchange, the same component of the warp's next row is copied into it, a whole row
// ahead of its use.  Q = 3 (three blocks) reads plainly, all through one buffer.
// Measured at 512^3, tile form -> this: Q = 3 753 -> 569 us (590 with asynchronous copies), Q = 4
// 829 -> 703 us (851 with plain loads), against 550 and 640 us for their bytes at the copy
// bandwidth.
//
// H: the FP16 force mesh (pm_config.half_force): per cell four halves, each field of a row
// scaled by 2^-e so that the row's largest magnitude lies in [2^14, 2^15), e stored as one int8
// per (row, field) in fexp ([rows][4]).
template <int Q> constexpr int kRows4Bufs = Q == 4 ? Q : 1;   // buffers per row
template <int L, int Q> constexpr int kRows4Smem = (RowShape<L>::RPB * kRows4Bufs<Q> * RowShape<L>::BUF + RowShape<L>::TW + L) *
                                                   (int)sizeof(float2);
template <int L, int Q, bool H>
__global__ void __launch_bounds__(RowShape<L>::NT, Q == 4 ? 2 : 3)
k_rows_c2r4(RowJob<float> job, int nrows, int dq, void* __restrict__ out, signed char* __restrict__ fexp,
            const float2* __restrict__ twL, const float2* __restrict__ twN) {
  using S = RowShape<L>;
  constexpr int N = 2 * L, P = S::P, LN = S::LANES;
  constexpr int NB = kRows4Bufs<Q>;
  constexpr bool ASYNC = NB > 1;
  static_assert(S::BUF > L, "room for the side element");
  extern __shared__ __align__(16) float2 rsm[];
  float2* t = rsm + S::RPB * NB * S::BUF;
  float2* wn = t + S::TW;
  const int lane = threadIdx.x & 31, j = lane & (LN - 1);
  const int lrow = threadIdx.x / LN;
  float2* bufs = rsm + lrow * NB * S::BUF;
  const int groups = nrows / S::RPB;
  // component q of the row whose main and side offsets are given (main < 0: none), as one group
  auto fetch = [&](int q, long long main, long long side) {
    if (main >= 0) {
      float2* b = bufs + q * S::BUF;
      const float2* in = job.b[q].spec + main;
#pragma unroll
      for (int r = 0; r < P / 2; ++r) cp_async16(b + 2 * (j + LN * r), in + 2 * (j + LN * r));
      if (j == 0) cp_async8(b + L, job.b[q].spec + side);
    }
    cp_async_commit();
  };
  auto place = [&](int g, long long& main, long long& side) {
    if (g < groups) {
      const RowPlace<L> pl(g * S::RPB + lrow, job.lzb);
      main = pl.main, side = pl.side;
    } else {
      main = side = -1;
    }
  };
  long long nmain, nside;
  place(blockIdx.x, nmain, nside);
  if constexpr (ASYNC) {
#pragma unroll
    for (int q = 0; q < Q; ++q) fetch(q, nmain, nside);
  }
  row_tables<L>(t, wn, twL, twN);
  for (int g = blockIdx.x; g < groups; g += gridDim.x) {
    const int row = g * S::RPB + lrow;
    const long long main = nmain, side = nside;
    place(g + gridDim.x, nmain, nside);
    float2 f[Q][P];
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      float2* b = bufs + (ASYNC ? q : 0) * S::BUF;
      float2 xl;
      if constexpr (ASYNC) {
        cp_async_wait<Q - 1>();      // this component's copies; the Q - 1 groups behind it may be in flight
        __syncwarp();
#pragma unroll
        for (int r = 0; r < P; ++r) f[q][r] = b[j + LN * r];
        xl = b[L];
        __syncwarp();                // read by every lane before the exchange overwrites it
      } else {
        const float2* in = job.b[q].spec + main;
#pragma unroll
        for (int r = 0; r < P; ++r) f[q][r] = in[j + LN * r];
        xl = job.b[q].spec[side];
      }
      row_untangle<L>(f[q], xl, j, q == dq, wn);
      row_fft<L, +1>(f[q], b, j, t);
      if constexpr (ASYNC) fetch(q, nmain, nside);
    }
    if constexpr (!H) {
      V4<float>* o = reinterpret_cast<V4<float>*>(out) + (long long)row * N;
#pragma unroll
      for (int r = 0; r < P; ++r) {
        const float2 f3 = Q == 4 ? f[Q - 1][r] : cmake<float2>(0, 0);
        store_cells(o + 2 * (j + LN * r), V4<float>{f[0][r].x, f[1][r].x, f[2][r].x, f3.x},
                    V4<float>{f[0][r].y, f[1][r].y, f[2][r].y, f3.y});
      }
    } else {
      float sc[4];
      int ew = 0;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        float m = 0.f;
        if (q < Q) {
#pragma unroll
          for (int r = 0; r < P; ++r) m = fmaxf(m, fmaxf(fabsf(f[q < Q ? q : 0][r].x), fabsf(f[q < Q ? q : 0][r].y)));
#pragma unroll
          for (int d = LN / 2; d > 0; d >>= 1) m = fmaxf(m, __shfl_xor_sync(0xFFFFFFFFu, m, d, LN));
        }
        int e = m > 0.f ? ilogbf(m) - 14 : 0;   // m 2^-e in [2^14, 2^15)
        e = e < -120 ? -120 : (e > 120 ? 120 : e);
        sc[q] = __int_as_float((127 - e) << 23);   // 2^-e
        ew |= (e & 0xFF) << (8 * q);
      }
      if (j == 0) reinterpret_cast<int*>(fexp)[row] = ew;
      uint4* o = reinterpret_cast<uint4*>(out) + (long long)row * L;
#pragma unroll
      for (int r = 0; r < P; ++r) {
        const float2 f3 = Q == 4 ? f[Q - 1][r] : cmake<float2>(0, 0);
        const __half2 a0 = __floats2half2_rn(f[0][r].x * sc[0], f[1][r].x * sc[1]);
        const __half2 a1 = __floats2half2_rn(f[2][r].x * sc[2], f3.x * sc[3]);
        const __half2 b0 = __floats2half2_rn(f[0][r].y * sc[0], f[1][r].y * sc[1]);
        const __half2 b1 = __floats2half2_rn(f[2][r].y * sc[2], f3.y * sc[3]);
        o[j + LN * r] = make_uint4(*reinterpret_cast<const unsigned*>(&a0), *reinterpret_cast<const unsigned*>(&a1),
                                   *reinterpret_cast<const unsigned*>(&b0), *reinterpret_cast<const unsigned*>(&b1));
      }
    }
  }
}

template <class F> inline void row_smem(F fn, int smem) {
  if (smem > 48 * 1024) ensure_smem_attr((const void*)fn, smem);
}
// resident blocks: as many as fit on all SMs (each builds its tables once)
template <class F> inline int row_grid(F fn, int threads, int smem) {
  int occ = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, fn, threads, smem) != cudaSuccess || occ < 1) {
    (void)cudaGetLastError();
    occ = 1;
  }
  return occ * kNumSms;
}

template <int L>
static void launch_rows_r2c(const RowJob<float>& job, int nbuf, int nrows, const float2* tw, cudaStream_t st) {
  using S = RowShape<L>;
  row_smem(k_rows_r2c<L>, S::SMEM);
  static const int grid = row_grid(k_rows_r2c<L>, S::NT, S::SMEM);
  const int groups = nrows / S::RPB * nbuf;
  k_rows_r2c<L><<<groups < grid ? groups : grid, S::NT, S::SMEM, st>>>(job, nrows, nbuf, tw + L, tw + 2 * L);
}
template <int L>
static void launch_rows_c2r(const RowJob<float>& job, int nbuf, int nrows, const float2* tw, cudaStream_t st) {
  using S = RowShape<L>;
  row_smem(k_rows_c2r<L>, S::SMEM);
  static const int grid = row_grid(k_rows_c2r<L>, S::NT, S::SMEM);
  const int groups = nrows / S::RPB * nbuf;
  k_rows_c2r<L><<<groups < grid ? groups : grid, S::NT, S::SMEM, st>>>(job, nrows, nbuf, tw + L, tw + 2 * L);
}
template <int L, int Q, bool H>
static void launch_rows_c2r4_H(const RowJob<float>& job, int nrows, int dq, void* out, signed char* fexp, const float2* tw,
                               cudaStream_t st) {
  using S = RowShape<L>;
  constexpr int smem = kRows4Smem<L, Q>;
  row_smem(k_rows_c2r4<L, Q, H>, smem);
  static const int grid = row_grid(k_rows_c2r4<L, Q, H>, S::NT, smem);
  const int groups = nrows / S::RPB;
  k_rows_c2r4<L, Q, H><<<groups < grid ? groups : grid, S::NT, smem, st>>>(job, nrows, dq, out, fexp, tw + L,
                                                                            tw + 2 * L);
}
template <int L, int Q>
static void launch_rows_c2r4(const RowJob<float>& job, int nrows, int dq, void* out, signed char* fexp, const float2* tw,
                             cudaStream_t st) {
  if (fexp) launch_rows_c2r4_H<L, Q, true>(job, nrows, dq, out, fexp, tw, st);
  else launch_rows_c2r4_H<L, Q, false>(job, nrows, dq, out, fexp, tw, st);
}

}  // namespace pmgb
