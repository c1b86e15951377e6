// Shared-memory transform stages of a register block (padded columns, radix-2^r groups in
// registers): used by the clock passes of hhl_fft.cu and the one-block solves of hhl_batch.cu.
#pragma once

#include <type_traits>

#include "hhl_common.cuh"

namespace hhl {

namespace {

__device__ __forceinline__ int pad16(int p) { return p + (p >> 4); }
__device__ __forceinline__ int bitrev_m(int x, int m) { return (int)(__brev((unsigned)x) >> (32 - m)); }

template <class T>
struct Twiddle {
  const T* t0;  // exp(-2 pi i j / L), j < 64
  const T* t1;  // exp(-2 pi i 64 j / L)
  __device__ __forceinline__ T operator()(int q, bool conj) const {
    T f = cmul(t1[q >> 6], t0[q & 63]);
    if (conj) f.y = -f.y;
    return f;
  }
};

__host__ __device__ constexpr int twiddle_entries(int m) { return 64 + ((1 << m) / 64 > 1 ? (1 << m) / 64 : 1); }

template <class R>
__device__ void fill_twiddles(typename Cx<R>::T* t0, typename Cx<R>::T* t1, int m) {
  const int L = 1 << m;
  const int n1 = twiddle_entries(m) - 64;
  for (int j = threadIdx.x; j < 64 + n1; j += blockDim.x) {
    const int e = j < 64 ? j : 64 * (j - 64);
    if constexpr (std::is_same<R, df>::value) {  // double-float from the FP64 values
      double s, c;
      sincospi(-2.0 * (double)(e & (L - 1)) / (double)L, &s, &c);
      if (j < 64) t0[j] = mk<df>(df_of(c), df_of(s));
      else t1[j - 64] = mk<df>(df_of(c), df_of(s));
    } else {
      R s, c;
      if constexpr (sizeof(R) == 4) {
        sincospif(-2.0f * (float)(e & (L - 1)) / (float)L, &s, &c);
      } else {
        sincospi(-2.0 * (double)(e & (L - 1)) / (double)L, &s, &c);
      }
      if (j < 64) t0[j] = mk<R>(c, s);
      else t1[j - 64] = mk<R>(c, s);
    }
  }
}

// e^{-2 pi i k / 16}, k < 16 (the in-group factors of the twiddles, see butterflies()).
__constant__ double kRoot16[16][2] = {
    {1.0, 0.0}, {0.92387953251128674, -0.38268343236508978}, {0.70710678118654752, -0.70710678118654752},
    {0.38268343236508978, -0.92387953251128674}, {0.0, -1.0}, {-0.38268343236508978, -0.92387953251128674},
    {-0.70710678118654752, -0.70710678118654752}, {-0.92387953251128674, -0.38268343236508978}, {-1.0, 0.0},
    {-0.92387953251128674, 0.38268343236508978}, {-0.70710678118654752, 0.70710678118654752},
    {-0.38268343236508978, 0.92387953251128674}, {0.0, 1.0}, {0.38268343236508978, 0.92387953251128674},
    {0.70710678118654752, 0.70710678118654752}, {0.92387953251128674, 0.38268343236508978}};
__constant__ float kRoot16f[16][2] = {
    {1.0f, 0.0f}, {0.92387953251128674f, -0.38268343236508978f}, {0.70710678118654752f, -0.70710678118654752f},
    {0.38268343236508978f, -0.92387953251128674f}, {0.0f, -1.0f}, {-0.38268343236508978f, -0.92387953251128674f},
    {-0.70710678118654752f, -0.70710678118654752f}, {-0.92387953251128674f, -0.38268343236508978f}, {-1.0f, 0.0f},
    {-0.92387953251128674f, 0.38268343236508978f}, {-0.70710678118654752f, 0.70710678118654752f},
    {-0.38268343236508978f, 0.92387953251128674f}, {0.0f, 1.0f}, {0.38268343236508978f, 0.92387953251128674f},
    {0.70710678118654752f, 0.70710678118654752f}, {0.92387953251128674f, 0.38268343236508978f}};

// The root for the amplitude precision (FP32 kernels read FP32 constants: converting an FP64
// constant costs a pass through GB300's narrow FP64 pipe).
// Double-float remainders of those roots (kRoot16 - kRoot16f, evaluated in FP64 at compile time).
#define HHL_DFL(v) ((float)((v) - (double)(float)(v)))
#define HHL_R16(c, s) {HHL_DFL(c), HHL_DFL(s)}
__constant__ float kRoot16l[16][2] = {
    HHL_R16(1.0, 0.0), HHL_R16(0.92387953251128674, -0.38268343236508978),
    HHL_R16(0.70710678118654752, -0.70710678118654752), HHL_R16(0.38268343236508978, -0.92387953251128674),
    HHL_R16(0.0, -1.0), HHL_R16(-0.38268343236508978, -0.92387953251128674),
    HHL_R16(-0.70710678118654752, -0.70710678118654752), HHL_R16(-0.92387953251128674, -0.38268343236508978),
    HHL_R16(-1.0, 0.0), HHL_R16(-0.92387953251128674, 0.38268343236508978),
    HHL_R16(-0.70710678118654752, 0.70710678118654752), HHL_R16(-0.38268343236508978, 0.92387953251128674),
    HHL_R16(0.0, 1.0), HHL_R16(0.38268343236508978, 0.92387953251128674),
    HHL_R16(0.70710678118654752, 0.70710678118654752), HHL_R16(0.92387953251128674, 0.38268343236508978)};
#undef HHL_R16
#undef HHL_DFL

template <class R>
__device__ __forceinline__ R root16(int k, int part) {
  if constexpr (std::is_same<R, df>::value) return df{kRoot16f[k][part], kRoot16l[k][part]};
  else if constexpr (sizeof(R) == 4) return kRoot16f[k][part];
  else return (R)kRoot16[k][part];
}

// The RB radix-2 stages of one group: v[x] = element lo + x * 2^lo_bits (+ a multiple of
// 2^(lo_bits + RB)); local bit t is global stage s = t + 1 + lo_bits of an m-stage transform.
// MODE 0: DFT butterflies, MODE 1: Hadamard butterflies. DIF runs t from high to low.
// The twiddle of butterfly x at bit t, exp(-2 pi i ((x mod 2^t) 2^lo_bits + lo) 2^(m-s) / L),
// factors into exp(-2 pi i lo 2^(m-s) / L) (one table lookup per stage) times
// exp(-2 pi i (x mod 2^t) / 2^(t+1)) (a sixteenth root of unity, from constant memory).
// PIN (complex64): the products' roundings spelled out. The compiler fuses one of a complex product's
// two multiplications into the addition and picks which by context, so the same source gives other
// last bits in another kernel; a pinned kernel gives those that k_clock_block, which is not pinned, has
// from the CUDA 13.0 compiler (the tests compare the two).
template <bool PIN, bool SECOND, class T>
__device__ __forceinline__ T cmul_as(T a, T b) {  // SECOND: the imaginary part rounds a.x b.y first
  if constexpr (PIN && sizeof(T) == 8) {
    T z;
    z.x = __fmaf_rn(a.x, b.x, -__fmul_rn(a.y, b.y));
    z.y = SECOND ? __fmaf_rn(a.y, b.x, __fmul_rn(a.x, b.y)) : __fmaf_rn(a.x, b.y, __fmul_rn(a.y, b.x));
    return z;
  } else {
    return cmul(a, b);
  }
}

template <class T, int RB, bool DIT, int MODE, bool PIN = false>
__device__ __forceinline__ void butterflies(T (&v)[1 << RB], int lo, int lo_bits, int m, const Twiddle<T>& tw,
                                            bool conj) {
  constexpr int G = 1 << RB;
  using R = decltype(T().x);
#pragma unroll
  for (int tt = 0; tt < RB; ++tt) {
    const int t = DIT ? tt : (RB - 1 - tt);
    const int s = t + 1 + lo_bits;
    T base;
    if (MODE == 0) base = tw(lo << (m - s), conj);
#pragma unroll
    for (int x = 0; x < G; ++x) {
      if (x & (1 << t)) continue;
      const int x1 = x | (1 << t);
      T a = v[x], b = v[x1];
      if (MODE == 0) {
        const int xr = x & ((1 << t) - 1);
        T f = base;
        if (xr != 0) {
          const int k16 = xr << (3 - t);
          T w;
          w.x = root16<R>(k16, 0);
          w.y = conj ? -root16<R>(k16, 1) : root16<R>(k16, 1);
          f = cmul_as<PIN, true>(base, w);
        }
        if (DIT) {
          b = cmul_as<PIN, true>(b, f);
          v[x] = cadd(a, b);
          v[x1] = csub(a, b);
        } else {
          v[x] = cadd(a, b);
          v[x1] = cmul_as<PIN, RB != 4>(csub(a, b), f);
        }
      } else {
        v[x] = cadd(a, b);
        v[x1] = csub(a, b);
      }
    }
  }
}

// One local pass of RB stages (global stages s0-RB+1 .. s0 <= m_loc) on every group of the
// W local columns of 2^m_loc rows.
template <class T, int RB, bool DIT, int MODE, bool PIN = false>
__device__ void radix_pass(T* X, int Lp, int W, const Twiddle<T>& tw, int m, int m_loc, int s0, bool conj) {
  constexpr int G = 1 << RB;
  const int lo_bits = s0 - RB;
  const int gpc_bits = m_loc - RB;
  const int total = W << gpc_bits;
  for (int g = threadIdx.x; g < total; g += blockDim.x) {
    const int w = g >> gpc_bits;
    const int gg = g & ((1 << gpc_bits) - 1);
    const int lo = gg & ((1 << lo_bits) - 1);
    const int hi = gg >> lo_bits;
    const int base = (hi << s0) + lo;
    T* col = X + w * Lp;
    T v[G];
#pragma unroll
    for (int x = 0; x < G; ++x) v[x] = col[pad16(base + (x << lo_bits))];
    butterflies<T, RB, DIT, MODE, PIN>(v, lo, lo_bits, m, tw, conj);
#pragma unroll
    for (int x = 0; x < G; ++x) col[pad16(base + (x << lo_bits))] = v[x];
  }
}

template <class T, bool DIT, int MODE, bool PIN = false>
__device__ void local_stages(T* X, int Lp, int W, const Twiddle<T>& tw, int m, int m_loc, bool conj) {
  const int npass = (m_loc + 3) / 4;
  int done = 0;
  for (int p = 0; p < npass; ++p) {
    const int r = (m_loc - done) / (npass - p);  // balanced pass sizes, each <= 4
    const int s0 = DIT ? done + r : m_loc - done;
    switch (r) {
      case 4: radix_pass<T, 4, DIT, MODE, PIN>(X, Lp, W, tw, m, m_loc, s0, conj); break;
      case 3: radix_pass<T, 3, DIT, MODE, PIN>(X, Lp, W, tw, m, m_loc, s0, conj); break;
      case 2: radix_pass<T, 2, DIT, MODE, PIN>(X, Lp, W, tw, m, m_loc, s0, conj); break;
      default: radix_pass<T, 1, DIT, MODE, PIN>(X, Lp, W, tw, m, m_loc, s0, conj); break;
    }
    done += r;
    __syncthreads();
  }
}

}  // namespace
}  // namespace hhl
