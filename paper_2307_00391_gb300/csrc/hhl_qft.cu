// Whole-register QFT / inverse QFT of complex64 states (hhl_qft_whole; App. B, the circuit of the
// Fig. 1c experiment) as few passes over HBM as the shared memory allows: the low 12 bits in one
// pass over contiguous 32 KiB chunks, the bits above in passes of up to 9 bits, so a 30-qubit
// transform moves its state three times and a 20-qubit one twice.
//
// A pass of NB bits at bit position b transforms tiles of 2^NB rows (stride 2^b) by 2^(13 - NB)
// consecutive columns, 64 KiB a block (half that at NB = 4), as two register transforms of 2^A and 2^B points, A + B =
// NB: the first takes its points from HBM straight into registers, the second writes its own
// straight back, and the tile crosses shared memory once in between. Radix-2 circuits of the
// QFT's Hadamard and phase layers factor this way exactly: a 2^A-point transform on the upper A
// bits (constant roots), then the phase e^{2 pi i k r / 2^(b + NB)} on output k with r the index
// below those bits, then the same on the lower B bits. The phases come from the exact fraction
// k r 2^-(b + NB) of a turn: one sine / cosine pair for each power-of-two k, the others as
// products of at most five of them.
//
// Bound: HBM latency in the passes (2^NB rows of 128 bytes at NB = 9; 16 warps an SM, issue slots half
// full) and the shared-memory data path in the low bits (72% of its wavefronts). Measured on 2^30 amplitudes: 3.0 ms for the low bits, 3.2 ms a 9-bit pass, three passes a transform (the
// previous form: 4.75 ms for the low bits, 3 x 3.4 ms for passes of 6 bits).
#include <math.h>
#include <stdlib.h>

#include "hhl_common.cuh"

namespace hhl {

namespace {

constexpr int kQftThreads = 256;
// log2 of the amplitudes of a tile: 32 a thread, 16 where a tile of 4 bits would be wider than the block
constexpr int tile_bits(int nb) { return nb < 5 ? 12 : 13; }
constexpr int kLowBits = 12;   // bits of the chunk pass: 16 amplitudes a thread

// e^{2 pi i u / 2^32}: reduced to an eighth of a turn around a quarter, Taylor polynomials of sine and
// cosine on |x| <= pi / 4 (truncation below 4e-9), exact octant arithmetic on the integer.
__device__ __forceinline__ float2 turn_cis(unsigned u) {
  const unsigned q = (u + 0x20000000u) >> 30;
  const float x = (float)(int)(u - (q << 30)) * 1.4629180792671596e-9f;  // 2 pi 2^-32
  const float x2 = x * x;
  float s = fmaf(x2, 2.7557319e-6f, -1.9841270e-4f);
  s = fmaf(x2, s, 8.3333333e-3f);
  s = fmaf(x2, s, -0.16666667f);
  s = fmaf(x * x2, s, x);
  float c = fmaf(x2, -2.7557319e-7f, 2.4801587e-5f);
  c = fmaf(x2, c, -1.3888889e-3f);
  c = fmaf(x2, c, 4.1666667e-2f);
  c = fmaf(x2, c, -0.5f);
  c = fmaf(x2, c, 1.0f);
  const float2 r = (q & 1u) ? make_float2(-s, c) : make_float2(c, s);  // a quarter turn
  return (q & 2u) ? make_float2(-r.x, -r.y) : r;
}

// cos, sin of 2 pi e / 32
__device__ __forceinline__ constexpr float c32(int e) {
  constexpr float t[16] = {1.0f, 0.98078528f, 0.92387953f, 0.83146961f, 0.70710678f, 0.55557023f, 0.38268343f, 0.19509032f,
                           0.0f, -0.19509032f, -0.38268343f, -0.55557023f, -0.70710678f, -0.83146961f, -0.92387953f,
                           -0.98078528f};
  return t[e];
}
__device__ __forceinline__ constexpr float s32(int e) { return e <= 8 ? c32(8 - e) : c32(e - 8); }

// v e^{(+-) 2 pi i e / 32}, e a compile-time value in [0, 16)
template <bool NEG>
__device__ __forceinline__ float2 mul_root(float2 v, int e) {
  if (e == 0) return v;
  if (e == 8) return NEG ? make_float2(v.y, -v.x) : make_float2(-v.y, v.x);
  const float c = c32(e), s = NEG ? -s32(e) : s32(e);
  return make_float2(fmaf(c, v.x, -(s * v.y)), fmaf(c, v.y, s * v.x));
}

// 2^A-point transforms in registers: DIF with e^{+2 pi i x k}, natural order in, bit-reversed out
// (the QFT), and DIT with e^{-2 pi i x k}, bit-reversed in, natural out (its inverse).
template <int A, bool DIT>
__device__ __forceinline__ void point_transform(float2 (&v)[1 << A]) {
#pragma unroll
  for (int q = 0; q < A; ++q) {
    const int t = DIT ? q : A - 1 - q, half = 1 << t;
#pragma unroll
    for (int x = 0; x < (1 << A); ++x) {
      if (x & half) continue;
      const int e = (x & (half - 1)) << (4 - t);  // of 32: (x mod 2^t) / 2^(t + 1)
      const float2 a = v[x];
      if (DIT) {
        const float2 b = mul_root<true>(v[x + half], e);
        v[x] = make_float2(a.x + b.x, a.y + b.y);
        v[x + half] = make_float2(a.x - b.x, a.y - b.y);
      } else {
        const float2 b = v[x + half];
        v[x] = make_float2(a.x + b.x, a.y + b.y);
        v[x + half] = mul_root<false>(make_float2(a.x - b.x, a.y - b.y), e);
      }
    }
  }
}

template <int A>
__device__ __forceinline__ constexpr int rev_bits(int p) {
  int r = 0;
  for (int i = 0; i < A; ++i) r |= ((p >> i) & 1) << (A - 1 - i);
  return r;
}

// w[k] = e^{2 pi i k u / 2^32}, k < 2^A
template <int A>
__device__ __forceinline__ void phase_powers(unsigned u, float2 (&w)[1 << A]) {
  w[0] = make_float2(1.f, 0.f);
#pragma unroll
  for (int q = 0; q < A; ++q) {
    const float2 f = turn_cis(u << q);
    w[1 << q] = f;
#pragma unroll
    for (int k = 1; k < (1 << q); ++k) w[(1 << q) + k] = cmul(w[k], f);
  }
}

template <int A, bool CONJ>
__device__ __forceinline__ void apply_phases(float2 (&v)[1 << A], const float2 (&w)[1 << A]) {
#pragma unroll
  for (int p = 1; p < (1 << A); ++p) {  // position p holds frequency rev(p)
    const float2 f = w[rev_bits<A>(p)];
    v[p] = CONJ ? cconjmul(v[p], f) : cmul(v[p], f);
  }
}

// Bits [b, b + A + B) of every 2^n-amplitude state. Block t: column block t mod 2^(b - WB), then the
// index above the pass's bits.
template <int A, int B, bool DIT>
__global__ void __launch_bounds__(kQftThreads, 2) k_qft_pass(float2* __restrict__ S, int b) {
  constexpr int NB = A + B, TB = tile_bits(NB), WB = TB - NB, W = 1 << WB;
  constexpr int RA = 1 << A, RB = 1 << B;
  constexpr int PT = (1 << TB) / kQftThreads, GA = PT / RA, GB = PT / RB;  // transforms of each kind a thread does
  extern __shared__ __align__(16) float2 qft_tile[];
  const unsigned cb = blockIdx.x & ((1u << (b - WB)) - 1u);
  const size_t hi = (size_t)(blockIdx.x >> (b - WB));
  float2* base = S + (hi << (b + NB)) + ((size_t)cb << WB);
  const int w = threadIdx.x & (W - 1), g0 = threadIdx.x >> WB;  // column; first group
  constexpr int GS = kQftThreads >> WB;                         // groups of one round of the block
  const unsigned inner = (cb << WB) + (unsigned)w;              // index below the pass's bits
  if (!DIT) {
#pragma unroll
    for (int q = 0; q < GA; ++q) {
      const int jl = g0 + q * GS;  // lower B row bits
      float2 v[RA], f[RA];
#pragma unroll
      for (int x = 0; x < RA; ++x) v[x] = base[((size_t)((x << B) + jl) << b) + w];
      phase_powers<A>((inner + ((unsigned)jl << b)) << (32 - b - NB), f);
      point_transform<A, false>(v);
      apply_phases<A, false>(v, f);
#pragma unroll
      for (int x = 0; x < RA; ++x) qft_tile[(((x << B) + jl) << WB) + w] = v[x];
    }
    float2 f[RB];
    phase_powers<B>(inner << (32 - b - B), f);
    __syncthreads();
#pragma unroll
    for (int q = 0; q < GB; ++q) {
      const int row = (g0 + q * GS) << B;
      float2 v[RB];
#pragma unroll
      for (int x = 0; x < RB; ++x) v[x] = qft_tile[((row + x) << WB) + w];
      point_transform<B, false>(v);
      apply_phases<B, false>(v, f);
#pragma unroll
      for (int x = 0; x < RB; ++x) base[((size_t)(row + x) << b) + w] = v[x];
    }
  } else {
    float2 f[RB];
    phase_powers<B>(inner << (32 - b - B), f);
#pragma unroll
    for (int q = 0; q < GB; ++q) {
      const int row = (g0 + q * GS) << B;
      float2 v[RB];
#pragma unroll
      for (int x = 0; x < RB; ++x) v[x] = base[((size_t)(row + x) << b) + w];
      apply_phases<B, true>(v, f);
      point_transform<B, true>(v);
#pragma unroll
      for (int x = 0; x < RB; ++x) qft_tile[((row + x) << WB) + w] = v[x];
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < GA; ++q) {
      const int jl = g0 + q * GS;
      float2 v[RA], p[RA];
      phase_powers<A>((inner + ((unsigned)jl << b)) << (32 - b - NB), p);
#pragma unroll
      for (int x = 0; x < RA; ++x) v[x] = qft_tile[(((x << B) + jl) << WB) + w];
      apply_phases<A, true>(v, p);
      point_transform<A, true>(v);
#pragma unroll
      for (int x = 0; x < RA; ++x) base[((size_t)((x << B) + jl) << b) + w] = v[x];
    }
  }
}

// The low 12 bits of contiguous 2^12-amplitude chunks, scaled: three 16-point transforms a thread.
// The end of the chunk that HBM sees in 16-byte units a lane goes through shared memory, the
// other (amplitudes 256 apart a thread) straight between registers and HBM.
__device__ __forceinline__ int low_pad(int i) { return i + (i >> 4); }

template <bool DIT>
__global__ void __launch_bounds__(kQftThreads, 3) k_qft_low(float2* __restrict__ S, float scale) {
  __shared__ float2 X[(1 << kLowBits) + (1 << (kLowBits - 4))];
  __shared__ float2 roots[256];  // e^{2 pi i q / 256}
  const int t = threadIdx.x;
  float2* base = S + ((size_t)blockIdx.x << kLowBits);
  float4* base4 = reinterpret_cast<float4*>(base);
  float2 v[16], w[16];
  const int row = (t >> 4) * 256, l = t & 15;  // the middle transform's points: row + 16 x + l
  if (!DIT) {
#pragma unroll
    for (int x = 0; x < 16; ++x) v[x] = base[x * 256 + t];
    roots[t] = turn_cis((unsigned)t << 24);
    phase_powers<4>((unsigned)t << 20, w);
    point_transform<4, false>(v);
    apply_phases<4, false>(v, w);
#pragma unroll
    for (int x = 0; x < 16; ++x) X[low_pad(x * 256 + t)] = v[x];
    __syncthreads();
#pragma unroll
    for (int x = 0; x < 16; ++x) v[x] = X[low_pad(row + 16 * x + l)];
    point_transform<4, false>(v);
#pragma unroll
    for (int p = 0; p < 16; ++p) X[low_pad(row + 16 * p + l)] = cmul(v[p], roots[rev_bits<4>(p) * l]);
    __syncthreads();
#pragma unroll
    for (int x = 0; x < 16; ++x) v[x] = X[low_pad(16 * t + x)];
    point_transform<4, false>(v);
#pragma unroll
    for (int x = 0; x < 16; ++x) X[low_pad(16 * t + x)] = v[x];
    __syncthreads();
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int i = 2 * (q * kQftThreads + t);
      const float2 a = X[low_pad(i)], c = X[low_pad(i + 1)];
      base4[q * kQftThreads + t] = make_float4(a.x * scale, a.y * scale, c.x * scale, c.y * scale);
    }
  } else {
    roots[t] = turn_cis((unsigned)t << 24);
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int i = 2 * (q * kQftThreads + t);
      const float4 z = base4[q * kQftThreads + t];
      X[low_pad(i)] = make_float2(z.x, z.y);
      X[low_pad(i + 1)] = make_float2(z.z, z.w);
    }
    __syncthreads();
#pragma unroll
    for (int x = 0; x < 16; ++x) v[x] = X[low_pad(16 * t + x)];
    point_transform<4, true>(v);
#pragma unroll
    for (int x = 0; x < 16; ++x) X[low_pad(16 * t + x)] = v[x];
    __syncthreads();
#pragma unroll
    for (int p = 0; p < 16; ++p) v[p] = cconjmul(X[low_pad(row + 16 * p + l)], roots[rev_bits<4>(p) * l]);
    point_transform<4, true>(v);
#pragma unroll
    for (int x = 0; x < 16; ++x) X[low_pad(row + 16 * x + l)] = v[x];
    phase_powers<4>((unsigned)t << 20, w);
    __syncthreads();
#pragma unroll
    for (int x = 0; x < 16; ++x) v[x] = X[low_pad(x * 256 + t)];
    apply_phases<4, true>(v, w);
    point_transform<4, true>(v);
#pragma unroll
    for (int x = 0; x < 16; ++x) base[x * 256 + t] = make_float2(v[x].x * scale, v[x].y * scale);
  }
}

template <int A, int B, bool DIT>
hhl_status pass_launch(float2* S, int n, int log_states, int b, cudaStream_t st) {
  constexpr int TB = tile_bits(A + B);
  constexpr size_t smem = sizeof(float2) << TB;
  auto kern = k_qft_pass<A, B, DIT>;
  HHL_CUDA_TRY(raise_dyn_smem((const void*)kern, smem));
  HHL_PROF_BEGIN(st);
  kern<<<1u << (n + log_states - TB), kQftThreads, smem, st>>>(S, b);
  HHL_LAUNCH_CHECK("k_qft_pass");
  return HHL_OK;
}

template <bool DIT>
hhl_status pass_bits(float2* S, int n, int log_states, int b, int nb, cudaStream_t st) {
  switch (nb) {
    case 4: return pass_launch<2, 2, DIT>(S, n, log_states, b, st);
    case 5: return pass_launch<3, 2, DIT>(S, n, log_states, b, st);
    case 6: return pass_launch<3, 3, DIT>(S, n, log_states, b, st);
    case 7: return pass_launch<4, 3, DIT>(S, n, log_states, b, st);
    case 8: return pass_launch<4, 4, DIT>(S, n, log_states, b, st);
    default: return pass_launch<5, 4, DIT>(S, n, log_states, b, st);
  }
}

hhl_status low_launch(float2* S, int n, int log_states, float scale, bool dit, cudaStream_t st) {
  const unsigned grid = 1u << (n + log_states - kLowBits);
  HHL_PROF_BEGIN(st);
  if (dit) k_qft_low<true><<<grid, kQftThreads, 0, st>>>(S, scale);
  else k_qft_low<false><<<grid, kQftThreads, 0, st>>>(S, scale);
  HHL_LAUNCH_CHECK("k_qft_low");
  return HHL_OK;
}

}  // namespace

// From 2^20 amplitudes in all (and 16 bits, the low chunk and four more): below that a tile of 2^13
// leaves most SMs without one, and the passes of hhl_fft.cu (2^9 to 2^12 amplitudes a tile) are as fast.
bool qft_whole_tiles(int n, int log_states) {
  return n >= kLowBits + 4 && n + log_states >= 20 && getenv("HHL_LOWBITS_PLAIN") == nullptr;
}

hhl_status launch_qft_whole_tiles(void* state, int n, int log_states, int direction, cudaStream_t st) {
  float2* S = (float2*)state;
  const float scale = (float)(1.0 / sqrt(ldexp(1.0, n)));
  const int high = n - kLowBits, passes = (high + 8) / 9;
  int first[4], bits[4];  // low to high, balanced
  for (int q = 0, done = 0; q < passes; ++q) {
    first[q] = kLowBits + done;
    bits[q] = (high - done) / (passes - q);
    done += bits[q];
  }
  hhl_status s = HHL_OK;
  if (direction == 0) {
    for (int q = passes - 1; q >= 0 && s == HHL_OK; --q) s = pass_bits<false>(S, n, log_states, first[q], bits[q], st);
    return s == HHL_OK ? low_launch(S, n, log_states, scale, false, st) : s;
  }
  s = low_launch(S, n, log_states, scale, true, st);
  for (int q = 0; q < passes && s == HHL_OK; ++q) s = pass_bits<true>(S, n, log_states, first[q], bits[q], st);
  return s;
}

}  // namespace hhl
