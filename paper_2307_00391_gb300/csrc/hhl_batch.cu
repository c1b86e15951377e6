// Batched HHL: many instances of uneven size (system register n_s, clock n_c, right-hand
// side, T0), complex64 amplitudes, run as one CUDA graph.
//
// Each instance runs the postselected solve of the single-plan path (hhl_solve_postselected:
// QPE by doubling from the prepared clock = 0 row, the clock block with the anc = 0 weights
// summed, the uncompute and final Hadamards folded by halving into one row). What changes is
// how the controlled products get their operands: a batch of a few hundred instances cannot
// hold every U_k (at N = 4096 the split-FP16 operands of one instance alone are ~6.4 GB), so
// every U_k comes from the eigen-decomposition of the Toeplitz tridiagonal A. With
// v_j(i) = sqrt(2/(N+1)) sin(i j pi/(N+1)), the product formula
// sin a sin b = (cos(a-b) - cos(a+b))/2 turns U_k = V diag(e^{i lambdahat_j t_k}) V^T into
//     U_k[n][m] = g_k(|n - m|) - g_k(n + m)   (1-based n, m),
//     g_k(d) = 1/(N+1) sum_{j=1..N} cos(d j pi/(N+1)) e^{i lambdahat_j t_k}.
// The g_k of every instance (2N+2 values per k, O(N^2) FP64 work each, kept as double-float
// pairs: n_c (2N+2) x 16 bytes per instance) depend on A, T0 and k only, so one FP64 kernel
// computes them when the batch is created, as a plan computes its U_k. The tree steps on
// fewer than 128 rows generate U_k on the fly from g_k (k_toeplitz_rows); the larger ones get
// their GEMM operand (the split-FP16 real embedding for the tensor-core GEMM, or the complex64
// matrix for the CUDA-core GEMM) from one expansion kernel into a per-stream workspace right
// before it is used.
//
// Instances are spread over worker streams by decreasing GEMM work (longest processing
// time first); every stream owns a workspace sized for its largest instance. The whole
// batch (every instance's solve, from the preparation of its right-hand side to its
// dissipation) is captured once into a graph, forked over the worker streams, and replayed
// with one launch per run. The GEMM implementation of each instance (CUDA cores, or tcgen05
// with 128- or 256-column tiles) is given by the caller (an autotuned table) or by a size rule.
#include <math.h>
#include <string.h>

#include <algorithm>
#include <numeric>
#include <vector>

#include <cooperative_groups.h>
#include <cuda_fp16.h>

#include "hhl_fft_core.cuh"

namespace cg = cooperative_groups;

namespace hhl {
namespace {

constexpr double kPiB = 3.14159265358979323846;

// g_k(d) for d in [0, 2N+2) and every k: block (x = d chunk, y = k, z = instance).
struct GenInst {
  int N, n_c;
  const double2* ph;      // n_c x N
  const double* cos_tab;  // 2N+2
  float4* g;              // n_c x (2N+2)
};
__global__ void __launch_bounds__(256) k_ugen_g(const GenInst* __restrict__ inst) {
  extern __shared__ double2 sh_ph[];
  const GenInst in = inst[blockIdx.z];
  const int N = in.N, k = blockIdx.y;
  if (k >= in.n_c) return;  // block-uniform
  const double* __restrict__ cos_tab = in.cos_tab;
  const int M = 2 * N + 2;
  for (int j = threadIdx.x; j < N; j += blockDim.x) sh_ph[j] = in.ph[(size_t)k * N + j];
  __syncthreads();
  const double inv = 1.0 / (double)(N + 1);
  for (int d = blockIdx.x * blockDim.x + threadIdx.x; d < M; d += gridDim.x * blockDim.x) {
    double re = 0.0, im = 0.0;
    int q = 0;  // (d * j) mod M, j = 1..N
    for (int j = 1; j <= N; ++j) {
      q += d;
      if (q >= M) q -= M;
      const double c = cos_tab[q];
      const double2 p = sh_ph[j - 1];
      re = fma(c, p.x, re);
      im = fma(c, p.y, im);
    }
    // double-float (hi + lo) in FP32, so that the expansion below runs in FP32 arithmetic
    const double gr = re * inv, gi = im * inv;
    const float rh = (float)gr, ih = (float)gi;
    in.g[(size_t)k * M + d] = make_float4(rh, (float)(gr - (double)rh), ih, (float)(gi - (double)ih));
  }
}

// v (scaled by 2^15) -> FP16 hi = nearest(v), lo = nearest(v - hi), as the tcgen05 GEMM expects.
__device__ __forceinline__ void f16_split(float v, __half& hi, __half& lo) {
  hi = __float2half_rn(v);
  lo = __float2half_rn(v - __half2float(hi));
}

__device__ __forceinline__ uint32_t pack_h2(__half a, __half b) {
  return (uint32_t)__half_as_ushort(a) | ((uint32_t)__half_as_ushort(b) << 16);
}

__device__ __forceinline__ float2 u_elem(const float4* __restrict__ g, int n, int m) { return toeplitz_u(g, n, m); }

// Split-FP16 real embedding of U_k (adjoint: U_k^dagger = conj(U_k), A real symmetric),
// scaled by 2^15: hi / lo (2N x 2N), rows = output real column, columns = input real index.
// One thread per (n, m) writes the 2 x 2 block [[Re, -Im], [Im, Re]] at rows 2n, 2n+1 and
// columns 2m, 2m+1.
__global__ void k_ugen_embed_tc(int n_s, const float4* __restrict__ g, int adjoint, __half* __restrict__ hi,
                                __half* __restrict__ lo) {
  const int N = 1 << n_s;
  const int64_t N2 = 2LL * N;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < (int64_t)N * N;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int n = (int)(e >> n_s), m = (int)(e & (N - 1));
    float2 u = u_elem(g, n, m);
    if (adjoint) u.y = -u.y;
    __half hr, hi_, lr, li;
    f16_split(u.x * 32768.0f, hr, lr);
    f16_split(u.y * 32768.0f, hi_, li);
    const __half nhi = __hneg(hi_), nli = __hneg(li);
    const int64_t r0 = (2LL * n) * N2 + 2LL * m, r1 = r0 + N2;
    *reinterpret_cast<uint32_t*>(hi + r0) = pack_h2(hr, nhi);
    *reinterpret_cast<uint32_t*>(hi + r1) = pack_h2(hi_, hr);
    *reinterpret_cast<uint32_t*>(lo + r0) = pack_h2(lr, nli);
    *reinterpret_cast<uint32_t*>(lo + r1) = pack_h2(li, lr);
  }
}

// Complex64 operand of the CUDA-core GEMM: B[m][n] = U_k[n][m] (= U_k[m][n]) or conj.
__global__ void k_ugen_embed_simt(int n_s, const float4* __restrict__ g, int adjoint, float2* __restrict__ B) {
  const int N = 1 << n_s;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < (int64_t)N * N;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int m = (int)(e >> n_s), n = (int)(e & (N - 1));
    float2 u = u_elem(g, n, m);
    if (adjoint) u.y = -u.y;
    B[e] = u;
  }
}

// ------------------------------------------------------------------ one-block solves
// Instances whose clock and system registers fit one block's shared memory (n_c <= 7, N <= 128): the
// whole postselected solve in one launch for all of them, a block each, instead of about 17
// launches per instance (384 instances of 2^3..2^6 points: 6,900 launches of 0.6 us each on 8
// streams, 3.95 ms; one launch takes 85 us). Bound by issue within an SM and the latency of the 2 n_c
// dependent products: a block takes 21 us at 4 + 4 qubits and 360 us at 7 + 7, where the launches on eight
// streams took 79 us for one instance, 109 for 8 and 192 for 16. So while there are few, a
// cluster of up to 8 blocks shares an instance: 7 + 7 qubits 89 us for up to 8 instances, 120 for
// 16 and 32, 190 for 64 (the streams 360 and 697); 6 + 6 qubits 45 us up to 32 (84 by one block, the
// streams 72 to 297). In a batch with larger instances these launches are a branch of its graph (8 of
// 8 + 8 qubits with 16 of 7 + 7: 344 us; after the graph, a block each, 766). The
// arithmetic is that of the launches it replaces, operation for operation: U_k from its g table,
// every output of a product as 32 partial sums over m (mod 32) added in the order of
// k_toeplitz_rows' shuffles and warps, the transform stages of k_clock_block, the squares of
// k_measure_sums.
struct SmallInst {
  int n_s, n_c;
  long long b_off, out_off;  // doubles into the packed arrays
  const float4* g;           // n_c x (2N + 2)
  const float2* rot;         // R: (cos, sin)(theta_y / 2)
  double inv_c_lam, wall_lo, wall_hi, nu_over_h;
  int index, pad;            // position of the dissipation rate
};

constexpr int kSmallBits = 7;       // n_s and n_c at most
constexpr int kSmallThreads = 256;
constexpr int kSmallColumns = 16;   // system columns of a block at least, where a cluster shares an instance
constexpr int kSmallCluster = 8;    // blocks of a cluster at most

__host__ __device__ constexpr int small_column(int n_c) { return (1 << n_c) + (1 << n_c) / 16 + 1; }
size_t small_smem(int n_s, int n_c) {
  return ((size_t)twiddle_entries(n_c) + ((size_t)small_column(n_c) << n_s)) * sizeof(float2) +
         2 * (2 * ((size_t)1 << n_s) + 2) * sizeof(float4) + 16;
}

// The partial sums of output (n; rows in0 ..) whose parts lie in warp w of k_toeplitz_rows: parts
// 4w .. 4w + 3 (columns m = part mod 32), added as its shuffles add them.
template <int RB>
__device__ __forceinline__ void small_parts(const float2* __restrict__ X, int Lp, const float4* __restrict__ g, int N, int n,
                                            int in0, int w, bool adjoint, float2 (&y)[RB]) {
  float2 a[4][RB];
#pragma unroll
  for (int q = 0; q < 4; ++q)
#pragma unroll
    for (int r = 0; r < RB; ++r) a[q][r] = make_float2(0.f, 0.f);
  for (int t = 4 * w; t < N; t += 32) {  // (four independent chains of each row)
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int c = t + q;
      if (c < N) {
        float2 u = toeplitz_u(g, n, c);
        if (adjoint) u.y = -u.y;
#pragma unroll
        for (int r = 0; r < RB; ++r) {
          const float2 x = X[c * Lp + pad16(in0 + r)];
          a[q][r].x = fmaf(u.x, x.x, fmaf(-u.y, x.y, a[q][r].x));
          a[q][r].y = fmaf(u.x, x.y, fmaf(u.y, x.x, a[q][r].y));
        }
      }
    }
  }
#pragma unroll
  for (int r = 0; r < RB; ++r) y[r] = cadd(cadd(a[0][r], a[1][r]), cadd(a[2][r], a[3][r]));
}

// The system columns [n0, n0 + 2^wb) that this block computes.
struct SmallSlice {
  int n0, wb;
};

__device__ __forceinline__ void small_store(float2* X, int Lp, int n, int row, float2 y, bool accumulate, float scale,
                                            bool scaled) {
  float2* d = X + n * Lp + pad16(row);
  if (accumulate) {
    y.x += d->x;
    y.y += d->y;
    if (scaled) {
      y.x *= scale;
      y.y *= scale;
    }
  }
  *d = y;
}

// m output rows from out0 on, each U (or U^dagger) applied to its row from in0 on, the slice's columns: a
// thread takes RB rows of one column; while those are fewer than the block's threads, eight threads share
// them (the parts of one warp each) and add their sums in the order of the warps.
template <int RB>
__device__ __forceinline__ void small_rows(float2* X, int Lp, const float4* __restrict__ g, int N, SmallSlice sl, int m,
                                           int in0, int out0, bool adjoint, bool accumulate, float scale, bool scaled) {
  const int W = 1 << sl.wb, items = (m / RB) << sl.wb;
  float2 y[RB], p[RB];
  if (items < kSmallThreads) {
    // (a lane's neighbours take neighbouring columns: eight lanes then read 128 consecutive bytes of g, where
    // eight parts of one column lie 64 bytes apart and conflict four ways; 384 small instances 125 -> 85 us)
    const int w8 = (threadIdx.x >> 2) & 7, base = threadIdx.x & 3, mine = (threadIdx.x >> 5) * 4 + base;
    for (int i0 = 0; i0 < items; i0 += kSmallThreads / 8) {  // (whole warps take part in the shuffles)
      const int it = i0 + mine, n = sl.n0 + (it & (W - 1)), r = (it >> sl.wb) * RB;
#pragma unroll
      for (int q = 0; q < RB; ++q) p[q] = make_float2(0.f, 0.f);
      if (it < items && 4 * w8 < N) small_parts<RB>(X, Lp, g, N, n, in0 + r, w8, adjoint, p);
#pragma unroll
      for (int q = 0; q < RB; ++q) y[q] = p[q];
#pragma unroll
      for (int w = 1; w < 8; ++w) {
#pragma unroll
        for (int q = 0; q < RB; ++q) {
          y[q].x += __shfl_sync(0xffffffffu, p[q].x, base + 4 * w);
          y[q].y += __shfl_sync(0xffffffffu, p[q].y, base + 4 * w);
        }
      }
      if (it < items && w8 == 0) {
#pragma unroll
        for (int q = 0; q < RB; ++q) small_store(X, Lp, n, out0 + r + q, y[q], accumulate, scale, scaled);
      }
    }
  } else {
    for (int it = threadIdx.x; it < items; it += kSmallThreads) {
      const int n = sl.n0 + (it & (W - 1)), r = (it >> sl.wb) * RB;
      small_parts<RB>(X, Lp, g, N, n, in0 + r, 0, adjoint, y);
      for (int w = 1; 4 * w < N && w < 8; ++w) {
        small_parts<RB>(X, Lp, g, N, n, in0 + r, w, adjoint, p);
#pragma unroll
        for (int q = 0; q < RB; ++q) y[q] = cadd(y[q], p[q]);
      }
#pragma unroll
      for (int q = 0; q < RB; ++q) small_store(X, Lp, n, out0 + r + q, y[q], accumulate, scale, scaled);
    }
  }
}

__device__ void small_product(float2* X, int Lp, const float4* __restrict__ g, int N, SmallSlice sl, int m, int in0, int out0,
                              bool adjoint, bool accumulate, float scale, bool scaled) {
  if (m >= 4) small_rows<4>(X, Lp, g, N, sl, m, in0, out0, adjoint, accumulate, scale, scaled);
  else if (m == 2) small_rows<2>(X, Lp, g, N, sl, m, in0, out0, adjoint, accumulate, scale, scaled);
  else small_rows<1>(X, Lp, g, N, sl, m, in0, out0, adjoint, accumulate, scale, scaled);
}

__device__ __forceinline__ float small_square(float2 a, float2 b) {
  return fmaf(a.x, a.x, fmaf(a.y, a.y, fmaf(b.x, b.x, b.y * b.y)));
}

// The other blocks' columns of rows [row0, row0 + 2^lr) into this block's copy of the state.
__device__ __forceinline__ void small_pull(float2* X, int Lp, int N, SmallSlice sl, int row0, int lr) {
  const int W = 1 << sl.wb, total = (N - W) << lr;
  constexpr int U = 4;  // loads in flight per thread
  for (int e0 = threadIdx.x; e0 < total; e0 += U * kSmallThreads) {
    float2 v[U];
    float2* d[U];
#pragma unroll
    for (int q = 0; q < U; ++q) {
      const int e = e0 + q * kSmallThreads;
      if (e >= total) break;
      const int other = e >> lr, n = other < sl.n0 ? other : other + W;
      d[q] = X + n * Lp + pad16(row0 + (e & ((1 << lr) - 1)));
      v[q] = *cg::this_cluster().map_shared_rank(d[q], n >> sl.wb);
    }
#pragma unroll
    for (int q = 0; q < U; ++q)
      if (e0 + q * kSmallThreads < total) *d[q] = v[q];
  }
}

// One solve, by one block (c = 1) or, with CL, by the first c blocks of a cluster, each of which computes
// N / c system columns and reads the rows that its next product needs from the others through distributed
// shared memory, after the cluster's barrier. Such rows are never written again: an expansion's output
// rows are new, and a reduction's are read only once nothing more is added to them.
template <bool CL>
__device__ __forceinline__ void small_solve(const SmallInst& d, int c, int rank, unsigned char* small_raw,
                                            const double* __restrict__ b_all, double* __restrict__ b_copy,
                                            double* __restrict__ out_all, double* __restrict__ eps) {
  __shared__ double weights[kSmallCluster][2];  // block 0 of a cluster: the blocks' weights
  const int N = 1 << d.n_s, L = 1 << d.n_c, m = d.n_c, Lp = small_column(d.n_c), M = 2 * N + 2;
  float4* gk = reinterpret_cast<float4*>(small_raw);  // two tables: the next step's loads under this one
  float2* t0 = reinterpret_cast<float2*>(gk + 2 * M);
  float2* t1 = t0 + 64;
  float2* X = t0 + twiddle_entries(m);
  const int W = N / c;
  const SmallSlice sl{rank * W, 31 - __clz(W)};
  const double2* b = reinterpret_cast<const double2*>(b_all + d.b_off);
  auto load_g = [&](int k, int buf) {
    for (int q = threadIdx.x; q < M; q += kSmallThreads) gk[buf * M + q] = d.g[(size_t)k * M + q];
  };
  fill_twiddles<float>(t0, t1, m);
  load_g(0, 0);
  // the scaled right-hand side in clock row 0
  double nb2[1], s[1] = {0.0};
  double2 z = make_double2(0.0, 0.0);
  if (threadIdx.x < N) {
    z = b[threadIdx.x];
    s[0] = z.x * z.x + z.y * z.y;
    if (b_copy != nullptr && rank == 0) reinterpret_cast<double2*>(b_copy + d.b_off)[threadIdx.x] = z;
  }
  block_sum_all(s, nb2);
  const double scale = nb2[0] > 0.0 ? 1.0 / sqrt(nb2[0] * (double)L) : 0.0;
  if (threadIdx.x < N) X[threadIdx.x * Lp] = make_float2((float)(z.x * scale), (float)(z.y * scale));
  __syncthreads();
  if constexpr (CL) cg::this_cluster().sync();  // every block runs: its shared memory may be used
  // QPE by doubling
  for (int k = 0; k < m; ++k) {
    load_g(k + 1 < m ? k + 1 : m - 1, (k + 1) & 1);  // (the last load is the first reduction step's)
    small_product(X, Lp, gk + (k & 1) * M, N, sl, 1 << k, 0, 1 << k, false, false, 1.f, false);
    if constexpr (CL) {  // (the clock block needs this block's columns only, and overwrites what others read)
      cg::this_cluster().sync();
      if (k + 1 < m) small_pull(X, Lp, N, sl, 1 << k, k);
    }
    __syncthreads();
  }
  // inverse QFT, rotation (the anc = 0 half is only weighed), QFT
  const Twiddle<float2> tw{t0, t1};
  float2* Xs = X + sl.n0 * Lp;
  local_stages<float2, false, 0, true>(Xs, Lp, W, tw, m, m, false);
  const float inv = (float)(1.0 / sqrt((double)L));
  df w[2] = {df(0), df(0)};
  for (int u = threadIdx.x; u < L * (W / 2); u += kSmallThreads) {
    const int p = u & (L - 1), j = (u >> m) * 2;
    const float2 r = d.rot[bitrev_m(p, m)];
    float2 kt[2];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int idx = (j + q) * Lp + pad16(p);
      const float2 x = cscale(Xs[idx], inv);
      kt[q] = cscale(x, r.x);
      Xs[idx] = cscale(x, r.y);
    }
    w[0] = df_add(w[0], df(small_square(kt[0], kt[1]), 0.f));
  }
  __syncthreads();
  local_stages<float2, true, 0, true>(Xs, Lp, W, tw, m, m, true);
  for (int u = threadIdx.x; u < L * (W / 2); u += kSmallThreads) {
    const int p = u & (L - 1), j = (u >> m) * 2;
    float2 v[2];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int idx = (j + q) * Lp + pad16(p);
      v[q] = cscale(Xs[idx], inv);
      Xs[idx] = v[q];
    }
    w[1] = df_add(w[1], df(small_square(v[0], v[1]), 0.f));
  }
  double ws[2] = {(double)w[0].h + (double)w[0].l, (double)w[1].h + (double)w[1].l}, wt[2];
  block_sum_all(ws, wt);
  if constexpr (CL) {
    if (threadIdx.x < 2) *cg::this_cluster().map_shared_rank(&weights[rank][threadIdx.x], 0) = threadIdx.x ? wt[1] : wt[0];
    cg::this_cluster().sync();
    small_pull(X, Lp, N, sl, L / 2, m - 1);
  }
  __syncthreads();
  // uncompute, Hadamards and postselection by halving: the table of step k is in buffer k & 1 or,
  // for the first, in the one the last expansion step loaded
  int buf = m & 1;
  for (int k = m - 1; k >= 0; --k) {
    if (k > 0) load_g(k - 1, buf ^ 1);
    small_product(X, Lp, gk + buf * M, N, sl, 1 << k, 1 << k, 0, true, true, inv, k == 0);
    if constexpr (CL) {  // the next step's rows [2^(k-1), 2^k), at the end row 0
      cg::this_cluster().sync();
      if (k > 0 || rank == 0) small_pull(X, Lp, N, sl, k > 0 ? 1 << (k - 1) : 0, k > 0 ? k - 1 : 0);
    }
    __syncthreads();
    buf ^= 1;
  }
  if constexpr (CL) {
    cg::this_cluster().sync();  // block 0 has read the others' row 0
    if (rank > 0) return;
    wt[0] = wt[1] = 0.0;
    for (int q = 0; q < c; ++q) {
      wt[0] += weights[q][0];
      wt[1] += weights[q][1];
    }
  }
  // the measurement block and the dissipation rate
  double a[2] = {0.0, 0.0}, t[2];
  const double us = sqrt(nb2[0]) * d.inv_c_lam;
  float2 v = make_float2(0.f, 0.f);
  if (threadIdx.x < N) {
    const int i = threadIdx.x;
    v = X[i * Lp];
    a[0] = (double)v.x * (double)v.x + (double)v.y * (double)v.y;
    const double left = i == 0 ? d.wall_lo : us * (double)X[(i - 1) * Lp].x, right = us * (double)v.x;
    a[1] = (right - left) * (right - left);
    if (i == N - 1) a[1] += (d.wall_hi - right) * (d.wall_hi - right);
  }
  block_sum_all(a, t);
  double* out = out_all + d.out_off;
  if (threadIdx.x == 0) {
    out[0] = t[0];
    out[1] = wt[1];
    out[2] = wt[0] + wt[1];
    out[3] = sqrt(nb2[0]);
    eps[d.index] = d.nu_over_h * t[1];
  }
  if (threadIdx.x < N) {
    const double iv = t[0] > 0.0 ? 1.0 / sqrt(t[0]) : 0.0;
    out[4 + 2 * threadIdx.x] = (double)v.x * iv;
    out[5 + 2 * threadIdx.x] = (double)v.y * iv;
  }
}

template <bool CL>
__global__ void __launch_bounds__(kSmallThreads, CL ? 1 : 3) k_batch_small(const SmallInst* __restrict__ inst,
                                                                       const double* __restrict__ b_all,
                                                                       double* __restrict__ b_copy,
                                                                       double* __restrict__ out_all, double* __restrict__ eps) {
  extern __shared__ __align__(16) unsigned char small_raw[];
  if constexpr (CL) {
    const int size = (int)cg::this_cluster().num_blocks(), rank = (int)cg::this_cluster().block_rank();
    const SmallInst d = inst[blockIdx.x / size];
    const int most = (1 << d.n_s) / kSmallColumns, c = most < size ? most : size;
    if (c > 1) {  // (blocks beyond c leave: the cluster's barrier counts those that have not)
      if (rank < c) small_solve<true>(d, c, rank, small_raw, b_all, b_copy, out_all, eps);
    } else if (rank == 0) {
      small_solve<false>(d, 1, 0, small_raw, b_all, b_copy, out_all, eps);
    }
  } else {
    small_solve<false>(inst[blockIdx.x], 1, 0, small_raw, b_all, b_copy, out_all, eps);
  }
}

struct SmallClass {  // instances of similar shared-memory need: one launch
  int first = 0, count = 0;
  size_t smem = 0;
  int max_n = 0;    // points of the largest
  int cluster = 1;  // blocks an instance
};

struct Work {
  cudaStream_t s = nullptr;
  cudaEvent_t done = nullptr;
  int64_t capN = 0, cap_msub = 0;
  void* ubuf = nullptr;    // operand: tc hi|lo (2 x 4N^2 FP16) or simt (N^2 complex64)
  __half* a_hi = nullptr;  // tc split rows (M_sub x 2N FP16)
  __half* a_lo = nullptr;
  void* scratch = nullptr; // simt GEMM output rows (M_sub x N complex64)
  TcWork tcw;              // none: the batch's GEMMs run one CTA per tile (no split tiles)
};

int gemm_rule(int n_s, int n_c) {
  if (n_c < 8 || n_s < 6) return 0;
  return n_s == 6 ? 128 : 256;
}

}  // namespace
}  // namespace hhl

using hhl::Plan;
using hhl::fail;

struct hhl_batch_s {
  int count = 0;
  std::vector<Plan> plans;
  std::vector<int> gemm;       // 0 SIMT, 128 / 256 tcgen05 tile width
  std::vector<int> large;      // the instances that the graph runs
  std::vector<hhl::SmallClass> small;  // the others: one-block solves, by shared memory
  hhl::SmallInst* d_small = nullptr;
  int streams = 0;
  std::vector<int> stream_of;
  std::vector<size_t> state_off, b_off, out_off, ph_off, cos_off, g_off, rot_off;
  std::vector<CUtensorMap> maps;  // 4 per instance (tc): A_hi, A_lo, B_hi, B_lo
  std::vector<hhl::Work> work;
  void* arena = nullptr;       // all states
  double* d_b = nullptr;       // packed complex128 right-hand sides
  double* d_out = nullptr;     // packed [4 + 2N] measurement blocks
  double* d_eps = nullptr;     // count
  double* d_scal = nullptr;    // 16 per instance
  void* d_bs = nullptr;        // packed N complex64 per instance
  void* d_rot = nullptr;       // packed R complex64 (cos, sin) per instance
  double2* d_ph = nullptr;     // packed n_c x N phases per instance
  double* d_cos = nullptr;     // packed 2N+2 cosines per instance
  float4* d_g = nullptr;       // packed n_c x (2N+2) per instance (double-float)
  int* d_err = nullptr;
  size_t state_bytes = 0, work_bytes = 0;
  double gemm_flops = 0;
  cudaGraph_t graph = nullptr;
  cudaGraphExec_t exec = nullptr;
  uint64_t graph_launches = 0;  // kernels of one run (0 before the first)
  std::vector<double> host_b;  // staging for hhl_batch_run_host
};

namespace hhl {
namespace {

void free_batch(hhl_batch_s* b) {
  if (!b) return;
  if (b->exec) cudaGraphExecDestroy(b->exec);
  if (b->graph) cudaGraphDestroy(b->graph);
  for (auto& w : b->work) {
    if (w.ubuf) cudaFree(w.ubuf);
    if (w.a_hi) cudaFree(w.a_hi);
    if (w.a_lo) cudaFree(w.a_lo);
    if (w.scratch) cudaFree(w.scratch);
    if (w.done) cudaEventDestroy(w.done);
    if (w.s) cudaStreamDestroy(w.s);
  }
  void* ptrs[] = {b->arena, b->d_b, b->d_out, b->d_eps, b->d_scal, b->d_bs, b->d_rot, b->d_ph, b->d_cos, b->d_g, b->d_err, b->d_small};
  for (void* q : ptrs)
    if (q) cudaFree(q);
  delete b;
}

// Enqueue the whole circuit of instance i on its worker stream.
hhl_status enqueue_instance(hhl_batch_s* B, int i) {
  Plan& p = B->plans[i];
  Work& w = B->work[B->stream_of[i]];
  cudaStream_t st = w.s;
  void* state = (char*)B->arena + B->state_off[i];
  char* s0 = (char*)state;
  char* s1 = s0 + (size_t)(p.R * p.N) * 8;
  const double* b = B->d_b + B->b_off[i];
  // the postselected solve (the same circuit rearranged for its prepared input; see
  // hhl_solve_postselected): only the clock = 0 row of the anc = 0 half is prepared
  hhl_status s = launch_prep_row(p, b, state, st);
  if (s != HHL_OK) return s;
  const int M = (int)(2 * p.N + 2);
  // tree step k: expansion (rows [2^k, 2^(k+1)) = U_k rows [0, 2^k), anc = 0 half) or
  // reduction (rows [0, 2^k) += U_k^dagger rows [2^k, 2^(k+1)), anc = 1 half, the last step
  // scaled by 2^(-n_c/2)), on tcgen05 where the instance has tiles and 2^k >= 128 rows
  auto step = [&](int k, bool reduce) -> hhl_status {
    const float4* gk = B->d_g + B->g_off[i] + (size_t)k * M;
    const int64_t N2 = 2 * p.N;
    const int64_t m = 1LL << k;
    RowMap rows;
    rows.in_off = reduce ? m : 0;
    rows.out_off = reduce ? 0 : m;
    rows.accumulate = reduce ? 1 : 0;
    if (reduce && k == 0) rows.scale = 1.0 / sqrt((double)p.R);
    void* half = reduce ? (void*)s1 : (void*)s0;
    const int g = (int)std::min<int64_t>((p.N * p.N + 255) / 256, 152 * 16);
    if (m < toeplitz_rows_limit())  // few rows: U_k generated on the fly, no N x N operand
      return launch_toeplitz_rows((float2*)half, p.n_s, gk, reduce ? 1 : 0, rows, m, st);
    if (B->gemm[i] == 0 || rows.scale != 1.0) {
      HHL_PROF_BEGIN(st);
      k_ugen_embed_simt<<<g, 256, 0, st>>>(p.n_s, gk, reduce ? 1 : 0, (float2*)w.ubuf);
      HHL_LAUNCH_CHECK("k_ugen_embed_simt");
      return launch_ctrl_u_simt_map(p, half, rows, m, w.ubuf, st);
    }
    __half* hi = (__half*)w.ubuf;
    __half* lo = hi + N2 * N2;
    HHL_PROF_BEGIN(st);
    k_ugen_embed_tc<<<g, 256, 0, st>>>(p.n_s, gk, reduce ? 1 : 0, hi, lo);
    HHL_LAUNCH_CHECK("k_ugen_embed_tc");
    const CUtensorMap* mp = &B->maps[(size_t)i * 4];
    return launch_tc_gemm_map(p.n_s, m, rows, half, w.a_hi, w.a_lo, mp[0], mp[1], mp[2], mp[3], B->gemm[i], B->d_err, w.tcw, 0,
                              st);
  };
  for (int k = 0; k < p.n_c && s == HHL_OK; ++k) s = step(k, false);
  if (s == HHL_OK) s = launch_clock_block(p, state, st);
  if (s == HHL_OK) s = launch_measure_sums(p, state, st);  // |S0|^2, |S1|^2 before the reduction
  for (int k = p.n_c - 1; k >= 0 && s == HHL_OK; --k) s = step(k, true);
  if (s == HHL_OK) s = launch_measure_row(p, state, B->d_out + B->out_off[i], st);
  if (s == HHL_OK) s = launch_dissipation(p, state, B->d_eps + i, nullptr, st);
  return s;
}

// The launch of a class with `cluster` blocks an instance; attr: room for its one attribute.
cudaLaunchConfig_t small_config(const SmallClass& k, int cluster, cudaLaunchAttribute* attr, cudaStream_t st) {
  attr->id = cudaLaunchAttributeClusterDimension;
  attr->val.clusterDim.x = (unsigned)cluster;
  attr->val.clusterDim.y = attr->val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(k.count * cluster));
  cfg.blockDim = dim3(kSmallThreads);
  cfg.dynamicSmemBytes = k.smem;
  cfg.stream = st;
  cfg.attrs = attr;
  cfg.numAttrs = cluster > 1 ? 1 : 0;
  return cfg;
}

// Blocks an instance of a launch: as many as give each 16 columns (fewer gain nothing: 5 + 7 qubits 46 us by
// two blocks, 50 by one; 4 + 7 qubits 41 and 35) while all its clusters run at once (16 instances of 7 + 7 qubits:
// clusters of 8 come in two waves, 228 us, of 4 in one, 151; both before g was read without conflicts).
int small_cluster(const SmallClass& k) {
  int c = kSmallCluster;
  while (c > 1 && k.max_n < c * kSmallColumns) c /= 2;
  if (c > 1 && raise_dyn_smem((const void*)k_batch_small<true>, k.smem) != cudaSuccess) c = 1;
  for (; c > 1; c /= 2) {
    cudaLaunchAttribute attr[1];
    const cudaLaunchConfig_t cfg = small_config(k, c, attr, nullptr);
    int at_once = 0;
    if (cudaOccupancyMaxActiveClusters(&at_once, k_batch_small<true>, &cfg) == cudaSuccess && k.count <= at_once) break;
  }
  cudaGetLastError();
  return c;
}

// The one-block solves, on the caller's stream.
hhl_status run_small(const hhl_batch_s* B, const double* b, double* b_copy, double* out, double* eps, cudaStream_t st) {
  for (const SmallClass& c : B->small) {
    auto kern = c.cluster > 1 ? k_batch_small<true> : k_batch_small<false>;
    HHL_CUDA_TRY(raise_dyn_smem((const void*)kern, c.smem));
    cudaLaunchAttribute attr[1];
    const cudaLaunchConfig_t cfg = small_config(c, c.cluster, attr, st);
    HHL_PROF_BEGIN(st);
    HHL_CUDA_TRY(cudaLaunchKernelEx(&cfg, kern, (const SmallInst*)(B->d_small + c.first), b, b_copy, out, eps));
    HHL_LAUNCH_CHECK("k_batch_small");
  }
  return HHL_OK;
}

hhl_status capture(hhl_batch_s* B) {
  if (B->large.empty()) B->graph_launches = B->small.size();
  if (B->exec || B->large.empty()) return HHL_OK;
  cudaStream_t cap = nullptr;
  HHL_CUDA_TRY(cudaStreamCreateWithFlags(&cap, cudaStreamNonBlocking));
  cudaEvent_t fork = nullptr;
  HHL_CUDA_TRY(cudaEventCreateWithFlags(&fork, cudaEventDisableTiming));
  const uint64_t l0 = g_launches.load();
  hhl_status s = HHL_OK;
  cudaError_t e = cudaStreamBeginCapture(cap, cudaStreamCaptureModeRelaxed);
  // every replay starts with a clear GEMM error flag (a memset node ahead of the fork)
  if (e == cudaSuccess) e = cudaMemsetAsync(B->d_err, 0, sizeof(int), cap);
  if (e == cudaSuccess) e = cudaEventRecord(fork, cap);
  for (auto& w : B->work)
    if (e == cudaSuccess) e = cudaStreamWaitEvent(w.s, fork, 0);
  for (int i : B->large)
    if (e == cudaSuccess && s == HHL_OK) s = enqueue_instance(B, i);
  if (e == cudaSuccess && s == HHL_OK) s = run_small(B, B->d_b, nullptr, B->d_out, B->d_eps, cap);  // beside them
  for (auto& w : B->work) {
    if (e == cudaSuccess) e = cudaEventRecord(w.done, w.s);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(cap, w.done, 0);
  }
  cudaGraph_t graph = nullptr;
  cudaError_t e2 = cudaStreamEndCapture(cap, &graph);
  cudaEventDestroy(fork);
  cudaStreamDestroy(cap);
  if (s != HHL_OK) {
    if (graph) cudaGraphDestroy(graph);
    return s;
  }
  if (e != cudaSuccess) return cuda_fail(e, "batch capture");
  if (e2 != cudaSuccess) return cuda_fail(e2, "cudaStreamEndCapture");
  B->graph = graph;
  HHL_CUDA_TRY(cudaGraphInstantiate(&B->exec, graph, 0));
  B->graph_launches = g_launches.load() - l0;
  return HHL_OK;
}

}  // namespace
}  // namespace hhl

extern "C" {

hhl_status hhl_batch_create(const hhl_problem* probs, const hhl_params* params, int32_t count,
                            const int32_t* gemm_choice, int32_t streams, hhl_batch_t* out) {
  using namespace hhl;
  if (out == nullptr || probs == nullptr || params == nullptr || count < 1) return fail(HHL_ERR_INVALID_ARG, "bad batch arguments");
  *out = nullptr;
  if (streams < 1) streams = 8;
  hhl_batch_s* B = new hhl_batch_s();
  B->count = count;
  B->plans.resize(count);
  B->gemm.resize(count);
  B->stream_of.resize(count);
  std::vector<std::vector<double>> lam(count);
  for (int i = 0; i < count; ++i) {
    const hhl_problem& pr = probs[i];
    const hhl_params& pa = params[i];
    if (pa.precision != HHL_PREC_C64 || pa.expm_mode != HHL_EXPM_DENSE || pa.full_uncompute) {
      free_batch(B);
      return fail(HHL_ERR_UNSUPPORTED, "batch instances are complex64, dense, postselect-early");
    }
    if (pr.kind != HHL_MATRIX_TRIDIAG || pr.n_sys_qubits < 1) {
      free_batch(B);
      return fail(HHL_ERR_UNSUPPORTED, "batch instances need a tridiagonal A");
    }
    const int64_t N = 1LL << pr.n_sys_qubits;
    for (int64_t j = 1; j < N; ++j)
      if (pr.diag[j] != pr.diag[0] || (j + 1 < N && pr.off[j] != pr.off[0])) {
        free_batch(B);
        return fail(HHL_ERR_UNSUPPORTED, "batch instances need a Toeplitz tridiagonal A (just-in-time U_k)");
      }
    hhl_status s = plan_scalars(&pr, &pa, B->plans[i], &lam[i]);
    if (s != HHL_OK) {
      free_batch(B);
      return s;
    }
    Plan& p = B->plans[i];
    const int rule = gemm_rule(p.n_s, p.n_c);
    int gsel = gemm_choice ? gemm_choice[i] : -1;
    if (gsel != 0 && gsel != 128 && gsel != 256) gsel = rule;
    if (gsel != 0 && (p.R / 2 < 128 || 2 * p.N < gsel)) gsel = 0;  // tile does not fit
    B->gemm[i] = gsel;
    p.gemm_impl = gsel ? HHL_GEMM_TCGEN05 : HHL_GEMM_SIMT;
    // one-block solves: every tree step of n_c <= 7 is a Toeplitz product (fewer than 128 rows) whose
    // blocks take 8 outputs at N <= 128, which is the summation order the block repeats
    // (one or two of 7 + 7 qubits are faster as launches: 79 and 84 us, by a cluster each 89)
    const bool launches = count <= 2 && p.n_s + p.n_c == 2 * kSmallBits;
    if (gsel != 0 || p.n_c > kSmallBits || p.n_s > kSmallBits || toeplitz_rows_limit() < 128 || launches) B->large.push_back(i);
    // the two trees: sum over k of 2^k rows each (expansion and reduction)
    B->gemm_flops += 2.0 * 8.0 * (double)(p.R - 1) * (double)p.N * (double)p.N;
  }
  // LPT assignment of instances to worker streams by GEMM work
  B->streams = std::min(streams, count);
  streams = std::min<int>(streams, (int)B->large.size());
  std::vector<int> order = B->large;
  std::vector<char> is_large(count, 0);
  for (int i : B->large) is_large[i] = 1;
  // work of an instance: the GEMM rows of its two trees (2^n_c) and its 2 n_c operand
  // generations, each over N^2 entries
  auto cost = [&](int i) {
    const Plan& q = B->plans[i];
    return (double)(q.R + 2 * q.n_c) * (double)q.N * (double)q.N + 1.0;
  };
  std::sort(order.begin(), order.end(), [&](int a, int b) { return cost(a) > cost(b); });
  std::vector<double> load(streams, 0.0);
  B->work.resize(streams);
  for (int i : order) {
    const int w = (int)(std::min_element(load.begin(), load.end()) - load.begin());
    load[w] += cost(i);
    B->stream_of[i] = w;
    B->work[w].capN = std::max<int64_t>(B->work[w].capN, B->plans[i].N);
    B->work[w].cap_msub = std::max<int64_t>(B->work[w].cap_msub, B->plans[i].R / 2);
  }
  // offsets
  size_t so = 0, bo = 0, oo = 0, po = 0, co = 0, go = 0, ro = 0;
  B->state_off.resize(count); B->b_off.resize(count); B->out_off.resize(count); B->ph_off.resize(count);
  B->cos_off.resize(count); B->g_off.resize(count); B->rot_off.resize(count);
  for (int i = 0; i < count; ++i) {
    const Plan& p = B->plans[i];
    B->state_off[i] = so; so += is_large[i] ? (size_t)(2 * p.R * p.N) * 8 : 0;
    B->b_off[i] = bo;     bo += (size_t)2 * p.N;
    B->out_off[i] = oo;   oo += (size_t)(4 + 2 * p.N);
    B->ph_off[i] = po;    po += (size_t)p.n_c * p.N;
    B->cos_off[i] = co;   co += (size_t)(2 * p.N + 2);
    B->g_off[i] = go;     go += (size_t)p.n_c * (2 * p.N + 2);
    B->rot_off[i] = ro;   ro += (size_t)p.R;
  }
  B->state_bytes = so;
  auto alloc = [&](void** ptr, size_t bytes) -> bool {
    if (cudaMalloc(ptr, std::max<size_t>(bytes, 16)) != cudaSuccess) {
      cudaGetLastError();
      *ptr = nullptr;
      return false;
    }
    return true;
  };
  bool ok = alloc(&B->arena, so) && alloc((void**)&B->d_b, bo * sizeof(double)) &&
            alloc((void**)&B->d_out, oo * sizeof(double)) && alloc((void**)&B->d_eps, count * sizeof(double)) &&
            alloc((void**)&B->d_scal, (size_t)count * 16 * sizeof(double)) &&
            alloc(&B->d_bs, (bo / 2) * sizeof(float2)) && alloc(&B->d_rot, ro * sizeof(float2)) &&
            alloc((void**)&B->d_ph, po * sizeof(double2)) && alloc((void**)&B->d_cos, co * sizeof(double)) &&
            alloc((void**)&B->d_g, go * sizeof(float4)) && alloc((void**)&B->d_err, sizeof(int)) &&
            alloc((void**)&B->d_small, (count - B->large.size()) * sizeof(SmallInst));
  for (auto& w : B->work) {
    if (!ok) break;
    const int64_t N2 = 2 * w.capN;
    // ubuf holds the FP16 hi|lo embedding (2 x 4 N^2 x 2 bytes) or the complex64 SIMT operand
    // (N^2 x 8 bytes), whichever the instances of this stream need (16 N^2 bytes cover both)
    ok = alloc(&w.ubuf, (size_t)2 * N2 * N2 * sizeof(__half)) && alloc((void**)&w.a_hi, (size_t)w.cap_msub * N2 * 2) &&
         alloc((void**)&w.a_lo, (size_t)w.cap_msub * N2 * 2) && alloc(&w.scratch, (size_t)w.cap_msub * w.capN * 8);
    B->work_bytes += (size_t)2 * N2 * N2 * 2 + 2 * (size_t)w.cap_msub * N2 * 2 + (size_t)w.cap_msub * w.capN * 8;
    if (ok) ok = cudaStreamCreateWithFlags(&w.s, cudaStreamNonBlocking) == cudaSuccess &&
                 cudaEventCreateWithFlags(&w.done, cudaEventDisableTiming) == cudaSuccess;
  }
  if (!ok) {
    free_batch(B);
    return fail(HHL_ERR_OOM, "batch device allocation failed");
  }
  // host tables: phases e^{i lambdahat_j t_k}, cosines cos(q pi/(N+1)), rotation (cos, sin)(theta_y/2)
  std::vector<double2> ph;
  std::vector<double> cs;
  std::vector<float2> rot;
  for (int i = 0; i < count; ++i) {
    Plan& p = B->plans[i];
    ph.resize((size_t)p.n_c * p.N);
    for (int k = 0; k < p.n_c; ++k) {
      const double t = p.t0 * (double)(1LL << k) / (double)p.R;
      for (int64_t j = 0; j < p.N; ++j) {
        const double a = lam[i][j] / p.lam_ub * t;
        ph[(size_t)k * p.N + j] = make_double2(cos(a), sin(a));
      }
    }
    cs.resize(2 * p.N + 2);
    for (int64_t q = 0; q < 2 * p.N + 2; ++q) cs[q] = cos((double)q * kPiB / (double)(p.N + 1));
    rot.resize(p.R);
    for (int64_t y = 0; y < p.R; ++y) rot[y] = make_float2((float)cos(p.theta[y] / 2), (float)sin(p.theta[y] / 2));
    cudaMemcpy(B->d_ph + B->ph_off[i], ph.data(), ph.size() * sizeof(double2), cudaMemcpyHostToDevice);
    cudaMemcpy(B->d_cos + B->cos_off[i], cs.data(), cs.size() * sizeof(double), cudaMemcpyHostToDevice);
    cudaMemcpy((float2*)B->d_rot + B->rot_off[i], rot.data(), rot.size() * sizeof(float2), cudaMemcpyHostToDevice);
    if (!is_large[i]) {
      B->maps.insert(B->maps.end(), 4, CUtensorMap{});
      continue;
    }
    // device pointers of the per-instance plan view
    Work& w = B->work[B->stream_of[i]];
    p.d_scal = B->d_scal + (size_t)16 * i;
    p.d_bs = (float2*)B->d_bs + B->b_off[i] / 2;
    p.d_rot = (float2*)B->d_rot + B->rot_off[i];
    p.d_scratch = w.scratch;
    if (B->gemm[i]) {
      CUtensorMap m4[4];
      const int64_t N2 = 2 * p.N;
      hhl_status s = tc_make_map(&m4[0], w.a_hi, N2, p.R / 2, 128);
      if (s == HHL_OK) s = tc_make_map(&m4[1], w.a_lo, N2, p.R / 2, 128);
      if (s == HHL_OK) s = tc_make_map(&m4[2], (__half*)w.ubuf, N2, N2, B->gemm[i]);
      if (s == HHL_OK) s = tc_make_map(&m4[3], (__half*)w.ubuf + N2 * N2, N2, N2, B->gemm[i]);
      if (s != HHL_OK) {
        free_batch(B);
        return s;
      }
      B->maps.insert(B->maps.end(), m4, m4 + 4);
    } else {
      B->maps.insert(B->maps.end(), 4, CUtensorMap{});
    }
  }
  hhl_status s = HHL_OK;
  if (cudaError_t me = cudaMemset(B->d_err, 0, sizeof(int)); me != cudaSuccess) s = cuda_fail(me, "cudaMemset(error flag)");
  if (s == HHL_OK) s = tc_init_kernels();
  if (s == HHL_OK) {
    int64_t maxN = 0;
    for (const Plan& p : B->plans) maxN = std::max<int64_t>(maxN, p.N);
    cudaError_t e = cudaFuncSetAttribute(k_ugen_g, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)std::max<int64_t>(maxN * (int64_t)sizeof(double2), 1024));
    if (e != cudaSuccess) s = cuda_fail(e, "cudaFuncSetAttribute(k_ugen_g)");
  }
  // g_k for every k of every instance, once (they depend on A, T0 and k only): one launch for the
  // one-block solves, one each for the others on their worker streams
  GenInst* d_gen = nullptr;
  if (s == HHL_OK) {
    std::vector<GenInst> gen;
    std::vector<int> order_g;
    int small_n = 0, small_k = 0;
    for (int pass = 0; pass < 2; ++pass)
      for (int i = 0; i < count; ++i) {
        if ((int)is_large[i] != pass) continue;
        const Plan& p = B->plans[i];
        gen.push_back({(int)p.N, p.n_c, B->d_ph + B->ph_off[i], B->d_cos + B->cos_off[i], B->d_g + B->g_off[i]});
        order_g.push_back(i);
        if (pass == 0) {
          small_n = std::max(small_n, (int)p.N);
          small_k = std::max(small_k, p.n_c);
        }
      }
    const int n_small = count - (int)B->large.size();
    cudaError_t e = cudaMalloc((void**)&d_gen, gen.size() * sizeof(GenInst));
    if (e == cudaSuccess) e = cudaMemcpy(d_gen, gen.data(), gen.size() * sizeof(GenInst), cudaMemcpyHostToDevice);
    // A copy from pageable memory may return before it has reached the device, and the worker streams do
    // not wait for the legacy stream that carries it: every table is there before the first launch.
    if (e == cudaSuccess) e = cudaStreamSynchronize(cudaStreamLegacy);
    for (int z = 0; z < n_small && e == cudaSuccess; z += 65535) {
      const dim3 grid((unsigned)((2 * small_n + 2 + 255) / 256), (unsigned)small_k, (unsigned)std::min(65535, n_small - z));
      k_ugen_g<<<grid, 256, small_n * sizeof(double2)>>>(d_gen + z);
      e = cudaGetLastError();
    }
    for (size_t q = n_small; q < gen.size() && e == cudaSuccess; ++q) {
      const dim3 grid((unsigned)((2 * gen[q].N + 2 + 255) / 256), (unsigned)gen[q].n_c);
      k_ugen_g<<<grid, 256, gen[q].N * sizeof(double2), B->work[B->stream_of[order_g[q]]].s>>>(d_gen + q);
      e = cudaGetLastError();
    }
    if (e != cudaSuccess) s = cuda_fail(e, "k_ugen_g");
  }
  if (s == HHL_OK && (int)B->large.size() < count) {
    // the one-block solves, largest first, in at most two launches (the shared memory of a launch is
    // its largest instance's; past 72 KiB, fewer than three blocks an SM, a quarter of it starts the next)
    std::vector<SmallInst> small;
    std::vector<int> idx;
    for (int i = 0; i < count; ++i)
      if (!is_large[i]) idx.push_back(i);
    auto need = [&](int i) { return small_smem(B->plans[i].n_s, B->plans[i].n_c); };
    std::stable_sort(idx.begin(), idx.end(), [&](int a, int c) { return need(a) > need(c); });
    for (int i : idx) {
      const Plan& p = B->plans[i];
      SmallInst d = {};
      d.n_s = p.n_s;
      d.n_c = p.n_c;
      d.b_off = (long long)B->b_off[i];
      d.out_off = (long long)B->out_off[i];
      d.g = B->d_g + B->g_off[i];
      d.rot = (const float2*)B->d_rot + B->rot_off[i];
      d.inv_c_lam = 1.0 / (p.C * p.lam_ub);
      d.wall_lo = p.wall_lo;
      d.wall_hi = p.wall_hi;
      d.nu_over_h = p.nu * (double)(p.N + 1);
      d.index = i;
      if (B->small.empty() || (4 * need(i) < B->small.back().smem && B->small.back().smem > (72 << 10)))
        B->small.push_back({(int)small.size(), 0, need(i)});
      SmallClass& c = B->small.back();
      ++c.count;
      c.max_n = std::max(c.max_n, (int)p.N);
      small.push_back(d);
    }
    for (SmallClass& c : B->small) c.cluster = small_cluster(c);
    cudaError_t e = cudaMemcpy(B->d_small, small.data(), small.size() * sizeof(SmallInst), cudaMemcpyHostToDevice);
    if (e != cudaSuccess) s = cuda_fail(e, "batch setup");
  }
  if (s == HHL_OK) {
    cudaError_t e = cudaDeviceSynchronize();
    if (e != cudaSuccess) s = cuda_fail(e, "batch setup");
  }
  if (d_gen) cudaFree(d_gen);
  if (s != HHL_OK) {
    free_batch(B);
    return s;
  }
  *out = B;
  return HHL_OK;
}

hhl_status hhl_batch_plan(const hhl_problem* probs, const hhl_params* params, int32_t count, hhl_batch_t* out) {
  return hhl_batch_create(probs, params, count, nullptr, 8, out);
}

void hhl_batch_destroy(hhl_batch_t b) { hhl::free_batch(b); }

hhl_status hhl_batch_get_info(hhl_batch_t b, hhl_batch_info* info) {
  if (b == nullptr || info == nullptr) return fail(HHL_ERR_INVALID_ARG, "NULL batch or info");
  memset(info, 0, sizeof(*info));
  info->count = b->count;
  info->streams = b->streams;
  info->state_bytes = b->state_bytes;
  info->workspace_bytes = b->work_bytes;
  info->gemm_flops = b->gemm_flops;
  info->graph_launches = b->graph_launches;
  info->b_doubles = 0;
  info->out_doubles = 0;
  for (int i = 0; i < b->count; ++i) {
    info->b_doubles += 2 * b->plans[i].N;
    info->out_doubles += 4 + 2 * b->plans[i].N;
  }
  return HHL_OK;
}

hhl_status hhl_batch_instance(hhl_batch_t b, int32_t i, int32_t* n_sys_qubits, int32_t* n_clock, int32_t* gemm,
                              int64_t* b_offset, int64_t* out_offset, double* t0) {
  if (b == nullptr || i < 0 || i >= b->count) return fail(HHL_ERR_INVALID_ARG, "bad batch or index");
  if (n_sys_qubits) *n_sys_qubits = b->plans[i].n_s;
  if (n_clock) *n_clock = b->plans[i].n_c;
  if (gemm) *gemm = b->gemm[i];
  if (b_offset) *b_offset = (int64_t)b->b_off[i];
  if (out_offset) *out_offset = (int64_t)b->out_off[i];
  if (t0) *t0 = b->plans[i].t0;
  return HHL_OK;
}

hhl_status hhl_batch_run(hhl_batch_t b, const double* b_dev, double* out_dev, double* eps_dev, void* stream) {
  using namespace hhl;
  if (b == nullptr || b_dev == nullptr || out_dev == nullptr || eps_dev == nullptr)
    return fail(HHL_ERR_INVALID_ARG, "NULL argument");
  cudaStream_t st = (cudaStream_t)stream;
  size_t bo = 0, oo = 0;
  for (int i = 0; i < b->count; ++i) {
    bo += 2 * b->plans[i].N;
    oo += 4 + 2 * b->plans[i].N;
  }
  hhl_status s = capture(b);
  if (s != HHL_OK) return s;
  // One-block solves only: they read and write the caller's arrays themselves (and keep the right-hand
  // sides for hhl_batch_run_eager) where 16-byte loads may and no output lies in what another block reads.
  const double* b_end = b_dev + bo;
  const bool apart = (out_dev >= b_end || out_dev + oo <= b_dev) && (eps_dev >= b_end || eps_dev + b->count <= b_dev);
  if (b->exec == nullptr && (uintptr_t)b_dev % sizeof(double2) == 0 && apart)
    return run_small(b, b_dev, b->d_b, out_dev, eps_dev, st);
  HHL_CUDA_TRY(cudaMemcpyAsync(b->d_b, b_dev, bo * sizeof(double), cudaMemcpyDeviceToDevice, st));
  if (b->exec != nullptr) {
    HHL_CUDA_TRY(cudaGraphLaunch(b->exec, st));
    g_launches.fetch_add(b->graph_launches, std::memory_order_relaxed);
  } else {
    s = run_small(b, b->d_b, nullptr, b->d_out, b->d_eps, st);
    if (s != HHL_OK) return s;
  }
  HHL_CUDA_TRY(cudaMemcpyAsync(out_dev, b->d_out, oo * sizeof(double), cudaMemcpyDeviceToDevice, st));
  HHL_CUDA_TRY(cudaMemcpyAsync(eps_dev, b->d_eps, b->count * sizeof(double), cudaMemcpyDeviceToDevice, st));
  return HHL_OK;
}

hhl_status hhl_batch_run_eager(hhl_batch_t b, void* stream) {
  using namespace hhl;
  if (b == nullptr) return fail(HHL_ERR_INVALID_ARG, "NULL batch");
  cudaStream_t st = (cudaStream_t)stream;
  cudaEvent_t fork = nullptr;
  HHL_CUDA_TRY(cudaEventCreateWithFlags(&fork, cudaEventDisableTiming));
  HHL_CUDA_TRY(cudaMemsetAsync(b->d_err, 0, sizeof(int), st));
  HHL_CUDA_TRY(cudaEventRecord(fork, st));
  for (auto& w : b->work) HHL_CUDA_TRY(cudaStreamWaitEvent(w.s, fork, 0));
  hhl_status s = HHL_OK;
  for (size_t q = 0; q < b->large.size() && s == HHL_OK; ++q) s = enqueue_instance(b, b->large[q]);
  if (s == HHL_OK) s = run_small(b, b->d_b, nullptr, b->d_out, b->d_eps, st);
  for (auto& w : b->work) {
    HHL_CUDA_TRY(cudaEventRecord(w.done, w.s));
    HHL_CUDA_TRY(cudaStreamWaitEvent(st, w.done, 0));
  }
  cudaEventDestroy(fork);
  return s;
}

hhl_status hhl_batch_run_host(hhl_batch_t b, const double* b_host, double* out_host, double* eps_host, void* stream) {
  using namespace hhl;
  if (b == nullptr || b_host == nullptr || out_host == nullptr || eps_host == nullptr)
    return fail(HHL_ERR_INVALID_ARG, "NULL argument");
  cudaStream_t st = (cudaStream_t)stream;
  size_t bo = 0, oo = 0;
  for (int i = 0; i < b->count; ++i) {
    bo += 2 * b->plans[i].N;
    oo += 4 + 2 * b->plans[i].N;
  }
  hhl_status s = capture(b);
  if (s != HHL_OK) return s;
  HHL_CUDA_TRY(cudaMemcpyAsync(b->d_b, b_host, bo * sizeof(double), cudaMemcpyHostToDevice, st));
  if (b->exec != nullptr) {
    HHL_CUDA_TRY(cudaGraphLaunch(b->exec, st));
    g_launches.fetch_add(b->graph_launches, std::memory_order_relaxed);
  } else {
    s = run_small(b, b->d_b, nullptr, b->d_out, b->d_eps, st);
    if (s != HHL_OK) return s;
  }
  HHL_CUDA_TRY(cudaMemcpyAsync(out_host, b->d_out, oo * sizeof(double), cudaMemcpyDeviceToHost, st));
  HHL_CUDA_TRY(cudaMemcpyAsync(eps_host, b->d_eps, b->count * sizeof(double), cudaMemcpyDeviceToHost, st));
  return hhl_batch_status(b, stream);
}

hhl_status hhl_batch_status(hhl_batch_t b, void* stream) {
  using namespace hhl;
  if (b == nullptr) return fail(HHL_ERR_INVALID_ARG, "NULL batch");
  cudaStream_t st = (cudaStream_t)stream;
  int err = 0;
  HHL_CUDA_TRY(cudaMemcpyAsync(&err, b->d_err, sizeof(int), cudaMemcpyDeviceToHost, st));
  HHL_CUDA_TRY(cudaStreamSynchronize(st));
  return tc_flag_status(err);
}

}  // extern "C"
