// Complex128 dense plans in the eigenbasis of A.
//
// U_k = V diag(e^{i lambdahat_j t_k}) V^T for every k with one orthogonal V (the analytic sine
// basis of a Toeplitz tridiagonal A, Jacobi vectors of another real symmetric A), and V acts on
// the system register only, so it commutes with every gate on the clock and the ancilla. The
// whole circuit is therefore V on every clock row, then per eigenvector j a circuit on the clock
// and the ancilla alone (the controlled U_k are the phases e^{i phi_j c} of clock row c, phi_j =
// lambdahat_j T0 / 2^{n_c}), then V^T on every row of both halves: three real N x N products
// instead of 2 n_c complex ones on half the rows. GB300's FP64 pipe is about 1/32 of its FP32
// one, so the products bound these plans: N = 16, 2^6 clock rows (11 qubits) took 12 products of
// 70 us each, 0.93 ms a solve, and takes 35 us this way. complex64 plans keep their gate products:
// their read-outs are FP64 values of FP32 states, and this form rounds those states differently
// (nearer to the exact circuit, but by 1e-7 to 4e-5 of the read-out).
//
// The postselected solve starts from the product state of n_c Hadamards, and the controlled
// phases keep the clock one: qubit k holds (|0> + e^{i 2^k phi}|1>) / sqrt 2. The inverse QFT
// resolves the bits of the clock value y from the least significant up, bit m from qubit n_c-1-m
// after the phase of the lower bits of y, so the weight of y is a product of n_c factors,
//     |psi_j(y)|^2 = prod_m cos^2(pi a_m(y)),  a_m(y) = 2^{n_c-1-m} phi / 2 pi - (y mod 2^{m+1}) / 2^{m+1},
// where y and y + 2^m share a_m up to half a turn (cos^2 becomes sin^2): a binary tree with one
// sine / cosine pair per inner node. What follows the inversion rotation (QFT, uncompute,
// Hadamards, clock = 0) is the adjoint of what precedes it, so the postselected amplitude is
// v_j = beta_j sum_y sin(theta_y / 2) |psi_j(y)|^2 with beta = V^T bhat, and the weights of the two
// ancilla halves are sum_j |beta_j|^2 sum_y {cos^2, sin^2}(theta_y / 2) |psi_j(y)|^2.
#include <math.h>

#include <algorithm>
#include <vector>

#include "hhl_common.cuh"

namespace hhl {

struct SpecState {
  void* mem = nullptr;        // one allocation for everything below
  double* basis = nullptr;    // V, N x N row-major (column j: eigenvector j)
  double* basis_t = nullptr;  // V^T (the same buffer for the symmetric sine basis)
  unsigned long long* frac = nullptr;  // N: phi_j / (2 pi) mod 1 in units of 2^-64
  double2* ph_lo = nullptr;   // N x 32: e^{i phi_j c}, c < 32
  double2* ph_hi = nullptr;   // N x (R / 32, at least 1): e^{i phi_j 32 q}
  double2* tw = nullptr;      // R: e^{-2 pi i q / R}
  double* sin_half = nullptr; // R: sin(theta_y / 2)
  double2* x = nullptr;       // N: bhat
  double2* beta = nullptr;    // N: V^T bhat, then the postselected eigen-amplitudes
  double2* wts = nullptr;     // N: the weights of the two ancilla halves per eigenvector
};

namespace {

constexpr double kPiS = 3.14159265358979323846;
constexpr int kSpecThreads = 256;
constexpr size_t kSpecRowSmem = 128 * 1024;  // system rows of one block of the row products
constexpr int kClockThreads = 128;
constexpr int kClockBits = 7;                // log2 of the threads of one column (at most)

// ------------------------------------------------------------------ plan tables
// V of the sine basis from its table w sin(q pi / (N + 1)), q < 2N + 2.
__global__ void k_spec_sine_basis(int N, const double* __restrict__ tab, double* __restrict__ V) {
  const int M = 2 * N + 2;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < (long long)N * N;
       e += (long long)gridDim.x * blockDim.x) {
    const long long i = e / N, j = e - i * N;
    V[e] = tab[(int)(((i + 1) * (j + 1)) % M)];
  }
}

// Phases of every eigenvector (lo, hi) and the roots of the clock transform.
__global__ void k_spec_phases(int N, int R, const unsigned long long* __restrict__ frac, double2* __restrict__ lo,
                              double2* __restrict__ hi, double2* __restrict__ tw) {
  const int nh = R > 32 ? R / 32 : 1, per = 32 + nh;
  const long long total = (long long)N * per + R;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total;
       e += (long long)gridDim.x * blockDim.x) {
    double s, c;
    if (e < (long long)N * per) {
      const int j = (int)(e / per), q = (int)(e - (long long)j * per);
      const unsigned long long t = frac[j] * (unsigned long long)(q < 32 ? q : 32 * (q - 32));  // exact mod 1
      sincospi((double)(long long)t * 1.0842021724855044e-19, &s, &c);  // 2 t 2^-64 half turns
      if (q < 32) lo[(size_t)j * 32 + q] = make_double2(c, s);
      else hi[(size_t)j * nh + (q - 32)] = make_double2(c, s);
    } else {
      const int q = (int)(e - (long long)N * per);
      sincospi(-2.0 * (double)q / (double)R, &s, &c);
      tw[q] = make_double2(c, s);
    }
  }
}

// ------------------------------------------------------------------ products on the clock rows
// X[r][:] <- X[r][:] B for every row r (B real, N x N), in place: a block owns BM rows, holds them
// in shared memory and writes them back when every output is formed, so no second buffer is
// needed. A thread takes RPT rows of one output column; B streams from L2 (each element serves BM
// rows). Bound by the FP64 pipe.
template <int RPT>
__global__ void __launch_bounds__(kSpecThreads) k_spec_rows(double2* __restrict__ X, const double* __restrict__ B, int N,
                                                            long long rows) {
  dep_begin();
  extern __shared__ __align__(16) unsigned char spec_smem[];
  double2* xs = reinterpret_cast<double2*>(spec_smem);
  const int tn = N < kSpecThreads ? N : kSpecThreads, rg = kSpecThreads / tn, BM = RPT * rg;
  const long long r0 = (long long)blockIdx.x * BM;
  const int nr = (int)(rows - r0 < BM ? rows - r0 : BM);
  for (int e = threadIdx.x; e < nr * N; e += kSpecThreads) xs[e] = X[r0 * N + e];
  __syncthreads();
  const int g = threadIdx.x / tn;
  const double2* xr[RPT];
#pragma unroll
  for (int q = 0; q < RPT; ++q) xr[q] = xs + (size_t)(g + q * rg < nr ? g + q * rg : 0) * N;
  for (int n = threadIdx.x % tn; n < N; n += tn) {
    double2 acc[RPT];
#pragma unroll
    for (int q = 0; q < RPT; ++q) acc[q] = make_double2(0.0, 0.0);
#pragma unroll 4
    for (int m = 0; m < N; ++m) {
      const double v = B[(size_t)m * N + n];
#pragma unroll
      for (int q = 0; q < RPT; ++q) {
        const double2 z = xr[q][m];
        acc[q].x = fma(v, z.x, acc[q].x);
        acc[q].y = fma(v, z.y, acc[q].y);
      }
    }
#pragma unroll
    for (int q = 0; q < RPT; ++q)
      if (g + q * rg < nr) X[(r0 + g + q * rg) * N + n] = acc[q];
  }
}

template <int RPT>
hhl_status rows_launch(double2* X, const double* B, int N, long long rows, cudaStream_t st) {
  const int tn = std::min(N, kSpecThreads), bm = RPT * (kSpecThreads / tn);
  const size_t smem = (size_t)bm * N * sizeof(double2);
  HHL_CUDA_TRY(raise_dyn_smem((const void*)k_spec_rows<RPT>, smem));
  HHL_PROF_BEGIN(st);
  launch_dep(k_spec_rows<RPT>, (unsigned)((rows + bm - 1) / bm), kSpecThreads, smem, st, X, B, N, rows);
  HHL_LAUNCH_CHECK("k_spec_rows");
  return HHL_OK;
}

// Rows per thread: as many as keep a block's rows within kSpecRowSmem while the blocks still cover
// the SMs (few rows: one each, the product is then bound by latency, not by reads of B).
hhl_status spec_rows(double2* X, const double* B, int N, long long rows, cudaStream_t st) {
  const int rg = kSpecThreads / std::min(N, kSpecThreads);
  int rpt = 8;
  while (rpt > 1 && ((size_t)rpt * rg * N * sizeof(double2) > kSpecRowSmem || rows < 152LL * rpt * rg)) rpt /= 2;
  switch (rpt) {
    case 8: return rows_launch<8>(X, B, N, rows, st);
    case 4: return rows_launch<4>(X, B, N, rows, st);
    case 2: return rows_launch<2>(X, B, N, rows, st);
    default: return rows_launch<1>(X, B, N, rows, st);
  }
}

// ------------------------------------------------------------------ the postselected solve
// |b|^2 and bhat = b / |b|; one block.
__global__ void __launch_bounds__(kSpecThreads) k_spec_prep(const double2* b, int N,
                                                            double* __restrict__ scal, double2* __restrict__ x) {
  dep_begin();
  double s[1] = {0.0}, nb2[1];
  for (int i = threadIdx.x; i < N; i += kSpecThreads) {
    const double2 z = b[i];
    s[0] += z.x * z.x + z.y * z.y;
  }
  block_sum_all(s, nb2);
  if (threadIdx.x == 0) scal[0] = nb2[0];
  const double scale = nb2[0] > 0.0 ? 1.0 / sqrt(nb2[0]) : 0.0;
  for (int i = threadIdx.x; i < N; i += kSpecThreads) x[i] = make_double2(b[i].x * scale, b[i].y * scale);
}

// y = B^T x, B N x N row-major: a block takes 8 outputs and splits the sum over its 32 groups of
// 8 threads, whose partial sums are added in a fixed order.
__global__ void __launch_bounds__(kSpecThreads) k_spec_matvec(const double* __restrict__ B, const double2* x,
                                                              int N, double2* __restrict__ y) {
  dep_begin();
  __shared__ double2 part[kSpecThreads / 32][8];
  const int o = blockIdx.x * 8 + (threadIdx.x & 7), p = threadIdx.x >> 3;
  double2 acc = make_double2(0.0, 0.0);
  if (o < N) {
#pragma unroll 4
    for (int m = p; m < N; m += 32) {
      const double v = B[(size_t)m * N + o];
      acc.x = fma(v, x[m].x, acc.x);
      acc.y = fma(v, x[m].y, acc.y);
    }
  }
#pragma unroll
  for (int off = 8; off < 32; off <<= 1) {
    acc.x += __shfl_xor_sync(0xffffffffu, acc.x, off);
    acc.y += __shfl_xor_sync(0xffffffffu, acc.y, off);
  }
  if ((threadIdx.x & 31) < 8) part[threadIdx.x >> 5][threadIdx.x & 7] = acc;
  __syncthreads();
  if (threadIdx.x < 8 && o < N) {
    double2 v = part[0][threadIdx.x];
#pragma unroll
    for (int w = 1; w < kSpecThreads / 32; ++w) v = cadd(v, part[w][threadIdx.x]);
    y[o] = v;
  }
}

// The clock trees, one column (eigenvector) per group of 2^nb threads: each thread owns one value of
// the lowest nb bits of y (at most kClockBits) and walks the bits above, an inner node per step of a
// depth-first search, so that a weight is one product of its path. Angles are 64-bit fractions
// of a half turn.
__global__ void __launch_bounds__(kClockThreads) k_spec_tree(const unsigned long long* __restrict__ frac,
                                                             const double* __restrict__ rot, int n_c, int N,
                                                             double2* __restrict__ beta, double2* __restrict__ wts) {
  dep_begin();
  __shared__ double red[4][3];
  const int nb = n_c < kClockBits ? n_c : kClockBits, lb = n_c - nb;
  const int tpc = 1 << nb, t = threadIdx.x & (tpc - 1);
  const int j = blockIdx.x * (kClockThreads >> nb) + (threadIdx.x >> nb);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const bool live = j < N;
  double g = 0.0, w1 = 0.0, sum = 0.0;
  if (live) {
    const unsigned long long f = frac[j];
    auto factors = [&](int m, unsigned low, double& c2, double& s2) {  // of bit m for the lower bits of y
      const unsigned long long a = (f << (n_c - 1 - m)) - ((unsigned long long)low << (63 - m));
      double s, c;
      sincospi((double)(long long)a * 5.4210108624275222e-20, &s, &c);
      c2 = c * c;
      s2 = s * s;
    };
    double p = 1.0, c2, s2;
    for (int m = 0; m < nb; ++m) {
      factors(m, (unsigned)t & ((1u << m) - 1u), c2, s2);
      p *= ((t >> m) & 1) ? s2 : c2;
    }
    // path[q]: the weight of the current prefix of nb + q bits; alt[q]: that of its sibling with
    // bit nb + q - 1 set. Leaves in the order of a counter whose top bit is the lowest bit above nb.
    double path[8], alt[8];
    path[0] = p;
    unsigned y = (unsigned)t;
    int q = 0;
    for (unsigned leaf = 0; leaf < (1u << lb); ++leaf) {
      for (; q < lb; ++q) {  // descend with zero bits
        factors(nb + q, y, c2, s2);
        alt[q + 1] = path[q] * s2;
        path[q + 1] = path[q] * c2;
      }
      const double r = rot[y], pr = path[lb] * r;
      g += pr;
      w1 = fma(pr, r, w1);
      sum += path[lb];
      while (q > 0 && (y >> (nb + q - 1)) & 1u) {  // climb out of finished siblings
        y &= ~(1u << (nb + q - 1));
        --q;
      }
      if (q > 0) {
        y |= 1u << (nb + q - 1);
        path[q] = alt[q];
      }
    }
  }
  const int span = tpc < 32 ? tpc : 32;
  for (int o = span >> 1; o > 0; o >>= 1) {
    g += __shfl_xor_sync(0xffffffffu, g, o);
    w1 += __shfl_xor_sync(0xffffffffu, w1, o);
    sum += __shfl_xor_sync(0xffffffffu, sum, o);
  }
  if (tpc > 32) {
    if (lane == 0) {
      red[warp][0] = g;
      red[warp][1] = w1;
      red[warp][2] = sum;
    }
    __syncthreads();
    const int w0 = warp & ~((tpc >> 5) - 1);
    g = w1 = sum = 0.0;
    for (int w = 0; w < (tpc >> 5); ++w) {
      g += red[w0 + w][0];
      w1 += red[w0 + w][1];
      sum += red[w0 + w][2];
    }
  }
  if (live && t == 0) {
    const double2 z = beta[j];
    const double m2 = z.x * z.x + z.y * z.y;
    wts[j] = make_double2(m2 * (sum - w1), m2 * w1);
    beta[j] = make_double2(z.x * g, z.y * g);
  }
}

// The measurement block and the dissipation rate (layout of hhl_measure_async /
// hhl_dissipation_async). Every block forms |v|^2 itself and writes its share of xhat; block 0 writes
// the scalars.
__global__ void __launch_bounds__(kSpecThreads) k_spec_finish(const double2* v, const double2* wts,
                                                              int N, double* __restrict__ scal, double inv_c_lam,
                                                              double wall_lo, double wall_hi, double nu_over_h,
                                                              double* __restrict__ out, double* __restrict__ eps) {
  dep_begin();
  const double scale = sqrt(scal[0]) * inv_c_lam;  // u = |b| Re(v) / (C lambda_ub)
  double s[4] = {0.0, 0.0, 0.0, 0.0}, tot[4];
  for (int i = threadIdx.x; i < N; i += kSpecThreads) {
    const double2 z = v[i];
    s[0] += z.x * z.x + z.y * z.y;
    if (blockIdx.x == 0) {
      s[1] += wts[i].x;
      s[2] += wts[i].y;
      const double left = i == 0 ? wall_lo : scale * v[i - 1].x, d = scale * z.x - left;
      s[3] += d * d;
      if (i == N - 1) {
        const double e = wall_hi - scale * z.x;
        s[3] += e * e;
      }
    }
  }
  block_sum_all(s, tot);
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    scal[1] = tot[1];
    scal[2] = tot[2];
    scal[3] = tot[0];
    out[0] = tot[0];
    out[1] = tot[2];
    out[2] = tot[1] + tot[2];
    out[3] = sqrt(scal[0]);
    if (eps != nullptr) eps[0] = nu_over_h * tot[3];
  }
  const double inv = tot[0] > 0.0 ? 1.0 / sqrt(tot[0]) : 0.0;
  for (int i = blockIdx.x * kSpecThreads + threadIdx.x; i < N; i += gridDim.x * kSpecThreads) {
    out[4 + 2 * i] = v[i].x * inv;
    out[5 + 2 * i] = v[i].y * inv;
  }
}

}  // namespace

hhl_status launch_spec_circuit(const Plan& p, void* state, cudaStream_t st) {
  const SpecState& s = *p.spec;
  const int N = (int)p.N;
  hhl_status r = spec_rows((double2*)state, s.basis, N, p.R, st);  // the anc = 0 half to the eigenbasis
  if (r == HHL_OK) r = launch_clock_spec(p, state, s.ph_lo, s.ph_hi, s.tw, st);
  if (r == HHL_OK) r = spec_rows((double2*)state, s.basis_t, N, 2 * p.R, st);  // both halves back
  return r;
}

hhl_status launch_spec_solve(const Plan& p, const double* b, double2* v_row, double* out, double* eps, cudaStream_t st) {
  const SpecState& s = *p.spec;
  const int N = (int)p.N;
  HHL_PROF_BEGIN(st);
  launch_dep(k_spec_prep, 1, kSpecThreads, 0, st, (const double2*)b, N, p.d_scal, s.x);
  HHL_LAUNCH_CHECK("k_spec_prep");
  HHL_PROF_BEGIN(st);
  launch_dep(k_spec_matvec, (N + 7) / 8, kSpecThreads, 0, st, s.basis, s.x, N, s.beta);
  HHL_LAUNCH_CHECK("k_spec_matvec");
  const int cols = kClockThreads >> std::min(p.n_c, kClockBits);
  HHL_PROF_BEGIN(st);
  launch_dep(k_spec_tree, (N + cols - 1) / cols, kClockThreads, 0, st, s.frac, s.sin_half, p.n_c, N, s.beta, s.wts);
  HHL_LAUNCH_CHECK("k_spec_tree");
  HHL_PROF_BEGIN(st);
  launch_dep(k_spec_matvec, (N + 7) / 8, kSpecThreads, 0, st, s.basis_t, s.beta, N, v_row);
  HHL_LAUNCH_CHECK("k_spec_matvec");
  HHL_PROF_BEGIN(st);
  launch_dep(k_spec_finish, std::max(1, std::min(16, N / kSpecThreads)), kSpecThreads, 0, st, 
      v_row, s.wts, N, p.d_scal, 1.0 / (p.C * p.lam_ub), p.wall_lo, p.wall_hi, p.nu * (double)(p.N + 1), out, eps);
  HHL_LAUNCH_CHECK("k_spec_finish");
  return HHL_OK;
}

void spec_free(Plan& p) {
  if (p.spec == nullptr) return;
  if (p.spec->mem) cudaFree(p.spec->mem);
  delete p.spec;
  p.spec = nullptr;
}

hhl_status spec_create(Plan& p, const std::vector<double>& lam, const std::vector<double>* vec, cudaStream_t st) {
  const size_t N = (size_t)p.N, R = (size_t)p.R, nh = R > 32 ? R / 32 : 1, mat = N * N;
  SpecState* s = new SpecState();
  p.spec = s;  // the plan's destructor frees what a failure below leaves
  // What the host computes comes first and is copied at once (in units of 8 bytes): the phase
  // fractions, sin(theta_y / 2), and V, V^T or the sine table.
  std::vector<double> host(N + R + (vec != nullptr ? 2 * mat : 2 * N + 2));
  unsigned long long* frac = reinterpret_cast<unsigned long long*>(host.data());
  double *sh = host.data() + N, *basis = sh + R;
  for (size_t j = 0; j < N; ++j) {
    double t = lam[j] / p.lam_ub * p.t0 / (2.0 * kPiS * (double)R);
    t -= floor(t);
    frac[j] = t < 1.0 ? (unsigned long long)(t * 18446744073709551616.0) : 0ULL;
  }
  for (size_t y = 0; y < R; ++y) sh[y] = sin(p.theta[y] / 2.0);
  if (vec != nullptr) {
    std::copy(vec->begin(), vec->end(), basis);
    for (size_t a = 0; a < N; ++a)
      for (size_t c = 0; c < N; ++c) basis[mat + c * N + a] = (*vec)[a * N + c];
  } else {
    const double w = sqrt(2.0 / (double)(N + 1));
    for (size_t q = 0; q < 2 * N + 2; ++q) basis[q] = w * sin((double)q * kPiS / (double)(N + 1));
  }
  const size_t host_units = (host.size() + 1) & ~(size_t)1;  // (complex tables from a 16-byte boundary)
  const size_t cplx = N * 32 + N * nh + R + 3 * N;
  const size_t bytes = (host_units + (vec != nullptr ? 0 : mat) + 2 * cplx) * sizeof(double);
  if (!alloc_optional(&s->mem, bytes, &p.table_bytes)) {
    spec_free(p);  // no room beside the operands: the plan runs its gate products
    return HHL_OK;
  }
  double* d = static_cast<double*>(s->mem);
  s->frac = reinterpret_cast<unsigned long long*>(d);
  s->sin_half = d + N;
  double2* z = reinterpret_cast<double2*>(d + host_units);
  s->ph_lo = z;
  s->ph_hi = s->ph_lo + N * 32;
  s->tw = s->ph_hi + N * nh;
  s->x = s->tw + R;
  s->beta = s->x + N;
  s->wts = s->beta + N;
  s->basis = vec != nullptr ? d + N + R : reinterpret_cast<double*>(s->wts + N);
  s->basis_t = vec != nullptr ? s->basis + mat : s->basis;  // (the sine basis is symmetric)
  HHL_CUDA_TRY(cudaMemcpyAsync(d, host.data(), host.size() * sizeof(double), cudaMemcpyHostToDevice, st));
  if (vec == nullptr) {
    HHL_PROF_BEGIN(st);
    k_spec_sine_basis<<<(unsigned)std::min<size_t>((mat + 255) / 256, 152 * 16), 256, 0, st>>>((int)N, d + N + R, s->basis);
    HHL_LAUNCH_CHECK("k_spec_sine_basis");
  }
  HHL_PROF_BEGIN(st);
  k_spec_phases<<<(unsigned)std::min<size_t>((N * (32 + nh) + R + 255) / 256, 152 * 16), 256, 0, st>>>(
      (int)N, (int)R, s->frac, s->ph_lo, s->ph_hi, s->tw);
  HHL_LAUNCH_CHECK("k_spec_phases");
  HHL_CUDA_TRY(cudaStreamSynchronize(st));  // the host copy goes out of scope
  return HHL_OK;
}

}  // namespace hhl
