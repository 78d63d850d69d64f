// k_bisp.cu - the bispectrum hot path (Sec. III.B of the paper).
//
//   counts     exact N_T (eq. NT) by integer enumeration of closed triangles,
//              one block per cubic-symmetry orbit of q_1 (48-element group),
//   export     F_0, F_2, F_4 on the shells (z-pass MODE 1, k_power.cu),
//   shot noise shell means of Re F_l F^w_0* and Re F_0 F^w_l* (z-pass MODE 2)
//              for the thin-shell form of eq. SNbisp2thin,
//   shell IFFT F_k^(l)(x) = sum_{q in shell} F_l(q) e^{+iq.x} (eq. F_k): z and
//              y passes over each shell's ball only (host-built work lists),
//              then a complex-to-real x pass,
//   contract   T^(l)(a,b,c) = sum_x F_a^(l) F_b^(0) F_c^(0) (eq. Factorize):
//              here the FP32 CUDA-core form with compensated accumulation, FP64
//              across x slices (the tensor-core form is in k_contract_tc.cu),
//   finalize   B^(l) = (2l+1) T^(l) / (N^3 N_T I_33) - N^(l) (eqs. BispMono,
//              BispQuad) on the host in FP64.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <map>
#include <mutex>
#include <vector>

#include "fkp_internal.h"

namespace fkp {

constexpr int kCTK = 64;     // x points per contraction chunk
constexpr int kCA = 16;      // outputs (values of a) per contraction thread

struct ContractItem {
  int ell_i, b, c, a0, na;
  int out[kCA];              // triangle index * nq + quantity, or -1
};

struct BispState {
  int S = 0, mm = 0, nsh2 = 0;
  int M = 0;                         // side of the grid that the triangle sums are formed on (sum_grid)
  FftPlan fp{};                      // transforms of length M
  std::vector<double> lo, hi, cen;
  std::vector<int> ta, tb, tc;       // triangle list
  std::vector<long long> nt;         // exact counts
  std::vector<unsigned char> cc;     // centre closed
  // CUDA graph of the device part of a call (catalogs and contraction it was
  // captured with; the previous call's, to capture on a repeat)
  cudaGraphExec_t graph_exec = nullptr;
  CatDev graph_key[2] = {}, last_key[2] = {};
  int graph_contraction = -1, last_contraction = -1;
  bool last_valid = false;
  int nl = 0;                        // number of multipoles computed (1..3)
  int nq = 3;                        // triangle sums per triangle: T0, T2, T4 (and T22 for FKP_B4B)
  bool zero_area = false;            // FKP_B4B: T22 = sum_x F_a^(2) F_b^(2) F_c^(0) (eq. Bhexa2)
  int ells[3] = {0, 2, 4};
  std::vector<ContractItem> items;
  int nslices = 1;
  long long slice_len = 0;
  // device
  float2* d_tw = nullptr;            // twiddles of length M
  signed char* d_slut = nullptr;
  float2* d_E = nullptr;
  float2* d_T1 = nullptr;
  float2* d_T2 = nullptr;
  float* d_I = nullptr;
  ContractItem* d_items = nullptr;
  double* d_cpart = nullptr;
  double* d_T = nullptr;
  double* d_spart = nullptr;
  int* d_spartc = nullptr;
  double* d_shell = nullptr;
  long long* d_shellc = nullptr;
  // tensor-core contraction: tiles of pairs (b >= c), groups of tiles, outputs -> partials
  int tc_groups = 0, tc_ncols = 0, tc_slices = 0, tc_chunks = 0;
  short2* d_pairs = nullptr;
  TcGroup* d_groups = nullptr;
  int* d_off = nullptr;
  float* d_tcpart = nullptr;
  // shell IFFT work lists: z tiles (s, n_y + mm, n_x0), y tiles (s, n_x0, |n_y| range); floor(r_s)
  int nzjobs = 0, nyjobs = 0;
  int4 *d_zjobs = nullptr, *d_yjobs = nullptr;
  int* d_kmax = nullptr;
  void* h_out = nullptr;             // host copy of d_T, d_shell, d_shellc (one allocation)
};

__device__ __forceinline__ int wrap_mode(int n, int N) { return n < 0 ? n + N : n; }

// ----------------------------------------------------------------------------
// exact triangle counts
// ----------------------------------------------------------------------------

// ball: packed n2 vectors with |n2| < hi_max sorted by |n2|^2 (shells are
// contiguous); shb: their shells.  reps: q1 orbit representatives
// (nx >= ny >= nz >= 0) with shell and orbit size.  For each rep and each n2
// in shells <= shell(q1), c = shell(|q1 + n2|); counts with c <= b add the
// orbit size to N_T(a, b, c).
__global__ void __launch_bounds__(256) k_counts(const int* __restrict__ ball, const signed char* __restrict__ shb,
                                                const int* __restrict__ upto, const int4* __restrict__ reps,
                                                const signed char* __restrict__ slut, int nsq, int S,
                                                unsigned long long* __restrict__ NT) {
  extern __shared__ int sh_counts[];  // [S][S]
  signed char* sl = reinterpret_cast<signed char*>(sh_counts + S * S);
  for (int t = threadIdx.x; t < S * S; t += blockDim.x) sh_counts[t] = 0;
  for (int t = threadIdx.x; t < nsq; t += blockDim.x) sl[t] = slut[t];
  __syncthreads();
  const int4 r = reps[blockIdx.x];
  const int a = r.w & 0xff, orbit = r.w >> 8;
  const int lim = upto[a];
  for (int i = threadIdx.x; i < lim; i += blockDim.x) {
    const int p = __ldg(ball + i);
    const int x = ((p >> 20) & 1023) - 512, y = ((p >> 10) & 1023) - 512, z = (p & 1023) - 512;
    const int sx = r.x + x, sy = r.y + y, sz = r.z + z;
    const int q = sx * sx + sy * sy + sz * sz;
    if (q < nsq) {
      const int c = sl[q];
      const int b = __ldg(shb + i);
      if (c >= 0 && c <= b) atomicAdd(sh_counts + b * S + c, 1);
    }
  }
  __syncthreads();
  for (int t = threadIdx.x; t < S * S; t += blockDim.x) {
    const int v = sh_counts[t];
    if (v) atomicAdd(NT + (size_t)a * S * S + t, (unsigned long long)v * (unsigned long long)orbit);
  }
}

// ----------------------------------------------------------------------------
// shell-filtered inverse FFTs (eq. F_k)
//
// F_k^(l)(x) = sum_{q in shell} F_l(q) e^{iq.x} is an unnormalised inverse
// DFT of F_l restricted to shell s, which is zero outside the ball |n| <= r_s
// (r_s^2 = the largest n^2 the shell holds).  The three passes visit only
// what that ball reaches, from work lists built with the plan:
//   z   per tile (s, n_y, 8 consecutive n_x) with n_x0^2 + n_y^2 <= r_s^2:
//       the 8 pencils along n_z, filled from E on the shell;  T1[s][z][n_y][n_x]
//   y   per tile (s, 8 consecutive n_x) with n_x0^2 <= r_s^2 and per z: the
//       8 pencils along n_y over |n_y| <= sqrt(r_s^2 - n_x0^2);  T2[s][z][y][n_x]
//   x   per pair of rows (s, z, y): complex-to-real along x from
//       n_x <= floor(r_s) (Hermitian extension), two real rows per complex
//       pencil;  I[s][z][y][x]
// Pencils are interleaved 8 to a block (element i of pencil p at i * 8 + p)
// (this form for sides without a compiled transform).
// ----------------------------------------------------------------------------

constexpr int kSP = 8;      // pencils per block
constexpr int kSNT = 256;   // threads per block: (kSP, 32)
static_assert(kSNT % kSP == 0, "a thread keeps its pencil across a pass");
constexpr int kSRL = 16;    // points per thread along a pencil (N <= 512)
constexpr int kXGap = 16;   // float2 of slack after each FFT buffer of the x shell pass

struct ShellParams {
  int N, mm, S, nsh2;
  const signed char* slut;
  const int* kmax;          // per shell: floor(r_s)
};

// One multipole's shell passes.
struct BispLaunch {
  ShellParams sp;
  FftPlan fp;
  const float2* tw;
  const float2* E;          // F_l on the ball |n| <= mm: [n_z + mm][n_y + mm][n_x]
  const int4* zjobs;
  int nz;
  const int4* yjobs;
  int ny;
  float2 *T1, *T2;
  float* I;                 // this multipole's S real shell fields
  int xblocks;
};

__global__ void __launch_bounds__(kSNT) k_shell_z(const float2* __restrict__ E, ShellParams sp, FftPlan fp,
                                                  const float2* __restrict__ twg, const int4* __restrict__ jobs,
                                                  float2* __restrict__ T1) {
  extern __shared__ float2 sm[];
  const int N = sp.N;
  float2* tw = sm;
  float2* A = sm + N;
  float2* B = A + kSP * N;
  const int tid = threadIdx.y * kSP + threadIdx.x;
  const int4 job = jobs[blockIdx.x];
  const int s = job.x, kyp = job.y, kx0 = job.z;
  const int mm = sp.mm, w2 = 2 * mm + 1, m1 = mm + 1, ny = kyp - mm;
  for (int i = tid; i < N; i += kSNT) tw[i] = twg[i];
  for (int i = tid; i < kSP * N; i += kSNT) A[i] = make_float2(0.f, 0.f);
  __syncthreads();
  for (int t = tid; t < w2 * kSP; t += kSNT) {
    const int kzp = t / kSP, c = t - kzp * kSP, kx = kx0 + c;
    if (kx < m1) {
      const int nz = kzp - mm;
      const int n2 = kx * kx + ny * ny + nz * nz;
      if (n2 < sp.nsh2 && sp.slut[n2] == s) A[wrap_mode(nz, N) * kSP + c] = E[((size_t)kzp * w2 + kyp) * m1 + kx];
    }
  }
  __syncthreads();
  const float2* R = fft_any<0, kSP, kSNT, 1>(A, B, fp, tw);
  const int c = threadIdx.x, run = threadIdx.y, rl = (N + 31) / 32;
  if (kx0 + c < m1) {
#pragma unroll
    for (int i = 0; i < kSRL; ++i) {
      const int z = i * 32 + run;
      if (i < rl && z < N) T1[(((size_t)s * N + z) * w2 + kyp) * m1 + kx0 + c] = R[z * kSP + c];
    }
  }
}

__global__ void __launch_bounds__(kSNT) k_shell_y(const float2* __restrict__ T1, ShellParams sp, FftPlan fp,
                                                  const float2* __restrict__ twg, const int4* __restrict__ jobs,
                                                  float2* __restrict__ T2) {
  extern __shared__ float2 sm[];
  const int N = sp.N;
  float2* tw = sm;
  float2* A = sm + N;
  float2* B = A + kSP * N;
  const int tid = threadIdx.y * kSP + threadIdx.x;
  const int4 job = jobs[blockIdx.x];
  const int s = job.x, kx0 = job.y, nyr = job.z, z = blockIdx.y;
  const int mm = sp.mm, w2 = 2 * mm + 1, m1 = mm + 1;
  for (int i = tid; i < N; i += kSNT) tw[i] = twg[i];
  for (int i = tid; i < kSP * N; i += kSNT) A[i] = make_float2(0.f, 0.f);
  __syncthreads();
  for (int t = tid; t < (2 * nyr + 1) * kSP; t += kSNT) {
    const int j = t / kSP, c = t - j * kSP, ny = j - nyr;
    if (kx0 + c < m1) A[wrap_mode(ny, N) * kSP + c] = T1[(((size_t)s * N + z) * w2 + ny + mm) * m1 + kx0 + c];
  }
  __syncthreads();
  const float2* R = fft_any<0, kSP, kSNT, 1>(A, B, fp, tw);
  const int c = threadIdx.x, run = threadIdx.y, rl = (N + 31) / 32;
  if (kx0 + c < m1) {
#pragma unroll
    for (int i = 0; i < kSRL; ++i) {
      const int y = i * 32 + run;
      if (i < rl && y < N) T2[(((size_t)s * N + z) * N + y) * m1 + kx0 + c] = R[y * kSP + c];
    }
  }
}

// Rows r = (s N + z) N + y; pencil p of a block iteration holds rows 2(g0+p)
// and 2(g0+p)+1 (same shell: N^2 is even) as x1 + i x2.
__global__ void __launch_bounds__(kSNT) k_shell_x(const float2* __restrict__ T2, ShellParams sp, FftPlan fp,
                                                  const float2* __restrict__ twg, float* __restrict__ I) {
  extern __shared__ float2 sm[];
  const int N = sp.N;
  float2* tw = sm;
  // A and B each followed by kXGap float2 of slack: the transposed rows
  // (stride N + 2 floats, so that the eight pencils' stores fall in distinct
  // banks) need 2 kSP (N + 2) floats of the free buffer
  float2* A = sm + N;
  float2* B = A + kSP * N + kXGap;
  // the next iteration's rows of T2: its 2 kSP rows are one contiguous span
  // (row 2 g0 with g0 a multiple of kSP = 8, so 16-byte aligned) fetched with
  // cp.async while this iteration transforms and stores
  float2* stg = B + kSP * N + kXGap;
  const int tid = threadIdx.y * kSP + threadIdx.x;
  const int m1 = sp.mm + 1;
  for (int i = tid; i < N; i += kSNT) tw[i] = twg[i];
  const long long pairs = (long long)sp.S * N * N / 2;
  auto stage = [&](long long gn) {
    if (gn < pairs) {
      const int npn = (int)(pairs - gn < kSP ? pairs - gn : kSP);
      const float2* src = T2 + 2 * gn * m1;
      for (int t = tid; t < npn * m1; t += kSNT)  // 16-byte chunks
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(stg + 2 * t)), "l"(src + 2 * t)
                     : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  stage((long long)blockIdx.x * kSP);
  for (long long g0 = (long long)blockIdx.x * kSP; g0 < pairs; g0 += (long long)gridDim.x * kSP) {
    const int np = (int)(pairs - g0 < kSP ? pairs - g0 : kSP);
    const int s = (int)((2 * g0) / ((long long)N * N));
    const int km = sp.kmax[s < sp.S ? s : sp.S - 1];
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();
    // p fastest: contiguous shared-memory stores, 32-byte row segments read.
    // A thread's pencil p = tid mod kSP is the same at every k; the shell (and
    // its reach kmp) is the iteration's unless the iteration straddles two
    // shells (N^2 not a multiple of 2 kSP)
    const int p = tid % kSP;
    const bool valid = p < np;
    int kmp = km;
    if (valid && (2 * g0 + 2 * np - 1) / ((long long)N * N) != s) {
      const int sp0 = (int)((2 * (g0 + p)) / ((long long)N * N));
      kmp = sp.kmax[sp0 < sp.S ? sp0 : sp.S - 1];
    }
    const float2* h0 = stg + (size_t)(2 * p) * m1;
    const float2* h1 = h0 + m1;
    for (int k = tid / kSP; k < N; k += kSNT / kSP) {
      float2 v = make_float2(0.f, 0.f);
      if (valid) {
        float2 x1 = make_float2(0.f, 0.f), x2 = x1;
        if (k == 0) {
          x1 = make_float2(h0[0].x, 0.f);
          x2 = make_float2(h1[0].x, 0.f);
        } else if (k <= kmp) {
          x1 = h0[k];
          x2 = h1[k];
        } else if (k >= N - kmp) {
          const float2 a = h0[N - k], b = h1[N - k];
          x1 = make_float2(a.x, -a.y);
          x2 = make_float2(b.x, -b.y);
        }
        v = make_float2(x1.x - x2.y, x1.y + x2.x);  // x1 + i x2
      }
      A[k * kSP + p] = v;
    }
    __syncthreads();
    stage(g0 + (long long)gridDim.x * kSP);
    const float2* R = fft_any<0, kSP, kSNT, 1>(A, B, fp, tw);
    // transpose through the free buffer into rows of stride N + 2 floats
    // (row 2p starts 20p banks further on: a warp's 8 pencils x 4 points hit
    // 32 distinct banks), then coalesced 8-byte stores (N even)
    float* rows = reinterpret_cast<float*>(R == A ? B : A);
    const int rs = N + 2;
    for (int t = tid; t < kSP * N; t += kSNT) {
      const int p = t % kSP, x = t / kSP;
      const float2 v = R[t];
      rows[(2 * p) * rs + x] = v.x;
      rows[(2 * p + 1) * rs + x] = v.y;
    }
    __syncthreads();
    const long long r0 = 2 * g0;
    const int hn = N / 2;
    float2* dst = reinterpret_cast<float2*>(I + r0 * N);
    for (int t = tid; t < 2 * np * hn; t += kSNT) {
      const int row = t / hn, x2 = t - row * hn;
      dst[t] = *reinterpret_cast<const float2*>(rows + row * rs + 2 * x2);
    }
  }
}

// The same three passes at compiled lengths, as N = R0 R1 in two stages with
// both radices in registers: the first stage takes its inputs where they lie
// (E, T1, the staged rows) and the second hands its outputs on (T1, T2, the
// transposed rows), so a transform crosses shared memory once instead of once
// per radix 8, 5, 3 stage and twice more for its fill and its result.  Those
// crossings and their barriers set the time of the staged form: 360^3, 37
// shells, per multipole z 0.55, y 1.64, x 3.81 ms; here the three together
// 6.0 -> 3.8 ms (with the F^w passes 20.4 -> 13.5 ms per mock).
// Block (8, kTY): threadIdx.x is the pencil, threadIdx.y the butterfly.
template <int N>
__global__ void __launch_bounds__(kSP * TwoStage<N>::kTY) k_shell_zc(const float2* __restrict__ E, ShellParams sp,
                                                                     const float2* __restrict__ twg,
                                                                     const int4* __restrict__ jobs,
                                                                     float2* __restrict__ T1) {
  using T = TwoStage<N>;
  __shared__ float2 tw[N], buf[kSP * N];
  const int c = threadIdx.x, j = threadIdx.y;
  for (int i = j * kSP + c; i < N; i += kSP * T::kTY) tw[i] = twg[i];
  const int4 job = jobs[blockIdx.x];
  const int s = job.x, kyp = job.y, kx = job.z + c;
  const int mm = sp.mm, w2 = 2 * mm + 1, m1 = mm + 1, ny = kyp - mm;
  if (j < T::R1) {
    float2 v[T::R0];
#pragma unroll
    for (int r = 0; r < T::R0; ++r) {
      const int i = j + r * T::R1, nz = i <= N / 2 ? i : i - N;
      const int n2 = kx * kx + ny * ny + nz * nz;
      v[r] = make_float2(0.f, 0.f);
      if (kx < m1 && n2 < sp.nsh2 && sp.slut[n2] == s) v[r] = __ldg(E + ((size_t)(nz + mm) * w2 + kyp) * m1 + kx);
    }
    two_stage_first<N, kSP, 1>(v, buf, c, j);
  }
  __syncthreads();
  if (j < T::R0) {
    float2 v[T::R1];
    two_stage_second<N, kSP, 1>(v, buf, tw, c, j);
    if (kx < m1) {
#pragma unroll
      for (int r = 0; r < T::R1; ++r) T1[(((size_t)s * N + j + r * T::R0) * w2 + kyp) * m1 + kx] = v[r];
    }
  }
}

template <int N>
__global__ void __launch_bounds__(kSP * TwoStage<N>::kTY) k_shell_yc(const float2* __restrict__ T1, ShellParams sp,
                                                                     const float2* __restrict__ twg,
                                                                     const int4* __restrict__ jobs,
                                                                     float2* __restrict__ T2) {
  using T = TwoStage<N>;
  __shared__ float2 tw[N], buf[kSP * N];
  const int c = threadIdx.x, j = threadIdx.y;
  for (int i = j * kSP + c; i < N; i += kSP * T::kTY) tw[i] = twg[i];
  const int4 job = jobs[blockIdx.x];
  const int s = job.x, kx = job.y + c, nyr = job.z, z = blockIdx.y;
  const int mm = sp.mm, w2 = 2 * mm + 1, m1 = mm + 1;
  if (j < T::R1) {
    const float2* src = T1 + (((size_t)s * N + z) * w2 + mm) * m1 + kx;
    float2 v[T::R0];
#pragma unroll
    for (int r = 0; r < T::R0; ++r) {
      const int i = j + r * T::R1, ny = i <= N / 2 ? i : i - N;
      v[r] = make_float2(0.f, 0.f);
      if (kx < m1 && ny <= nyr && ny >= -nyr) v[r] = __ldg(src + (long long)ny * m1);
    }
    two_stage_first<N, kSP, 1>(v, buf, c, j);
  }
  __syncthreads();
  if (j < T::R0) {
    float2 v[T::R1];
    two_stage_second<N, kSP, 1>(v, buf, tw, c, j);
    if (kx < m1) {
      float2* dst = T2 + (((size_t)s * N + z) * N + j) * m1 + kx;
#pragma unroll
      for (int r = 0; r < T::R1; ++r) dst[(size_t)(r * T::R0) * m1] = v[r];
    }
  }
}

template <int N>
__global__ void __launch_bounds__(kSP * TwoStage<N>::kTY) k_shell_xc(const float2* __restrict__ T2, ShellParams sp,
                                                                     const float2* __restrict__ twg,
                                                                     float* __restrict__ I) {
  using T = TwoStage<N>;
  constexpr int NT = kSP * T::kTY, rs = N + 2;
  extern __shared__ __align__(16) float2 sm[];
  float2* tw = sm;
  float2* buf = tw + N;
  float* rows = reinterpret_cast<float*>(buf + kSP * N);        // 2 kSP rows of stride N + 2 floats
  float2* stg = reinterpret_cast<float2*>(rows + 2 * kSP * rs);  // the next iteration's rows of T2
  const int p = threadIdx.x, j = threadIdx.y, tid = j * kSP + p;
  const int m1 = sp.mm + 1;
  for (int i = tid; i < N; i += NT) tw[i] = twg[i];
  const long long pairs = (long long)sp.S * N * N / 2;
  // 2 kSP rows of T2 are one contiguous span from row 2 g0 (g0 a multiple of 8: 16-byte aligned)
  auto stage = [&](long long gn) {
    if (gn < pairs) {
      const int npn = (int)(pairs - gn < kSP ? pairs - gn : kSP);
      const float2* src = T2 + 2 * gn * m1;
      for (int t = tid; t < npn * m1; t += NT)  // 16-byte chunks
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(stg + 2 * t)), "l"(src + 2 * t)
                     : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  stage((long long)blockIdx.x * kSP);
  for (long long g0 = (long long)blockIdx.x * kSP; g0 < pairs; g0 += (long long)gridDim.x * kSP) {
    const int np = (int)(pairs - g0 < kSP ? pairs - g0 : kSP);
    // the pencil's shell (an iteration may straddle two) and its reach
    const int s = (int)((2 * (g0 + p)) / ((long long)N * N));
    const int km = p < np ? sp.kmax[s < sp.S ? s : sp.S - 1] : -1;
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();
    if (j < T::R1) {
      const float2 *h0 = stg + (size_t)(2 * p) * m1, *h1 = h0 + m1;
      float2 v[T::R0];
#pragma unroll
      for (int r = 0; r < T::R0; ++r) {
        // x1 + i x2 of the Hermitian rows x1, x2: n_x and -n_x from the stored half
        const int i = j + r * T::R1, k = i <= N / 2 ? i : N - i;
        v[r] = make_float2(0.f, 0.f);
        if (k <= km) {
          float2 a = h0[k], b = h1[k];
          if (i == 0) a.y = b.y = 0.f;
          v[r] = i <= N / 2 ? make_float2(a.x - b.y, a.y + b.x) : make_float2(a.x + b.y, b.x - a.y);
        }
      }
      two_stage_first<N, kSP, 1>(v, buf, p, j);
    }
    __syncthreads();
    stage(g0 + (long long)gridDim.x * kSP);
    if (j < T::R0) {
      float2 v[T::R1];
      two_stage_second<N, kSP, 1>(v, buf, tw, p, j);
      // rows of stride N + 2 floats: a warp's 8 pencils x 4 points hit distinct banks
#pragma unroll
      for (int r = 0; r < T::R1; ++r) {
        rows[(2 * p) * rs + j + r * T::R0] = v[r].x;
        rows[(2 * p + 1) * rs + j + r * T::R0] = v[r].y;
      }
    }
    __syncthreads();
    float2* dst = reinterpret_cast<float2*>(I + 2 * g0 * N);
    for (int t = tid; t < 2 * np * (N / 2); t += NT) {
      const int row = t / (N / 2), x2 = t - row * (N / 2);
      dst[t] = *reinterpret_cast<const float2*>(rows + row * rs + 2 * x2);
    }
  }
}

template <int N>
static cudaError_t shell_passes_c(const BispLaunch& L, cudaStream_t s) {
  const dim3 blk(kSP, TwoStage<N>::kTY);
  cudaError_t e;
  if (L.nz > 0) k_shell_zc<N><<<L.nz, blk, 0, s>>>(L.E, L.sp, L.tw, L.zjobs, L.T1);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  if (L.ny > 0) k_shell_yc<N><<<dim3(L.ny, N), blk, 0, s>>>(L.T1, L.sp, L.tw, L.yjobs, L.T2);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  const size_t sm = sizeof(float2) * ((size_t)N * (1 + kSP) + 2 * kSP * (size_t)(L.sp.mm + 1)) +
                    sizeof(float) * 2 * kSP * (N + 2);
  if ((e = raise_smem_limit((const void*)k_shell_xc<N>, sm)) != cudaSuccess) return e;
  k_shell_xc<N><<<L.xblocks, blk, sm, s>>>(L.T2, L.sp, L.tw, L.I);
  return cudaGetLastError();
}

static cudaError_t shell_passes_n(const BispLaunch& L, cudaStream_t s) {
  const size_t sm = sizeof(float2) * (size_t)L.sp.N * (1 + 2 * kSP);
  cudaError_t e;
  if ((e = raise_smem_limit((const void*)k_shell_z, sm)) != cudaSuccess) return e;
  if ((e = raise_smem_limit((const void*)k_shell_y, sm)) != cudaSuccess) return e;
  const dim3 blk(kSP, kSNT / kSP);
  if (L.nz > 0) k_shell_z<<<L.nz, blk, sm, s>>>(L.E, L.sp, L.fp, L.tw, L.zjobs, L.T1);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  if (L.ny > 0) k_shell_y<<<dim3(L.ny, L.sp.N), blk, sm, s>>>(L.T1, L.sp, L.fp, L.tw, L.yjobs, L.T2);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  // + the slack after A and B, and the row staging
  const size_t smx = sm + sizeof(float2) * (2 * kXGap + 2 * kSP * (size_t)(L.sp.mm + 1));
  if ((e = raise_smem_limit((const void*)k_shell_x, smx)) != cudaSuccess) return e;
  k_shell_x<<<L.xblocks, blk, smx, s>>>(L.T2, L.sp, L.fp, L.tw, L.I);
  return cudaGetLastError();
}

static cudaError_t shell_passes(const BispLaunch& L, cudaStream_t s) {
  switch (L.sp.N) {
    case 512: return shell_passes_c<512>(L, s);
    case 384: return shell_passes_c<384>(L, s);
    case 360: return shell_passes_c<360>(L, s);
    case 256: return shell_passes_c<256>(L, s);
    case 192: return shell_passes_c<192>(L, s);
    case 128: return shell_passes_c<128>(L, s);
    case 64: return shell_passes_c<64>(L, s);
    default: return shell_passes_n(L, s);
  }
}

// ----------------------------------------------------------------------------
// triangle contraction, FP32 on CUDA cores
// ----------------------------------------------------------------------------

// blockIdx.x: item block (one item per thread), blockIdx.y: x slice.  The
// slice's fields are staged in shared memory kCTK points at a time, layout
// [x][field] with an odd row stride.  Each thread forms I_b I_c once per x
// and multiplies it into up to kCA values of a.  Chunk sums are FP32 and
// are added to compensated per-output accumulators.
__global__ void __launch_bounds__(256) k_contract_fp32(const float* __restrict__ I, long long N3, int nf, int S,
                                                       const ContractItem* __restrict__ items, int nitems,
                                                       long long slice_len, double* __restrict__ part, int nout) {
  extern __shared__ float ism[];
  const int stride = nf | 1;
  const int it = blockIdx.x * blockDim.x + threadIdx.x;
  ContractItem item;
  if (it < nitems) item = items[it];
  else { item.na = 0; item.b = 0; item.c = 0; item.a0 = 0; item.ell_i = 0; }
  const int base = item.ell_i * S + item.a0;
  float ks[kCA], kc[kCA];
#pragma unroll
  for (int i = 0; i < kCA; ++i) { ks[i] = 0.f; kc[i] = 0.f; }
  const long long x0 = (long long)blockIdx.y * slice_len;
  const long long x1 = (N3 < x0 + slice_len) ? N3 : x0 + slice_len;
  for (long long xc = x0; xc < x1; xc += kCTK) {
    const int nx = (int)(x1 - xc < kCTK ? x1 - xc : kCTK);
    __syncthreads();
    for (int t = threadIdx.x; t < nf * kCTK; t += blockDim.x) {
      const int f = t / kCTK, xl = t - f * kCTK;
      ism[xl * stride + f] = xl < nx ? __ldg(I + (size_t)f * N3 + xc + xl) : 0.f;
    }
    __syncthreads();
    if (item.na > 0) {
      float cs[kCA];
#pragma unroll
      for (int i = 0; i < kCA; ++i) cs[i] = 0.f;
      for (int xl = 0; xl < kCTK; ++xl) {
        const float* row = ism + xl * stride;
        const float p = row[item.b] * row[item.c];
#pragma unroll
        for (int i = 0; i < kCA; ++i)
          if (i < item.na) cs[i] = fmaf(row[base + i], p, cs[i]);
      }
#pragma unroll
      for (int i = 0; i < kCA; ++i) {
        const float y = cs[i] - kc[i];
        const float t = ks[i] + y;
        kc[i] = (t - ks[i]) - y;
        ks[i] = t;
      }
    }
  }
  if (it < nitems) {
#pragma unroll
    for (int i = 0; i < kCA; ++i)
      if (i < item.na && item.out[i] >= 0)
        part[(size_t)blockIdx.y * nout + item.out[i]] = (double)ks[i] - (double)kc[i];
  }
}

// Sums over the slices, a block 32 outputs: 16 threads each every sixteenth
// slice, then in a fixed order (one thread per output took 125 us for the 1,216
// slices of a 64^3 case, as long as the contraction).
__global__ void __launch_bounds__(512) k_reduce_slices(const double* __restrict__ part, int nslices, int nout,
                                                       double* __restrict__ out) {
  __shared__ double sh[16][33];
  const int o = blockIdx.x * 32 + threadIdx.x;
  double s = 0.0;
  if (o < nout) {
#pragma unroll 4
    for (int k = threadIdx.y; k < nslices; k += 16) s += part[(size_t)k * nout + o];
  }
  sh[threadIdx.y][threadIdx.x] = s;
  __syncthreads();
  if (threadIdx.y == 0 && o < nout) {
    for (int k = 1; k < 16; ++k) s += sh[k][threadIdx.x];
    out[o] = s;
  }
}

// ----------------------------------------------------------------------------
// host side
// ----------------------------------------------------------------------------

#define BCK(call)                                                                                   \
  do {                                                                                              \
    cudaError_t e_ = (call);                                                                        \
    if (e_ != cudaSuccess)                                                                          \
      return set_error(FKP_ECUDA, "%s:%d %s: %s", __FILE__, __LINE__, #call, cudaGetErrorString(e_)); \
  } while (0)

static int pack(int x, int y, int z) { return ((x + 512) << 20) | ((y + 512) << 10) | (z + 512); }

// Exact closed-triangle counts for shells lo_s <= |n| < hi_s (k_f units).
static int compute_counts(BispState& st, cudaStream_t s, std::vector<long long>& NT) {
  const int S = st.S;
  const double hmax = st.hi[S - 1];
  const int R = (int)std::ceil(hmax);
  struct Pt { int n2, x, y, z; };
  std::vector<Pt> ball;
  for (int x = -R; x <= R; ++x)
    for (int y = -R; y <= R; ++y)
      for (int z = -R; z <= R; ++z) {
        const int n2 = x * x + y * y + z * z;
        if (n2 > 0 && n2 < st.nsh2) ball.push_back({n2, x, y, z});
      }
  std::vector<signed char> slut(st.nsh2 > 0 ? st.nsh2 : 1, -1);
  for (int q = 1; q < st.nsh2; ++q)
    for (int k = 0; k < S; ++k)
      if (q >= st.lo[k] * st.lo[k] && q < st.hi[k] * st.hi[k]) { slut[q] = (signed char)k; break; }
  std::vector<Pt> pts;
  for (auto& p : ball) if (slut[p.n2] >= 0) pts.push_back(p);
  std::stable_sort(pts.begin(), pts.end(), [](const Pt& a, const Pt& b) { return a.n2 < b.n2; });
  std::vector<int> packed(pts.size());
  std::vector<signed char> shb(pts.size());
  std::vector<int> upto(S, 0);
  for (size_t i = 0; i < pts.size(); ++i) {
    packed[i] = pack(pts[i].x, pts[i].y, pts[i].z);
    shb[i] = slut[pts[i].n2];
  }
  for (int k = 0; k < S; ++k) {
    int c = 0;
    for (size_t i = 0; i < pts.size(); ++i) if (shb[i] <= k) c = (int)i + 1;
    upto[k] = c;
  }
  // orbit representatives x >= y >= z >= 0 and orbit sizes (signs x permutations)
  std::vector<int4> reps;
  for (int x = 0; x <= R; ++x)
    for (int y = 0; y <= x; ++y)
      for (int z = 0; z <= y; ++z) {
        const int n2 = x * x + y * y + z * z;
        if (n2 == 0 || n2 >= st.nsh2 || slut[n2] < 0) continue;
        const int nz = (x != 0) + (y != 0) + (z != 0);
        int perms = (x == y && y == z) ? 1 : ((x == y || y == z) ? 3 : 6);
        const int orbit = (1 << nz) * perms;
        reps.push_back(make_int4(x, y, z, (orbit << 8) | slut[n2]));
      }
  // the largest query |q1 + n2|^2 < (2 hmax)^2; entries past nsh2 are outside every shell
  const int nsq = st.nsh2;
  int *d_ball = nullptr, *d_upto = nullptr;
  signed char *d_shb = nullptr, *d_sl = nullptr;
  int4* d_reps = nullptr;
  unsigned long long* d_NT = nullptr;
  const size_t nt3 = (size_t)S * S * S;
  BCK(cudaMalloc(&d_ball, sizeof(int) * std::max<size_t>(1, packed.size())));
  BCK(cudaMalloc(&d_shb, std::max<size_t>(1, shb.size())));
  BCK(cudaMalloc(&d_upto, sizeof(int) * S));
  BCK(cudaMalloc(&d_reps, sizeof(int4) * std::max<size_t>(1, reps.size())));
  BCK(cudaMalloc(&d_sl, slut.size()));
  BCK(cudaMalloc(&d_NT, sizeof(unsigned long long) * nt3));
  BCK(cudaMemcpyAsync(d_ball, packed.data(), sizeof(int) * packed.size(), cudaMemcpyHostToDevice, s));
  BCK(cudaMemcpyAsync(d_shb, shb.data(), shb.size(), cudaMemcpyHostToDevice, s));
  BCK(cudaMemcpyAsync(d_upto, upto.data(), sizeof(int) * S, cudaMemcpyHostToDevice, s));
  BCK(cudaMemcpyAsync(d_reps, reps.data(), sizeof(int4) * reps.size(), cudaMemcpyHostToDevice, s));
  BCK(cudaMemcpyAsync(d_sl, slut.data(), slut.size(), cudaMemcpyHostToDevice, s));
  BCK(cudaMemsetAsync(d_NT, 0, sizeof(unsigned long long) * nt3, s));
  const size_t sm = sizeof(int) * S * S + slut.size();
  BCK(raise_smem_limit((const void*)k_counts, sm));
  if (!reps.empty()) k_counts<<<(unsigned)reps.size(), 256, sm, s>>>(d_ball, d_shb, d_upto, d_reps, d_sl, nsq, S, d_NT);
  BCK(cudaGetLastError());
  std::vector<unsigned long long> h(nt3);
  BCK(cudaMemcpyAsync(h.data(), d_NT, sizeof(unsigned long long) * nt3, cudaMemcpyDeviceToHost, s));
  BCK(cudaStreamSynchronize(s));
  cudaFree(d_ball); cudaFree(d_shb); cudaFree(d_upto); cudaFree(d_reps); cudaFree(d_sl); cudaFree(d_NT);
  NT.assign(nt3, 0);
  for (size_t i = 0; i < nt3; ++i) NT[i] = (long long)h[i];
  return FKP_OK;
}

// Exact counts depend on the shells only (the grid is large enough that
// n1 + n2 + n3 = 0 mod N means = 0), so they are cached per shell set.
static std::mutex g_count_mu;
static std::map<std::vector<int>, std::vector<long long>> g_count_cache;

// Side of the grid on which the triangle sums of shells with |n_a| <= mm are
// formed.  A product of three shell fields holds modes up to 3 mm per axis, so
// its sum over an M^3 grid with M > 3 mm is M^3 times its n = 0 mode, the sum
// over the closed triangles (eq. Factorize): the same on every such grid, up
// to the factor (N/M)^3 of a sum over N^3 nodes.  The smallest grid costs
// least (transforms and contraction go with M^3), but the operands' and
// transforms' random rounding averages over M^3 points only, so no grid is
// made smaller than 128^3, where the sums cost little.  A side with a compiled
// transform is taken up to 1.35 times the points of the smallest smooth side:
// the runtime-size passes take 2.4 times as long per point (27 shells x 3: 6.8 ms
// on 250^3, 3.0 on 256^3, beside 3.4 and 3.7 ms of contraction, so up to 1.6 times
// the points would pay there).  27 shells on 512^3: M = 256 (250 is the smallest),
// the whole mock 102 -> 18 ms; 37 shells on 360^3: M = 360 as before.
int sum_grid(int N, int mm) {
  auto smooth = [](int n) {
    for (int f : {2, 3, 5}) while (n % f == 0) n /= f;
    return n == 1;
  };
  int m = std::max(128, 3 * std::min(mm, N) + 1);
  while (m < N && ((m & 1) || !smooth(m))) ++m;
  m = std::min(m, N);
  for (int c : {128, 192, 256, 360, 384, 512})
    if (c >= m && c <= N && (double)c * c * c <= 1.35 * m * m * m) return c;
  return m;
}

int bisp_plan_init(Plan* P) {
  auto* st = new BispState();
  P->bisp = st;
  const fkp_bshells_t& bs = P->bs;
  if (bs.step < bs.width) return set_error(FKP_EINVAL, "bispectrum shells must not overlap (step >= width)");
  const int S = st->S = bs.nshells;
  const int N = P->g.N;
  for (int s = 0; s < S; ++s) {
    const double c = bs.first + (double)s * bs.step;
    st->cen.push_back(c);
    st->lo.push_back(c - 0.5 * bs.width);
    st->hi.push_back(c + 0.5 * bs.width);
  }
  const double hmax = st->hi[S - 1];
  st->nsh2 = (int)std::ceil(hmax * hmax);
  st->mm = (int)std::ceil(hmax) - 1;
  while ((double)(st->mm + 1) * (st->mm + 1) < hmax * hmax) ++st->mm;
  const int M = st->M = sum_grid(N, st->mm);
  if (!radix_plan(M, st->fp)) return set_error(FKP_EINVAL, "no radix plan for the sum grid M=%d", M);
  st->nl = 1;
  if (P->want & (FKP_B2 | FKP_B4B)) st->nl = 2;
  if (P->want & FKP_B4) st->nl = 3;
  st->zero_area = (P->want & FKP_B4B) != 0;
  st->nq = st->zero_area ? 4 : 3;
  if (st->nl > 1 && P->lmax < 2 * (st->nl - 1)) return set_error(FKP_EINVAL, "internal: lmax too small");

  cudaStream_t s0 = nullptr;
  std::vector<int> key = {bs.first, bs.step, bs.width, bs.nshells};
  std::vector<long long> NT;
  {
    std::lock_guard<std::mutex> lk(g_count_mu);
    auto itc = g_count_cache.find(key);
    if (itc != g_count_cache.end()) NT = itc->second;
  }
  if (NT.empty()) {
    int rc = compute_counts(*st, s0, NT);
    if (rc) return rc;
    std::lock_guard<std::mutex> lk(g_count_mu);
    g_count_cache[key] = NT;
  }
  for (int a = 0; a < S; ++a)
    for (int b = 0; b <= a; ++b)
      for (int c = 0; c <= b; ++c) {
        const long long n = NT[((size_t)a * S + b) * S + c];
        if (n <= 0) continue;
        st->ta.push_back(a);
        st->tb.push_back(b);
        st->tc.push_back(c);
        st->nt.push_back(n);
        st->cc.push_back(st->cen[b] + st->cen[c] >= st->cen[a] ? 1 : 0);
      }
  const int ntri = P->ntri = (int)st->ta.size();
  // contraction items: for each multipole and pair (b >= c), the values of a
  // with N_T > 0 in runs of kCA
  std::map<long long, int> tindex;
  for (int t = 0; t < ntri; ++t) tindex[((long long)st->ta[t] * S + st->tb[t]) * S + st->tc[t]] = t;
  // quantity q < nl: rows F^(2q)_a, second factor F^(0)_b; q = 3 (T22): rows
  // F^(2)_a, second factor F^(2)_b (field index S + b)
  const int nq = st->nq;
  std::vector<int> qs;
  for (int li = 0; li < st->nl; ++li) qs.push_back(li);
  if (st->zero_area) qs.push_back(3);
  for (int q : qs) {
    const int li = q == 3 ? 1 : q;
    for (int b = 0; b < S; ++b)
      for (int c = 0; c <= b; ++c) {
        int amin = -1, amax = -1;
        for (int a = b; a < S; ++a)
          if (tindex.count(((long long)a * S + b) * S + c)) { if (amin < 0) amin = a; amax = a; }
        if (amin < 0) continue;
        for (int a0 = amin; a0 <= amax; a0 += kCA) {
          ContractItem it;
          it.ell_i = li; it.b = q == 3 ? S + b : b; it.c = c; it.a0 = a0; it.na = std::min(kCA, amax - a0 + 1);
          for (int i = 0; i < kCA; ++i) {
            auto f = tindex.find(((long long)(a0 + i) * S + b) * S + c);
            it.out[i] = (i < it.na && f != tindex.end()) ? f->second * nq + q : -1;
          }
          st->items.push_back(it);
        }
      }
  }
  // tensor-core contraction: output (triangle t, quantity q) is a field row and
  // a pair of factors (field indices); quantities that are not computed have none
  std::vector<int> arow, orow;
  std::vector<short2> opair;
  const bool tc_ok = st->nl * S <= tc_rows();
  for (int t = 0; t < ntri && tc_ok; ++t)
    for (int q : qs) {
      arow.push_back((q == 3 ? S : q * S) + st->ta[t]);
      opair.push_back(make_short2((short)((q == 3 ? S : 0) + st->tb[t]), (short)st->tc[t]));
      orow.push_back(t * nq + q);
    }
  TcPlan tcp;
  if (!arow.empty()) tcp = tc_plan(S, st->nl, arow, opair);
  std::vector<int> off(std::max(1, ntri) * nq, -1);
  for (size_t o = 0; o < orow.size(); ++o) off[orow[o]] = tcp.off[o];
  st->tc_groups = (int)tcp.groups.size();
  st->tc_ncols = tcp.ncols;
  const long long N3 = (long long)st->M * st->M * st->M;
  tc_slicing(N3, std::max(1, st->tc_groups), P->ctx->nsm, &st->tc_slices, &st->tc_chunks);
  const int iblocks = std::max<int>(1, ((int)st->items.size() + 255) / 256);
  st->nslices = std::max(1, (P->ctx->nsm * 8) / iblocks);
  st->slice_len = ((N3 + st->nslices - 1) / st->nslices + kCTK - 1) / kCTK * kCTK;
  st->nslices = (int)((N3 + st->slice_len - 1) / st->slice_len);

  // shell LUT (n^2 -> shell), the same rule as the counts
  std::vector<signed char> slut(st->nsh2, -1);
  for (int q = 1; q < st->nsh2; ++q)
    for (int k = 0; k < S; ++k)
      if (q >= st->lo[k] * st->lo[k] && q < st->hi[k] * st->hi[k]) { slut[q] = (signed char)k; break; }

  const int mm = st->mm, w2 = 2 * mm + 1, m1 = mm + 1;
  // shell radii and the shell passes' work lists
  std::vector<int> r2max(S, -1), kmax(S, 0);
  for (int q = 1; q < st->nsh2; ++q)
    if (slut[q] >= 0) r2max[slut[q]] = q;
  std::vector<int4> zj, yj;
  for (int s = 0; s < S; ++s) {
    if (r2max[s] < 0) continue;
    int k = 0;
    while ((k + 1) * (k + 1) <= r2max[s]) ++k;
    kmax[s] = std::min(k, mm);
    for (int kyp = 0; kyp < w2; ++kyp) {
      const int ny = kyp - mm;
      for (int kx0 = 0; kx0 < m1; kx0 += 8)
        if (kx0 * kx0 + ny * ny <= r2max[s]) zj.push_back(make_int4(s, kyp, kx0, 0));
    }
    for (int kx0 = 0; kx0 < m1; kx0 += 8)
      if (kx0 * kx0 <= r2max[s]) {
        int nyr = 0;
        while ((nyr + 1) * (nyr + 1) + kx0 * kx0 <= r2max[s]) ++nyr;
        yj.push_back(make_int4(s, kx0, std::min(nyr, mm), 0));
      }
  }
  st->nzjobs = (int)zj.size();
  st->nyjobs = (int)yj.size();
  bool ok = true;
  auto A = [&](size_t bytes) { void* p = P->alloc(bytes); if (!p) ok = false; return p; };
  st->d_slut = (signed char*)A(st->nsh2);
  st->d_zjobs = (int4*)A(sizeof(int4) * std::max<size_t>(1, zj.size()));
  st->d_yjobs = (int4*)A(sizeof(int4) * std::max<size_t>(1, yj.size()));
  st->d_kmax = (int*)A(sizeof(int) * S);
  st->d_E = (float2*)A(sizeof(float2) * 3 * (size_t)w2 * w2 * m1);
  st->d_tw = (float2*)A(sizeof(float2) * M);
  st->d_T1 = (float2*)A(sizeof(float2) * (size_t)S * M * w2 * m1);
  st->d_T2 = (float2*)A(sizeof(float2) * (size_t)S * M * M * m1);
  st->d_I = (float*)A(sizeof(float) * (size_t)st->nl * S * N3);
  st->d_items = (ContractItem*)A(sizeof(ContractItem) * std::max<size_t>(1, st->items.size()));
  st->d_cpart = (double*)A(sizeof(double) * (size_t)st->nslices * std::max(1, ntri) * st->nq);
  st->d_T = (double*)A(sizeof(double) * (std::max(1, ntri) * st->nq + (BQ_N + 1) * S));
  st->d_shell = st->d_T ? st->d_T + std::max(1, ntri) * st->nq : nullptr;
  st->d_shellc = reinterpret_cast<long long*>(st->d_T ? st->d_shell + BQ_N * S : nullptr);
  st->d_spart = (double*)A(sizeof(double) * BQ_N * S * (size_t)P->nblk_z);
  st->d_spartc = (int*)A(sizeof(int) * S * (size_t)P->nblk_z);
  if (st->tc_groups > 0) {
    st->d_pairs = (short2*)A(sizeof(short2) * tcp.pairs.size());
    st->d_groups = (TcGroup*)A(sizeof(TcGroup) * tcp.groups.size());
    st->d_off = (int*)A(sizeof(int) * off.size());
    st->d_tcpart = (float*)A(sizeof(float) * (size_t)st->tc_slices * st->tc_ncols * 128);
  }
  if (!ok) return set_error(FKP_ENOMEM, "device allocation failed for the bispectrum workspace (%.2f GB in plan)",
                            P->bytes_total / 1e9);
  if (P->ctx->budget && P->bytes_total > P->ctx->budget)
    return set_error(FKP_ENOMEM, "plan needs %.2f GB, over the HBM budget", P->bytes_total / 1e9);
  std::vector<float2> tw(M);
  for (int m = 0; m < M; ++m) {
    const double a = 2.0 * M_PI * (double)m / (double)M;
    tw[m] = make_float2((float)std::cos(a), (float)-std::sin(a));
  }
  BCK(cudaMemcpy(st->d_tw, tw.data(), sizeof(float2) * M, cudaMemcpyHostToDevice));
  BCK(cudaMallocHost(&st->h_out, sizeof(double) * (std::max(1, ntri) * st->nq + (BQ_N + 1) * S)));
  BCK(cudaMemcpy(st->d_slut, slut.data(), st->nsh2, cudaMemcpyHostToDevice));
  if (!zj.empty()) BCK(cudaMemcpy(st->d_zjobs, zj.data(), sizeof(int4) * zj.size(), cudaMemcpyHostToDevice));
  if (!yj.empty()) BCK(cudaMemcpy(st->d_yjobs, yj.data(), sizeof(int4) * yj.size(), cudaMemcpyHostToDevice));
  BCK(cudaMemcpy(st->d_kmax, kmax.data(), sizeof(int) * S, cudaMemcpyHostToDevice));
  if (!st->items.empty())
    BCK(cudaMemcpy(st->d_items, st->items.data(), sizeof(ContractItem) * st->items.size(), cudaMemcpyHostToDevice));
  BCK(cudaMemset(st->d_cpart, 0, sizeof(double) * (size_t)st->nslices * std::max(1, ntri) * st->nq));
  if (st->d_pairs) {
    BCK(cudaMemcpy(st->d_pairs, tcp.pairs.data(), sizeof(short2) * tcp.pairs.size(), cudaMemcpyHostToDevice));
    BCK(cudaMemcpy(st->d_groups, tcp.groups.data(), sizeof(TcGroup) * tcp.groups.size(), cudaMemcpyHostToDevice));
    BCK(cudaMemcpy(st->d_off, off.data(), sizeof(int) * off.size(), cudaMemcpyHostToDevice));
  }
  return FKP_OK;
}

void bisp_plan_free(Plan* P) {
  bisp_drop_graph(P);
  if (P->bisp && static_cast<BispState*>(P->bisp)->h_out) cudaFreeHost(static_cast<BispState*>(P->bisp)->h_out);
  delete static_cast<BispState*>(P->bisp);
  P->bisp = nullptr;
}

void bisp_drop_graph(Plan* P) {
  auto* st = static_cast<BispState*>(P->bisp);
  if (!st) return;
  if (st->graph_exec) cudaGraphExecDestroy(st->graph_exec);
  st->graph_exec = nullptr;
}

}  // namespace fkp

using namespace fkp;

// Enqueues the device part of one bispectrum call (gridding, the F and F^w
// passes, the shell IFFTs, the contraction) on s.
static int enqueue_bisp(Plan* P, const CatDev& g, const CatDev& r, int contraction, cudaStream_t s) {
  auto* st = static_cast<BispState*>(P->bisp);
  const bool tensor = contraction == FKP_CONTRACT_BF16X3 || contraction == FKP_CONTRACT_BF16X6;
  int rc = enqueue_grids(P, g, r, s);
  if (rc) return rc;
  const int S = st->S, mm = st->mm, M = st->M;
  ZParams zp = zparams(P, 1);
  zp.nshells = S;
  zp.nsh2 = st->nsh2;
  zp.slut = st->d_slut;
  zp.E = st->d_E;
  zp.mm = mm;
  // F: P bins and export on the shells
  rc = enqueue_xy(P, P->d_grid, P->d_grid2, nullptr, s, P->reach, true);
  if (rc) return rc;
  const int nbz = zpass_blocks(P->reach, P->sched.z_threads, P->ctx->nsm);
  const int nbw = zpass_blocks(P->reach_w, P->sched.z_threads, P->ctx->nsm);
  BCK(launch_zpass(P->d_S2, P->g, P->mt, P->fp, P->d_tw, zp, P->reach, P->d_zpart, P->d_zpartc, P->d_err + 1, s,
                   P->ctx->nsm, P->sched.z_threads));
  BCK(launch_reduce_bins(P->d_zpart, P->d_zpartc, nbz, P->pb.nbins, P->d_bins, P->d_binc, s));
  BCK(record_stage(P->ev[5], s));
  // F^w: shell sums against the exported F_l
  rc = enqueue_xy(P, P->d_gridw, P->d_gridw2, nullptr, s, P->reach_w, false);
  if (rc) return rc;
  zp.mode = 2;
  BCK(launch_zpass(P->d_S2, P->g, P->mt, P->fp, P->d_tw, zp, P->reach_w, st->d_spart, st->d_spartc, P->d_err + 1, s,
                   P->ctx->nsm, P->sched.z_threads));
  BCK(launch_reduce_bins(st->d_spart, st->d_spartc, nbw, S, st->d_shell, st->d_shellc, s));
  BCK(record_stage(P->ev[6], s));
  // shell IFFTs, onto the grid of the triangle sums
  const long long N3 = (long long)M * M * M;
  {
    const size_t es = (size_t)(2 * mm + 1) * (2 * mm + 1) * (mm + 1);
    BispLaunch L;
    L.sp = ShellParams{M, mm, S, st->nsh2, st->d_slut, st->d_kmax};
    L.fp = st->fp;
    L.tw = st->d_tw;
    L.zjobs = st->d_zjobs;
    L.nz = st->nzjobs;
    L.yjobs = st->d_yjobs;
    L.ny = st->nyjobs;
    L.T1 = st->d_T1;
    L.T2 = st->d_T2;
    L.xblocks = P->ctx->nsm * 6;
    for (int li = 0; li < st->nl; ++li) {
      L.E = st->d_E + li * es;
      L.I = st->d_I + (size_t)li * S * N3;
      BCK(shell_passes(L, s));
    }
  }
  BCK(record_stage(P->ev[7], s));
  // contraction
  const int ntri = P->ntri, nout = std::max(1, ntri) * st->nq;
  if (tensor && st->d_pairs) {
    // The hi/lo split's dropped terms average over the points of the sum grid.
    // On one smaller than the plan's its T_4 was further from FP64 than sums over
    // N^3 points (400^3 -> 216^3, 22 shells: 1.9e-6 -> 2.4e-6; 300^3, 16 shells: 1.9e-6
    // -> 2.4e-6), so there it takes the six products of the 3-way split too (1.2e-6).
    const int nsplit = contraction == FKP_CONTRACT_BF16X3 && M == P->g.N ? 2 : 3;
    BCK(launch_contract_tc(st->d_I, N3, S, st->nl, st->d_groups, st->tc_groups, st->d_pairs, st->tc_ncols,
                           st->d_tcpart, P->d_err + 1, st->tc_slices, st->tc_chunks, nsplit, s));
    BCK(launch_tc_reduce(st->d_tcpart, st->tc_slices, st->tc_ncols, st->d_off, nout, st->d_T, s));
  } else if (!st->items.empty()) {
    const int nf = st->nl * S;
    const size_t smc = sizeof(float) * (size_t)kCTK * (nf | 1);
    BCK(raise_smem_limit((const void*)k_contract_fp32, smc));
    const int iblocks = ((int)st->items.size() + 255) / 256;
    k_contract_fp32<<<dim3(iblocks, st->nslices), 256, smc, s>>>(st->d_I, N3, nf, S, st->d_items,
                                                                 (int)st->items.size(), st->slice_len, st->d_cpart,
                                                                 nout);
    BCK(cudaGetLastError());
    k_reduce_slices<<<(nout + 31) / 32, dim3(32, 16), 0, s>>>(st->d_cpart, st->nslices, nout, st->d_T);
    BCK(cudaGetLastError());
  }
  BCK(record_stage(P->ev[8], s));
  return FKP_OK;
}

// Captures enqueue_bisp for these catalogs and contraction into the plan's
// bispectrum graph, on the plan's own capture stream.
static int capture_bisp(Plan* P, const CatDev& g, const CatDev& r, int contraction) {
  auto* st = static_cast<BispState*>(P->bisp);
  if (!P->cap_stream) BCK(cudaStreamCreateWithFlags(&P->cap_stream, cudaStreamNonBlocking));
  if (st->graph_exec) cudaGraphExecDestroy(st->graph_exec);
  st->graph_exec = nullptr;
  BCK(cudaStreamBeginCapture(P->cap_stream, cudaStreamCaptureModeThreadLocal));
  const int rc = enqueue_bisp(P, g, r, contraction, P->cap_stream);
  cudaGraph_t graph = nullptr;
  const cudaError_t e = cudaStreamEndCapture(P->cap_stream, &graph);
  if (rc || e != cudaSuccess || !graph) {
    if (graph) cudaGraphDestroy(graph);
    return rc ? rc : set_error(FKP_ECUDA, "bispectrum graph capture failed: %s", cudaGetErrorString(e));
  }
  const cudaError_t ei = cudaGraphInstantiate(&st->graph_exec, graph, 0);
  cudaGraphDestroy(graph);
  if (ei != cudaSuccess) {
    st->graph_exec = nullptr;
    return set_error(FKP_ECUDA, "bispectrum graph instantiation failed: %s", cudaGetErrorString(ei));
  }
  st->graph_key[0] = g;
  st->graph_key[1] = r;
  st->graph_contraction = contraction;
  return FKP_OK;
}

static bool same_cat_b(const CatDev& a, const CatDev& b) { return std::memcmp(&a, &b, sizeof(CatDev)) == 0; }

extern "C" int fkp_bispectrum(void* plan, const fkp_catalog_t* gal, const fkp_catalog_t* ran, int contraction,
                              void* stream, fkp_power_out* pout, fkp_bisp_out* bout) {
  auto* P = static_cast<Plan*>(plan);
  if (!P) return set_error(FKP_EINVAL, "NULL plan");
  if (!P->wantB || !P->bisp) return set_error(FKP_ESTATE, "plan was created without FKP_B* flags");
  if (contraction != FKP_CONTRACT_FP32 && contraction != FKP_CONTRACT_BF16X3 && contraction != FKP_CONTRACT_BF16X6)
    return set_error(FKP_EINVAL, "unknown contraction mode %d", contraction);
  auto* st = static_cast<BispState*>(P->bisp);
  const bool tensor = contraction == FKP_CONTRACT_BF16X3 || contraction == FKP_CONTRACT_BF16X6;
  if (tensor && !st->d_pairs && P->ntri > 0)
    return set_error(FKP_EINVAL, "the tensor-core contraction needs (multipoles x shells) <= %d rows", tc_rows());
  BCK(cudaSetDevice(P->ctx->device));
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  CatDev g, r;
  int rc = stage_catalog(P, gal, 0, g, s);
  if (rc) return rc;
  rc = randoms_of(P, ran, r, s);
  if (rc) return rc;
  const bool device_cats = (gal->on_device || gal->n == 0) && (!ran || ran->on_device || ran->n == 0);
  // CUDA graph of the device part: replayed when the catalogs and the
  // contraction are those it was captured with; captured on the second
  // identical call in a row (the same rule as the power path)
  bool replayed = false;
  if (P->graphs && device_cats) {
    const bool hit = st->graph_exec && same_cat_b(g, st->graph_key[0]) && same_cat_b(r, st->graph_key[1]) &&
                     st->graph_contraction == contraction;
    if (!hit && st->last_valid && same_cat_b(g, st->last_key[0]) && same_cat_b(r, st->last_key[1]) &&
        st->last_contraction == contraction) {
      if (capture_bisp(P, g, r, contraction) != FKP_OK) {
        cudaGetLastError();
        if (st->graph_exec) cudaGraphExecDestroy(st->graph_exec);
        st->graph_exec = nullptr;
      }
    }
    if (st->graph_exec && same_cat_b(g, st->graph_key[0]) && same_cat_b(r, st->graph_key[1]) &&
        st->graph_contraction == contraction) {
      BCK(cudaGraphLaunch(st->graph_exec, s));
      replayed = true;
    } else {
      st->last_key[0] = g;
      st->last_key[1] = r;
      st->last_contraction = contraction;
      st->last_valid = true;
    }
  }
  if (!replayed) {
    rc = enqueue_bisp(P, g, r, contraction, s);
    if (rc) return rc;
  }
  const int N = P->g.N, S = st->S;
  const long long N3 = (long long)N * N * N;
  const int ntri = P->ntri, nout = std::max(1, ntri) * st->nq;
  // triangle sums and shell sums back in one copy, read after finish_power's synchronization
  BCK(cudaMemcpyAsync(st->h_out, st->d_T, sizeof(double) * (nout + (BQ_N + 1) * S), cudaMemcpyDeviceToHost, s));
  const double *T = static_cast<const double*>(st->h_out), *sh = T + nout;
  const long long* shc = reinterpret_cast<const long long*>(sh + BQ_N * S);
  rc = finish_power(P, s, pout, true, 0, 0);
  if (rc) return rc;
  float t = 0.f;
  if (pout) {
    pout->graph = replayed ? 1 : 0;
    if (cudaEventElapsedTime(&t, P->ev[5], P->ev[7]) == cudaSuccess) pout->timing_ms[5] = t;  // F^w + shell IFFTs
    if (cudaEventElapsedTime(&t, P->ev[7], P->ev[8]) == cudaSuccess) pout->timing_ms[6] = t;
    if (cudaEventElapsedTime(&t, P->ev[0], P->ev[8]) == cudaSuccess) pout->timing_ms[7] = t;
  }
  // scalars for the finalize
  const double* hds = static_cast<const double*>(P->h_pinned) + (BQ_N + 1) * P->pb.nbins;
  const double I33 = hds[DS_I33], S3 = hds[DS_S3];
  if (!bout) return FKP_OK;
  bout->I33 = I33;
  bout->S3 = S3;
  auto L = [](int l, double mu) {
    return l == 0 ? 1.0 : (l == 2 ? 0.5 * (3 * mu * mu - 1) : (35 * mu * mu * mu * mu - 30 * mu * mu + 3) / 8.0);
  };
  const double N3d = (double)N3;
  const double toN = std::pow((double)N / (double)st->M, 3);  // the sums over M^3 nodes as sums over N^3
  for (int t = 0; t < ntri; ++t) {
    const int a = st->ta[t], b = st->tb[t], c = st->tc[t];
    if (bout->tri) { bout->tri[3 * t] = (int16_t)a; bout->tri[3 * t + 1] = (int16_t)b; bout->tri[3 * t + 2] = (int16_t)c; }
    if (bout->NT) bout->NT[t] = st->nt[t];
    if (bout->centre_closed) bout->centre_closed[t] = st->cc[t];
    const double ca = st->cen[a], cb = st->cen[b], cc = st->cen[c];
    const double mu12 = std::max(-1.0, std::min(1.0, (cc * cc - ca * ca - cb * cb) / (2 * ca * cb)));
    const double mu13 = std::max(-1.0, std::min(1.0, (cb * cb - ca * ca - cc * cc) / (2 * ca * cc)));
    for (int li = 0; li < 3; ++li) {
      const int l = 2 * li;
      double* Bp = li == 0 ? bout->B0 : (li == 1 ? bout->B2 : bout->B4);
      double* Np = li == 0 ? bout->N0 : (li == 1 ? bout->N2 : bout->N4);
      double* Tp = li == 0 ? bout->T0 : (li == 1 ? bout->T2 : bout->T4);
      if (li >= st->nl) {
        if (Bp) Bp[t] = std::nan("");
        if (Np) Np[t] = std::nan("");
        if (Tp) Tp[t] = std::nan("");
        continue;
      }
      // shell means: SQ_00 = <Re F0 Fw0*>, SQ_20/40 = <Re F_l Fw0*>, SQ_02/04 = <Re F0 Fw_l*>
      auto mean = [&](int q, int sI) { return shc[sI] > 0 ? sh[q * S + sI] / (double)shc[sI] : 0.0; };
      const int q1 = li == 0 ? SQ_00 : (li == 1 ? SQ_20 : SQ_40);
      const int q2 = li == 0 ? SQ_00 : (li == 1 ? SQ_02 : SQ_04);
      double noise = (2 * l + 1) / I33 * (mean(q1, a) + L(l, mu12) * mean(q2, b) + L(l, mu13) * mean(q2, c));
      if (l == 0) noise -= 2.0 * S3 / I33;
      const double Tv = toN * T[st->nq * t + li];
      if (Tp) Tp[t] = Tv;
      if (Np) Np[t] = noise;
      if (Bp) Bp[t] = (2 * l + 1) * Tv / (N3d * (double)st->nt[t] * I33) - noise;
    }
    // split hexadecapole (eq. Bhexa2) from the raw sums
    const double T22 = st->zero_area ? toN * T[st->nq * t + 3] : std::nan("");
    if (bout->T22) bout->T22[t] = T22;
    if (bout->B4b)
      bout->B4b[t] = st->zero_area ? (17.5 * T22 - toN * (5.0 * T[st->nq * t + 1] + 3.5 * T[st->nq * t])) /
                                         (N3d * (double)st->nt[t] * I33)
                                   : std::nan("");
  }
  return FKP_OK;
}
