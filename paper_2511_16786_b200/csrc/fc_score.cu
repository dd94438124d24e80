// fc_score_layer: Outlier KV Recognition Module (Sec. 3.2.1, Eq. 5-10) plus the
// energy sums of Eq. 11-12, for one layer.
//
// How the score is computed.  For one head, channel c, the complex sequence
// z[i] = K[i,c] + j V[i,c] carries both matrices through one transform (the DCT is a
// real linear map, so real and imaginary parts never mix).  The orthonormal DCT-II of
// Eq. 6-7 of a length-N sequence equals Re(exp(-j*pi*m/(2N)) * W[m]) * alpha[m], where W
// is the N-point DFT of the even/odd reordering  w[n] = z[2n], w[N-1-n] = z[2n+1].
// Low-pass filtering (Eq. 8) and the inverse DCT (Eq. 9) are linear, so the
// spectrum of the residual  z - z_base  in that DFT domain is, with P = W[q],
// Q = W[N-q], u = exp(j*pi*q/N):
//     E[q] = P - [q <= omega] (P + uQ)/2 - [N-q <= omega] (P - uQ)/2,   E[0] = 0,
// and the residual itself is the inverse DFT of E.  Dev[x] (Eq. 10) is then
// (1/d) * sum_c |residual|^2 with the real part belonging to K and the imaginary
// part to V; K and V are read exactly once and no Base KV is ever stored.
//
// The N-point DFT is done in three passes over an intermediate that stays in L2
// (N = N1*N2, n = n1*N2 + n2, q = k1 + N1*k2):
//   pass 1  for every n2: DFT over n1                      -> A[k1][n2]
//   pass 2  for every k1 (with N1-k1, which holds the partner bins N-q):
//           twiddle, DFT over n2, the filter above, inverse DFT over k2, twiddle -> B[k1][n2]
//   pass 3  for every n2: inverse DFT over k1, |.|^2 summed over the channels -> scores
// 16-bit sequences from 513 tokens on whose kept band fits a grid of a power of two points between a quarter and half of the
// tokens do not take these passes: they are scored on that grid between two banded matrix products (fc_band.cuh).
// Every other length up to 65536 takes the same three passes on a longer transform with the residual written as one
// padded convolution (fc_score_fast.cuh); the spectrum diagnostics run on the same passes.  The generic kernels of this
// file serve the power of two 131072, spectra of short powers of two and the entry point without allocation; there,
// lengths that are not a power of two (or are below 16) go through Bluestein's chirp convolution on a power-of-two
// length M >= 2N-1.
#include "fc_common.cuh"
#include "fc_score_fast.cuh"
#include "fc_band.h"
#include "fc_score_small.cuh"

#include <math.h>
#include <mutex>
#include <type_traits>
#include <unordered_map>
#include <vector>

namespace {

constexpr int kThreads = 256;

// ---------------------------------------------------------------------------
// index helpers
// ---------------------------------------------------------------------------
// Reordered index p -> token (w[n] = z[2n] for n < ceil(N/2), w[N-1-n] = z[2n+1]).
__device__ __forceinline__ int perm_token(int p, int N) {
  const int half = (N + 1) >> 1;
  return p < half ? 2 * p : 2 * (N - 1 - p) + 1;
}

using fast::chirp;

template <typename T> struct Elem;
template <> struct Elem<float> {
  static constexpr int VEC = 4;
  __device__ static void load(const float *p, float (&out)[4]) {
    const float4 v = *reinterpret_cast<const float4 *>(p);
    out[0] = v.x; out[1] = v.y; out[2] = v.z; out[3] = v.w;
  }
};
template <> struct Elem<__half> {
  static constexpr int VEC = 8;
  __device__ static void load(const __half *p, float (&out)[8]) {
    const uint4 v = *reinterpret_cast<const uint4 *>(p);
    const __half2 *h = reinterpret_cast<const __half2 *>(&v);
#pragma unroll
    for (int i = 0; i < 4; ++i) { const float2 f = __half22float2(h[i]); out[2 * i] = f.x; out[2 * i + 1] = f.y; }
  }
};
template <> struct Elem<__nv_bfloat16> {
  static constexpr int VEC = 8;
  __device__ static void load(const __nv_bfloat16 *p, float (&out)[8]) {
    const uint4 v = *reinterpret_cast<const uint4 *>(p);
    const __nv_bfloat162 *h = reinterpret_cast<const __nv_bfloat162 *>(&v);
#pragma unroll
    for (int i = 0; i < 4; ++i) { const float2 f = __bfloat1622float2(h[i]); out[2 * i] = f.x; out[2 * i + 1] = f.y; }
  }
};

// ---------------------------------------------------------------------------
// pass-1 loaders: value of transform input p for VEC consecutive workspace columns
// ---------------------------------------------------------------------------
// K/V rows of one sequence.  Column gc of the group maps to head h0 + gc/d, channel gc%d.
template <typename T, bool BLUE>
struct KvLoader {
  static constexpr int VEC = Elem<T>::VEC;
  const T *k, *v;          // already offset to the first token of the sequence
  long long stride_token, stride_head;
  int head0, head_dim, N;
  float accK, accV;        // running sums of squares (per thread)
  __device__ void init() { accK = 0.f; accV = 0.f; }
  __device__ void load(int p, int gc, float2 (&out)[VEC]) {
    if (BLUE && p >= N) {
#pragma unroll
      for (int i = 0; i < VEC; ++i) out[i] = make_float2(0.f, 0.f);
      return;
    }
    const int t = perm_token(p, N);
    const int h = head0 + gc / head_dim, c = gc % head_dim;
    const long long off = (long long)t * stride_token + (long long)h * stride_head + c;
    float a[VEC], b[VEC];
    Elem<T>::load(k + off, a);
    Elem<T>::load(v + off, b);
#pragma unroll
    for (int i = 0; i < VEC; ++i) { accK = fmaf(a[i], a[i], accK); accV = fmaf(b[i], b[i], accV); }
    if (BLUE) {
      const float2 ch = chirp(p, N);
#pragma unroll
      for (int i = 0; i < VEC; ++i) out[i] = cmul_conj(make_float2(a[i], b[i]), ch);
    } else {
#pragma unroll
      for (int i = 0; i < VEC; ++i) out[i] = make_float2(a[i], b[i]);
    }
  }
};

// Bluestein, second half: reads the N-point spectrum W[q][col], applies the
// low-pass residual filter, and feeds conj(E[q]) * conj(chirp) to the forward
// machinery (an inverse DFT is the conjugate of the forward DFT of the conjugate).
struct FilterLoader {
  static constexpr int VEC = 2;
  const float2 *spec;      // [N][ncol]
  int ncol, N, omega;
  __device__ void init() {}
  __device__ void load(int p, int gc, float2 (&out)[2]) {
    if (p >= N) { out[0] = out[1] = make_float2(0.f, 0.f); return; }
    const int q = p, qp = (N - q) % N;
    const float4 P4 = *reinterpret_cast<const float4 *>(spec + (size_t)q * ncol + gc);
    const float4 Q4 = *reinterpret_cast<const float4 *>(spec + (size_t)qp * ncol + gc);
    float s, c;
    sincospif(__fdiv_rn((float)q, (float)N), &s, &c);
    const float2 u = make_float2(c, s);
    const float inL = (q <= omega) ? 0.5f : 0.f;
    const float inH = (q != 0 && N - q <= omega) ? 0.5f : 0.f;
    const float2 ch = chirp(p, N);
    const float2 Pv[2] = {make_float2(P4.x, P4.y), make_float2(P4.z, P4.w)};
    const float2 Qv[2] = {make_float2(Q4.x, Q4.y), make_float2(Q4.z, Q4.w)};
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const float2 uQ = cmul(Qv[i], u);
      float2 E = Pv[i];
      E = csub(E, cscale(cadd(Pv[i], uQ), inL));
      E = csub(E, cscale(csub(Pv[i], uQ), inH));
      out[i] = cmul_conj(cconj(E), ch);
    }
  }
};

// Bluestein convolution kernel h[p] = chirp(|p|) wrapped to length M, in column 0.
struct ChirpKernelLoader {
  static constexpr int VEC = 2;
  int N, M;
  __device__ void init() {}
  __device__ void load(int p, int gc, float2 (&out)[2]) {
    out[0] = out[1] = make_float2(0.f, 0.f);
    if (gc != 0) return;
    if (p < N) out[0] = chirp(p, N);
    else if (p > M - N) out[0] = chirp(M - p, N);
  }
};

// ---------------------------------------------------------------------------
// pass 1: DFT over n1 for one n2 and one slice of cs columns
// grid (N2, ncol_ws/cs)
// ---------------------------------------------------------------------------
template <class Loader>
__global__ void __launch_bounds__(kThreads)
k_pass1(Loader ld, FftPlan plan, int N2, int ncol_ws, int cs_log2, float2 *__restrict__ ws,
        const float2 *__restrict__ master, int master_len, double *__restrict__ partial) {
  extern __shared__ float2 smem[];
  const int N1 = plan.len, cs = 1 << cs_log2;
  float2 *S = smem;
  float2 *tw = S + (size_t)N1 * cs;
  int *rev = reinterpret_cast<int *>(tw + N1);
  const int tid = threadIdx.x;
  const int n2 = blockIdx.x, gc0 = blockIdx.y * cs;

  for (int i = tid; i < N1; i += kThreads) {
    tw[i] = master[(size_t)i * (master_len / N1)];
    rev[i] = digit_rev(plan, i);
  }
  ld.init();
  constexpr int VEC = Loader::VEC;
  const int vec_per_row = cs / VEC;
  for (int it = tid; it < N1 * vec_per_row; it += kThreads) {
    const int row = it / vec_per_row, cv = it - row * vec_per_row;
    float2 vals[VEC];
    ld.load(row * N2 + n2, gc0 + cv * VEC, vals);
    float2 *dst = S + (size_t)row * cs + cv * VEC;
#pragma unroll
    for (int i = 0; i < VEC; i += 2)
      *reinterpret_cast<float4 *>(dst + i) = make_float4(vals[i].x, vals[i].y, vals[i + 1].x, vals[i + 1].y);
  }
  __syncthreads();
  fft_forward_tile(plan, S, cs_log2, tw, tid, kThreads);
  for (int w = tid; w < N1 * cs; w += kThreads) {
    const int pos = w >> cs_log2, c = w & (cs - 1);
    ws[((size_t)rev[pos] * N2 + n2) * ncol_ws + gc0 + c] = S[w];
  }
  if constexpr (!std::is_same<Loader, FilterLoader>::value && !std::is_same<Loader, ChirpKernelLoader>::value) {
    if (partial != nullptr) {
      __shared__ double red[2][kThreads / 32];
      double a = warp_sum_d((double)ld.accK), b = warp_sum_d((double)ld.accV);
      if ((tid & 31) == 0) { red[0][tid >> 5] = a; red[1][tid >> 5] = b; }
      __syncthreads();
      if (tid == 0) {
        double sa = 0, sb = 0;
        for (int i = 0; i < kThreads / 32; ++i) { sa += red[0][i]; sb += red[1][i]; }
        const size_t slot = (size_t)blockIdx.y * gridDim.x + blockIdx.x;
        partial[2 * slot] = sa;
        partial[2 * slot + 1] = sb;
      }
    }
  }
}

// ---------------------------------------------------------------------------
// pass 2: for one k1 (and its partner N1-k1): twiddle, DFT over n2, middle step,
// inverse DFT over k2, twiddle, scale.  In place in the workspace.
// MID_DCT   : low-pass residual filter between bins q and N-q   grid (N1/2+1, ncol_ws/cs2)
// MID_MULH  : pointwise product with the chirp spectrum          grid (N1, ncol_ws/cs2)
// MID_SPEC  : forward only; column 0 written to hhat[k]          grid (N1, 1)
// ---------------------------------------------------------------------------
enum { MID_DCT = 0, MID_MULH = 1, MID_SPEC = 2 };

template <int MID>
__global__ void __launch_bounds__(kThreads)
k_pass2(FftPlan plan, int N1, int ncol_ws, int cs2_log2, float2 *__restrict__ ws,
        const float2 *__restrict__ master, int master_len, int omega,
        float2 *__restrict__ hhat, float scale) {
  extern __shared__ float2 smem[];
  const int N2 = plan.len, cs2 = 1 << cs2_log2;
  const int Nfft = N1 * N2;
  const int tid = threadIdx.x;
  int k1a = blockIdx.x, k1b = blockIdx.x;
  int halves = 1;
  if (MID == MID_DCT) {
    k1b = (N1 - k1a) % N1;
    halves = (k1b != k1a) ? 2 : 1;
  }
  const int ncolT_log2 = cs2_log2 + (halves - 1);
  const int ncolT = 1 << ncolT_log2;
  const int gc0 = blockIdx.y * cs2;

  float2 *S = smem;                                    // [N2][2*cs2] for the paired rows of MID_DCT, else [N2][cs2]
  float2 *tw = S + (size_t)N2 * (MID == MID_DCT ? 2 : 1) * cs2;   // [N2]
  float2 *twN = tw + N2;                               // [2][N2]
  unsigned short *rev = reinterpret_cast<unsigned short *>(twN + 2 * N2);   // [N2]
  unsigned short *pos_of = rev + N2;                                       // [N2]

  const int mstepN = master_len / Nfft;
  for (int i = tid; i < N2; i += kThreads) {
    tw[i] = master[(size_t)i * (master_len / N2)];
    twN[i] = master[(size_t)(((long long)i * k1a) % Nfft) * mstepN];
    twN[N2 + i] = master[(size_t)(((long long)i * k1b) % Nfft) * mstepN];
    const int k = digit_rev(plan, i);
    rev[i] = (unsigned short)k;
    pos_of[k] = (unsigned short)i;
  }
  __syncthreads();

  // load with the forward inter-pass twiddle w_N^(n2*k1)
  for (int w = tid; w < N2 * ncolT; w += kThreads) {
    const int n2 = w >> ncolT_log2, col = w & (ncolT - 1);
    const int hf = col >> cs2_log2, c = col & (cs2 - 1);
    const int k1 = hf ? k1b : k1a;
    const float2 a = ws[((size_t)k1 * N2 + n2) * ncol_ws + gc0 + c];
    S[w] = cmul(a, twN[hf * N2 + n2]);
  }
  __syncthreads();
  fft_forward_tile(plan, S, ncolT_log2, tw, tid, kThreads);

  if (MID == MID_SPEC) {
    for (int pos = tid; pos < N2; pos += kThreads)
      hhat[k1a + N1 * (int)rev[pos]] = S[(size_t)pos << ncolT_log2];
    return;
  }
  if (MID == MID_MULH) {
    for (int w = tid; w < N2 * ncolT; w += kThreads) {
      const int pos = w >> ncolT_log2;
      S[w] = cmul(S[w], hhat[k1a + N1 * (int)rev[pos]]);
    }
  } else {
    // Every pair {q, N-q} is owned by the thread that meets the smaller bin.
    const int N = Nfft;
    const int ustep = master_len / (2 * N);
    for (int w = tid; w < N2 * ncolT; w += kThreads) {
      const int pos = w >> ncolT_log2, col = w & (ncolT - 1);
      const int hf = col >> cs2_log2, c = col & (cs2 - 1);
      const int k1 = hf ? k1b : k1a;
      const int q = k1 + N1 * (int)rev[pos];
      const int qp = (N - q) % N;
      if (q > qp) continue;
      const int k1p = qp % N1, k2p = qp / N1;
      const int hfp = (k1p == k1) ? hf : 1 - hf;
      const int wp = ((int)pos_of[k2p] << ncolT_log2) + (hfp << cs2_log2) + c;
      const float2 P = S[w], Q = S[wp];
      if (q == 0) { S[w] = make_float2(0.f, 0.f); continue; }
      const float2 u = cconj(master[(size_t)q * ustep]);           // exp(+j*pi*q/N)
      const float2 uQ = cmul(Q, u);
      const float inLq = (q <= omega) ? 0.5f : 0.f, inHq = (N - q <= omega) ? 0.5f : 0.f;
      float2 Eq = P;
      Eq = csub(Eq, cscale(cadd(P, uQ), inLq));
      Eq = csub(Eq, cscale(csub(P, uQ), inHq));
      S[w] = Eq;
      if (qp != q) {
        // bin N-q: u' = exp(j*pi*(N-q)/N) = -conj(u)
        const float2 upP = cscale(cmul_conj(P, u), -1.f);
        const float inLp = (qp <= omega) ? 0.5f : 0.f, inHp = (q <= omega) ? 0.5f : 0.f;
        float2 Ep = Q;
        Ep = csub(Ep, cscale(cadd(Q, upP), inLp));
        Ep = csub(Ep, cscale(csub(Q, upP), inHp));
        S[wp] = Ep;
      }
    }
  }
  __syncthreads();
  fft_inverse_tile(plan, S, ncolT_log2, tw, tid, kThreads);
  for (int w = tid; w < N2 * ncolT; w += kThreads) {
    const int n2 = w >> ncolT_log2, col = w & (ncolT - 1);
    const int hf = col >> cs2_log2, c = col & (cs2 - 1);
    const int k1 = hf ? k1b : k1a;
    const float2 r = cscale(cmul_conj(S[w], twN[hf * N2 + n2]), scale);
    ws[((size_t)k1 * N2 + n2) * ncol_ws + gc0 + c] = r;
  }
}

// ---------------------------------------------------------------------------
// pass 3: inverse DFT over k1 for one n2.
// EPI_SCORE : loops over the head's column slices, accumulates sum_c |.|^2 per row,
//             writes scores and the per-block outlier-energy partials.  grid (N2, heads)
// EPI_SPEC  : multiplies by conj(chirp) and stores rows p < N of the N-point
//             spectrum to spec[p][col] (Bluestein, first half).    grid (N2, ncol_ws/cs)
// ---------------------------------------------------------------------------
enum { EPI_SCORE = 0, EPI_SPEC = 1 };

template <int EPI, bool BLUE>
__global__ void __launch_bounds__(kThreads)
k_pass3(FftPlan plan, int N2, int N, int ncol_ws, int cs_log2, const float2 *__restrict__ ws,
        const float2 *__restrict__ master, int master_len,
        float2 *__restrict__ spec, float *__restrict__ scores, int head0, int head_dim,
        long long score_stride, float inv_scale, double *__restrict__ partial,
        float energy_scale, int accumulate) {
  // EPI_SCORE sums the head_dim columns starting at blockIdx.y * head_dim; when a head is
  // transformed in several column groups, head_dim is the group width, energy_scale the
  // true number of channels, and every group after the first adds to the stored score.
  extern __shared__ float2 smem[];
  const int N1 = plan.len, cs = 1 << cs_log2;
  float2 *S = smem;
  float2 *tw = S + (size_t)N1 * cs;
  int *rev = reinterpret_cast<int *>(tw + N1);
  float *accK = reinterpret_cast<float *>(rev + N1);
  float *accV = accK + N1;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int n2 = blockIdx.x;

  for (int i = tid; i < N1; i += kThreads) {
    tw[i] = master[(size_t)i * (master_len / N1)];
    rev[i] = digit_rev(plan, i);
    accK[i] = 0.f;
    accV[i] = 0.f;
  }
  __syncthreads();

  const int nslices = (EPI == EPI_SCORE) ? head_dim / cs : 1;
  for (int sl = 0; sl < nslices; ++sl) {
    const int gc0 = (EPI == EPI_SCORE) ? (blockIdx.y * head_dim + sl * cs) : blockIdx.y * cs;
    for (int w = tid; w < N1 * cs; w += kThreads) {
      const int pos = w >> cs_log2, c = w & (cs - 1);
      S[w] = ws[((size_t)rev[pos] * N2 + n2) * ncol_ws + gc0 + c];
    }
    __syncthreads();
    fft_inverse_tile(plan, S, cs_log2, tw, tid, kThreads);
    if (EPI == EPI_SPEC) {
      for (int w = tid; w < N1 * cs; w += kThreads) {
        const int n1 = w >> cs_log2, c = w & (cs - 1);
        const int p = n1 * N2 + n2;
        if (p < N) spec[(size_t)p * ncol_ws + gc0 + c] = cmul_conj(S[w], chirp(p, N));
      }
    } else {
      for (int n1 = warp; n1 < N1; n1 += kThreads / 32) {
        const int p = n1 * N2 + n2;
        float sk = 0.f, sv = 0.f;
        if (!BLUE || p < N) {
          float2 ch = make_float2(1.f, 0.f);
          if (BLUE) ch = chirp(p, N);
          for (int c = lane; c < cs; c += 32) {
            float2 e = S[((size_t)n1 << cs_log2) + c];
            if (BLUE) e = cmul_conj(e, ch);
            sk = fmaf(e.x, e.x, sk);
            sv = fmaf(e.y, e.y, sv);
          }
        }
        sk = warp_sum(sk);
        sv = warp_sum(sv);
        if (lane == 0) { accK[n1] += sk; accV[n1] += sv; }
      }
    }
    __syncthreads();
  }

  if (EPI == EPI_SCORE) {
    const int h = head0 + blockIdx.y;
    double dk = 0.0, dv = 0.0;
    for (int n1 = tid; n1 < N1; n1 += kThreads) {
      const int p = n1 * N2 + n2;
      if (p < N) {
        const float k = accK[n1] * inv_scale, v = accV[n1] * inv_scale;   // already divided by d
        float *dst = scores + (long long)h * score_stride + perm_token(p, N);
        *dst = accumulate ? *dst + (k + v) : k + v;
        dk += (double)k;
        dv += (double)v;
      }
    }
    __shared__ double red[2][kThreads / 32];
    dk = warp_sum_d(dk);
    dv = warp_sum_d(dv);
    if (lane == 0) { red[0][warp] = dk; red[1][warp] = dv; }
    __syncthreads();
    if (tid == 0) {
      double sa = 0, sb = 0;
      for (int i = 0; i < kThreads / 32; ++i) { sa += red[0][i]; sb += red[1][i]; }
      const size_t slot = (size_t)blockIdx.y * gridDim.x + blockIdx.x;
      partial[2 * slot] = sa * (double)energy_scale;      // d * sum Dev_k = outlier-band energy
      partial[2 * slot + 1] = sb * (double)energy_scale;
    }
  }
}

// Fixed-order reduction of the per-block partial sums of one sequence into
// energy[4] = (hiK, totK, hiV, totV).  One block.
__global__ void __launch_bounds__(256)
k_energy_finalize(const double *__restrict__ part_tot, int n_tot, const double *__restrict__ part_hi,
                  int n_hi, double *__restrict__ energy) {
  __shared__ double red[4][256];
  const int tid = threadIdx.x;
  double a0 = 0, a1 = 0, b0 = 0, b1 = 0;
  for (int i = tid; i < n_tot; i += 256) { a0 += part_tot[2 * i]; a1 += part_tot[2 * i + 1]; }
  for (int i = tid; i < n_hi; i += 256) { b0 += part_hi[2 * i]; b1 += part_hi[2 * i + 1]; }
  red[0][tid] = b0; red[1][tid] = a0; red[2][tid] = b1; red[3][tid] = a1;
  __syncthreads();
  for (int s = 128; s > 0; s >>= 1) {
    if (tid < s)
      for (int j = 0; j < 4; ++j) red[j][tid] += red[j][tid + s];
    __syncthreads();
  }
  if (tid < 4) energy[tid] = red[tid][0];
}

// ---------------------------------------------------------------------------
// Power spectrum of a layer (Eq. 11): P_k[m], P_v[m] = sum over heads and channels of C[m,c]^2.
// With z = k + j*v reordered as in pass 1 and Z its unnormalised N-point DFT, the spectra of the two
// real sequences are Y_k[q] = (Z[q] + conj(Z[N-q]))/2 and Y_v[q] = (Z[q] - conj(Z[N-q]))/(2j), and with
// w = exp(-j*pi*q/(2N)) * Y[q]:  C[q] = alpha[q]*Re(w),  C[N-q] = -alpha[N-q]*Im(w)  (alpha of Eq. 7).
// ---------------------------------------------------------------------------
// (P, Q) = (Z[q], Z[N-q]), t = exp(-j*pi*q/(2N)).  lo = (P_k[q], P_v[q]), hi = (P_k[N-q], P_v[N-q]).
__device__ __forceinline__ void power_of_pair(float2 P, float2 Q, float2 t, int q, float invN, float2 &lo, float2 &hi) {
  if (q == 0) {
    lo = make_float2(P.x * P.x * invN, P.y * P.y * invN);
    hi = lo;
    return;
  }
  const float2 yk = make_float2(0.5f * (P.x + Q.x), 0.5f * (P.y - Q.y));
  const float2 yv = make_float2(0.5f * (P.y + Q.y), 0.5f * (Q.x - P.x));
  const float2 wk = cmul(yk, t), wv = cmul(yv, t);
  const float a2 = 2.f * invN;
  lo = make_float2(a2 * wk.x * wk.x, a2 * wv.x * wv.x);
  hi = make_float2(a2 * wk.y * wk.y, a2 * wv.y * wv.y);
}

// Power-of-two N: pass 2 without the way back.  grid (N1/2 + 1, NY); block y works through the column
// slices y, y + NY, ... of the group and writes its sums over them to partial[y][q].
__global__ void __launch_bounds__(kThreads)
k_pass2_power(FftPlan plan, int N1, int ncol_ws, int cs2_log2, const float2 *__restrict__ ws,
              const float2 *__restrict__ master, int master_len, float2 *__restrict__ partial) {
  extern __shared__ float2 smem[];
  const int N2 = plan.len, cs2 = 1 << cs2_log2;
  const int N = N1 * N2;
  const int tid = threadIdx.x;
  const int k1a = blockIdx.x, k1b = (N1 - k1a) % N1;
  const int halves = (k1b != k1a) ? 2 : 1;
  const int ncolT_log2 = cs2_log2 + (halves - 1);
  const int ncolT = 1 << ncolT_log2;

  float2 *S = smem;                                    // [N2][2*cs2] at most
  float2 *tw = S + (size_t)N2 * 2 * cs2;               // [N2]
  float2 *twN = tw + N2;                               // [2][N2]
  unsigned short *rev = reinterpret_cast<unsigned short *>(twN + 2 * N2);   // [N2]
  unsigned short *pos_of = rev + N2;                                       // [N2]
  float2 *acc = reinterpret_cast<float2 *>(pos_of + N2);                   // [N2][2]: (P_k, P_v) of row (pos, half)

  const int mstepN = master_len / N;
  for (int i = tid; i < N2; i += kThreads) {
    tw[i] = master[(size_t)i * (master_len / N2)];
    twN[i] = master[(size_t)(((long long)i * k1a) % N) * mstepN];
    twN[N2 + i] = master[(size_t)(((long long)i * k1b) % N) * mstepN];
    const int k = digit_rev(plan, i);
    rev[i] = (unsigned short)k;
    pos_of[k] = (unsigned short)i;
    acc[2 * i] = make_float2(0.f, 0.f);
    acc[2 * i + 1] = make_float2(0.f, 0.f);
  }
  __syncthreads();

  const int tstep = master_len / (4 * N);
  const float invN = 1.f / (float)N;
  for (int sl = blockIdx.y; sl < ncol_ws / cs2; sl += gridDim.y) {
    const int gc0 = sl * cs2;
    for (int w = tid; w < N2 * ncolT; w += kThreads) {
      const int n2 = w >> ncolT_log2, col = w & (ncolT - 1);
      const int hf = col >> cs2_log2, c = col & (cs2 - 1);
      const int k1 = hf ? k1b : k1a;
      S[w] = cmul(ws[((size_t)k1 * N2 + n2) * ncol_ws + gc0 + c], twN[hf * N2 + n2]);
    }
    __syncthreads();
    fft_forward_tile(plan, S, ncolT_log2, tw, tid, kThreads);
    // every pair {q, N-q} is owned by the thread that meets the smaller bin; each location of S receives
    // the contribution of its own bin
    for (int w = tid; w < N2 * ncolT; w += kThreads) {
      const int pos = w >> ncolT_log2, col = w & (ncolT - 1);
      const int hf = col >> cs2_log2, c = col & (cs2 - 1);
      const int k1 = hf ? k1b : k1a;
      const int q = k1 + N1 * (int)rev[pos];
      const int qp = (N - q) % N;
      if (q > qp) continue;
      const int k1p = qp % N1, k2p = qp / N1;
      const int hfp = (k1p == k1) ? hf : 1 - hf;
      const int wp = ((int)pos_of[k2p] << ncolT_log2) + (hfp << cs2_log2) + c;
      float2 lo, hi;
      power_of_pair(S[w], S[wp], master[(size_t)q * tstep], q, invN, lo, hi);
      S[w] = lo;
      if (qp != q) S[wp] = hi;
    }
    __syncthreads();
    for (int r = tid; r < N2 * halves; r += kThreads) {      // row r = (pos, half): sum its cs2 columns in order
      const int pos = r / halves, hf = r - pos * halves;
      const float2 *row = S + ((size_t)pos << ncolT_log2) + (hf << cs2_log2);
      float2 a = acc[2 * pos + hf];
      for (int c = 0; c < cs2; ++c) { a.x += row[c].x; a.y += row[c].y; }
      acc[2 * pos + hf] = a;
    }
    __syncthreads();
  }
  for (int r = tid; r < N2 * halves; r += kThreads) {
    const int pos = r / halves, hf = r - pos * halves;
    const int q = (hf ? k1b : k1a) + N1 * (int)rev[pos];
    partial[(size_t)blockIdx.y * N + q] = acc[2 * pos + hf];
  }
}

// Chirp convolutions: from the N-point spectrum spec[q][col].  grid (N/2 + 1): block q sums the pair
// {q, N-q} over all columns of the group and writes partial[q], partial[N-q].
__global__ void __launch_bounds__(kThreads)
k_spec_power(const float2 *__restrict__ spec, int ncol, int N, float2 *__restrict__ partial) {
  const int q = blockIdx.x, qp = (N - q) % N;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  float s, c;
  sincospif(-__fdiv_rn((float)q, (float)(2 * N)), &s, &c);
  const float2 t = make_float2(c, s);
  const float invN = 1.f / (float)N;
  float a[4] = {0.f, 0.f, 0.f, 0.f};
  for (int col = tid; col < ncol; col += kThreads) {
    float2 lo, hi;
    power_of_pair(spec[(size_t)q * ncol + col], spec[(size_t)qp * ncol + col], t, q, invN, lo, hi);
    a[0] += lo.x; a[1] += lo.y; a[2] += hi.x; a[3] += hi.y;
  }
  __shared__ float red[4][kThreads / 32];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    a[i] = warp_sum(a[i]);
    if (lane == 0) red[i][warp] = a[i];
  }
  __syncthreads();
  if (tid == 0) {
    float r[4] = {0.f, 0.f, 0.f, 0.f};
    for (int w = 0; w < kThreads / 32; ++w)
      for (int i = 0; i < 4; ++i) r[i] += red[i][w];
    partial[q] = make_float2(r[0], r[1]);
    if (qp != q) partial[qp] = make_float2(r[2], r[3]);
  }
}

// spectrum[m] (+)= sum over y of partial[y][m], in fp64 and in a fixed order.  The partial sums of the direct form are in
// the order [k1][k2] of pass 2, bin k1 + N1*k2; N1 == 1: in the order of the bins.
__global__ void k_power_accumulate(const float2 *__restrict__ partial, int ny, int N, int N1, double *__restrict__ spectrum,
                                   int first) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= N) return;
  const int N2 = N / N1, m = N1 == 1 ? i : i / N2 + N1 * (i % N2);
  double a = first ? 0.0 : spectrum[2 * m], b = first ? 0.0 : spectrum[2 * m + 1];
#pragma unroll 4
  for (int y = 0; y < ny; ++y) {
    const float2 p = __ldcs(partial + (size_t)y * N + i);
    a += (double)p.x;
    b += (double)p.y;
  }
  spectrum[2 * m] = a;
  spectrum[2 * m + 1] = b;
}

// energy[l*stride .. +3] = 0 for the n layers of an empty sequence
__global__ void k_zero_energy(double *energy, int n, long long stride) {
  if ((int)threadIdx.x < 4 * n) energy[(threadIdx.x >> 2) * stride + (threadIdx.x & 3)] = 0.0;
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
inline int ilog2(int x) { int b = 0; while ((1 << b) < x) ++b; return b; }
inline bool is_pow2(int x) { return x > 0 && (x & (x - 1)) == 0; }
inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

// ---- generic kernels: the power of two 131072, spectra of powers of two below 1024, the no-allocation entry point ----
struct SeqPlan {
  bool bluestein;
  int N, Nfft, N1, N2;
  int cs, cs2;               // columns per tile in pass 1/3 and pass 2
};

SeqPlan plan_sequence(int N) {
  SeqPlan s;
  s.N = N;
  s.bluestein = !(is_pow2(N) && N >= 16);
  s.Nfft = N;
  if (s.bluestein) {
    s.Nfft = 64;
    while (s.Nfft < 2 * N - 1) s.Nfft <<= 1;
  }
  const int bits = ilog2(s.Nfft);
  int b1 = bits / 2;
  if (b1 > 7) b1 = 7;
  s.cs = 64;
  // 131072 points: 256 x 512 with 32-column tiles in passes 1 and 3 beats 128 x 1024, whose pass 2 has
  // room for only 4 columns per block
  if (bits == 17) { b1 = 8; s.cs = 32; }
  s.N1 = 1 << b1;
  s.N2 = s.Nfft / s.N1;
  int cs2 = 4096 / s.N2;      // 2*N2*cs2*8 bytes = 64 KiB
  if (cs2 > 64) cs2 = 64;
  if (cs2 < 4) cs2 = 4;
  s.cs2 = cs2;
  return s;
}

struct GenericLayout {
  size_t off_ws, off_spec, off_hhat, off_hcol, off_part_tot, off_part_hi, total;
  int heads_per_group;
  int sub_cols;              // chirp form: columns of one head transformed together (head_dim = all of them)
};

// Workspace carve-up for one sequence (all sequences share the regions; the query takes the maximum over the view).
GenericLayout generic_layout(const fc_handle *h, const SeqPlan &sp, int num_heads, int head_dim) {
  GenericLayout L;
  const size_t per_head = (size_t)sp.Nfft * head_dim * sizeof(float2);
  int hg = (int)(h->group_bytes / per_head);
  if (hg < 1) hg = 1;
  if (hg > num_heads) hg = num_heads;
  const int groups = (num_heads + hg - 1) / hg;
  hg = (num_heads + groups - 1) / groups;                      // balanced groups
  L.heads_per_group = hg;
  // A single head whose intermediates pass four times the budget is split into column groups: a workspace saving
  // (narrower tiles cost 2..8 % of the time).
  int sub = head_dim;
  const size_t split_above = h->group_bytes > ((size_t)1 << 60) ? h->group_bytes : 4 * h->group_bytes;
  if (sp.bluestein && hg == 1)
    while (sub % 64 == 0 && (size_t)sp.Nfft * sub * sizeof(float2) > split_above) sub /= 2;
  L.sub_cols = sub;
  size_t off = 0;
  L.off_ws = off;       off += align_up((size_t)sp.Nfft * sub * hg * sizeof(float2), 256);
  L.off_spec = off;     off += sp.bluestein ? align_up((size_t)sp.N * sub * hg * sizeof(float2), 256) : 0;
  L.off_hhat = off;     off += sp.bluestein ? align_up((size_t)sp.Nfft * sizeof(float2), 256) : 0;
  L.off_hcol = off;     off += sp.bluestein ? align_up((size_t)sp.Nfft * 8 * sizeof(float2), 256) : 0;
  const size_t slices = (size_t)num_heads * head_dim / 32;   // finest slicing any kernel variant uses
  L.off_part_tot = off; off += align_up(slices * sp.N2 * 2 * sizeof(double), 256);
  L.off_part_hi = off;  off += align_up((size_t)num_heads * (head_dim / sub) * sp.N2 * 2 * sizeof(double), 256);
  L.total = off;
  return L;
}

// ---- the specialised passes (fc_score_fast.cuh) ----
struct PassPlan {
  bool ok;                   // false: the length is left to the generic kernels
  bool small;                // one kernel does it all (fc_score_small.cuh); only pad, N and M are set besides
  bool pad;                  // padded form (else direct: M == N)
  int N, M, N1, N2;
  int a, r1b, r2b;           // N1 = a * r1b, N2 = 16 * r2b (32 * r2b with dbl)
  bool dbl;                  // pass 2 takes its rows in two halves
  int cpw, cp;               // channel pairs per block of passes 1 and 3, per row tile of pass 2
};

// Shapes of the padded form: M = 2^k * {1, 5/4, 3/2, 7/4} from 1024 to 131072 (27 lengths, so that 2N-1 is padded by
// 1.12 on average).  a = 10 and 12 with rows of 128 or 256 points run 3..10 % faster on a radix-8 second stage
// (80 or 96 x N2) than on 160 or 192 x N2/2; a = 14 loses 8 % that way, and rows of 512 points lose 14 % against 160 or
// 192 x 256.
inline PassPlan pad_shape(int M) {
  PassPlan p = {};
  p.pad = true;
  p.M = M;
  p.a = is_pow2(M) ? 16 : (M % 5 == 0) ? 10 : (M % 3 == 0) ? 12 : 14;
  if (p.a == 16) {
    if (M < 1024 || M > 131072) return p;
    const int bits = ilog2(M), b1 = bits / 2 > 8 ? 8 : bits / 2;
    p.r1b = (1 << b1) / 16;
  } else {
    const int rest = M / p.a;                    // r1b * N2
    if (M % (128 * p.a) != 0 || !is_pow2(rest)) return p;
    if (rest <= 512) p.r1b = rest / 32;          // rows of 32 points
    else if (p.a != 14 && (rest == 1024 || rest == 2048)) p.r1b = 8;
    else p.r1b = 16;
  }
  p.N1 = p.a * p.r1b;
  p.N2 = M / p.N1;
  if (p.N2 < 32 || p.N2 > 512 || p.r1b < 2) return p;
  p.dbl = p.N2 == 512;
  p.r2b = p.dbl ? 16 : p.N2 / 16;
  // radix-16 second stage and rows of 128 points or more: 16 pairs (256-thread blocks, two or three per SM) instead of
  // 32 (512 threads, one per SM), 10..14 % on transforms of 57344..98304 points; shorter rows lose 4 % that way
  p.cpw = (p.r1b == 16 && p.N2 >= 128) ? 16 : 32;
  // 256-thread blocks in pass 2
  p.cp = p.dbl ? 4 : p.r2b == 16 ? 8 : p.r2b == 8 ? 16 : 32;
  p.ok = true;
  return p;
}

// The smallest padded length >= 2N - 1, N <= 65536.
PassPlan plan_padded(int N) {
  int best = 0;
  const int need = 2 * N - 1;
  for (int k = 10; k <= 17; ++k)
    for (int f = 4; f <= 7; ++f) {
      const int M = (1 << k) / 4 * f;
      if (M >= need && (best == 0 || M < best) && pad_shape(M).ok) best = M;
    }
  PassPlan p = pad_shape(best);
  p.N = N;
  return p;
}

// Channel pairs per block of the small kernel for M points.
constexpr int small_cp(int M) { return M <= 128 ? 32 : 4096 / M; }

// How a sequence of N tokens and head_dim channels is transformed (head_dim 0: the three passes wherever they apply).
PassPlan plan_passes(int N, int head_dim) {
  PassPlan p = {};
  // one kernel where a cluster of at most 16 blocks holds a head
  if (N <= 1024 && head_dim > 0) {
    int M = 64;
    const bool pad = !(is_pow2(N) && N >= 64);
    while (M < (pad ? 2 * N - 1 : N)) M <<= 1;
    if (M <= 1024) {
      const int width = 2 * small_cp(M), blocks = head_dim / width;
      if (head_dim % width == 0 && is_pow2(blocks) && blocks <= 16) {
        p.ok = p.small = true;
        p.pad = pad;
        p.N = N;
        p.M = M;
        return p;
      }
    }
  }
  if (is_pow2(N) && N >= 1024) {
    if (N > 65536) return p;
    const int bits = ilog2(N);
    // 8192 points: 128 x 64 keeps every pass at 256-thread blocks (2 % over 64 x 128)
    const int b1 = bits == 13 ? 7 : bits / 2;
    p.N = p.M = N;
    p.a = 16;
    p.r1b = (1 << b1) / 16;
    p.N1 = 1 << b1;
    p.N2 = N / p.N1;
    p.r2b = p.N2 / 16;
    // every pass runs 256-thread blocks from 8192 points on, the measured optimum
    p.cpw = p.N1 == 256 ? 16 : 32;
    p.cp = (N == 8192) ? 32 : (N == 16384) ? 16 : 8;
    p.ok = true;
    return p;
  }
  return N > 65536 ? p : plan_padded(N);
}

// How one sequence's units (layer, head) are grouped into launches.
struct GroupPlan {
  int units;                 // units per launch
  int sub, ngr;              // columns of a unit per launch and launches per unit (ngr > 1 only with units == 1)
  size_t buf_bytes;          // intermediates of one launch (one copy per internal stream)
  size_t layer_bytes;        // intermediates of all heads of one layer together
};

GroupPlan plan_groups(const fc_handle *h, const PassPlan &p, int num_units, int num_heads, int head_dim) {
  GroupPlan g;
  const size_t per_unit = (size_t)p.M * head_dim * sizeof(float2);
  g.layer_bytes = per_unit * (size_t)num_heads;
  int nu = (int)(h->group_bytes / per_unit);
  if (nu < 1) nu = 1;
  if (nu > num_units) nu = num_units;
  int groups = (num_units + nu - 1) / nu;
  const int nu_alloc = nu;                                     // the workspace does not depend on the mode
  // All units fit one group: they stay one group (fuller launches) and consecutive calls alternate over the internal
  // streams, where calls overlap (fc_set_score_overlap: 28 calls of 4 heads of 8192 tokens 1.31 -> 1.11 ms) or the
  // whole call is tiny (8 MiB: 44 -> 31 us per call at 4 heads of 1024 tokens); otherwise a call that has to finish
  // before it returns is faster with its units on both streams (49 against 56 us per layer of 4 heads of 8192 tokens).
  const bool one_group = groups == 1 && (h->score_overlap || per_unit * (size_t)num_units <= ((size_t)8 << 20));
  if (groups < h->num_aux && num_units >= h->num_aux && !one_group) groups = h->num_aux;
  g.units = (num_units + groups - 1) / groups;                 // balanced groups
  g.sub = head_dim;
  if (nu_alloc == 1) {
    // the intermediates of the groups in flight (one per internal stream) should stay in the cache, so a unit is
    // halved down to 64 columns while they exceed three times the budget (two times: 20000 and 38000 tokens 7..11 %
    // slower; four and a half: 28000 and 32000 tokens 12 % slower)
    while (g.sub % 128 == 0 && (size_t)h->num_aux * p.M * g.sub * sizeof(float2) > 3 * h->group_bytes) g.sub /= 2;
  }
  g.ngr = head_dim / g.sub;
  g.buf_bytes = align_up((size_t)p.M * g.sub * nu_alloc * sizeof(float2), 256);
  return g;
}

// Workspace carve-up of one scoring call: the regions hold the largest sequence of the view.
struct ScoreLayout {
  size_t buf_bytes;          // intermediates, one buffer per internal stream
  size_t off_buf, off_tab, off_band, off_tot, off_hi, off_small, total;
  size_t tot_bytes, hi_bytes;   // per-block partial sums of one step; two copies, used in turn
};

// Cutoff index omega of Eq. 8 for a sequence of N tokens.
inline int cutoff_index(double gamma, int N) {
  long long om = (long long)floor(gamma * (double)N);
  if (om > N - 1) om = N - 1;
  if (om < 0) om = 0;
  return (int)om;
}

inline bool first_of_its_length(const fc_kv_view *kv, int b) {
  const int N = kv->cu_seqlens[b + 1] - kv->cu_seqlens[b];
  for (int i = 0; i < b; ++i)
    if (kv->cu_seqlens[i + 1] - kv->cu_seqlens[i] == N) return false;
  return true;
}

ScoreLayout score_layout(const fc_handle *h, const fc_kv_view *kv, int num_layers) {
  ScoreLayout L = {};
  const int H = kv->num_heads, d = kv->head_dim, nl = num_layers < FC_LAYER_CHUNK ? num_layers : FC_LAYER_CHUNK;
  size_t tab = 0, generic = 0, nsmall = 0, band = 0;
  for (int b = 0; b < kv->batch; ++b) {
    const int N = kv->cu_seqlens[b + 1] - kv->cu_seqlens[b];
    if (N == 0) continue;
    const PassPlan p = plan_passes(N, kv->head_dim);
    FcBandSizes bs;
    if (!h->generic_only && fc_band_bounds(kv, N, &bs)) {      // whether it is taken depends on the cutoff: room for both
      if (first_of_its_length(kv, b)) band += bs.tables;
      const size_t buf = fc_band_buffer_bytes(h, &bs, nl * H);
      const size_t part = (size_t)nl * H * bs.steps * 4 * sizeof(double);
      if (align_up(buf, 256) > L.buf_bytes) L.buf_bytes = align_up(buf, 256);
      if (part > L.tot_bytes) L.tot_bytes = part;
    }
    if (!p.ok || h->generic_only) {
      const size_t t = generic_layout(h, plan_sequence(N), H, d).total;
      if (t > generic) generic = t;
      continue;
    }
    if (p.pad && first_of_its_length(kv, b)) tab += (size_t)p.M * sizeof(float4);
    if (p.small) { ++nsmall; continue; }
    const GroupPlan g = plan_groups(h, p, nl * H, H, d);
    const size_t tot = (size_t)nl * H * (d / (2 * p.cpw)) * p.N2 * 2 * sizeof(double);
    const size_t hi = (size_t)nl * H * g.ngr * p.N2 * 2 * sizeof(double);
    if (g.buf_bytes > L.buf_bytes) L.buf_bytes = g.buf_bytes;
    if (tot > L.tot_bytes) L.tot_bytes = tot;
    if (hi > L.hi_bytes) L.hi_bytes = hi;
  }
  L.tot_bytes = align_up(L.tot_bytes, 256);
  L.hi_bytes = align_up(L.hi_bytes, 256);
  size_t off = 0;
  L.off_buf = off; off += L.buf_bytes * h->num_aux;
  if (off < generic) off = generic;            // tables outlive a sequence on the generic kernels
  L.off_tab = off; off += align_up(tab, 256);
  L.off_band = off; off += band;
  L.off_tot = off; off += 2 * L.tot_bytes;
  L.off_hi = off;  off += 2 * L.hi_bytes;
  L.off_small = off; off += align_up(nl * nsmall * H * 4 * sizeof(double), 256);
  L.total = off < 256 ? 256 : off;
  return L;
}

// Each internal stream's intermediate buffer is kept in the persisting part of L2, on the direct path only.
// Not where the intermediates of all heads of the sequence are small against the cache (48 MiB: they stay
// resident anyway and the set-aside only takes cache from the rows and scores; measured -2.5 % at 4 heads of 8192
// tokens with the window, +1.6 % and +4 % at 2 and 4 heads of 32768, no difference at 64 MiB).
bool window_fits(const fc_handle *h, const PassPlan &p, const GroupPlan &g) {
  return h->l2_persist && p.ok && !p.pad && g.layer_bytes > ((size_t)48 << 20) && g.buf_bytes <= h->window_max &&
         g.buf_bytes * (size_t)h->num_aux <= h->persist_max;
}

// The persisting part of L2 is a limit of the whole context, shared by the handles of a device (fc_persist_acquire):
// held while calls contain a sequence that wants it, let go when a call has none.  Decided once per call; left as it is
// while `st` is being captured into a graph, where device-wide settings cannot change.
void claim_persisting_l2(fc_handle *h, const fc_kv_view *kv, int num_layers, double gamma, cudaStream_t st) {
  if (!h->l2_persist) return;
  const int nl = num_layers < FC_LAYER_CHUNK ? num_layers : FC_LAYER_CHUNK;
  bool claim = false;
  for (int b = 0; b < kv->batch && !claim; ++b) {
    const int N = kv->cu_seqlens[b + 1] - kv->cu_seqlens[b];
    if (N == 0) continue;
    const PassPlan p = plan_passes(N, kv->head_dim);
    if (!p.ok || p.pad || p.small || fc_band_grid(kv, N, cutoff_index(gamma, N)) != 0) continue;
    claim = window_fits(h, p, plan_groups(h, p, nl * kv->num_heads, kv->num_heads, kv->head_dim));
  }
  if (claim == (h->persist_on != 0)) return;
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(st, &cap) != cudaSuccess) { cudaGetLastError(); return; }
  if (cap != cudaStreamCaptureStatusNone) return;
  if (claim) {
    if (!fc_persist_acquire(h)) h->l2_persist = 0;      // not available here: never try again
  } else {
    fc_persist_release(h);
  }
}

// `pointers`: the view's own k and v are checked too
fc_status validate_view(const fc_handle *h, const fc_kv_view *kv, bool pointers) {
  if (!h || !kv || !kv->cu_seqlens || (pointers && (!kv->k || !kv->v))) return FC_ERR_INVALID_ARG;
  if (kv->num_heads <= 0 || kv->head_dim <= 0 || kv->batch < 0) return FC_ERR_INVALID_ARG;
  if (kv->dtype != FC_F32 && kv->dtype != FC_F16 && kv->dtype != FC_BF16) return FC_ERR_UNSUPPORTED;
  if (kv->head_dim % 64 != 0) return FC_ERR_UNSUPPORTED;
  const size_t es = kv->dtype == FC_F32 ? 4 : 2;
  if (kv->cu_seqlens[0] != 0) return FC_ERR_INVALID_ARG;
  for (int b = 0; b < kv->batch; ++b) {
    const long long n = (long long)kv->cu_seqlens[b + 1] - kv->cu_seqlens[b];
    if (n < 0) return FC_ERR_INVALID_ARG;
    if (n > h->max_seqlen) return FC_ERR_UNSUPPORTED;
    if (n > 65536 && !is_pow2((int)n)) return FC_ERR_UNSUPPORTED;
  }
  if (kv->stride_token < (long long)kv->head_dim || kv->stride_head < (long long)kv->head_dim)
    return FC_ERR_INVALID_ARG;
  if (pointers && (((uintptr_t)kv->k & 15) || ((uintptr_t)kv->v & 15))) return FC_ERR_INVALID_ARG;
  if ((kv->stride_token * es) % 16 || (kv->stride_head * es) % 16) return FC_ERR_INVALID_ARG;
  return FC_OK;
}

// Function attributes are set once per kernel and device (and again only if a launch needs more shared
// memory than the last time), not before every launch.
template <class Kern>
fc_status set_smem(Kern kern, size_t bytes) {
  static std::mutex mu;
  static std::unordered_map<unsigned long long, size_t> done;     // (device, kernel) -> bytes already allowed
  int dev = 0;
  FC_CUDA_TRY(cudaGetDevice(&dev));
  const unsigned long long key = (unsigned long long)reinterpret_cast<uintptr_t>(reinterpret_cast<const void *>(kern)) ^
                                 ((unsigned long long)dev << 56);
  std::lock_guard<std::mutex> lock(mu);
  auto it = done.find(key);
  if (it != done.end() && it->second >= bytes) return FC_OK;
  if (bytes > 48 * 1024) FC_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes));
  // as much of the L1/shared array as shared memory as the device offers: these kernels do not rely on L1
  if (it == done.end())
    FC_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared));
  done[key] = bytes;
  return FC_OK;
}

// Clusters of more than 8 blocks, once per kernel and device.
template <class Kern>
fc_status allow_wide_clusters(Kern kern) {
  static std::mutex mu;
  static std::unordered_map<unsigned long long, bool> done;
  int dev = 0;
  FC_CUDA_TRY(cudaGetDevice(&dev));
  const unsigned long long key = (unsigned long long)reinterpret_cast<uintptr_t>(reinterpret_cast<const void *>(kern)) ^
                                 ((unsigned long long)dev << 56);
  std::lock_guard<std::mutex> lock(mu);
  if (done[key]) return FC_OK;
  FC_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
  done[key] = true;
  return FC_OK;
}

size_t smem_pass13(const SeqPlan &sp, int cs) {
  return (size_t)sp.N1 * cs * sizeof(float2) + sp.N1 * sizeof(float2) + sp.N1 * sizeof(int) + 2 * sp.N1 * sizeof(float);
}
size_t smem_pass2(const SeqPlan &sp, int cs2, int halves = 2) {
  return (size_t)sp.N2 * halves * cs2 * sizeof(float2) + 3 * (size_t)sp.N2 * sizeof(float2) + 2 * (size_t)sp.N2 * sizeof(unsigned short);
}

template <class Loader>
fc_status launch_pass1(fc_handle *h, cudaStream_t st, const Loader &ld, const SeqPlan &sp, int ncol_ws, int cs,
                       float2 *ws, double *partial) {
  const FftPlan p1 = make_plan(sp.N1);
  const size_t sm = smem_pass13(sp, cs);
  fc_status s = set_smem(k_pass1<Loader>, sm);
  if (s != FC_OK) return s;
  dim3 grid(sp.N2, ncol_ws / cs);
  ProfScope ps(h, FC_K_PASS1, st);
  k_pass1<Loader><<<grid, kThreads, sm, st>>>(ld, p1, sp.N2, ncol_ws, ilog2(cs), ws, h->master, h->master_len, partial);
  return fc_after_launch(h);
}

template <int MID>
fc_status launch_pass2(fc_handle *h, cudaStream_t st, const SeqPlan &sp, int ncol_ws, int cs2, float2 *ws,
                       int omega, float2 *hhat, float scale) {
  const FftPlan p2 = make_plan(sp.N2);
  const size_t sm = smem_pass2(sp, cs2, MID == MID_DCT ? 2 : 1);
  fc_status s = set_smem(k_pass2<MID>, sm);
  if (s != FC_OK) return s;
  dim3 grid(MID == MID_DCT ? sp.N1 / 2 + 1 : sp.N1, ncol_ws / cs2);
  ProfScope ps(h, FC_K_PASS2, st);
  k_pass2<MID><<<grid, kThreads, sm, st>>>(p2, sp.N1, ncol_ws, ilog2(cs2), ws, h->master, h->master_len, omega, hhat, scale);
  return fc_after_launch(h);
}

// ---- launches of the specialised passes ----
struct PassArgs {
  fc_handle *h;
  cudaStream_t st;
  const PassPlan *p;
  const fast::LayerPtrs *lp;
  const fc_kv_view *kv;
  int u0, nu, c0, cols;      // units of the launch; first channel and channels per unit
  int omega;
  float2 *ws;
  const float4 *tab;
};

inline size_t smem_outer(const PassPlan &p) { return (size_t)p.N1 * p.cpw * sizeof(float4) + p.N1 * sizeof(float2); }

template <typename T, int A, int R1B, int CPW, int LD>
fc_status launch_p1(const PassArgs &x, double *part_tot, int layer_slots) {
  const PassPlan &p = *x.p;
  const size_t sm = smem_outer(p);
  const int ncol = LD == fast::LD_TABLE ? 2 * CPW : x.nu * x.cols;
  fc_status s = set_smem(fast::k_p1<T, R1B, CPW, LD, A>, sm);
  if (s != FC_OK) return s;
  ProfScope ps(x.h, FC_K_PASS1, x.st);
  fast::k_p1<T, R1B, CPW, LD, A><<<dim3(p.N2, ncol / (2 * CPW)), CPW * R1B, sm, x.st>>>(
      *x.lp, x.kv->stride_token, x.kv->stride_head, x.kv->num_heads, x.kv->head_dim, x.u0, x.c0, x.cols, p.N, p.N2, ncol,
      x.ws, x.h->master, x.h->master_len, part_tot, layer_slots, x.omega, x.tab);
  return fc_after_launch(x.h);
}

// first-stage radix, second-stage radix and channel pairs of passes 1 and 3: the shapes plan_passes gives
#define FC_OUTER_PAD_SHAPES(X)                                                                                \
  X(16, 2, 32) X(16, 4, 32) X(16, 8, 32) X(16, 16, 16) X(14, 4, 32) X(14, 8, 32) X(14, 16, 32) X(14, 16, 16) \
  X(12, 4, 32) X(12, 8, 32) X(12, 16, 32) X(12, 16, 16) X(10, 4, 32) X(10, 8, 32) X(10, 16, 32) X(10, 16, 16)
#define FC_OUTER_DIRECT_SHAPES(X) X(16, 2, 32) X(16, 4, 32) X(16, 8, 32) X(16, 16, 16)

template <typename T>
fc_status run_p1(const PassArgs &x, double *part_tot, int layer_slots) {
  const PassPlan &p = *x.p;
#define FC_P1(A_, R_, C_)                                                  \
  if (p.pad && p.a == A_ && p.r1b == R_ && p.cpw == C_)                    \
    return launch_p1<T, A_, R_, C_, fast::LD_PAD>(x, part_tot, layer_slots);
  FC_OUTER_PAD_SHAPES(FC_P1)
#undef FC_P1
#define FC_P1(A_, R_, C_)                                                  \
  if (!p.pad && p.a == A_ && p.r1b == R_ && p.cpw == C_)                   \
    return launch_p1<T, A_, R_, C_, fast::LD_KV>(x, part_tot, layer_slots);
  FC_OUTER_DIRECT_SHAPES(FC_P1)
#undef FC_P1
  return FC_ERR_INTERNAL;
}

// The rows of a chirp convolution (spectrum diagnostics).
template <typename T>
fc_status run_p1_chirp(const PassArgs &x) {
  const PassPlan &p = *x.p;
#define FC_P1(A_, R_, C_) \
  if (p.a == A_ && p.r1b == R_ && p.cpw == C_) return launch_p1<T, A_, R_, C_, fast::LD_CHIRP>(x, nullptr, 0);
  FC_OUTER_PAD_SHAPES(FC_P1)
#undef FC_P1
  return FC_ERR_INTERNAL;
}

fc_status run_p1_table(const PassArgs &x) {
  const PassPlan &p = *x.p;
#define FC_P1(A_, R_, C_) \
  if (p.a == A_ && p.r1b == R_ && p.cpw == C_) return launch_p1<float, A_, R_, C_, fast::LD_TABLE>(x, nullptr, 0);
  FC_OUTER_PAD_SHAPES(FC_P1)
#undef FC_P1
  return FC_ERR_INTERNAL;
}

// tab_out != nullptr: the forward half on the two kernel columns, `ncol` columns wide (run_p1_table)
template <int R2B, int CP, int MODE>
fc_status launch_p2(const PassArgs &x, int ncol, float4 *tab_out, float2 *power) {
  const PassPlan &p = *x.p;
  constexpr bool TAB = MODE == fast::MODE_PAD || MODE == fast::MODE_MUL;
  const size_t sm = (size_t)2 * (16 * R2B) * CP * sizeof(float4) + (4 * R2B + 4) * sizeof(float2) +
                    (TAB ? 2 * (16 * R2B) * sizeof(float4) : (2 * (16 * R2B) + 4) * sizeof(float2));
  fc_status s = set_smem(fast::k_p2<R2B, CP, MODE>, sm);
  if (s != FC_OK) return s;
  ProfScope ps(x.h, FC_K_PASS2, x.st);
  fast::k_p2<R2B, CP, MODE><<<dim3(p.N1 / 2, tab_out ? 1 : ncol / (2 * CP)), 2 * CP * R2B, sm, x.st>>>(
      p.N1, ncol, x.ws, x.h->master, x.h->master_len, x.omega, x.tab, tab_out, power, p.N);
  return fc_after_launch(x.h);
}

template <int MODE>
fc_status launch_p2_512(const PassArgs &x, int ncol, float4 *tab_out) {
  const PassPlan &p = *x.p;
  constexpr int C = 8;
  const size_t sm = (size_t)2 * 16 * (32 * C + C) * sizeof(float2) + 1024 * sizeof(float4) + (64 + 68) * sizeof(float2);
  fc_status s = set_smem(fast::k_p2_512<C, MODE>, sm);
  if (s != FC_OK) return s;
  ProfScope ps(x.h, FC_K_PASS2, x.st);
  fast::k_p2_512<C, MODE><<<dim3(p.N1 / 2, tab_out ? 1 : ncol / C), 32 * C, sm, x.st>>>(
      p.N1, ncol, x.ws, x.h->master, x.h->master_len, x.tab, tab_out, p.N);
  return fc_after_launch(x.h);
}

fc_status run_p2(const PassArgs &x, int ncol, int mode, float4 *tab_out = nullptr, float2 *power = nullptr) {
  const PassPlan &p = *x.p;
  using namespace fast;
  if (p.N2 == 512) return mode == MODE_PAD ? launch_p2_512<MODE_PAD>(x, ncol, tab_out) : launch_p2_512<MODE_MUL>(x, ncol, tab_out);
#define FC_P2(R_, C_, M_) \
  if (mode == M_ && p.r2b == R_ && p.cp == C_) return launch_p2<R_, C_, M_>(x, ncol, tab_out, power);
  FC_P2(2, 32, MODE_PAD) FC_P2(4, 32, MODE_PAD) FC_P2(8, 16, MODE_PAD) FC_P2(16, 8, MODE_PAD)
  FC_P2(2, 32, MODE_MUL) FC_P2(4, 32, MODE_MUL) FC_P2(8, 16, MODE_MUL) FC_P2(16, 8, MODE_MUL)
  FC_P2(2, 8, MODE_FILTER) FC_P2(4, 8, MODE_FILTER) FC_P2(4, 32, MODE_FILTER) FC_P2(8, 16, MODE_FILTER) FC_P2(16, 8, MODE_FILTER)
  FC_P2(2, 8, MODE_POWER) FC_P2(4, 8, MODE_POWER) FC_P2(4, 32, MODE_POWER) FC_P2(8, 16, MODE_POWER) FC_P2(16, 8, MODE_POWER)
#undef FC_P2
  return FC_ERR_INTERNAL;
}

template <int A, int R1B, int CPW, int OUT>
fc_status launch_p3(const PassArgs &x, long long score_stride, int accumulate, int hi_base, const fast::EnergyOut &eo,
                    float2 *spec = nullptr) {
  const PassPlan &p = *x.p;
  const size_t sm = smem_outer(p);
  fc_status s = set_smem(fast::k_p3<R1B, CPW, OUT, A>, sm);
  if (s != FC_OK) return s;
  const float inv = OUT == fast::OUT_SPEC ? 1.f / (float)p.M : (float)(1.0 / ((double)p.M * (double)p.M * (double)x.kv->head_dim));
  ProfScope ps(x.h, FC_K_PASS3, x.st);
  fast::k_p3<R1B, CPW, OUT, A><<<dim3(p.N2, x.nu), CPW * R1B, sm, x.st>>>(
      *x.lp, x.kv->num_heads, x.kv->head_dim, x.u0, x.cols, p.N, p.N2, x.nu * x.cols, x.ws, x.h->master, x.h->master_len,
      score_stride, inv, accumulate, hi_base, eo, spec, x.tab);
  return fc_after_launch(x.h);
}

fc_status run_p3(const PassArgs &x, long long score_stride, int accumulate, int hi_base, const fast::EnergyOut &eo) {
  const PassPlan &p = *x.p;
#define FC_P3(A_, R_, C_)                               \
  if (p.pad && p.a == A_ && p.r1b == R_ && p.cpw == C_) \
    return launch_p3<A_, R_, C_, fast::OUT_PAD>(x, score_stride, accumulate, hi_base, eo);
  FC_OUTER_PAD_SHAPES(FC_P3)
#undef FC_P3
#define FC_P3(A_, R_, C_)                                \
  if (!p.pad && p.a == A_ && p.r1b == R_ && p.cpw == C_) \
    return launch_p3<A_, R_, C_, fast::OUT_SCORE>(x, score_stride, accumulate, hi_base, eo);
  FC_OUTER_DIRECT_SHAPES(FC_P3)
#undef FC_P3
  return FC_ERR_INTERNAL;
}

// The N-point spectrum at the end of a chirp convolution (spectrum diagnostics).
fc_status run_p3_spec(const PassArgs &x, float2 *spec) {
  const PassPlan &p = *x.p;
  static const fast::EnergyOut none = {};
#define FC_P3(A_, R_, C_) \
  if (p.a == A_ && p.r1b == R_ && p.cpw == C_) return launch_p3<A_, R_, C_, fast::OUT_SPEC>(x, 0, 0, 0, none, spec);
  FC_OUTER_PAD_SHAPES(FC_P3)
#undef FC_P3
  return FC_ERR_INTERNAL;
}

// How the spectrum diagnostics transform a sequence: a power of two from 1024 to 65536 directly, a length that is not a
// power of two by a chirp convolution of >= 2N - 1 points (plan.pad); 131072 points and powers of two below 1024, where
// launches count and a chirp would add two of them, are left to the generic kernels.
PassPlan plan_spectrum(int N) {
  static const PassPlan none = {};
  if (is_pow2(N) && N >= 16) return N >= 1024 && N <= 65536 ? plan_passes(N, 0) : none;
  return plan_padded(N);
}

// Tables of the padded form (filter) or of the chirp (spectrum = true: its spectrum and per-row factors) for every such
// sequence of the view, tabs[b].  A table depends on the length, the cutoff and the form (small kernel or passes) only, so
// the handle keeps the last FC_TAB_SLOTS (the layers of a prefill share theirs).  While the stream is being captured, and for lengths beyond the
// slots, tables go to the workspace (`spare`), every call: a graph must not depend on what the handle holds when it is
// replayed.  `buf`: an intermediate buffer to build them in.
fc_status prepare_tables(fc_handle *h, cudaStream_t st, const fc_kv_view *kv, double gamma, bool spectrum, float4 *spare,
                         float2 *buf, const float4 **tabs, const FcBandJob *const *band = nullptr) {
  bool cached = true, any = false, flushed = false;
  bool used[FC_TAB_SLOTS] = {};
  auto plan_of = [&](int N) { return spectrum ? plan_spectrum(N) : plan_passes(N, kv->head_dim); };
  auto omega_of = [&](int N) { return spectrum ? -1 : cutoff_index(gamma, N); };
  // head_dim decides between the small kernel and the passes, whose tables differ in length and order, so the form is
  // part of the key (with it N fixes the transform length)
  auto key_of = [&](int N) {
    return (long long)N + (plan_of(N).small ? 1ll << 24 : 0ll) + ((long long)(omega_of(N) + 2) << 32);
  };
  for (int b = 0; b < kv->batch; ++b) {
    tabs[b] = nullptr;
    const int N = kv->cu_seqlens[b + 1] - kv->cu_seqlens[b];
    if (N == 0) continue;
    const PassPlan p = plan_of(N);
    if (!p.ok || !p.pad || (band && band[b])) continue;
    if (!any) {
      any = true;
      cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
      if (cudaStreamIsCapturing(st, &cap) != cudaSuccess) { cudaGetLastError(); cap = cudaStreamCaptureStatusActive; }
      cached = cap == cudaStreamCaptureStatusNone;
    }
    if (cached)
      for (int i = 0; i < FC_TAB_SLOTS; ++i)
        if (h->tab_key[i] == key_of(N)) { tabs[b] = h->tab_cache + (size_t)i * h->tab_slot_len; used[i] = true; }
  }
  if (!any) return FC_OK;
  for (int b = 0; b < kv->batch; ++b) {
    const int N = kv->cu_seqlens[b + 1] - kv->cu_seqlens[b];
    if (N == 0 || tabs[b]) continue;
    const PassPlan p = plan_of(N);
    if (!p.ok || !p.pad || (band && band[b])) continue;
    if (!first_of_its_length(kv, b)) {
      for (int i = 0; i < b && !tabs[b]; ++i)
        if (kv->cu_seqlens[i + 1] - kv->cu_seqlens[i] == N) tabs[b] = tabs[i];
      continue;
    }
    fc_status s;
    // the table's place and the intermediate buffer may still be in use on the internal streams
    if (!flushed && (s = fc_flush_pending(h, st)) != FC_OK) return s;
    flushed = true;
    float4 *dst = nullptr;
    int slot = -1;
    for (int i = 0; cached && i < FC_TAB_SLOTS && slot < 0; ++i) {
      const int c = (h->tab_next + i) % FC_TAB_SLOTS;
      if (!used[c]) slot = c;
    }
    if (slot >= 0) {
      h->tab_next = (slot + 1) % FC_TAB_SLOTS;
      h->tab_key[slot] = 0;                                  // not valid until its launches are in the stream
      used[slot] = true;
      dst = h->tab_cache + (size_t)slot * h->tab_slot_len;
    } else {
      dst = spare;
      spare += p.M;
    }
    if (p.small) {
      small::k_small_table<<<(p.M + 63) / 64, 64, (N + 1) * sizeof(float), st>>>(dst, N, omega_of(N), p.M, h->master,
                                                                                h->master_len);
      if ((s = fc_after_launch(h)) != FC_OK) return s;
    } else {
      static const fast::LayerPtrs none = {};
      const PassArgs x{h, st, &p, &none, kv, 0, 1, 0, 2 * p.cpw, omega_of(N), buf, nullptr};
      if ((s = run_p1_table(x)) != FC_OK) return s;
      if ((s = run_p2(x, 2 * p.cpw, spectrum ? fast::MODE_MUL : fast::MODE_PAD, dst)) != FC_OK) return s;
    }
    if (slot >= 0) h->tab_key[slot] = key_of(N);
    tabs[b] = dst;
  }
  return FC_OK;
}

// One sequence on the specialised passes, for a chunk of layers.  `lp` points at the sequence's first token.
template <typename T>
fc_status score_sequence(fc_handle *h, cudaStream_t st, const fc_kv_view *kv, const PassPlan &p, int nl,
                         const fast::LayerPtrs &lp, double gamma, double *energy, long long energy_stride,
                         const ScoreLayout &L, char *wsb, const float4 *tab) {
  const int d = kv->head_dim, H = kv->num_heads, U = nl * H;
  const long long total_tokens = kv->cu_seqlens[kv->batch];
  const GroupPlan g = plan_groups(h, p, U, H, d);
  const unsigned par = h->step & 1u;               // consecutive steps alternate between two copies of the partial sums
  fc_status s;
  if (window_fits(h, p, g) && h->persist_on) {
    // keep each stream's intermediate in the persisting part of L2; everything else these streams touch
    // (the K/V rows, the scores) streams through
    for (int i = 0; i < h->num_aux; ++i) {
      const char *base = wsb + L.off_buf + (size_t)i * L.buf_bytes;
      if (h->window_base[i] == base && h->window_bytes[i] == g.buf_bytes) continue;
      cudaStreamAttrValue av = {};
      av.accessPolicyWindow.base_ptr = const_cast<char *>(base);
      av.accessPolicyWindow.num_bytes = g.buf_bytes;
      av.accessPolicyWindow.hitRatio = 1.0f;
      av.accessPolicyWindow.hitProp = cudaAccessPropertyPersisting;
      av.accessPolicyWindow.missProp = cudaAccessPropertyStreaming;
      if (cudaStreamSetAttribute(h->aux[i], cudaStreamAttributeAccessPolicyWindow, &av) != cudaSuccess) {
        cudaGetLastError();
        h->l2_persist = 0;               // not supported here: never try again
        break;
      }
      h->window_base[i] = base;
      h->window_bytes[i] = g.buf_bytes;
    }
  }
  // the partial sums and the block counters of this parity were last used two steps ago: the other streams must be
  // through with that step (this one is, by stream order)
  if (h->step >= 2)
    for (int i = 0; i < h->num_aux; ++i)
      for (int o = 0; o < h->num_aux; ++o)
        if (o != i) FC_CUDA_TRY(cudaStreamWaitEvent(h->aux[i], h->ev_done[par][o], 0));
  double *part_tot = reinterpret_cast<double *>(wsb + L.off_tot + par * L.tot_bytes);
  fast::EnergyOut eo;
  eo.part_hi = reinterpret_cast<double *>(wsb + L.off_hi + par * L.hi_bytes);
  eo.part_tot = part_tot;
  eo.hi_slots = H * g.ngr * p.N2;
  eo.tot_slots = H * (d / (2 * p.cpw)) * p.N2;
  eo.done = h->done_counter + par * FC_LAYER_CHUNK;
  eo.total_blocks = (unsigned)(H * g.ngr * p.N2);
  eo.energy = energy;
  eo.energy_stride = energy_stride;
  int group = 0;
  for (int u0 = 0; u0 < U; u0 += g.units, ++group) {
    const int nu = U - u0 < g.units ? U - u0 : g.units;
    const int si = (int)((group + h->step) % (unsigned)h->num_aux);   // a single group: steps alternate
    PassArgs x{h, h->aux[si], &p, &lp, kv, u0, nu, 0, g.sub, cutoff_index(gamma, p.N),
               reinterpret_cast<float2 *>(wsb + L.off_buf + (size_t)si * L.buf_bytes), tab};
    for (int cg = 0; cg < g.ngr; ++cg) {                      // column groups of one unit, in stream order
      x.c0 = cg * g.sub;
      if ((s = run_p1<T>(x, part_tot, eo.tot_slots)) != FC_OK) return s;
      if ((s = run_p2(x, nu * g.sub, p.pad ? fast::MODE_PAD : fast::MODE_FILTER)) != FC_OK) return s;
      if ((s = run_p3(x, total_tokens, cg > 0 ? 1 : 0, cg * H * p.N2, eo)) != FC_OK) return s;
    }
  }
  for (int i = 0; i < h->num_aux; ++i) FC_CUDA_TRY(cudaEventRecord(h->ev_done[par][i], h->aux[i]));
  h->step++;
  h->pending_join = true;
  return FC_OK;
}

struct Jobs : std::vector<FcBandJob *> {
  using std::vector<FcBandJob *>::vector;
  ~Jobs() { for (FcBandJob *j : *this) fc_band_release(j); }
};

// Tables of the sequences scored in the kept band, as prepare_tables does it: the handle keeps those of the last calls that it
// has room for, the others, and all while the stream is being captured, are built into the workspace.
fc_status band_tables(fc_handle *h, cudaStream_t st, const fc_kv_view *kv, const Jobs &band, char *spare, const char **tabs) {
  bool cached = true, any = false, flushed = false;
  bool used[FC_BAND_KEPT] = {};
  for (int b = 0; b < kv->batch; ++b) {
    if (!band[b]) continue;
    if (!any) {
      any = true;
      cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
      if (cudaStreamIsCapturing(st, &cap) != cudaSuccess) { cudaGetLastError(); cap = cudaStreamCaptureStatusActive; }
      cached = cap == cudaStreamCaptureStatusNone;
    }
    const int i = cached ? fc_band_kept(h, band[b]) : -1;
    if (i >= 0) { tabs[b] = h->band_pool + h->band_kept[i].off; used[i] = true; }
  }
  for (int b = 0; b < kv->batch; ++b) {
    if (!band[b] || tabs[b]) continue;
    for (int i = 0; i < b && !tabs[b]; ++i)
      if (band[i] && fc_band_table_key(band[i]) == fc_band_table_key(band[b])) tabs[b] = tabs[i];
    if (tabs[b]) continue;
    fc_status s;
    // the tables' place may still be in use on the internal streams
    if (!flushed && (s = fc_flush_pending(h, st)) != FC_OK) return s;
    flushed = true;
    const int place = cached ? fc_band_place(h, band[b], used) : -1;
    char *dst = spare;
    if (place >= 0) {
      used[place] = true;
      dst = h->band_pool + h->band_kept[place].off;
    } else {
      FcBandSizes bs;
      fc_band_bounds(kv, kv->cu_seqlens[b + 1] - kv->cu_seqlens[b], &bs);
      spare += bs.tables;
    }
    if ((s = fc_band_tables(h, st, band[b], dst)) != FC_OK) return s;
    if (place >= 0) h->band_kept[place].key = fc_band_table_key(band[b]);      // valid from here on in stream order
    tabs[b] = dst;
  }
  return FC_OK;
}

// One sequence in the kept band, for a chunk of layers, on the internal streams or, with on_caller, on `st`.  `lp` points at
// the sequence's first token.
fc_status score_band(fc_handle *h, cudaStream_t st, bool on_caller, const fc_kv_view *kv, FcBandJob *job, int nl, const fast::LayerPtrs &lp,
                     double *energy, long long energy_stride, const ScoreLayout &L, char *wsb, const char *tables) {
  const int U = nl * kv->num_heads;
  const int nu = fc_band_units(h, job, U, L.buf_bytes), groups = (U + nu - 1) / nu;
  const int ranges = fc_band_ranges(h, job, nu);
  const unsigned par = h->step & 1u;               // as in score_sequence
  if (!on_caller && h->step >= 2)
    for (int i = 0; i < h->num_aux; ++i)
      for (int o = 0; o < h->num_aux; ++o)
        if (o != i) FC_CUDA_TRY(cudaStreamWaitEvent(h->aux[i], h->ev_done[par][o], 0));
  FcBandLaunch l = {lp.k, lp.v, lp.scores, nl, tables, reinterpret_cast<double *>(wsb + L.off_tot + par * L.tot_bytes), energy,
                    h->done_counter + par * FC_LAYER_CHUNK, (long long)kv->cu_seqlens[kv->batch], energy_stride};
  fc_status s = fc_band_bind(h, job, kv, l);
  if (s != FC_OK) return s;
  int group = 0;
  for (int u0 = 0; u0 < U; u0 += nu, ++group) {
    const int si = on_caller ? 0 : (int)((group + h->step) % (unsigned)h->num_aux);
    s = fc_band_group(h, on_caller ? st : h->aux[si], job, l, u0, U - u0 < nu ? U - u0 : nu, nu, ranges,
                      on_caller || groups <= h->num_aux,
                      wsb + L.off_buf + (size_t)si * L.buf_bytes);
    if (s != FC_OK) return s;
  }
  if (on_caller) return FC_OK;
  for (int i = 0; i < h->num_aux; ++i) FC_CUDA_TRY(cudaEventRecord(h->ev_done[par][i], h->aux[i]));
  h->step++;
  h->pending_join = true;
  return FC_OK;
}

// The short sequences of a chunk of layers, one launch per transform length and form (and 32 sequences), on the caller's
// stream.
template <typename T, class S, bool PADDED>
fc_status launch_small(fc_handle *h, cudaStream_t st, const fc_kv_view *kv, const fast::LayerPtrs &lp, int nl,
                       const small::SeqTable &tab, int nseq, double *part, double *energy) {
  const size_t sm = S::smem(PADDED);
  fc_status s = set_smem(small::k_small<T, S, PADDED>, sm);
  if (s != FC_OK) return s;
  const unsigned blocks = (unsigned)(kv->head_dim / (2 * S::CP));
  if (blocks > 8 && (s = allow_wide_clusters(small::k_small<T, S, PADDED>)) != FC_OK) return s;
  cudaLaunchConfig_t lc = {};
  lc.gridDim = dim3(blocks, kv->num_heads, nl * nseq);
  lc.blockDim = dim3(S::NT);
  lc.dynamicSmemBytes = sm;
  lc.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = blocks;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  lc.attrs = at;
  lc.numAttrs = 1;
  ProfScope ps(h, FC_K_PASS2, st);
  if (cudaLaunchKernelEx(&lc, small::k_small<T, S, PADDED>, lp, tab, nseq, (long long)kv->stride_token,
                         (long long)kv->stride_head, (int)kv->num_heads, (int)kv->head_dim, (const float2 *)h->master,
                         h->master_len, (long long)kv->cu_seqlens[kv->batch], part, h->small_counter, energy,
                         4ll * kv->batch) != cudaSuccess) {
    cudaGetLastError();
    return FC_ERR_CUDA;
  }
  return fc_after_launch(h);
}

template <typename T>
fc_status score_small(fc_handle *h, cudaStream_t st, const fc_kv_view *kv, const fc_layer_buffers *layers, int nl,
                      const std::vector<PassPlan> &plans, const std::vector<const float4 *> &tabs, double gamma,
                      double *energy, double *part) {
  fast::LayerPtrs lp = {};
  for (int l = 0; l < nl; ++l) {
    lp.k[l] = layers[l].k;
    lp.v[l] = layers[l].v;
    lp.scores[l] = const_cast<float *>(layers[l].scores);
  }
  for (int M = 64; M <= 1024; M <<= 1)
    for (int pad = 0; pad < 2; ++pad) {
      small::SeqTable tab = {};
      int n = 0;
      for (int b = 0; b <= kv->batch; ++b) {
        if (n > 0 && (n == small::kSeqs || b == kv->batch)) {
          fc_status s = FC_ERR_INTERNAL;
#define FC_SMALL(M_, A_, B_, C_)                                                                                        \
  if (M == M_)                                                                                                          \
    s = pad ? launch_small<T, small::Shape<A_, B_, C_, small_cp(M_)>, true>(h, st, kv, lp, nl, tab, n, part, energy)    \
            : launch_small<T, small::Shape<A_, B_, C_, small_cp(M_)>, false>(h, st, kv, lp, nl, tab, n, part, energy);
          FC_SMALL(64, 8, 1, 8) FC_SMALL(128, 16, 1, 8) FC_SMALL(256, 16, 1, 16) FC_SMALL(512, 8, 8, 8)
          FC_SMALL(1024, 16, 8, 8)
#undef FC_SMALL
          if (s != FC_OK) return s;
          part += (size_t)nl * n * kv->num_heads * 4;
          n = 0;
        }
        if (b == kv->batch || !plans[b].small || plans[b].M != M || plans[b].pad != (pad != 0)) continue;
        tab.start[n] = kv->cu_seqlens[b];
        tab.N[n] = plans[b].N;
        tab.omega[n] = cutoff_index(gamma, plans[b].N);
        tab.index[n] = b;
        tab.tab[n] = tabs[b];
        ++n;
      }
    }
  return FC_OK;
}

// One sequence of one layer on the generic kernels, on the caller's stream.
template <typename T>
fc_status score_generic(fc_handle *h, cudaStream_t st, const fc_kv_view *kv, int b, double gamma, float *scores,
                        double *energy_b, char *wsb) {
  const int start = kv->cu_seqlens[b];
  const int N = kv->cu_seqlens[b + 1] - start;
  const long long total_tokens = kv->cu_seqlens[kv->batch];
  const int d = kv->head_dim, H = kv->num_heads;
  const SeqPlan sp = plan_sequence(N);
  const GenericLayout L = generic_layout(h, sp, H, d);
  const int omega = cutoff_index(gamma, N);
  float2 *ws = reinterpret_cast<float2 *>(wsb + L.off_ws);
  float2 *spec = reinterpret_cast<float2 *>(wsb + L.off_spec);
  float2 *hhat = reinterpret_cast<float2 *>(wsb + L.off_hhat);
  float2 *hcol = reinterpret_cast<float2 *>(wsb + L.off_hcol);
  double *part_tot = reinterpret_cast<double *>(wsb + L.off_part_tot);
  double *part_hi = reinterpret_cast<double *>(wsb + L.off_part_hi);
  const T *kp = static_cast<const T *>(kv->k) + (long long)start * kv->stride_token;
  const T *vp = static_cast<const T *>(kv->v) + (long long)start * kv->stride_token;
  const FftPlan p1 = make_plan(sp.N1);
  fc_status s;
  if (sp.bluestein) {
    ChirpKernelLoader cl{N, sp.Nfft};
    if ((s = launch_pass1(h, st, cl, sp, 8, 8, hcol, nullptr)) != FC_OK) return s;
    if ((s = launch_pass2<MID_SPEC>(h, st, sp, 8, 8, hcol, 0, hhat, 1.f)) != FC_OK) return s;
  }
  size_t tot_slots = 0, hi_slots = 0;
  for (int h0 = 0; h0 < H; h0 += L.heads_per_group) {
    const int hg = (H - h0 < L.heads_per_group) ? H - h0 : L.heads_per_group;
    double *ptot = part_tot + 2 * tot_slots;
    double *phi = part_hi + 2 * hi_slots;
    if (!sp.bluestein) {
      const int ncol_ws = hg * d;
      const size_t sm3 = smem_pass13(sp, sp.cs);
      KvLoader<T, false> ld{kp, vp, kv->stride_token, kv->stride_head, h0, d, N, 0.f, 0.f};
      if ((s = launch_pass1(h, st, ld, sp, ncol_ws, sp.cs, ws, ptot)) != FC_OK) return s;
      if ((s = launch_pass2<MID_DCT>(h, st, sp, ncol_ws, sp.cs2, ws, omega, nullptr, 1.f / (float)N)) != FC_OK) return s;
      if ((s = set_smem(k_pass3<EPI_SCORE, false>, sm3)) != FC_OK) return s;
      {
        ProfScope ps(h, FC_K_PASS3, st);
        k_pass3<EPI_SCORE, false><<<dim3(sp.N2, hg), kThreads, sm3, st>>>(
            p1, sp.N2, N, ncol_ws, ilog2(sp.cs), ws, h->master, h->master_len, nullptr, scores + start, h0, d,
            total_tokens, 1.f / (float)d, phi, (float)d, 0);
      }
      if ((s = fc_after_launch(h)) != FC_OK) return s;
      tot_slots += (size_t)sp.N2 * (ncol_ws / sp.cs);
      hi_slots += (size_t)sp.N2 * hg;
      continue;
    }
    // One head may be transformed in several column groups (sub < d) so that the padded length-Nfft intermediates of a
    // group stay within the budget; the groups run in stream order and the last pass adds their contributions to the
    // score in that order.
    const float invM = 1.f / (float)sp.Nfft;
    const float inv = (float)(1.0 / ((double)N * (double)N * (double)d));
    const int sub = L.sub_cols, cs = (sub % 64 == 0) ? sp.cs : 32;
    const int ngroups = (hg == 1) ? d / sub : 1;
    const int ncol = (hg == 1) ? sub : hg * d;
    int cs2 = 2 * sp.cs2 > 64 ? 64 : 2 * sp.cs2;       // the convolution pass holds single rows: twice the columns fit
    while (ncol % cs2) cs2 >>= 1;
    const size_t sm3c = smem_pass13(sp, cs);
    for (int cg = 0; cg < ngroups; ++cg) {
      const int c0 = cg * sub;
      double *ptot_c = ptot + 2 * (size_t)cg * sp.N2 * (ncol / cs);
      double *phi_c = phi + 2 * (size_t)cg * sp.N2 * hg;
      const int dd = (hg == 1) ? sub : d;           // columns the loader and the last pass see per head
      KvLoader<T, true> ld{kp + c0, vp + c0, kv->stride_token, kv->stride_head, h0, dd, N, 0.f, 0.f};
      if ((s = launch_pass1(h, st, ld, sp, ncol, cs, ws, ptot_c)) != FC_OK) return s;
      if ((s = launch_pass2<MID_MULH>(h, st, sp, ncol, cs2, ws, 0, hhat, invM)) != FC_OK) return s;
      if ((s = set_smem(k_pass3<EPI_SPEC, true>, sm3c)) != FC_OK) return s;
      {
        ProfScope ps(h, FC_K_PASS3, st);
        k_pass3<EPI_SPEC, true><<<dim3(sp.N2, ncol / cs), kThreads, sm3c, st>>>(
            p1, sp.N2, N, ncol, ilog2(cs), ws, h->master, h->master_len, spec, nullptr, 0, dd, 0, 0.f, nullptr, 0.f, 0);
      }
      if ((s = fc_after_launch(h)) != FC_OK) return s;
      FilterLoader fl{spec, ncol, N, omega};
      if ((s = launch_pass1(h, st, fl, sp, ncol, cs, ws, nullptr)) != FC_OK) return s;
      if ((s = launch_pass2<MID_MULH>(h, st, sp, ncol, cs2, ws, 0, hhat, invM)) != FC_OK) return s;
      if ((s = set_smem(k_pass3<EPI_SCORE, true>, sm3c)) != FC_OK) return s;
      {
        ProfScope ps(h, FC_K_PASS3, st);
        k_pass3<EPI_SCORE, true><<<dim3(sp.N2, hg), kThreads, sm3c, st>>>(
            p1, sp.N2, N, ncol, ilog2(cs), ws, h->master, h->master_len, nullptr, scores + start, h0, dd,
            total_tokens, inv, phi_c, (float)d, cg > 0 ? 1 : 0);
      }
      if ((s = fc_after_launch(h)) != FC_OK) return s;
    }
    tot_slots += (size_t)sp.N2 * (ncol / cs) * ngroups;
    hi_slots += (size_t)sp.N2 * hg * ngroups;
  }
  {
    ProfScope ps(h, FC_K_OTHER, st);
    k_energy_finalize<<<1, 256, 0, st>>>(part_tot, (int)tot_slots, part_hi, (int)hi_slots, energy_b);
  }
  return fc_after_launch(h);
}

// The internal streams wait for everything `st` has been given so far.
fc_status fork_streams(fc_handle *h, cudaStream_t st) {
  FC_CUDA_TRY(cudaEventRecord(h->ev_fork, st));
  for (int i = 0; i < h->num_aux; ++i) FC_CUDA_TRY(cudaStreamWaitEvent(h->aux[i], h->ev_fork, 0));
  return FC_OK;
}

// All sequences of `num_layers` layers that share the view's layout; energy[l][B][4].
template <typename T>
fc_status score_call(fc_handle *h, cudaStream_t st, const fc_kv_view *kv, const fc_layer_buffers *layers, int num_layers,
                     double gamma, double *energy, char *wsb) {
  const int B = kv->batch;
  const ScoreLayout L = score_layout(h, kv, num_layers);
  fc_status s;
  bool fork = true, direct_only = true, any_fast = false, any_small = false, any_passes = false, any_band = false;
  std::vector<PassPlan> plans(B);
  std::vector<const float4 *> tabs(B, nullptr);
  Jobs band;                                   // of 16-bit calls only
  std::vector<const char *> band_tabs;
  if (kv->dtype != FC_F32) {
    band.resize(B, nullptr);
    band_tabs.resize(B, nullptr);
  }
  for (int b = 0; b < B; ++b) {
    const int N = kv->cu_seqlens[b + 1] - kv->cu_seqlens[b];
    if (N == 0) continue;
    if (!h->generic_only) plans[b] = plan_passes(N, kv->head_dim);
    // what fc_set_score_overlap promises goes by the length, not by the form that scores it
    if (!plans[b].ok || (plans[b].pad && !plans[b].small)) direct_only = false;
    if (kv->dtype != FC_F32 && (band[b] = fc_band_plan(h, kv, N, cutoff_index(gamma, N))) != nullptr) {
      any_band = true;
      plans[b].ok = true;
      plans[b].small = plans[b].pad = false;
    }
    any_fast = any_fast || plans[b].ok;
    any_small = any_small || plans[b].small;
    any_passes = any_passes || (plans[b].ok && !plans[b].small);
  }
  if (any_fast && (s = prepare_tables(h, st, kv, gamma, false, reinterpret_cast<float4 *>(wsb + L.off_tab),
                                      reinterpret_cast<float2 *>(wsb + L.off_buf), tabs.data(), any_band ? band.data() : nullptr)) != FC_OK) return s;
  if (any_band && (s = band_tables(h, st, kv, band, wsb + L.off_band, band_tabs.data())) != FC_OK) return s;
  // A single sequence with little work (128-token steps per SM; from about two on, two streams are worth their fork) stays on
  // the caller's stream, without fork and join: one layer of 4 heads of 8192 tokens 81 -> 61 us by the host's clock.  Several
  // sequences run beside each other on the internal streams, and beside the short ones on the caller's: one layer of 4 heads
  // of 517, 1024, 64, 1999, 333, 4096, 100 and 2311 tokens 167 -> 93 us, of 600 and 700 45 -> 28.
  bool on_caller = false;
  if (any_band) {
    int seqs = 0;
    long long steps = 0;
    for (int b = 0; b < B; ++b) {
      const int N = kv->cu_seqlens[b + 1] - kv->cu_seqlens[b];
      if (N == 0) continue;
      ++seqs;
      steps += (long long)((N + 127) / 128) * (num_layers < FC_LAYER_CHUNK ? num_layers : FC_LAYER_CHUNK) * kv->num_heads;
    }
    on_caller = seqs == 1 && steps <= 2 * h->num_sms;
    if (on_caller && (s = fc_flush_pending(h, st)) != FC_OK) return s;
  }
  // a call that carves the workspace differently: nothing of the previous call may be in flight on the other streams
  const FcCarve carve = {wsb, L.buf_bytes, L.tot_bytes, L.hi_bytes, L.off_tot};
  const bool recarved = !(carve == h->last_carve);
  if (any_small && recarved && (s = fc_flush_pending(h, st)) != FC_OK) return s;
  if (any_fast && h->step >= 1 && recarved) {
    for (int i = 0; i < h->num_aux; ++i)
      for (int o = 0; o < h->num_aux; ++o)
        if (o != i) FC_CUDA_TRY(cudaStreamWaitEvent(h->aux[i], h->ev_done[(h->step - 1) & 1u][o], 0));
  }
  if (any_fast) h->last_carve = carve;
  for (int l0 = 0; l0 < num_layers; l0 += FC_LAYER_CHUNK) {
    const int nl = num_layers - l0 < FC_LAYER_CHUNK ? num_layers - l0 : FC_LAYER_CHUNK;
    if (any_small && any_passes && fork && !on_caller) {          // the internal streams need not wait for the short sequences
      if ((s = fork_streams(h, st)) != FC_OK) return s;
      fork = false;
    }
    if (any_small && (s = score_small<T>(h, st, kv, layers + l0, nl, plans, tabs, gamma, energy + 4 * (size_t)l0 * B,
                                         reinterpret_cast<double *>(wsb + L.off_small))) != FC_OK)
      return s;
    for (int b = 0; b < B; ++b) {
      const int start = kv->cu_seqlens[b];
      double *en = energy + 4 * ((size_t)l0 * B + b);
      if (kv->cu_seqlens[b + 1] == start) {
        k_zero_energy<<<1, 128, 0, st>>>(en, nl, 4ll * B);
        if ((s = fc_after_launch(h)) != FC_OK) return s;
        continue;
      }
      if (!plans[b].ok) {                       // generic kernels: they share the workspace and run on `st`
        if ((s = fc_flush_pending(h, st)) != FC_OK) return s;
        fork = true;
        for (int l = 0; l < nl; ++l) {
          fc_kv_view one = *kv;
          one.k = layers[l0 + l].k;
          one.v = layers[l0 + l].v;
          s = score_generic<T>(h, st, &one, b, gamma, const_cast<float *>(layers[l0 + l].scores), en + 4ll * B * l, wsb);
          if (s != FC_OK) return s;
        }
        continue;
      }
      if (plans[b].small) continue;
      if (fork && !on_caller) {
        if ((s = fork_streams(h, st)) != FC_OK) return s;
        fork = false;
      }
      fast::LayerPtrs lp = {};
      for (int l = 0; l < nl; ++l) {
        lp.k[l] = static_cast<const T *>(layers[l0 + l].k) + (long long)start * kv->stride_token;
        lp.v[l] = static_cast<const T *>(layers[l0 + l].v) + (long long)start * kv->stride_token;
        lp.scores[l] = const_cast<float *>(layers[l0 + l].scores) + start;
      }
      s = any_band && band[b] ? score_band(h, st, on_caller, kv, band[b], nl, lp, en, 4ll * B, L, wsb, band_tabs[b])
                  : score_sequence<T>(h, st, kv, plans[b], nl, lp, gamma, en, 4ll * B, L, wsb, tabs[b]);
      if (s != FC_OK) return s;
    }
  }
  // the caller's stream waits for this call's work right away, unless it asked to have that deferred
  if (!h->score_overlap || !direct_only) return fc_flush_pending(h, st);
  return FC_OK;
}

fc_status score_dispatch(fc_handle *h, cudaStream_t st, const fc_kv_view *kv, const fc_layer_buffers *layers,
                         int num_layers, double gamma, double *energy, void *workspace) {
  char *wsb = static_cast<char *>(workspace);
  switch (kv->dtype) {
    case FC_F32: return score_call<float>(h, st, kv, layers, num_layers, gamma, energy, wsb);
    case FC_F16: return score_call<__half>(h, st, kv, layers, num_layers, gamma, energy, wsb);
    default: return score_call<__nv_bfloat16>(h, st, kv, layers, num_layers, gamma, energy, wsb);
  }
}

// Column slices of one launch of k_pass2_power that run side by side (the rest are looped over).
constexpr int kPowerNY = 16;

size_t power_partial_bytes(int N) { return align_up((size_t)kPowerNY * N * sizeof(float2), 256); }

// Power spectrum of one sequence (Eq. 11) into spectrum[2*m .. 2*m+1], m < N, on the generic kernels (the power of two
// 131072) and the caller's stream.
template <typename T>
fc_status power_generic(fc_handle *h, cudaStream_t st, const fc_kv_view *kv, int b, double *spectrum, char *wsb) {
  const int start = kv->cu_seqlens[b];
  const int N = kv->cu_seqlens[b + 1] - start;
  const int d = kv->head_dim, H = kv->num_heads;
  const SeqPlan sp = plan_sequence(N);
  const GenericLayout L = generic_layout(h, sp, H, d);
  float2 *ws = reinterpret_cast<float2 *>(wsb + L.off_ws);
  float2 *partial = reinterpret_cast<float2 *>(wsb + L.total);
  double *out = spectrum + 2 * (size_t)start;
  const T *kp = static_cast<const T *>(kv->k) + (long long)start * kv->stride_token;
  const T *vp = static_cast<const T *>(kv->v) + (long long)start * kv->stride_token;
  fc_status s;
  for (int h0 = 0; h0 < H; h0 += L.heads_per_group) {
    const int hg = (H - h0 < L.heads_per_group) ? H - h0 : L.heads_per_group;
    const int ncol_ws = hg * d;
    KvLoader<T, false> ld{kp, vp, kv->stride_token, kv->stride_head, h0, d, N, 0.f, 0.f};
    if ((s = launch_pass1(h, st, ld, sp, ncol_ws, sp.cs, ws, nullptr)) != FC_OK) return s;
    const FftPlan p2 = make_plan(sp.N2);
    const size_t sm = smem_pass2(sp, sp.cs2) + (size_t)sp.N2 * 2 * sizeof(float2);
    if ((s = set_smem(k_pass2_power, sm)) != FC_OK) return s;
    const int slices = ncol_ws / sp.cs2, ny = slices < kPowerNY ? slices : kPowerNY;
    k_pass2_power<<<dim3(sp.N1 / 2 + 1, ny), kThreads, sm, st>>>(p2, sp.N1, ncol_ws, ilog2(sp.cs2), ws, h->master,
                                                                 h->master_len, partial);
    if ((s = fc_after_launch(h)) != FC_OK) return s;
    k_power_accumulate<<<(N + 255) / 256, 256, 0, st>>>(partial, ny, N, 1, out, h0 == 0 ? 1 : 0);
    if ((s = fc_after_launch(h)) != FC_OK) return s;
  }
  return FC_OK;
}

// Workspace of one fc_power_spectrum call: per internal stream an intermediate buffer and (chirp convolutions) an N-point
// spectrum, tables, and every sequence's partial sums.
struct PowerLayout {
  size_t buf_bytes, spec_bytes, off_spec, off_tab, off_part, total;
};

// Rows of partial sums of one sequence, at most: a 2*cp-channel slice each (direct), or a launch each (chirp).
inline int power_rows(const PassPlan &p, const GroupPlan &g, int H, int d) { return p.pad ? H * g.ngr : H * d / (2 * p.cp); }

PowerLayout power_layout(const fc_handle *h, const fc_kv_view *kv) {
  PowerLayout L = {};
  const int H = kv->num_heads, d = kv->head_dim;
  size_t tab = 0, part = 0, generic = 256;
  for (int b = 0; b < kv->batch; ++b) {
    const int N = kv->cu_seqlens[b + 1] - kv->cu_seqlens[b];
    if (N == 0) continue;
    const PassPlan p = plan_spectrum(N);
    if (!p.ok) {
      const size_t t = generic_layout(h, plan_sequence(N), H, d).total + power_partial_bytes(N);
      if (t > generic) generic = t;
      continue;
    }
    const GroupPlan g = plan_groups(h, p, H, H, d);
    if (g.buf_bytes > L.buf_bytes) L.buf_bytes = g.buf_bytes;
    if (p.pad) {
      const size_t sb = align_up(g.buf_bytes / p.M * N, 256);
      if (sb > L.spec_bytes) L.spec_bytes = sb;
      if (first_of_its_length(kv, b)) tab += (size_t)p.M * sizeof(float4);
    }
    part += align_up((size_t)power_rows(p, g, H, d) * N * sizeof(float2), 256);
  }
  L.off_spec = L.buf_bytes * h->num_aux;
  L.off_tab = L.off_spec + L.spec_bytes * h->num_aux;
  L.off_part = L.off_tab + align_up(tab, 256);
  L.total = L.off_part + part;
  if (generic > L.total) L.total = generic;
  return L;
}

// Power spectra of all sequences of a layer.  Launches alternate over the internal streams; each writes partial sums of
// its own, which are added in a fixed order once all streams have joined (4 layers of 32768 + 10000 tokens, 4 heads,
// cutoffs included: 3.59 ms on the generic kernels and one stream, 1.06 ms now).
template <typename T>
fc_status power_call(fc_handle *h, cudaStream_t st, const fc_kv_view *kv, double *spectrum, char *wsb) {
  const int B = kv->batch, H = kv->num_heads, d = kv->head_dim;
  const PowerLayout L = power_layout(h, kv);
  std::vector<const float4 *> tabs(B, nullptr);
  std::vector<int> ny(B, 0);
  fc_status s = FC_OK;
  bool passes = false;
  for (int b = 0; b < B; ++b) {
    const int N = kv->cu_seqlens[b + 1] - kv->cu_seqlens[b];
    if (N == 0) continue;
    if (plan_spectrum(N).ok) passes = true;
    else if ((s = power_generic<T>(h, st, kv, b, spectrum, wsb)) != FC_OK) return s;
  }
  if (!passes) return FC_OK;
  if ((s = prepare_tables(h, st, kv, 0.0, true, reinterpret_cast<float4 *>(wsb + L.off_tab), reinterpret_cast<float2 *>(wsb),
                          tabs.data())) != FC_OK)
    return s;
  if ((s = fork_streams(h, st)) != FC_OK) return s;
  size_t part = L.off_part;
  unsigned turn = 0;
  for (int b = 0; b < B; ++b) {
    const int start = kv->cu_seqlens[b], N = kv->cu_seqlens[b + 1] - start;
    if (N == 0) continue;
    const PassPlan p = plan_spectrum(N);
    if (!p.ok) continue;
    const GroupPlan g = plan_groups(h, p, H, H, d);
    fast::LayerPtrs lp = {};
    lp.k[0] = static_cast<const T *>(kv->k) + (long long)start * kv->stride_token;
    lp.v[0] = static_cast<const T *>(kv->v) + (long long)start * kv->stride_token;
    float2 *rows = reinterpret_cast<float2 *>(wsb + part);
    for (int u0 = 0; u0 < H; u0 += g.units)
      for (int cg = 0; cg < g.ngr; ++cg, ++turn) {
        const int nu = H - u0 < g.units ? H - u0 : g.units, si = (int)(turn % (unsigned)h->num_aux), ncol = nu * g.sub;
        PassArgs x{h, h->aux[si], &p, &lp, kv, u0, nu, cg * g.sub, g.sub, 0,
                   reinterpret_cast<float2 *>(wsb + (size_t)si * L.buf_bytes), tabs[b]};
        if (p.pad) {
          float2 *spec = reinterpret_cast<float2 *>(wsb + L.off_spec + (size_t)si * L.spec_bytes);
          if ((s = run_p1_chirp<T>(x)) != FC_OK) return s;
          if ((s = run_p2(x, ncol, fast::MODE_MUL)) != FC_OK) return s;
          if ((s = run_p3_spec(x, spec)) != FC_OK) return s;
          k_spec_power<<<N / 2 + 1, kThreads, 0, x.st>>>(spec, ncol, N, rows);
          if ((s = fc_after_launch(h)) != FC_OK) return s;
          rows += N;
          ++ny[b];
        } else {
          if ((s = run_p1<T>(x, nullptr, 0)) != FC_OK) return s;
          if ((s = run_p2(x, ncol, fast::MODE_POWER, nullptr, rows)) != FC_OK) return s;
          rows += (size_t)(ncol / (2 * p.cp)) * N;
          ny[b] += ncol / (2 * p.cp);
        }
      }
    part += align_up((size_t)power_rows(p, g, H, d) * N * sizeof(float2), 256);
  }
  h->pending_join = true;
  if ((s = fc_flush_pending(h, st)) != FC_OK) return s;
  part = L.off_part;
  for (int b = 0; b < B; ++b) {
    const int start = kv->cu_seqlens[b], N = kv->cu_seqlens[b + 1] - start;
    if (N == 0) continue;
    const PassPlan p = plan_spectrum(N);
    if (!p.ok) continue;
    k_power_accumulate<<<(N + 255) / 256, 256, 0, st>>>(reinterpret_cast<float2 *>(wsb + part), ny[b], N, p.pad ? 1 : p.N1,
                                                        spectrum + 2 * (size_t)start, 1);
    if ((s = fc_after_launch(h)) != FC_OK) return s;
    part += align_up((size_t)power_rows(p, plan_groups(h, p, H, H, d), H, d) * N * sizeof(float2), 256);
  }
  return FC_OK;
}

// Operation count of the chirp form: the yardstick fc_describe_plan reports for lengths that are not powers of two.
// Smallest of 2^k and 160, 192, 224 x 32..512 that is >= need (0 if none up to 131072).
inline int chirp_length(long long need) {
  int best = 0;
  for (int M = 1024; M <= 131072; M <<= 1)
    if (M >= need) { best = M; break; }
  for (int n1 = 160; n1 <= 224; n1 += 32)
    for (int n2 = 32; n2 <= 512; n2 <<= 1) {
      const int M = n1 * n2;
      if (M >= need && (best == 0 || M < best)) best = M;
    }
  return best;
}

}  // namespace

extern "C" fc_status fc_describe_plan(const fc_handle *h, int32_t seqlen, double gamma, int32_t out[4]) {
  if (!h || !out || seqlen < 1 || !(gamma >= 0.0 && gamma <= 1.0)) return FC_ERR_INVALID_ARG;
  if (seqlen > h->max_seqlen || (seqlen > 65536 && !is_pow2(seqlen))) return FC_ERR_UNSUPPORTED;
  const SeqPlan sp = plan_sequence(seqlen);
  out[0] = sp.bluestein ? 1 : 0;
  out[1] = sp.Nfft;
  const PassPlan p = plan_passes(seqlen, 0);
  out[2] = (p.ok && !p.pad) ? p.N1 : sp.N1;
  out[3] = (p.ok && !p.pad) ? p.N2 : sp.N2;
  if (sp.bluestein) {
    const int omega = cutoff_index(gamma, seqlen), Mf = chirp_length(2LL * seqlen - 1);
    bool shaped = Mf != 0 && Mf <= sp.Nfft;
    if (shaped) out[1] = Mf;
    if (h->band_form && 2LL * omega + 1 < seqlen) {
      const int Mb = chirp_length((long long)seqlen + 2LL * omega + 1);
      if (Mb != 0 && Mb < out[1]) { out[0] = 2; out[1] = Mb; shaped = true; }
    }
    if (shaped) {
      const PassPlan c = pad_shape(out[1]);
      out[2] = c.N1;
      out[3] = c.N2;
    }
  }
  return FC_OK;
}

extern "C" fc_status fc_scoring_form(const fc_handle *h, int32_t seqlen, fc_dtype dtype, int32_t head_dim, double gamma, int32_t out[2]) {
  if (!h || !out || seqlen < 1 || !(gamma >= 0.0 && gamma <= 1.0)) return FC_ERR_INVALID_ARG;
  fc_kv_view kv = {};
  const int32_t cu[2] = {0, seqlen};
  kv.dtype = dtype;
  kv.num_heads = 1;
  kv.batch = 1;
  kv.head_dim = head_dim;
  kv.stride_token = kv.stride_head = head_dim;
  kv.cu_seqlens = cu;
  const fc_status s = validate_view(h, &kv, false);
  if (s != FC_OK) return s;
  const PassPlan p = h->generic_only ? PassPlan{} : plan_passes(seqlen, head_dim);
  const int grid = h->generic_only ? 0 : fc_band_grid(&kv, seqlen, cutoff_index(gamma, seqlen));
  out[0] = grid ? FC_FORM_BAND : !p.ok ? FC_FORM_GENERIC : p.small ? FC_FORM_SHORT : p.pad ? FC_FORM_PADDED : FC_FORM_DIRECT;
  out[1] = grid ? grid : p.ok ? p.M : plan_sequence(seqlen).Nfft;
  return FC_OK;
}

extern "C" size_t fc_score_layers_workspace_bytes(const fc_handle *h, const fc_kv_view *shape, int32_t num_layers) {
  if (validate_view(h, shape, false) != FC_OK || num_layers < 1) return 0;
  return score_layout(h, shape, num_layers).total;
}

extern "C" size_t fc_score_workspace_bytes(const fc_handle *h, const fc_kv_view *kv) {
  if (validate_view(h, kv, true) != FC_OK) return 0;
  return score_layout(h, kv, 1).total;
}

extern "C" fc_status fc_score_layers(fc_handle *h, const fc_kv_view *shape, const fc_layer_buffers *layers,
                                     int32_t num_layers, double gamma, double *energy, void *workspace,
                                     size_t workspace_bytes, fc_stream stream) {
  fc_status s = validate_view(h, shape, false);
  if (s != FC_OK) return s;
  if (!layers || !energy || num_layers < 1) return FC_ERR_INVALID_ARG;
  if (!(gamma >= 0.0 && gamma <= 1.0)) return FC_ERR_INVALID_ARG;
  for (int l = 0; l < num_layers; ++l)
    if (!layers[l].k || !layers[l].v || !layers[l].scores || ((uintptr_t)layers[l].k & 15) || ((uintptr_t)layers[l].v & 15))
      return FC_ERR_INVALID_ARG;
  if (!workspace || ((uintptr_t)workspace & 255) || workspace_bytes < score_layout(h, shape, num_layers).total)
    return FC_ERR_WORKSPACE;
  int dev = -1;
  FC_CUDA_TRY(cudaGetDevice(&dev));
  if (dev != h->device) FC_CUDA_TRY(cudaSetDevice(h->device));
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  claim_persisting_l2(h, shape, num_layers, gamma, st);
  return score_dispatch(h, st, shape, layers, num_layers, gamma, energy, workspace);
}

extern "C" fc_status fc_score_layer(fc_handle *h, const fc_kv_view *kv, double gamma, float *scores,
                                    double *energy, void *workspace, size_t workspace_bytes,
                                    fc_stream stream) {
  const fc_status s = validate_view(h, kv, true);
  if (s != FC_OK) return s;
  if (!scores || !energy) return FC_ERR_INVALID_ARG;
  fc_layer_buffers one = {};
  one.k = kv->k;
  one.v = kv->v;
  one.scores = scores;
  return fc_score_layers(h, kv, &one, 1, gamma, energy, workspace, workspace_bytes, stream);
}

extern "C" size_t fc_power_spectrum_workspace_bytes(const fc_handle *h, const fc_kv_view *kv) {
  if (validate_view(h, kv, true) != FC_OK) return 0;
  return power_layout(h, kv).total;
}

extern "C" fc_status fc_power_spectrum(fc_handle *h, const fc_kv_view *kv, double *spectrum, void *workspace,
                                       size_t workspace_bytes, fc_stream stream) {
  fc_status s = validate_view(h, kv, true);
  if (s != FC_OK) return s;
  if (!spectrum) return FC_ERR_INVALID_ARG;
  const size_t need = fc_power_spectrum_workspace_bytes(h, kv);
  if (!workspace || ((uintptr_t)workspace & 255) || workspace_bytes < need) return FC_ERR_WORKSPACE;
  int dev = -1;
  FC_CUDA_TRY(cudaGetDevice(&dev));
  if (dev != h->device) FC_CUDA_TRY(cudaSetDevice(h->device));
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  if ((s = fc_flush_pending(h, st)) != FC_OK) return s;     // the workspace may still be in use on the internal streams
  switch (kv->dtype) {
    case FC_F32: return power_call<float>(h, st, kv, spectrum, (char *)workspace);
    case FC_F16: return power_call<__half>(h, st, kv, spectrum, (char *)workspace);
    default: return power_call<__nv_bfloat16>(h, st, kv, spectrum, (char *)workspace);
  }
}

// ---------------------------------------------------------------------------
// fc_cutoff_from_spectrum: the smallest omega whose kept band holds a given share of the energy.
// Bound by reading the spectrum once, so a cluster of 8 blocks shares a sequence: each of its 128 warps sums a contiguous
// segment of bins with coalesced loads, the segment totals meet in the first block's shared memory, and its first warp
// finds the segment in which the running sum first reaches share * total and walks that one (32768 + 10000 bins: 37.7 us
// with one block per sequence and a run of bins per thread, 4.2 us now).  Sums are fp64 in a fixed order (deterministic).
// ---------------------------------------------------------------------------
namespace {

constexpr int kCutThreads = 512, kCutCluster = 8, kCutSegs = kCutCluster * kCutThreads / 32;
struct CutTable { int start[65]; };

__device__ __forceinline__ double warp_inclusive(double v, int lane) {
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const double t = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += t;
  }
  return v;
}

__global__ void __cluster_dims__(kCutCluster, 1, 1) __launch_bounds__(kCutThreads)
k_cutoff_from_spectrum(const double *__restrict__ spectrum, const __grid_constant__ CutTable st, int b0, double share,
                       int *__restrict__ omega, double *__restrict__ gamma) {
  __shared__ double seg_sum[kCutSegs];
  cooperative_groups::cluster_group cluster = cooperative_groups::this_cluster();
  const int lane = threadIdx.x & 31, rank = (int)cluster.block_rank();
  const int seq = blockIdx.x / kCutCluster;
  const int s0 = st.start[seq], N = st.start[seq + 1] - s0;
  const int b = b0 + seq;
  if (N == 0) {                                       // the same for the whole cluster
    if (rank == 0 && threadIdx.x == 0) { omega[b] = 0; gamma[b] = 0.0; }
    return;
  }
  cluster.barrier_arrive();
  const double *P = spectrum + 2 * (size_t)s0;
  const int len = ((N + kCutSegs - 1) / kCutSegs + 31) & ~31;       // bins per segment
  {
    const int sg = rank * (kCutThreads / 32) + (threadIdx.x >> 5);
    const int lo = sg * len, hi = lo + len < N ? lo + len : N;
    double a = 0.0;
#pragma unroll 8
    for (int m = lo + lane; m < hi; m += 32) a += P[2 * m] + P[2 * m + 1];
    a = warp_sum_d(a);
    cluster.barrier_wait();                           // the first block has started: its memory may be written
    if (lane == 0) *cluster.map_shared_rank(&seg_sum[sg], 0) = a;
  }
  cluster.sync();
  if (rank != 0 || threadIdx.x >= 32) return;
  constexpr int PER = kCutSegs / 32;
  double run[PER], acc = 0.0;
#pragma unroll
  for (int i = 0; i < PER; ++i) { acc += seg_sum[lane * PER + i]; run[i] = acc; }
  const double incl = warp_inclusive(acc, lane);
  double before = __shfl_up_sync(0xffffffffu, incl, 1);
  if (lane == 0) before = 0.0;
  const double total = __shfl_sync(0xffffffffu, incl, 31), want = share * total;
  if (!(total > 0.0)) {
    if (lane == 0) { omega[b] = 0; gamma[b] = 0.5 / (double)N; }
    return;
  }
  // the segment that holds the crossing: the first non-empty one whose running sum has reached `want` (sums of one and
  // the same set can differ in the last bit, so "the last one reaches the total" is not relied on: without a qualifying
  // one the last non-empty one is taken)
  const int last = (N - 1) / len;
  int mine = kCutSegs;
#pragma unroll
  for (int i = PER - 1; i >= 0; --i)
    if (before + run[i] >= want) mine = lane * PER + i;
  const int first = __reduce_min_sync(0xffffffffu, mine);
  const int owner = first < last ? first : last;
  double base = before;
#pragma unroll
  for (int i = 1; i < PER; ++i)
    if (owner % PER == i) base = before + run[i - 1];
  base = __shfl_sync(0xffffffffu, base, owner / PER);
  const int lo = owner * len, hi = lo + len < N ? lo + len : N;
  int found = hi - 1;
  for (int m0 = lo; m0 < hi && found == hi - 1; m0 += 8 * 32) {
    double v[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int m = m0 + 32 * i + lane;
      const int at = 2 * (m < hi ? m : lo);
      v[i] = m < hi ? P[at] + P[at + 1] : 0.0;
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const double sum = base + warp_inclusive(v[i], lane);
      const int m = m0 + 32 * i + lane;
      const unsigned hit = __ballot_sync(0xffffffffu, m < hi && sum >= want);
      if (hit && found == hi - 1) found = m0 + 32 * i + __ffs(hit) - 1;
      base = __shfl_sync(0xffffffffu, sum, 31);
    }
  }
  if (lane == 0) {
    omega[b] = found;
    gamma[b] = ((double)found + 0.5) / (double)N;
  }
}

}  // namespace

extern "C" fc_status fc_cutoff_from_spectrum(fc_handle *h, const double *spectrum, int32_t batch,
                                             const int32_t *cu_seqlens, double share, int32_t *omega,
                                             double *gamma, fc_stream stream) {
  if (!h || !spectrum || !cu_seqlens || !omega || !gamma || batch < 0) return FC_ERR_INVALID_ARG;
  if (!(share >= 0.0 && share <= 1.0) || cu_seqlens[0] != 0) return FC_ERR_INVALID_ARG;
  for (int b = 0; b < batch; ++b)
    if (cu_seqlens[b + 1] < cu_seqlens[b]) return FC_ERR_INVALID_ARG;
  int dev = -1;
  FC_CUDA_TRY(cudaGetDevice(&dev));
  if (dev != h->device) FC_CUDA_TRY(cudaSetDevice(h->device));
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  fc_status s;
  for (int b0 = 0; b0 < batch; b0 += 64) {
    const int nseq = batch - b0 < 64 ? batch - b0 : 64;
    CutTable tab;
    for (int i = 0; i <= nseq; ++i) tab.start[i] = cu_seqlens[b0 + i];
    k_cutoff_from_spectrum<<<nseq * kCutCluster, kCutThreads, 0, st>>>(spectrum, tab, b0, share, omega, gamma);
    if ((s = fc_after_launch(h)) != FC_OK) return s;
  }
  return FC_OK;
}

// ---------------------------------------------------------------------------
// fc_score_layer_static: the same scoring with every byte of scratch in arrays that are
// part of the loaded library image, for callers that must not allocate device memory.
// ---------------------------------------------------------------------------
namespace {

constexpr int kStaticMaxSeqlen = 4096;                       // longest sequence accepted
constexpr int kStaticMasterLen = 4 * kStaticMaxSeqlen;       // same sizing rule as fc_create's table
constexpr size_t kStaticScratchBytes = FC_STATIC_SCRATCH_BYTES;

// Scratch shared by every call of fc_score_layer_static on a device; it keeps whatever the
// last call left there.  The kernels below write each region before they read it, so
// nothing has to be cleared between calls.
static __device__ __align__(256) unsigned char g_static_scratch[kStaticScratchBytes];
static __device__ __align__(256) float2 g_static_master[kStaticMasterLen];
static __device__ int g_static_status;
static __device__ unsigned g_static_counter;

// exp(-2*pi*j*i/len) in fp64, rounded once to fp32 (same definition as the handle's table).
__global__ void k_fill_static_master(float2 *master, int len) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= len) return;
  double s, c;
  sincospi(-2.0 * (double)i / (double)len, &s, &c);
  master[i] = make_float2((float)c, (float)s);
}

// Device addresses of the arrays above, looked up once per device.  In host code the
// array names stand for the symbols, not for device memory: they must never be passed
// to a kernel; cudaGetSymbolAddress gives the pointer a kernel can use.
struct StaticSetup {
  bool ready;
  unsigned char *scratch;
  float2 *master;
  int *status;
  unsigned *counter;
  int num_sms;
};
constexpr int kMaxDevices = 64;
StaticSetup g_setup[kMaxDevices];
std::mutex g_setup_mutex;

fc_status static_setup(int dev, StaticSetup *out) {
  if (dev < 0 || dev >= kMaxDevices) return FC_ERR_UNSUPPORTED;
  std::lock_guard<std::mutex> lock(g_setup_mutex);
  StaticSetup &s = g_setup[dev];
  if (!s.ready) {
    void *p_scratch = nullptr, *p_master = nullptr, *p_status = nullptr, *p_counter = nullptr;
    FC_CUDA_TRY(cudaGetSymbolAddress(&p_scratch, g_static_scratch));
    FC_CUDA_TRY(cudaGetSymbolAddress(&p_master, g_static_master));
    FC_CUDA_TRY(cudaGetSymbolAddress(&p_status, g_static_status));
    FC_CUDA_TRY(cudaGetSymbolAddress(&p_counter, g_static_counter));
    k_fill_static_master<<<(kStaticMasterLen + 255) / 256, 256>>>(static_cast<float2 *>(p_master), kStaticMasterLen);
    FC_CUDA_TRY(cudaGetLastError());
    FC_CUDA_TRY(cudaDeviceSynchronize());
    s.scratch = static_cast<unsigned char *>(p_scratch);
    s.master = static_cast<float2 *>(p_master);
    s.status = static_cast<int *>(p_status);
    s.counter = static_cast<unsigned *>(p_counter);
    FC_CUDA_TRY(cudaDeviceGetAttribute(&s.num_sms, cudaDevAttrMultiProcessorCount, dev));
    s.ready = true;
  }
  *out = s;
  return FC_OK;
}

}  // namespace

extern "C" size_t fc_static_scratch_bytes(void) { return kStaticScratchBytes; }

extern "C" fc_status fc_score_layer_static(const fc_kv_view *kv, double gamma, float *scores,
                                           double *energy, fc_stream stream) {
  if (!kv || !scores || !energy) return FC_ERR_INVALID_ARG;
  if (!(gamma >= 0.0 && gamma <= 1.0)) return FC_ERR_INVALID_ARG;
  int dev = -1;
  FC_CUDA_TRY(cudaGetDevice(&dev));
  StaticSetup su;
  fc_status s = static_setup(dev, &su);
  if (s != FC_OK) return s;
  // A handle that lives on this stack frame and owns nothing: its table, status word and
  // counter are the static arrays, and it is restricted to the single-stream kernels.
  fc_handle hs = {};
  hs.device = dev;
  hs.max_seqlen = kStaticMaxSeqlen;
  hs.master_len = kStaticMasterLen;
  hs.master = su.master;
  hs.status_word = su.status;
  hs.done_counter = su.counter;
  hs.group_bytes = 1;                 // one head per transform group: the smallest workspace
  hs.prof_class = FC_K_NONE;
  hs.generic_only = true;
  hs.num_sms = su.num_sms;
  s = validate_view(&hs, kv, true);         // lengths above kStaticMaxSeqlen come back as FC_ERR_UNSUPPORTED
  if (s != FC_OK) return s;
  if (score_layout(&hs, kv, 1).total > kStaticScratchBytes) return FC_ERR_WORKSPACE;
  fc_layer_buffers one = {};
  one.k = kv->k;
  one.v = kv->v;
  one.scores = scores;
  return score_dispatch(&hs, static_cast<cudaStream_t>(stream), kv, &one, 1, gamma, energy, su.scratch);
}

extern "C" fc_status fc_static_last_device_status(fc_stream stream) {
  int dev = -1;
  FC_CUDA_TRY(cudaGetDevice(&dev));
  StaticSetup su;
  fc_status s = static_setup(dev, &su);
  if (s != FC_OK) return s;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  FC_CUDA_TRY(cudaStreamSynchronize(st));
  int word = 0;
  FC_CUDA_TRY(cudaMemcpy(&word, su.status, sizeof(int), cudaMemcpyDeviceToHost));
  if (word != 0) FC_CUDA_TRY(cudaMemset(su.status, 0, sizeof(int)));
  if (word == 0) return FC_OK;
  return (word & FC_DEV_FLAG_INTERNAL) ? FC_ERR_INTERNAL : FC_ERR_TIMEOUT;
}
