// The three transform passes of the scoring path, for transform lengths M = N1*N2 with N1 = A*R1B (A = 16, 14, 12,
// 10; R1B = 2, 4, 8, 16) and N2 = 16*R2B, or 32*R2B where pass 2 takes its rows in two halves.  Same mathematics as
// the generic kernels in fc_score.cu (see the header comment there); what differs is the mapping:
//
//  * every thread owns two adjacent channels (one float4 = two complex values),
//    so all shared-memory and workspace accesses are 128-bit and a twiddle is
//    loaded once for two butterflies;
//  * a thread keeps a whole butterfly (A or 16 points x 2 channels) in
//    registers; the first stage of pass 1 is fed straight from the K/V rows in
//    global memory and the last stage of each pass is written straight to global
//    memory, so a tile crosses shared memory once per exchange;
//  * strides are compile-time constants;
//  * one launch covers a run of units, a unit being one KV head of one layer: the layers of a prefill share their
//    lengths, so short sequences fill the GPU layer by layer instead of launch by launch.
//
// Two forms share the kernels:
//  direct (M = N a power of two): the DCT/low-pass residual filter between the bins q and N-q (fc_score.cu).
//  padded (any N <= M/2): the residual operator I - P of Eq. 8-10 written out in the token domain.  With
//      g(t) = (1 + 2 sum_{m=1..omega} cos(pi*m*t/N)) / (2N)
//    the Base KV of Eq. 9 is  z_base[x] = sum_y (g(x-y) + g(x+y+1)) z[y]: a convolution and a correlation of the
//    tokens in their own order.  Both are products on the M-point spectrum Z of the zero-padded tokens, M >= 2N-1:
//      E[k] = c[k] Z[k] - h[k] Z[-k],   c = 1 - DFT of g wrapped around 0 (real),   h = DFT of g(t+1), t = 0..2N-2,
//    and the residual is the inverse transform's first N outputs.  One forward and one inverse transform of 2N points
//    where two chirp convolutions (four transforms of 1.4N..2N points, six launches) did the same before: a packed
//    batch of eight sequences of 7k..54k tokens went from 94.5 to 58.4 ms (28 layers x 4 heads).
//
// The transforms are left unnormalised; pass 3 folds 1/M^2 into the score.
#pragma once
#include "fc_common.cuh"

namespace fast {

__device__ __forceinline__ int perm_token(int p, int N) {
  const int half = (N + 1) >> 1;
  return p < half ? 2 * p : 2 * (N - 1 - p) + 1;
}

// two adjacent channels of one row
template <typename T> struct Load2;
template <> struct Load2<float> {
  __device__ static float2 ld(const float *p) { return __ldg(reinterpret_cast<const float2 *>(p)); }
};
template <> struct Load2<__half> {
  __device__ static float2 ld(const __half *p) {
    const unsigned u = __ldg(reinterpret_cast<const unsigned *>(p));
    return __half22float2(*reinterpret_cast<const __half2 *>(&u));
  }
};
template <> struct Load2<__nv_bfloat16> {
  __device__ static float2 ld(const __nv_bfloat16 *p) {
    const unsigned u = __ldg(reinterpret_cast<const unsigned *>(p));
    return make_float2(__uint_as_float(u << 16), __uint_as_float(u & 0xffff0000u));
  }
};

// exp(-2*pi*j*r/n) for table lengths the master table has no entries for (not a power of two)
__device__ __forceinline__ float2 root_of_unity(int r, int n) {
  double sn, cs;
  sincospi(-2.0 * (double)r / (double)n, &sn, &cs);
  return make_float2((float)cs, (float)sn);
}

// Where the layers of one launch keep their rows (first token of the sequence) and scores.
struct LayerPtrs {
  const void *k[FC_LAYER_CHUNK], *v[FC_LAYER_CHUNK];
  float *scores[FC_LAYER_CHUNK];
};

// g(t) of the padded form, |t| < 2N (even, period 2N); arguments are reduced in integers.
__device__ __forceinline__ float base_kernel(int t, int N, int omega) {
  if (t < 0) t = -t;
  if (t > N) t = 2 * N - t;
  const long long band = 2ll * omega + 1;
  if (t == 0) return (float)((double)band / (2.0 * (double)N));
  const long long r = (band * (long long)t) % (4ll * N);
  return (float)(sinpi((double)r / (2.0 * (double)N)) / (2.0 * (double)N * sinpi((double)t / (2.0 * (double)N))));
}

// exp(+j*pi*n*n/N); n*n is reduced modulo 2N (one period) in integers first.
__device__ __forceinline__ float2 chirp(int n, int N) {
  const unsigned long long r = ((unsigned long long)n * (unsigned long long)n) % (2ull * (unsigned long long)N);
  float s, c;
  sincospif(__fdiv_rn((float)(unsigned)r, (float)N), &s, &c);
  return make_float2(c, s);
}

// (|C_k[q]|^2, |C_v[q]|^2) of Eq. 11 from P = Z[q], Q = Z[N-q] of the packed sequence K + jV in the DCT's order and
// t = exp(-j*pi*q/(2N)): C[q] = alpha[q] Re(t Y[q]) with Y_k = (P + conj Q)/2, Y_v = (P - conj Q)/(2j) (alpha of Eq. 7).
__device__ __forceinline__ float2 power_of_bin(float2 P, float2 Q, float2 t, float alpha2) {
  const float ck = 0.5f * ((P.x + Q.x) * t.x - (P.y - Q.y) * t.y);
  const float cv = 0.5f * ((P.y + Q.y) * t.x - (Q.x - P.x) * t.y);
  return make_float2(alpha2 * ck * ck, alpha2 * cv * cv);
}

// What pass 1 transforms: the rows of a sequence whose length is the transform's (LD_KV), the rows of a shorter one
// with zeros behind (LD_PAD: at most half of the transform, so half of every first-stage butterfly), or the two
// convolution kernels of the padded form in the columns 0 and 1 (LD_TABLE).
// The spectrum diagnostics need the N-point spectrum itself: for lengths that are not a power of two LD_CHIRP and the
// modes MODE_MUL and OUT_SPEC compute it by one chirp convolution (rows in the DCT's even/odd order times the conjugate
// chirp, product with the chirp's spectrum, outputs times the conjugate chirp).
enum { LD_KV = 0, LD_PAD = 1, LD_TABLE = 2, LD_CHIRP = 3 };
// What pass 2 does between its halves: the residual filter of the direct form, of the padded form, a product with a
// spectrum (rows are independent), or nothing but the sums of the power spectrum (direct form, no way back).
enum { MODE_FILTER = 0, MODE_PAD = 1, MODE_MUL = 2, MODE_POWER = 3 };
// What pass 3 does with its rows: scores of the direct and of the padded form, or the N-point spectrum.
enum { OUT_SCORE = 0, OUT_PAD = 1, OUT_SPEC = 2 };

// x[p] *= w^p (CONJ: conj(w)^p), p = 1..15, for both channels, from w and w^4 alone: the other powers are products of
// at most three table values (w^p = w^(4g) * w^r), which replaces 13 of 15 shared-memory reads per use by arithmetic.
template <bool CONJ>
__device__ __forceinline__ void twiddle_powers16(float2 (&x0)[16], float2 (&x1)[16], float2 c1, float2 c4) {
  if (CONJ) { c1.y = -c1.y; c4.y = -c4.y; }
  const float2 c2 = cmul(c1, c1), c3 = cmul(c2, c1);
  float2 base = c4;
  x0[1] = cmul(x0[1], c1); x1[1] = cmul(x1[1], c1);
  x0[2] = cmul(x0[2], c2); x1[2] = cmul(x1[2], c2);
  x0[3] = cmul(x0[3], c3); x1[3] = cmul(x1[3], c3);
#pragma unroll
  for (int g = 1; g < 4; ++g) {
    const float2 b1 = cmul(base, c1), b2 = cmul(base, c2), b3 = cmul(base, c3);
    x0[4 * g] = cmul(x0[4 * g], base);     x1[4 * g] = cmul(x1[4 * g], base);
    x0[4 * g + 1] = cmul(x0[4 * g + 1], b1); x1[4 * g + 1] = cmul(x1[4 * g + 1], b1);
    x0[4 * g + 2] = cmul(x0[4 * g + 2], b2); x1[4 * g + 2] = cmul(x1[4 * g + 2], b2);
    x0[4 * g + 3] = cmul(x0[4 * g + 3], b3); x1[4 * g + 3] = cmul(x1[4 * g + 3], b3);
    if (g < 3) base = cmul(base, c4);
  }
}

// x[p] *= b * s^p (CONJ: the conjugate of that), p = 0..15, from b, s and s^4.
template <bool CONJ>
__device__ __forceinline__ void twiddle_affine16(float2 (&x0)[16], float2 (&x1)[16], float2 b, float2 s1, float2 s4) {
  if (CONJ) { b.y = -b.y; s1.y = -s1.y; s4.y = -s4.y; }
  const float2 s2 = cmul(s1, s1), s3 = cmul(s2, s1);
  float2 base = b;
#pragma unroll
  for (int g = 0; g < 4; ++g) {
    const float2 b1 = cmul(base, s1), b2 = cmul(base, s2), b3 = cmul(base, s3);
    x0[4 * g] = cmul(x0[4 * g], base);     x1[4 * g] = cmul(x1[4 * g], base);
    x0[4 * g + 1] = cmul(x0[4 * g + 1], b1); x1[4 * g + 1] = cmul(x1[4 * g + 1], b1);
    x0[4 * g + 2] = cmul(x0[4 * g + 2], b2); x1[4 * g + 2] = cmul(x1[4 * g + 2], b2);
    x0[4 * g + 3] = cmul(x0[4 * g + 3], b3); x1[4 * g + 3] = cmul(x1[4 * g + 3], b3);
    if (g < 3) base = cmul(base, s4);
  }
}

template <int R>
__device__ __forceinline__ void dft_fwd(float2 (&x)[R]) { dft_small<R, -1>(x); }
template <int R>
__device__ __forceinline__ void dft_inv(float2 (&x)[R]) { dft_small<R, +1>(x); }

// ---------------------------------------------------------------------------
// pass 1: grid (N2, columns of the launch / (2*CPW)), block CPW*R1B.
// Thread (cp = tid % CPW, j = tid / CPW): channels 2cp, 2cp+1 of the slice; first
// stage points n1 = j + R1B*p, p = 0..A-1, loaded from the K/V rows.
// The launch's columns are dcols channels, from channel c0 on, of each of the units u0, u0 + 1, ...; unit u is head
// u % H of layer u / H.  The sums of squares of a block go to slot [layer][head][64- or 32-channel slice][n2].
// ---------------------------------------------------------------------------
// Launch bounds: three resident blocks of 256 threads (80 registers), the measured best for the power-of-two path.
template <typename T, int R1B, int CPW, int LD = LD_KV, int A = 16>
__global__ void __launch_bounds__(CPW * R1B, (768 / (CPW * R1B)) > 0 ? 768 / (CPW * R1B) : 1)
k_p1(const __grid_constant__ LayerPtrs lp, long long stride_token, long long stride_head, int H, int head_dim, int u0,
     int c0, int dcols, int N, int N2, int ncol_ws, float2 *__restrict__ ws, const float2 *__restrict__ master,
     int master_len, double *__restrict__ partial, int layer_slots, int omega = 0, const float4 *__restrict__ tab = nullptr) {
  constexpr int N1 = A * R1B, NT = CPW * R1B, IT = (A + R1B - 1) / R1B, NW = (NT + 31) / 32;
  extern __shared__ float4 smem4[];
  float4 *S = smem4;                                        // [N1][CPW]
  float2 *tw = reinterpret_cast<float2 *>(S + N1 * CPW);    // [N1]
  __shared__ double red[2][NW];
  const int tid = threadIdx.x, cp = tid % CPW, j = tid / CPW;
  const int n2 = blockIdx.x, gc0 = blockIdx.y * (2 * CPW);
  int slot = 0;
  float2 x0[A], x1[A];
  float accK = 0.f, accV = 0.f;
  if (LD == LD_TABLE) {
    // columns 0 and 1, the N1 rows of this n2 shared out over the block (fp64 sines: 17 us at 96 rows with a column's own
    // threads, 5.3 us now)
    const int M = N1 * N2;
    for (int i = tid; i < N1 * CPW; i += NT) S[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    __syncthreads();
    if (gc0 == 0)
      for (int i = tid; i < 2 * N1; i += NT) {
        const int n = (i >> 1) * N2 + n2;
        float2 *at = reinterpret_cast<float2 *>(S + (i >> 1) * CPW) + (i & 1);
        if (omega < 0) {                                  // the chirp, wrapped, in column 0
          const int m = n < N ? n : n > M - N ? M - n : -1;
          if ((i & 1) == 0 && m >= 0) *at = chirp(m, N);
        } else if (i & 1) {
          if (n <= 2 * N - 2) at->x = base_kernel(n + 1, N, omega);
        } else if (n < N || n > M - N) {
          at->x = base_kernel(n < N ? n : M - n, N, omega);
        }
      }
    __syncthreads();
#pragma unroll
    for (int p = 0; p < A; ++p) {
      const float4 t = S[(j + R1B * p) * CPW + cp];
      x0[p] = make_float2(t.x, t.y);
      x1[p] = make_float2(t.z, t.w);
    }
  } else {
    const int unit = u0 + gc0 / dcols, layer = unit / H, head = unit - layer * H;
    const int ch = c0 + gc0 % dcols;
    slot = layer * layer_slots + (head * (head_dim / (2 * CPW)) + ch / (2 * CPW)) * gridDim.x + n2;
    const T *kb = static_cast<const T *>(lp.k[layer]) + (long long)head * stride_head + ch + 2 * cp;
    const T *vb = static_cast<const T *>(lp.v[layer]) + (long long)head * stride_head + ch + 2 * cp;
    if (LD == LD_PAD || LD == LD_CHIRP) {
      // rows past the sequence read row 0 and are zeroed
      float2 z0[A / 2], z1[A / 2];
#pragma unroll
      for (int p = 0; p < A / 2; ++p) {
        const int n = (j + R1B * p) * N2 + n2;
        const long long off = (long long)(n < N ? (LD == LD_CHIRP ? perm_token(n, N) : n) : 0) * stride_token;
        const float2 kk = Load2<T>::ld(kb + off), vv = Load2<T>::ld(vb + off);
        z0[p] = n < N ? make_float2(kk.x, vv.x) : make_float2(0.f, 0.f);
        z1[p] = n < N ? make_float2(kk.y, vv.y) : make_float2(0.f, 0.f);
      }
      for (int i = tid; i < N1; i += NT) tw[i] = (A == 16) ? master[(size_t)i * (master_len / N1)] : root_of_unity(i, N1);
      __syncthreads();
#pragma unroll
      for (int p = 0; p < A / 2; ++p) {
        accK = fmaf(z0[p].x, z0[p].x, fmaf(z1[p].x, z1[p].x, accK));
        accV = fmaf(z0[p].y, z0[p].y, fmaf(z1[p].y, z1[p].y, accV));
      }
      if (LD == LD_CHIRP) {
#pragma unroll
        for (int p = 0; p < A / 2; ++p) {
          const int n = (j + R1B * p) * N2 + n2;
          const float4 t = __ldg(tab + (n < N ? n : 0));
          z0[p] = cmul_conj(z0[p], make_float2(t.z, t.w));
          z1[p] = cmul_conj(z1[p], make_float2(t.z, t.w));
        }
      }
      dft_zero_tail<A>(z0, x0);
      dft_zero_tail<A>(z1, x1);
    } else {
#pragma unroll
      for (int p = 0; p < A; ++p) {
        const int n = (j + R1B * p) * N2 + n2;
        const long long off = (long long)perm_token(n, N) * stride_token;
        const float2 kk = Load2<T>::ld(kb + off), vv = Load2<T>::ld(vb + off);
        x0[p] = make_float2(kk.x, vv.x);
        x1[p] = make_float2(kk.y, vv.y);
      }
    }
  }
  if (LD != LD_PAD && LD != LD_CHIRP) {
    for (int i = tid; i < N1; i += NT) tw[i] = (A == 16) ? master[(size_t)i * (master_len / N1)] : root_of_unity(i, N1);
    __syncthreads();
    if (LD == LD_KV) {
#pragma unroll
      for (int p = 0; p < A; ++p) {
        accK = fmaf(x0[p].x, x0[p].x, fmaf(x1[p].x, x1[p].x, accK));
        accV = fmaf(x0[p].y, x0[p].y, fmaf(x1[p].y, x1[p].y, accV));
      }
    }
    dft_fwd<A>(x0);
    dft_fwd<A>(x1);
  }
#pragma unroll
  for (int p = 0; p < A; ++p) {
    if (p > 0) {
      const float2 w = tw[j * p];
      x0[p] = cmul(x0[p], w);
      x1[p] = cmul(x1[p], w);
    }
    S[(j + R1B * p) * CPW + cp] = make_float4(x0[p].x, x0[p].y, x1[p].x, x1[p].y);
  }
  __syncthreads();
  // second stage: radix R1B inside sub-block pp; bin k1 = pp + A*q
#pragma unroll
  for (int it = 0; it < IT; ++it) {
    const int pp = j + R1B * it;
    if (A % R1B != 0 && pp >= A) break;
    float2 y0[R1B], y1[R1B];
#pragma unroll
    for (int q = 0; q < R1B; ++q) {
      const float4 t = S[(q + R1B * pp) * CPW + cp];
      y0[q] = make_float2(t.x, t.y);
      y1[q] = make_float2(t.z, t.w);
    }
    dft_fwd<R1B>(y0);
    dft_fwd<R1B>(y1);
    float4 *dst = reinterpret_cast<float4 *>(ws + ((size_t)pp * N2 + n2) * ncol_ws + gc0 + 2 * cp);
#pragma unroll
    for (int q = 0; q < R1B; ++q) {
      *dst = make_float4(y0[q].x, y0[q].y, y1[q].x, y1[q].y);
      dst += (size_t)A * N2 * ncol_ws / 2;
    }
  }
  if (LD == LD_TABLE || LD == LD_CHIRP || partial == nullptr) return;
  // per-block sums of squares (total energy of Eq. 12, by Parseval)
  const double a = warp_sum_d((double)accK), b = warp_sum_d((double)accV);
  if ((tid & 31) == 0) { red[0][tid >> 5] = a; red[1][tid >> 5] = b; }
  __syncthreads();
  if (tid == 0) {
    double sa = 0, sb = 0;
#pragma unroll
    for (int i = 0; i < NW; ++i) { sa += red[0][i]; sb += red[1][i]; }
    partial[2 * (size_t)slot] = sa;
    partial[2 * (size_t)slot + 1] = sb;
  }
}

// ---------------------------------------------------------------------------
// pass 2: grid (N1/2, columns of the launch / (2*CP)); block 2*CP*R2B.
// Thread (cp = tid % CP, hf = (tid / CP) & 1, j = tid / (2*CP)): channel pair cp of
// the slice, half hf (k1 = blockIdx.x or N1 - blockIdx.x), first-stage points
// n2 = j + R2B*p.
// Between its forward and inverse halves: the DCT/low-pass residual filter (direct form), or E = c Z[k] - h Z[-k] with
// (c, h) from the table (padded form); either way bin k meets its partner M-k, which lies in the block's other row.
// tab_out (padded form): forward half only, of the convolution kernels in the columns 0 and 1; the table entries of
// this block's bins are written instead.  Tables are laid out [k1][k2].
// ---------------------------------------------------------------------------
template <int R2B, int CP, int MODE = MODE_FILTER>
__global__ void __launch_bounds__(2 * CP * R2B, 512 / (2 * CP * R2B > 32 ? 2 * CP * R2B : 32))
k_p2(int N1, int ncol_ws, float2 *__restrict__ ws, const float2 *__restrict__ master, int master_len, int omega,
     const float4 *__restrict__ tab, float4 *__restrict__ tab_out, float2 *__restrict__ power, int Nseq) {
  constexpr bool TAB = MODE == MODE_PAD || MODE == MODE_MUL;
  constexpr int N2 = 16 * R2B, NT = 2 * CP * R2B, IT = 16 / R2B;
  extern __shared__ float4 smem4[];
  float4 *S = smem4;                                         // [2][N2][CP]
  // only the table values the products below start from are kept: w_N2^j and w_N2^4j, and per row k1 the twiddles
  // w_N^(k1*j) with the steps w_N^(k1*R2B) and w_N^(k1*4*R2B) behind them
  constexpr int HN = R2B + 2;
  float2 *tw = reinterpret_cast<float2 *>(S + 2 * N2 * CP);  // [2][R2B]
  float2 *twN = tw + 2 * R2B;                                // [2][HN]
  // the second half starts H2 = N2 + 4 entries in, so that threads of the two halves reading the same index hit
  // different banks
  constexpr int H2 = N2 + 4;
  float2 *uT = twN + 2 * HN;                                 // [2][N2] exp(-j*pi*(k1 + N1*k2)/N)
  const int tid = threadIdx.x, cp = tid % CP, hf = (tid / CP) & 1, j = tid / (2 * CP);
  // block x > 0 holds the partner rows x and N1 - x, block 0 the two rows that are their own partners, 0 and N1/2
  // (each half then reads its partner bins from itself)
  const int k1a = blockIdx.x, k1b = k1a == 0 ? N1 / 2 : N1 - k1a;
  const bool self = k1a == 0;
  const int k1 = hf ? k1b : k1a;
  const int N = N1 * N2;
  const int gc0 = blockIdx.y * (2 * CP);
  // padded form: the (h, c) entries of the block's two rows in place of uT
  float4 *hc = reinterpret_cast<float4 *>(uT);               // [2][N2]
  {
    const int ustep = master_len / (2 * N);
    for (int i = tid; i < N2; i += NT) {
      if (TAB) {
        if (tab_out == nullptr) {
          hc[i] = __ldg(tab + (size_t)k1a * N2 + i);
          hc[N2 + i] = __ldg(tab + (size_t)k1b * N2 + i);
        }
      } else {
        // exp(-j*pi*q/N) of the filter, exp(-j*pi*q/(2N)) of the power spectrum
        uT[i] = master[(size_t)(k1a + N1 * i) * (MODE == MODE_POWER ? ustep / 2 : ustep)];
        uT[H2 + i] = master[(size_t)(k1b + N1 * i) * (MODE == MODE_POWER ? ustep / 2 : ustep)];
      }
    }
    for (int i = tid; i < 2 * R2B; i += NT)
      tw[i] = master[(size_t)(i < R2B ? i : 4 * (i - R2B)) * (master_len / N2)];
    // N is a power of two (every root is in the master table) or, in the padded form, 2^a * {3, 5, 7}
    const bool in_master = (master_len % N) == 0;
    for (int i = tid; i < 2 * HN; i += NT) {
      const int half = i / HN, e = i - half * HN;
      const int r = ((e < R2B ? e : e == R2B ? R2B : 4 * R2B) * (half ? k1b : k1a)) % N;
      twN[i] = in_master ? master[(size_t)r * (master_len / N)] : root_of_unity(r, N);
    }
  }
  float4 *Sh = S + hf * (N2 * CP);
  const float2 *twR = twN + hf * HN;
  float2 x0[16], x1[16];
  float4 *base = reinterpret_cast<float4 *>(ws + ((size_t)k1 * N2 + j) * ncol_ws + gc0 + 2 * cp);
  const float4 *src = base;
#pragma unroll
  for (int p = 0; p < 16; ++p) {
    const float4 t = __ldcg(src);
    src += (size_t)R2B * ncol_ws / 2;
    x0[p] = make_float2(t.x, t.y);
    x1[p] = make_float2(t.z, t.w);
  }
  __syncthreads();
  twiddle_affine16<false>(x0, x1, twR[j], twR[R2B], twR[R2B + 1]);
  dft_fwd<16>(x0);
  dft_fwd<16>(x1);
  twiddle_powers16<false>(x0, x1, tw[j], tw[R2B + j]);
#pragma unroll
  for (int p = 0; p < 16; ++p)
    Sh[(j + R2B * p) * CP + cp] = make_float4(x0[p].x, x0[p].y, x1[p].x, x1[p].y);
  __syncthreads();
  // second forward stage, written back in place (each sub-block is touched by one thread only);
  // registers keep bins k2 = pp + 16*q at index it*R2B + q
#pragma unroll
  for (int it = 0; it < IT; ++it) {
    const int pp = j + R2B * it;
    float2 y0[R2B], y1[R2B];
#pragma unroll
    for (int q = 0; q < R2B; ++q) {
      const float4 t = Sh[(q + R2B * pp) * CP + cp];
      y0[q] = make_float2(t.x, t.y);
      y1[q] = make_float2(t.z, t.w);
    }
    dft_fwd<R2B>(y0);
    dft_fwd<R2B>(y1);
#pragma unroll
    for (int q = 0; q < R2B; ++q) {
      x0[it * R2B + q] = y0[q];
      x1[it * R2B + q] = y1[q];
      // direct form: only bins inside the two bands are read by their partners (the partner of an in-band bin is
      // in the other band), so the rest, 1 - 2*gamma of them, is not written back
      bool wanted = MODE != MODE_MUL;
      if (MODE == MODE_FILTER) {
        const int bin = k1 + N1 * (pp + 16 * q);
        wanted = bin <= omega || N - bin <= omega;
      }
      if (wanted) Sh[(q + R2B * pp) * CP + cp] = make_float4(y0[q].x, y0[q].y, y1[q].x, y1[q].y);
    }
  }
  if (TAB && tab_out != nullptr) {            // x0: spectrum of g around 0 or of the chirp, x1: spectrum of g(t + 1)
    if (cp == 0 && blockIdx.y == 0) {
#pragma unroll
      for (int it = 0; it < IT; ++it)
#pragma unroll
        for (int q = 0; q < R2B; ++q) {
          const int at = k1 * N2 + j + R2B * it + 16 * q;
          const float2 a = x0[it * R2B + q], b = x1[it * R2B + q];
          if (MODE == MODE_MUL) {             // the chirp of row `at` beside it
            const float2 c = at < Nseq ? chirp(at, Nseq) : make_float2(0.f, 0.f);
            tab_out[at] = make_float4(a.x, a.y, c.x, c.y);
          } else {
            tab_out[at] = make_float4(b.x, b.y, 1.f - a.x, 0.f);
          }
        }
    }
    return;
  }
  if (MODE != MODE_MUL) __syncthreads();      // spectra of both rows are in shared memory
  const float4 *Sp = S + (self ? hf : 1 - hf) * (N2 * CP);
#pragma unroll
  for (int it = 0; it < IT; ++it) {
    const int pp = j + R2B * it;
#pragma unroll
    for (int q = 0; q < R2B; ++q) {
      const int k2 = pp + 16 * q;
      const int bin = k1 + N1 * k2;
      const int k2p = (k1 == 0) ? ((N2 - k2) & (N2 - 1)) : (N2 - 1 - k2);
      if (MODE == MODE_MUL) {
        const float4 w = hc[hf * N2 + k2];
        x0[it * R2B + q] = cmul(x0[it * R2B + q], make_float2(w.x, w.y));
        x1[it * R2B + q] = cmul(x1[it * R2B + q], make_float2(w.x, w.y));
        continue;
      }
      if (MODE == MODE_POWER) {               // both channels' powers replace the bins
        const float4 t = Sp[((k2p >> 4) + R2B * (k2p & 15)) * CP + cp];
        const float2 u = uT[hf * H2 + k2];
        const float alpha2 = (bin == 0 ? 1.f : 2.f) / (float)N;
        const float2 a = power_of_bin(x0[it * R2B + q], make_float2(t.x, t.y), u, alpha2);
        const float2 b = power_of_bin(x1[it * R2B + q], make_float2(t.z, t.w), u, alpha2);
        x0[it * R2B + q] = make_float2(a.x + b.x, a.y + b.y);
        continue;
      }
      if (MODE == MODE_PAD) {
        const float4 t = Sp[((k2p >> 4) + R2B * (k2p & 15)) * CP + cp], w = hc[hf * N2 + k2];
        float2 &P0 = x0[it * R2B + q], &P1 = x1[it * R2B + q];
        P0 = make_float2(fmaf(t.y, w.y, fmaf(-t.x, w.x, w.z * P0.x)), fmaf(-t.y, w.x, fmaf(-t.x, w.y, w.z * P0.y)));
        P1 = make_float2(fmaf(t.w, w.y, fmaf(-t.z, w.x, w.z * P1.x)), fmaf(-t.w, w.x, fmaf(-t.z, w.y, w.z * P1.y)));
        continue;
      }
      const bool inL = bin <= omega, inH = (N - bin) <= omega;
      float2 &P0 = x0[it * R2B + q], &P1 = x1[it * R2B + q];
      if (bin == 0 || (inL && inH)) {
        P0 = make_float2(0.f, 0.f);
        P1 = make_float2(0.f, 0.f);
      } else if (inL || inH) {
        const float4 t = Sp[((k2p >> 4) + R2B * (k2p & 15)) * CP + cp];
        float2 u = uT[hf * H2 + k2];                             // exp(-j*pi*bin/N)
        const float sgn = inL ? -0.5f : 0.5f;                   // E = (P -/+ uQ)/2 with u = exp(+j*pi*bin/N)
        u = make_float2(u.x * sgn, -u.y * sgn);
        const float2 q0 = make_float2(t.x, t.y), q1 = make_float2(t.z, t.w);
        P0 = make_float2(fmaf(q0.x, u.x, fmaf(-q0.y, u.y, 0.5f * P0.x)),
                         fmaf(q0.x, u.y, fmaf(q0.y, u.x, 0.5f * P0.y)));
        P1 = make_float2(fmaf(q1.x, u.x, fmaf(-q1.y, u.y, 0.5f * P1.x)),
                         fmaf(q1.x, u.y, fmaf(q1.y, u.x, 0.5f * P1.y)));
      }
    }
  }
  if (MODE == MODE_POWER) {
    // sums over the slice's channels: transposed reduction over the CP lanes that share (row, j), the 16 bins halved at
    // every step; bin index = it*R2B + q
    int count = 16, first = 0;
#pragma unroll
    for (int st = CP / 2; st >= 1; st >>= 1) {
      if (count > 1) {
        const int half = count / 2;
        const bool up = (cp & st) != 0;
#pragma unroll
        for (int i = 0; i < half; ++i) {
          const float2 send = up ? x0[i] : x0[i + half], keep = up ? x0[i + half] : x0[i];
          x0[i] = make_float2(keep.x + __shfl_xor_sync(0xffffffffu, send.x, st), keep.y + __shfl_xor_sync(0xffffffffu, send.y, st));
        }
        if (up) first += half;
        count = half;
      } else {
        x0[0] = make_float2(x0[0].x + __shfl_xor_sync(0xffffffffu, x0[0].x, st), x0[0].y + __shfl_xor_sync(0xffffffffu, x0[0].y, st));
      }
    }
    constexpr int KEEP = CP >= 16 ? 1 : 16 / CP;
    if (CP <= 16 || (cp & (CP / 16 - 1)) == 0) {
      float2 *dst = power + (size_t)blockIdx.y * N + (size_t)k1 * N2;
#pragma unroll
      for (int i = 0; i < KEEP; ++i) {
        const int e = first + i;
        dst[j + R2B * (e / R2B) + 16 * (e % R2B)] = x0[i];
      }
    }
    return;
  }
  // first inverse stage (mirror of the second forward stage)
#pragma unroll
  for (int it = 0; it < IT; ++it) {
    float2 y0[R2B], y1[R2B];
#pragma unroll
    for (int q = 0; q < R2B; ++q) { y0[q] = x0[it * R2B + q]; y1[q] = x1[it * R2B + q]; }
    dft_inv<R2B>(y0);
    dft_inv<R2B>(y1);
#pragma unroll
    for (int q = 0; q < R2B; ++q) { x0[it * R2B + q] = y0[q]; x1[it * R2B + q] = y1[q]; }
  }
  if (MODE != MODE_MUL) __syncthreads();      // all partner reads are done
#pragma unroll
  for (int it = 0; it < IT; ++it) {
    const int pp = j + R2B * it;
#pragma unroll
    for (int q = 0; q < R2B; ++q)
      Sh[(q + R2B * pp) * CP + cp] = make_float4(x0[it * R2B + q].x, x0[it * R2B + q].y,
                                                x1[it * R2B + q].x, x1[it * R2B + q].y);
  }
  __syncthreads();
#pragma unroll
  for (int p = 0; p < 16; ++p) {
    const float4 t = Sh[(j + R2B * p) * CP + cp];
    x0[p] = make_float2(t.x, t.y);
    x1[p] = make_float2(t.z, t.w);
  }
  twiddle_powers16<true>(x0, x1, tw[j], tw[R2B + j]);
  dft_inv<16>(x0);
  dft_inv<16>(x1);
  twiddle_affine16<true>(x0, x1, twR[j], twR[R2B], twR[R2B + 1]);
  asm volatile("" : "+r"(ncol_ws));           // the row addresses are formed again rather than kept from the loads
#pragma unroll
  for (int p = 0; p < 16; ++p) {
    *base = make_float4(x0[p].x, x0[p].y, x1[p].x, x1[p].y);
    base += (size_t)R2B * ncol_ws / 2;
  }
}


// ---------------------------------------------------------------------------
// pass 2 of the padded form for rows of 512 points: a thread holds 32 points of ONE channel (the same 64 data registers
// as 16 points of two), two radix-16 butterflies in the outer stage and one of radix 32 in the inner one, so a row
// crosses shared memory as often as one of 256 points.  grid (N1/2, columns / C), block 32*C: C = 8 channels are 64-byte
// pieces of the workspace rows and 256 threads with 75 KB, two blocks per SM like the other passes.  (Joining two
// 256-point transforms by a radix-2 step instead reads seven values per point around the filter: 28 layers x 4 heads of
// 38158 tokens took 16.2 ms against 13.4 ms.)
// ---------------------------------------------------------------------------
__device__ __forceinline__ void twiddle_powers16_one(float2 (&x)[16], float2 c1, float2 c4, bool conj) {
  if (conj) { c1.y = -c1.y; c4.y = -c4.y; }
  const float2 c2 = cmul(c1, c1), c3 = cmul(c2, c1);
  float2 base = c4;
  x[1] = cmul(x[1], c1); x[2] = cmul(x[2], c2); x[3] = cmul(x[3], c3);
#pragma unroll
  for (int g = 1; g < 4; ++g) {
    x[4 * g] = cmul(x[4 * g], base);
    x[4 * g + 1] = cmul(x[4 * g + 1], cmul(base, c1));
    x[4 * g + 2] = cmul(x[4 * g + 2], cmul(base, c2));
    x[4 * g + 3] = cmul(x[4 * g + 3], cmul(base, c3));
    if (g < 3) base = cmul(base, c4);
  }
}
__device__ __forceinline__ void twiddle_affine16_one(float2 (&x)[16], float2 b, float2 s1, float2 s4, bool conj) {
  if (conj) { b.y = -b.y; s1.y = -s1.y; s4.y = -s4.y; }
  const float2 s2 = cmul(s1, s1), s3 = cmul(s2, s1);
  float2 base = b;
#pragma unroll
  for (int g = 0; g < 4; ++g) {
    x[4 * g] = cmul(x[4 * g], base);
    x[4 * g + 1] = cmul(x[4 * g + 1], cmul(base, s1));
    x[4 * g + 2] = cmul(x[4 * g + 2], cmul(base, s2));
    x[4 * g + 3] = cmul(x[4 * g + 3], cmul(base, s3));
    if (g < 3) base = cmul(base, s4);
  }
}

template <int C, int MODE>
__global__ void __launch_bounds__(32 * C, 2)
k_p2_512(int N1, int ncol_ws, float2 *__restrict__ ws, const float2 *__restrict__ master, int master_len,
         const float4 *__restrict__ tab, float4 *__restrict__ tab_out, int Nseq) {
  constexpr int ROW = 512, NT = 32 * C;
  constexpr int SUB = 32 * C + (C < 16 ? C : 0);              // groups of 32 points, padded against bank conflicts
  constexpr int HALF = 16 * SUB;
  extern __shared__ float4 smem4[];
  float2 *S = reinterpret_cast<float2 *>(smem4);              // [row][HALF]
  float4 *hc = reinterpret_cast<float4 *>(S + 2 * HALF);      // [2][512] (h, c) of the two rows
  float2 *tw = reinterpret_cast<float2 *>(hc + 2 * ROW);      // [2][32] w_512^j, w_512^4j
  float2 *twN = tw + 64;                                      // [2][34] w_N^(k1*j) and its steps of 32 and 128 points
  const int tid = threadIdx.x, c = tid % C, j = (tid / C) % 16, row = tid / (16 * C);
  const int k1a = blockIdx.x, k1b = k1a == 0 ? N1 / 2 : N1 - k1a;
  const int k1 = row ? k1b : k1a;
  const int N = N1 * ROW;
  float2 x[2][16];                                            // points j + 16*b + 32*p
  float2 *base = ws + ((size_t)k1 * ROW + j) * ncol_ws + blockIdx.y * C + c;
#pragma unroll
  for (int b = 0; b < 2; ++b)
#pragma unroll
    for (int p = 0; p < 16; ++p) x[b][p] = __ldcg(base + (size_t)(16 * b + 32 * p) * ncol_ws);
  if (tab_out == nullptr)
    for (int i = tid; i < 2 * ROW; i += NT) hc[i] = __ldg(tab + (size_t)(i < ROW ? k1a : k1b) * ROW + (i & (ROW - 1)));
  for (int i = tid; i < 64; i += NT) tw[i] = master[(size_t)(i < 32 ? i : 4 * (i - 32)) * (master_len / ROW)];
  {
    const bool in_master = (master_len % N) == 0;
    for (int i = tid; i < 2 * 34; i += NT) {
      const int r2 = i / 34, e = i - r2 * 34;
      const int r = ((e < 32 ? e : e == 32 ? 32 : 128) * (r2 ? k1b : k1a)) % N;
      twN[i] = in_master ? master[(size_t)r * (master_len / N)] : root_of_unity(r, N);
    }
  }
  float2 *S1 = S + row * HALF + j * C + c;                    // + 16*b*C + p*SUB
  float2 *S2 = S + row * HALF + j * SUB + c;                  // + q*C
  const float2 *twR = twN + row * 34;
  __syncthreads();
#pragma unroll
  for (int b = 0; b < 2; ++b) {
    twiddle_affine16_one(x[b], twR[j + 16 * b], twR[32], twR[33], false);
    dft_fwd<16>(x[b]);
    twiddle_powers16_one(x[b], tw[j + 16 * b], tw[32 + j + 16 * b], false);
#pragma unroll
    for (int p = 0; p < 16; ++p) S1[16 * b * C + p * SUB] = x[b][p];
  }
  __syncthreads();
  // radix 32 over the points of group j: x[b][i] takes point 2i + b, then x[b][i] is bin k2 = j + 16*(i + 16*b)
#pragma unroll
  for (int b = 0; b < 2; ++b) {
#pragma unroll
    for (int i = 0; i < 16; ++i) x[b][i] = S2[(2 * i + b) * C];
    dft_fwd<16>(x[b]);
  }
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    const float2 o = cmul(x[1][i], make_float2(root32_cos(i), -root32_sin(i)));
    x[1][i] = csub(x[0][i], o);
    x[0][i] = cadd(x[0][i], o);
    S2[i * C] = x[0][i];
    S2[(i + 16) * C] = x[1][i];
  }
  if (tab_out != nullptr) {              // channel 0: spectrum of g around 0, channel 1: of g(t + 1)
    __syncthreads();
    if (c == 0 && blockIdx.y == 0)
      for (int q = 0; q < 32; ++q) {
        const float2 g0 = S2[q * C], g1 = S2[q * C + 1];
        const int at = k1 * ROW + j + 16 * q;
        if (MODE == MODE_MUL) {
          const float2 cf = at < Nseq ? chirp(at, Nseq) : make_float2(0.f, 0.f);
          tab_out[at] = make_float4(g0.x, g0.y, cf.x, cf.y);
        } else {
          tab_out[at] = make_float4(g1.x, g1.y, 1.f - g0.x, 0.f);
        }
      }
    return;
  }
  __syncthreads();
  {
    // partner of bin k2: 512 - k2 in row 0, 511 - k2 in the others; it sits in group 15 - j (row 0: -j mod 16) of the
    // partner row, at q' = 31 - q (row 0, j = 0: 32 - q, bin 0 with itself)
    const bool first = k1 == 0 && j == 0;
    const int prow = k1a == 0 ? row : 1 - row, pj = k1 == 0 ? ((16 - j) & 15) : 15 - j;
    const float2 *Sp = S + prow * HALF + pj * SUB + c + (first ? 32 : 31) * C;
    const float4 *hrow = hc + row * ROW + j;
#pragma unroll
    for (int q = 0; q < 32; ++q) {
      float2 &P = x[q >> 4][q & 15];
      if (MODE == MODE_MUL) {
        const float4 m = hrow[16 * q];
        P = cmul(P, make_float2(m.x, m.y));
        continue;
      }
      const float2 t = Sp[q == 0 && first ? -32 * C : -q * C];
      const float4 w = hrow[16 * q];
      P = make_float2(fmaf(t.y, w.y, fmaf(-t.x, w.x, w.z * P.x)), fmaf(-t.y, w.x, fmaf(-t.x, w.y, w.z * P.y)));
    }
  }
  __syncthreads();                       // all partner reads are done
  // inverse radix 32: point 2i + b from the sums (b = 0) and rotated differences (b = 1)
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    const float2 d = csub(x[0][i], x[1][i]);
    x[0][i] = cadd(x[0][i], x[1][i]);
    x[1][i] = cmul(d, make_float2(root32_cos(i), root32_sin(i)));
  }
#pragma unroll
  for (int b = 0; b < 2; ++b) {
    dft_inv<16>(x[b]);
#pragma unroll
    for (int i = 0; i < 16; ++i) S2[(2 * i + b) * C] = x[b][i];
  }
  __syncthreads();
#pragma unroll
  for (int b = 0; b < 2; ++b) {
#pragma unroll
    for (int p = 0; p < 16; ++p) x[b][p] = S1[16 * b * C + p * SUB];
    twiddle_powers16_one(x[b], tw[j + 16 * b], tw[32 + j + 16 * b], true);
    dft_inv<16>(x[b]);
    twiddle_affine16_one(x[b], twR[j + 16 * b], twR[32], twR[33], true);
#pragma unroll
    for (int p = 0; p < 16; ++p) base[(size_t)(16 * b + 32 * p) * ncol_ws] = x[b][p];
  }
}

// ---------------------------------------------------------------------------
// pass 3: grid (N2, units of the launch), block CPW*R1B.  Inverse DFT over k1,
// squared magnitude summed over the unit's channels, scores and the
// per-block outlier-energy partial sums.  The last block of a layer (over all launches of the sequence, on either
// stream) reduces that layer's partial sums to its energies.
// PAD: row n1*N2 + n2 is that token and only rows below N exist (at most the first half of the transform, so half of
// every last-stage butterfly); direct form: the rows are in the even/odd order of the DCT.
// A unit transformed in column groups: dcols is the group's width, accumulate adds to the stored score (groups after
// the first), hi_base is the group's first slot of the layer's outlier-energy sums.
// ---------------------------------------------------------------------------
struct EnergyOut {
  double *part_hi;               // [layer][hi_slots][2]
  const double *part_tot;        // [layer][tot_slots][2]
  int hi_slots, tot_slots;       // per layer
  unsigned *done;                // [layer], zero between sequences
  unsigned total_blocks;         // pass-3 blocks of one layer
  double *energy;                // [layer][energy_stride]
  long long energy_stride;
};

template <int R1B, int CPW, int OUT = OUT_SCORE, int A = 16>
__global__ void __launch_bounds__(CPW * R1B, 512 / (CPW * R1B))
k_p3(const __grid_constant__ LayerPtrs lp, int H, int head_dim, int u0, int dcols, int N, int N2, int ncol_ws,
     const float2 *__restrict__ ws, const float2 *__restrict__ master, int master_len, long long score_stride,
     float inv_scale, int accumulate, int hi_base, const __grid_constant__ EnergyOut eo,
     float2 *__restrict__ spec = nullptr, const float4 *__restrict__ tab = nullptr) {
  // OUT_SPEC: row n < N times conj(chirp(n)) and inv_scale to spec[n][column]; nothing else
  constexpr bool PAD = OUT != OUT_SCORE;
  constexpr int N1 = A * R1B, NT = CPW * R1B, IT = (A + R1B - 1) / R1B, NW = (NT + 31) / 32;
  constexpr int AO = PAD ? A / 2 : A;                       // rows a thread ends with
  constexpr int PR = PAD ? 8 : 16;                          // the same, rounded up to a power of two
  extern __shared__ float4 smem4[];
  float4 *S = smem4;                                        // [N1][CPW]
  float2 *tw = reinterpret_cast<float2 *>(S + N1 * CPW);    // [N1]
  __shared__ double red[2][NW];
  const int tid = threadIdx.x, cp = tid % CPW, j = tid / CPW;
  const int n2 = blockIdx.x, unit = u0 + blockIdx.y, layer = unit / H, head = unit - layer * H;
  for (int i = tid; i < N1; i += NT) tw[i] = (A == 16) ? master[(size_t)i * (master_len / N1)] : root_of_unity(i, N1);

  float acc[PR];            // |residual|^2 of rows j + R1B*p summed over this thread's channels (K and V)
#pragma unroll
  for (int i = 0; i < PR; ++i) acc[i] = 0.f;
  float totK = 0.f, totV = 0.f;

  const int nslices = dcols / (2 * CPW);
  for (int sl = 0; sl < nslices; ++sl) {
    const int gc0 = blockIdx.y * dcols + sl * (2 * CPW);
    // inverse radix-R1B stage on bins k1 = pp + A*q, straight from the workspace
#pragma unroll
    for (int it = 0; it < IT; ++it) {
      const int pp = j + R1B * it;
      if (A % R1B != 0 && pp >= A) break;
      float2 y0[R1B], y1[R1B];
      const float4 *src = reinterpret_cast<const float4 *>(ws + ((size_t)pp * N2 + n2) * ncol_ws + gc0 + 2 * cp);
#pragma unroll
      for (int q = 0; q < R1B; ++q) {
        const float4 t = __ldcg(src);
        src += (size_t)A * N2 * ncol_ws / 2;
        y0[q] = make_float2(t.x, t.y);
        y1[q] = make_float2(t.z, t.w);
      }
      dft_inv<R1B>(y0);
      dft_inv<R1B>(y1);
#pragma unroll
      for (int q = 0; q < R1B; ++q)
        S[(q + R1B * pp) * CPW + cp] = make_float4(y0[q].x, y0[q].y, y1[q].x, y1[q].y);
    }
    __syncthreads();
    float2 z0[AO], z1[AO];
    auto twiddled = [&](int p, float2 &a, float2 &b) {        // input p of the last stage, both channels
      const float4 t = S[(j + R1B * p) * CPW + cp];
      a = make_float2(t.x, t.y);
      b = make_float2(t.z, t.w);
      if (p > 0) {
        const float2 w = tw[j * p];
        a = cmul_conj(a, w);
        b = cmul_conj(b, w);
      }
    };
    if constexpr (PAD) {
      if constexpr (A < 14) {
        float2 x0[A], x1[A];
#pragma unroll
        for (int p = 0; p < A; ++p) twiddled(p, x0[p], x1[p]);
        idft_first_half<A>(x0, z0);
        idft_first_half<A>(x1, z1);
      } else {
        // the same with the odd inputs read after the even ones are transformed: 16 instead of 92 bytes of spills
        float2 o0[AO], o1[AO];
#pragma unroll
        for (int k = 0; k < AO; ++k) twiddled(2 * k, z0[k], z1[k]);
        dft_inv<AO>(z0);
        dft_inv<AO>(z1);
#pragma unroll
        for (int k = 0; k < AO; ++k) twiddled(2 * k + 1, o0[k], o1[k]);
        dft_inv<AO>(o0);
        dft_inv<AO>(o1);
        add_odd_half<A>(z0, o0);
        add_odd_half<A>(z1, o1);
      }
    } else {
#pragma unroll
      for (int p = 0; p < A; ++p) twiddled(p, z0[p], z1[p]);
      dft_inv<A>(z0);
      dft_inv<A>(z1);
    }
#pragma unroll
    for (int p = 0; p < AO; ++p) {
      if (PAD && (j + R1B * p) * N2 + n2 >= N) continue;
      if (OUT == OUT_SPEC) {
        const int n = (j + R1B * p) * N2 + n2;
        const float4 t = __ldg(tab + n);
        const float2 c = make_float2(t.z * inv_scale, t.w * inv_scale), a = cmul_conj(z0[p], c), b = cmul_conj(z1[p], c);
        *reinterpret_cast<float4 *>(spec + (size_t)n * ncol_ws + gc0 + 2 * cp) = make_float4(a.x, a.y, b.x, b.y);
        continue;
      }
      const float ek = fmaf(z0[p].x, z0[p].x, z1[p].x * z1[p].x);
      const float ev = fmaf(z0[p].y, z0[p].y, z1[p].y * z1[p].y);
      totK += ek;
      totV += ev;
      acc[p] += ek + ev;
    }
    __syncthreads();
  }
  if (OUT == OUT_SPEC) return;
  // transposed reduction over the CPW lanes that share j: the PR row sums are halved at every
  // step until one is left, further steps are plain adds; row p = cp >> log2(CPW/PR)
  {
    int count = PR;
#pragma unroll
    for (int s = CPW / 2; s >= 1; s >>= 1) {
      if (count > 1) {
        const int half = count / 2;
#pragma unroll
        for (int i = 0; i < half; ++i) {
          const bool up = (cp & s) != 0;
          const float send = up ? acc[i] : acc[i + half];
          const float keep = up ? acc[i + half] : acc[i];
          acc[i] = keep + __shfl_xor_sync(0xffffffffu, send, s);
        }
        count = half;
      } else {
        acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], s);
      }
    }
  }
  constexpr int DUP = CPW / PR;                             // lanes that end with the same row sum
  if ((cp & (DUP - 1)) == 0 && cp / DUP < AO) {             // rows AO.. of the reduction are padding
    const int p = (j + R1B * (cp / DUP)) * N2 + n2;
    if (!PAD || p < N) {
      float *dst = lp.scores[layer] + (long long)head * score_stride + (PAD ? p : perm_token(p, N));
      *dst = accumulate ? *dst + acc[0] * inv_scale : acc[0] * inv_scale;
    }
  }
  const double dk = warp_sum_d((double)(totK * inv_scale));
  const double dv = warp_sum_d((double)(totV * inv_scale));
  if ((tid & 31) == 0) { red[0][tid >> 5] = dk; red[1][tid >> 5] = dv; }
  __syncthreads();
  __shared__ bool is_last;
  if (tid == 0) {
    double sa = 0, sb = 0;
#pragma unroll
    for (int i = 0; i < NW; ++i) { sa += red[0][i]; sb += red[1][i]; }
    double *slot = eo.part_hi + 2 * ((size_t)layer * eo.hi_slots + hi_base + (size_t)head * gridDim.x + n2);
    slot[0] = sa * (double)head_dim;
    slot[1] = sb * (double)head_dim;
    __threadfence();
    is_last = (atomicAdd(eo.done + layer, 1u) + 1u == eo.total_blocks);
    if (is_last) eo.done[layer] = 0u;
  }
  __syncthreads();
  if (!is_last) return;
  // the layer's partial sums in a fixed order: energy = (hiK, totK, hiV, totV)
  __threadfence();
  const double *pt = eo.part_tot + 2 * (size_t)layer * eo.tot_slots, *ph = eo.part_hi + 2 * (size_t)layer * eo.hi_slots;
  double *redd = reinterpret_cast<double *>(smem4);        // [4][NT], the tile is no longer needed
  double a0 = 0, a1 = 0, b0 = 0, b1 = 0;
  for (int i = tid; i < eo.tot_slots; i += NT) { a0 += __ldcg(pt + 2 * i); a1 += __ldcg(pt + 2 * i + 1); }
  for (int i = tid; i < eo.hi_slots; i += NT) { b0 += __ldcg(ph + 2 * i); b1 += __ldcg(ph + 2 * i + 1); }
  redd[tid] = b0; redd[NT + tid] = a0; redd[2 * NT + tid] = b1; redd[3 * NT + tid] = a1;
  __syncthreads();
  for (int st = NT / 2; st > 0; st >>= 1) {
    if (tid < st)
      for (int q = 0; q < 4; ++q) redd[q * NT + tid] += redd[q * NT + tid + st];
    __syncthreads();
  }
  if (tid < 4) eo.energy[(long long)layer * eo.energy_stride + tid] = redd[tid * NT];
}

}  // namespace fast
