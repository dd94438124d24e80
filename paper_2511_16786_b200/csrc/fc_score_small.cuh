// Scoring of short sequences in one kernel: the whole transform of a few channels (M <= 1024 points, direct or padded
// form, see fc_score_fast.cuh) stays in one block's shared memory, one cluster of blocks holds a head, and the blocks'
// row sums meet through distributed shared memory, so a call is one launch on the caller's stream with no intermediate in
// global memory, no fork to the internal streams and no join.
//
// What bounds it: one layer of 4 heads is a chain of about ten barriers and three trips to memory in 64 blocks (nothing
// is near a throughput limit), many layers are bound like the three passes, by the shared-memory exchanges and the
// fp32 pipes, without their traffic to L2.  64 KB and 256 threads of 16 points x 2 channels per block, two blocks per SM:
// CP channel pairs with M * CP = 4096, d / (2 CP) blocks per cluster (16 for M = 1024 and 128 channels; wider heads at
// that length take the three passes).
#pragma once
#include <cooperative_groups.h>

#include "fc_score_fast.cuh"

namespace small {

using fast::Load2;

constexpr int kSeqs = 32;                 // sequences one launch can span (kernel-argument table)
struct SeqTable {
  int start[kSeqs], N[kSeqs], omega[kSeqs], index[kSeqs];      // first token, tokens, cutoff, sequence of the batch
  const float4 *tab[kSeqs];                                     // padded form: (h, c) of every bin
};

// (h, c) of every bin k of the M-point transform (fc_score_fast.cuh), by cosine sums over the kernel's symmetries:
//   c = 1 - g(0) - 2 sum_{t<N} g(t) cos(2 pi k t / M),   h = w^(k(N-1)) (g(N) + 2 sum_{u<N} g(N-u) cos(2 pi k u / M)).
__global__ void k_small_table(float4 *__restrict__ tab, int N, int omega, int M, const float2 *__restrict__ master,
                              int master_len) {
  extern __shared__ float g[];            // g(0) .. g(N)
  for (int t = threadIdx.x; t <= N; t += blockDim.x) g[t] = fast::base_kernel(t, N, omega);
  __syncthreads();
  const int k = blockIdx.x * blockDim.x + threadIdx.x, step = master_len / M;
  if (k >= M) return;
  double a = 0.0, b = 0.0;
  for (int t = 1, r = k; t < N; ++t, r = (r + k) & (M - 1)) {
    const double cs = (double)__ldg(&master[(size_t)r * step]).x;
    a += (double)g[t] * cs;
    b += (double)g[N - t] * cs;
  }
  const float hb = (float)((double)g[N] + 2.0 * b);
  const float2 w = master[(size_t)((long long)k * (N - 1) & (M - 1)) * step];
  tab[k] = make_float4(w.x * hb, w.y * hb, (float)(1.0 - (double)g[0] - 2.0 * a), 0.f);
}

// x[p] *= w^p, p = 1..R-1, both channels, from w and w^4.
template <int R, bool CONJ>
__device__ __forceinline__ void twiddle(float2 (&x0)[R], float2 (&x1)[R], float2 c1, float2 c4) {
  if (CONJ) { c1.y = -c1.y; c4.y = -c4.y; }
  const float2 c2 = cmul(c1, c1), c3 = cmul(c2, c1);
  x0[1] = cmul(x0[1], c1); x1[1] = cmul(x1[1], c1);
  x0[2] = cmul(x0[2], c2); x1[2] = cmul(x1[2], c2);
  x0[3] = cmul(x0[3], c3); x1[3] = cmul(x1[3], c3);
  float2 base = c4;
#pragma unroll
  for (int g = 1; g < R / 4; ++g) {
    const float2 b1 = cmul(base, c1), b2 = cmul(base, c2), b3 = cmul(base, c3);
    x0[4 * g] = cmul(x0[4 * g], base);       x1[4 * g] = cmul(x1[4 * g], base);
    x0[4 * g + 1] = cmul(x0[4 * g + 1], b1); x1[4 * g + 1] = cmul(x1[4 * g + 1], b1);
    x0[4 * g + 2] = cmul(x0[4 * g + 2], b2); x1[4 * g + 2] = cmul(x1[4 * g + 2], b2);
    x0[4 * g + 3] = cmul(x0[4 * g + 3], b3); x1[4 * g + 3] = cmul(x1[4 * g + 3], b3);
    if (4 * (g + 1) < R) base = cmul(base, c4);
  }
}

// Transform length M = RA*RB*RC (RB = 1: two stages), CP channel pairs per block.
template <int RA_, int RB_, int RC_, int CP_>
struct Shape {
  static constexpr int RA = RA_, RB = RB_, RC = RC_, CP = CP_, M = RA * RB * RC, LANES = M / 16, NT = LANES * CP;
  static constexpr int PAD = CP < 8 ? 1 : 0;                  // one row per RC rows: stage C strides RC rows
  static constexpr int ROWS = M + PAD * (M / RC);
  __device__ static int row(int pos) { return (pos + PAD * (pos / RC)) * CP; }
  static constexpr size_t smem(bool pad) {
    return (size_t)ROWS * CP * sizeof(float4) + (size_t)M * (pad ? sizeof(float4) : sizeof(float2));
  }
};

// One block: 2*CP channels of one head of one (layer, sequence).  grid (cluster, H, layers * sequences).
template <typename T, class S, bool PADDED>
__global__ void __launch_bounds__(S::NT, S::NT == 256 ? 2 : 4)
k_small(const __grid_constant__ fast::LayerPtrs lp, const __grid_constant__ SeqTable st, int nseq, long long stride_token,
        long long stride_head, int H, int head_dim, const float2 *__restrict__ master, int master_len,
        long long score_stride, double *__restrict__ part_en, unsigned *__restrict__ done, double *__restrict__ energy,
        long long energy_layer) {
  namespace cg = cooperative_groups;
  cg::cluster_group cluster = cg::this_cluster();
  constexpr int M = S::M, RA = S::RA, RB = S::RB, RC = S::RC, CP = S::CP, LANES = S::LANES, NT = S::NT;
  constexpr int L1 = M / RA, UA = 16 / RA, UB = RB > 1 ? 16 / RB : 1, UC = 16 / RC;
  extern __shared__ float4 smem4[];
  float4 *X = smem4;
  float4 *hc = X + S::ROWS * CP;                              // padded: (h, c) of every bin
  float2 *uT = reinterpret_cast<float2 *>(hc);                // direct: exp(-j*pi*q/N) of every bin
  __shared__ double red[4][NT / 32], sums[4];
  const int tid = threadIdx.x, cp = tid % CP, j = tid / CP, lane = tid & 31, warp = tid >> 5;
  const int slice = blockIdx.x, head = blockIdx.y, layer = blockIdx.z / nseq, sq = blockIdx.z - layer * nseq;
  const int N = st.N[sq], omega = st.omega[sq], start = st.start[sq];
  const int ch = slice * (2 * CP) + 2 * cp;
  const T *kb = static_cast<const T *>(lp.k[layer]) + (long long)start * stride_token + (long long)head * stride_head + ch;
  const T *vb = static_cast<const T *>(lp.v[layer]) + (long long)start * stride_token + (long long)head * stride_head + ch;

  asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");   // e.g. the allocation, which waits for this grid

  // stage A: butterfly j + LANES*u holds the points j + LANES*u + L1*p
  float2 x0[16], x1[16];
#pragma unroll
  for (int u = 0; u < UA; ++u)
#pragma unroll
    for (int p = 0; p < RA; ++p) {
      const int n = j + LANES * u + L1 * p;
      if (PADDED && p >= RA / 2) {                            // N <= M/2
        x0[u * RA + p] = x1[u * RA + p] = make_float2(0.f, 0.f);
        continue;
      }
      const long long off = (long long)(PADDED ? (n < N ? n : 0) : fast::perm_token(n, M)) * stride_token;
      const float2 kk = Load2<T>::ld(kb + off), vv = Load2<T>::ld(vb + off);
      const bool in = !PADDED || n < N;
      x0[u * RA + p] = in ? make_float2(kk.x, vv.x) : make_float2(0.f, 0.f);
      x1[u * RA + p] = in ? make_float2(kk.y, vv.y) : make_float2(0.f, 0.f);
    }
  const int mstep = master_len / M;
  if (PADDED) {
    for (int i = tid; i < M; i += NT) hc[i] = __ldg(st.tab[sq] + i);
  } else {
    for (int i = tid; i < M; i += NT) uT[i] = master[(size_t)i * (mstep / 2)];
  }
  float2 wa1[UA], wa4[UA], wb1[UB], wb4[UB];
#pragma unroll
  for (int u = 0; u < UA; ++u) {
    const int i = j + LANES * u;
    wa1[u] = __ldg(&master[(size_t)i * mstep]);
    wa4[u] = __ldg(&master[(size_t)((4 * i) & (M - 1)) * mstep]);
  }
  if constexpr (RB > 1) {
#pragma unroll
    for (int u = 0; u < UB; ++u) {
      const int i2 = (j + LANES * u) & (RC - 1);
      wb1[u] = __ldg(&master[(size_t)i2 * RA * mstep]);
      wb4[u] = __ldg(&master[(size_t)((4 * i2 * RA) & (M - 1)) * mstep]);
    }
  }
  float tot[4] = {0.f, 0.f, 0.f, 0.f};                        // (hiK, totK, hiV, totV)
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    tot[1] = fmaf(x0[i].x, x0[i].x, fmaf(x1[i].x, x1[i].x, tot[1]));
    tot[3] = fmaf(x0[i].y, x0[i].y, fmaf(x1[i].y, x1[i].y, tot[3]));
  }
  auto put = [&](int pos, float2 a, float2 b) { X[S::row(pos) + cp] = make_float4(a.x, a.y, b.x, b.y); };
  auto get = [&](int pos, float2 &a, float2 &b) {
    const float4 t = X[S::row(pos) + cp];
    a = make_float2(t.x, t.y);
    b = make_float2(t.z, t.w);
  };
  // ---- forward
#pragma unroll
  for (int u = 0; u < UA; ++u) {
    float2 y0[RA], y1[RA];
    if constexpr (PADDED && RA == 16) {
      float2 z0[8], z1[8];
#pragma unroll
      for (int p = 0; p < 8; ++p) { z0[p] = x0[p]; z1[p] = x1[p]; }
      dft_zero_tail<16>(z0, y0);
      dft_zero_tail<16>(z1, y1);
    } else {
#pragma unroll
      for (int p = 0; p < RA; ++p) { y0[p] = x0[u * RA + p]; y1[p] = x1[u * RA + p]; }
      fast::dft_fwd<RA>(y0);
      fast::dft_fwd<RA>(y1);
    }
    twiddle<RA, false>(y0, y1, wa1[u], wa4[u]);
#pragma unroll
    for (int p = 0; p < RA; ++p) put(j + LANES * u + L1 * p, y0[p], y1[p]);
  }
  __syncthreads();
  if constexpr (RB > 1) {
    // butterfly i of stage B: sub-block i / RC, inner index i % RC, points RC apart
#pragma unroll
    for (int u = 0; u < UB; ++u) {
      const int i = j + LANES * u, at = (i / RC) * L1 + (i & (RC - 1));
      float2 y0[RB], y1[RB];
#pragma unroll
      for (int p = 0; p < RB; ++p) get(at + RC * p, y0[p], y1[p]);
      fast::dft_fwd<RB>(y0);
      fast::dft_fwd<RB>(y1);
      twiddle<RB, false>(y0, y1, wb1[u], wb4[u]);
#pragma unroll
      for (int p = 0; p < RB; ++p) put(at + RC * p, y0[p], y1[p]);
    }
    __syncthreads();
  }
  // stage C: sub-block s = (bA, bB), bin bA + RA*(bB + RB*p)
#pragma unroll
  for (int u = 0; u < UC; ++u) {
    const int s = j + LANES * u;
    float2 y0[RC], y1[RC];
#pragma unroll
    for (int p = 0; p < RC; ++p) get(s * RC + p, y0[p], y1[p]);
    fast::dft_fwd<RC>(y0);
    fast::dft_fwd<RC>(y1);
#pragma unroll
    for (int p = 0; p < RC; ++p) {
      x0[u * RC + p] = y0[p];
      x1[u * RC + p] = y1[p];
      put(s * RC + p, y0[p], y1[p]);
    }
  }
  __syncthreads();
  // ---- the residual filter between the bins k and M-k
#pragma unroll
  for (int u = 0; u < UC; ++u) {
    // bins k = k0 + RA*RB*p; their partners are the sub-block of -k0 read backwards (k0 = 0: its own, shifted by one)
    const int s = j + LANES * u, k0 = s / RB + RA * (s % RB), kn = (RA * RB - k0) & (RA * RB - 1);
    const float4 *part = X + S::row(((kn & (RA - 1)) * RB + kn / RA) * RC) + cp;
#pragma unroll
    for (int p = 0; p < RC; ++p) {
      const int k = k0 + RA * RB * p;
      const float4 *other = part + (k0 == 0 ? (RC - p) & (RC - 1) : RC - 1 - p) * CP;
      float2 &P0 = x0[u * RC + p], &P1 = x1[u * RC + p];
      if (PADDED) {
        const float4 t = *other, w = hc[k];
        P0 = make_float2(fmaf(t.y, w.y, fmaf(-t.x, w.x, w.z * P0.x)), fmaf(-t.y, w.x, fmaf(-t.x, w.y, w.z * P0.y)));
        P1 = make_float2(fmaf(t.w, w.y, fmaf(-t.z, w.x, w.z * P1.x)), fmaf(-t.w, w.x, fmaf(-t.z, w.y, w.z * P1.y)));
      } else {
        const bool inL = k <= omega, inH = M - k <= omega;
        if (k == 0 || (inL && inH)) {
          P0 = P1 = make_float2(0.f, 0.f);
        } else if (inL || inH) {
          const float4 t = *other;
          const float2 e = uT[k];
          const float sgn = inL ? -0.5f : 0.5f;
          const float2 w = make_float2(e.x * sgn, -e.y * sgn);
          P0 = make_float2(fmaf(t.x, w.x, fmaf(-t.y, w.y, 0.5f * P0.x)), fmaf(t.x, w.y, fmaf(t.y, w.x, 0.5f * P0.y)));
          P1 = make_float2(fmaf(t.z, w.x, fmaf(-t.w, w.y, 0.5f * P1.x)), fmaf(t.z, w.y, fmaf(t.w, w.x, 0.5f * P1.y)));
        }
      }
    }
  }
  // ---- back
#pragma unroll
  for (int u = 0; u < UC; ++u) {
    float2 y0[RC], y1[RC];
#pragma unroll
    for (int p = 0; p < RC; ++p) { y0[p] = x0[u * RC + p]; y1[p] = x1[u * RC + p]; }
    fast::dft_inv<RC>(y0);
    fast::dft_inv<RC>(y1);
#pragma unroll
    for (int p = 0; p < RC; ++p) { x0[u * RC + p] = y0[p]; x1[u * RC + p] = y1[p]; }
  }
  __syncthreads();                                            // all partner reads are done
#pragma unroll
  for (int u = 0; u < UC; ++u)
#pragma unroll
    for (int p = 0; p < RC; ++p) put((j + LANES * u) * RC + p, x0[u * RC + p], x1[u * RC + p]);
  __syncthreads();
  if constexpr (RB > 1) {
#pragma unroll
    for (int u = 0; u < UB; ++u) {
      const int i = j + LANES * u, at = (i / RC) * L1 + (i & (RC - 1));
      float2 y0[RB], y1[RB];
#pragma unroll
      for (int p = 0; p < RB; ++p) get(at + RC * p, y0[p], y1[p]);
      twiddle<RB, true>(y0, y1, wb1[u], wb4[u]);
      fast::dft_inv<RB>(y0);
      fast::dft_inv<RB>(y1);
#pragma unroll
      for (int p = 0; p < RB; ++p) put(at + RC * p, y0[p], y1[p]);
    }
    __syncthreads();
  }
  float acc[16];                                              // |residual|^2 of row u*RA + p, this thread's two channels
#pragma unroll
  for (int u = 0; u < UA; ++u) {
    float2 y0[RA], y1[RA];
#pragma unroll
    for (int p = 0; p < RA; ++p) get(j + LANES * u + L1 * p, y0[p], y1[p]);
    twiddle<RA, true>(y0, y1, wa1[u], wa4[u]);
    fast::dft_inv<RA>(y0);
    fast::dft_inv<RA>(y1);
#pragma unroll
    for (int p = 0; p < RA; ++p) {
      const bool in = !PADDED || (p < RA / 2 && j + LANES * u + L1 * p < N);
      const float ek = in ? fmaf(y0[p].x, y0[p].x, y1[p].x * y1[p].x) : 0.f;
      const float ev = in ? fmaf(y0[p].y, y0[p].y, y1[p].y * y1[p].y) : 0.f;
      tot[0] += ek;
      tot[2] += ev;
      acc[u * RA + p] = ek + ev;
    }
  }
  // ---- sum over the block's channels (transposed reduction over the lanes of a row group), then over the cluster
  float *rowsum = reinterpret_cast<float *>(smem4);           // [M] point order
  __syncthreads();                                            // the tile is no longer needed
  {
    int count = 16, first = 0;                                // this lane keeps rows first .. first + count - 1
#pragma unroll
    for (int s = CP / 2; s >= 1; s >>= 1) {
      if (count > 1) {
        const int half = count / 2;
        const bool up = (cp & s) != 0;
#pragma unroll
        for (int i = 0; i < half; ++i) {
          const float send = up ? acc[i] : acc[i + half], keep = up ? acc[i + half] : acc[i];
          acc[i] = keep + __shfl_xor_sync(0xffffffffu, send, s);
        }
        if (up) first += half;
        count = half;
      } else {
        acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], s);
      }
    }
    constexpr int KEEP = CP >= 16 ? 1 : 16 / CP;
    if (CP <= 16 || (cp & (CP / 16 - 1)) == 0)
#pragma unroll
      for (int i = 0; i < KEEP; ++i) {
        const int e = first + i;
        rowsum[j + LANES * (e / RA) + L1 * (e % RA)] = acc[i];
      }
  }
  const float inv = 1.f / ((float)M * (float)M * (float)head_dim);
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const double v = warp_sum_d((double)((q & 1) ? tot[q] : tot[q] * inv));
    if (lane == 0) red[q][warp] = v;
  }
  __syncthreads();
  if (tid < 4) {
    double v = 0.0;
#pragma unroll
    for (int w = 0; w < NT / 32; ++w) v += red[tid][w];
    sums[tid] = v;
  }
  cluster.sync();
  const int nblk = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
  if (rank == 0 && tid < 32) {
    // energies: the head's sums, then, in the block of the (layer, sequence)'s last head, all heads' in order
    double *en = energy + layer * energy_layer + 4ll * st.index[sq];
    double v = 0.0;
    if (tid < 4) {
      for (int b = 0; b < nblk; ++b) v += *cluster.map_shared_rank(&sums[tid], b);
      if ((tid & 1) == 0) v *= (double)head_dim;              // d * sum Dev = outlier-band energy
      if (H == 1) en[tid] = v;
      else part_en[((size_t)blockIdx.z * H + head) * 4 + tid] = v;
    }
    if (H > 1) {
      __syncwarp();
      bool last = false;
      if (tid == 0) {
        __threadfence();
        last = atomicAdd(done + blockIdx.z, 1u) + 1u == (unsigned)H;
        if (last) done[blockIdx.z] = 0u;
        __threadfence();
      }
      if (__shfl_sync(0xffffffffu, last, 0) && tid < 4) {
        v = 0.0;
        for (int h = 0; h < H; ++h) v += __ldcg(part_en + ((size_t)blockIdx.z * H + h) * 4 + tid);
        en[tid] = v;
      }
    }
  }
  float *out = lp.scores[layer] + (long long)head * score_stride + start;
  const int per = (M + nblk - 1) / nblk;                      // rows of this block
  for (int i = NT - 1 - tid; i < per; i += NT) {              // (rank 0's first warp is busy with the energies)
    const int n = rank * per + i;
    if (n >= M || (PADDED && n >= N)) continue;
    float v = 0.f;
    for (int b = 0; b < nblk; ++b) v += *cluster.map_shared_rank(&rowsum[n], b);
    out[PADDED ? n : fast::perm_token(n, M)] = v * inv;
  }
  cluster.sync();                                             // remote reads of this block's memory are done
}

}  // namespace small
