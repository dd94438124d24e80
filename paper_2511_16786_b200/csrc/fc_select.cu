// fc_allocate_budgets (Dynamic Budget Allocation Module, Sec. 3.2.2) and
// fc_select_compact (keep the Outlier KVs by budget, Sec. 3.2.1 last sentence):
// fp64 budget arithmetic in one small kernel, an exact radix select per
// (sequence, head) on the fp32 score bits, an ordered compaction of the chosen
// token indices, and a row gather into the dense compacted cache.
//
// This file is compiled with -fmad=false so that the fp64 budget arithmetic is
// the plain IEEE sequence of multiplies, adds and divides it is written as.
#include "fc_common.cuh"

#include <cooperative_groups.h>
#include <math.h>
#include <mutex>
#include <unordered_map>

namespace {

constexpr int kSeqChunk = 64;          // sequences described per launch (kernel-argument table)
struct SeqTable {
  int start[kSeqChunk + 1];            // token offsets of the chunk's sequences (cu_seqlens slice)
};
constexpr int kLayerChunk = 32;        // layers selected by one launch (kernel-argument table)
struct LayerTable {                    // per layer of the chunk: where its scores, rows and outputs live (DEVICE pointers)
  const float *scores[kLayerChunk];
  const char *k[kLayerChunk], *v[kLayerChunk];
  char *out_k[kLayerChunk], *out_v[kLayerChunk];
  int *out_idx[kLayerChunk];
  long long cap[kLayerChunk];          // rows available in the layer's outputs
};

// ---------------------------------------------------------------------------
// budgets
// ---------------------------------------------------------------------------
__device__ double filled_sum(const double *w, int L, double lam, double lo, double hi) {
  double s = 0.0;
  for (int l = 0; l < L; ++l) {
    double q = lam * w[l];
    q = q < lo ? lo : (q > hi ? hi : q);
    s += q;
  }
  return s;
}

__device__ __forceinline__ double warp_min_d(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmin(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}
__device__ __forceinline__ double warp_max_d(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// One block per sequence of the chunk.  Shared memory: w[L], cand[2L], fval[2L], frac[L], bud[L], order[L].
// The sums whose rounding the rule fixes run in layer order (one thread, or one thread per candidate); everything else
// (searches over the candidates, the remainders' order and who gets one) is spread over the block, so that a call is a
// chain of a few L-step loops: 10.9 + 1.8 us (with the offsets as a second kernel) -> 9.0 us at 28 layers.
// The last block of the call writes the offsets.
constexpr int kAllocThreads = 256;
__global__ void __launch_bounds__(kAllocThreads)
k_allocate(const double *__restrict__ energy, int L, int B, int b0, SeqTable st, double rho,
           int min_keep, int *__restrict__ budgets, long long *__restrict__ out_offsets, unsigned *__restrict__ done,
           unsigned total_blocks) {
  extern __shared__ double sh[];
  double *w = sh;
  double *cand = w + L;
  double *fval = cand + 2 * L;
  double *frac = fval + 2 * L;
  int *bud = reinterpret_cast<int *>(frac + L);
  int *order = bud + L;
  __shared__ double s_sum, s_red[2][kAllocThreads / 32];
  __shared__ int s_bad, s_floor, s_last;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int b = b0 + blockIdx.x;
  asm volatile("griddepcontrol.wait;\n" ::: "memory");
  const int N = b < B ? st.start[blockIdx.x + 1] - st.start[blockIdx.x] : 0;
  if (N == 0) {
    if (b < B)
      for (int l = tid; l < L; l += kAllocThreads) budgets[(size_t)l * B + b] = 0;
  } else {
    const double lo = (double)(min_keep < N ? (min_keep < 0 ? 0 : min_keep) : N);
    const double hi = (double)N;
    double bt = floor(rho * (double)N * (double)L + 0.5);
    if (bt < (double)L * lo) bt = (double)L * lo;
    if (bt > (double)L * hi) bt = (double)L * hi;
    const long long B_tot = (long long)bt;

    // R^l = hiK/totK + hiV/totV   (Eq. 12)
    if (tid == 0) { s_bad = 0; s_floor = 0; }
    __syncthreads();
    for (int l = tid; l < L; l += kAllocThreads) {
      const double *e = energy + ((size_t)l * B + b) * 4;
      const double rk = e[1] > 0.0 ? e[0] / e[1] : 0.0;
      const double rv = e[3] > 0.0 ? e[2] / e[3] : 0.0;
      const double R = rk + rv;
      w[l] = R;
      if (!(R >= 0.0) || isinf(R)) s_bad = 1;
    }
    __syncthreads();
    if (tid == 0) {
      double s = 0.0;
#pragma unroll 4
      for (int l = 0; l < L; ++l) s += w[l];
      if (!(s > 0.0) || isinf(s) || isnan(s)) s_bad = 1;
      s_sum = s;
    }
    __syncthreads();
    const bool uniform = s_bad != 0;
    const double total = s_sum;
    for (int l = tid; l < L; l += kAllocThreads) w[l] = uniform ? 1.0 / (double)L : w[l] / total;
    __syncthreads();

    // kinks of f(lam) = sum clamp(lam*w, lo, hi) and f at each of them; the smallest kink b* > 0 with f(b*) >= B_tot
    // and the largest one in all
    double bstar = INFINITY, kmax = 0.0;
    for (int i = tid; i < 2 * L; i += kAllocThreads) {
      const double wl = w[i >> 1];
      const double c = wl > 0.0 ? ((i & 1) ? hi / wl : lo / wl) : INFINITY;
      double f = -1.0;
      if (!isinf(c)) {
        f = filled_sum(w, L, c, lo, hi);
        kmax = fmax(kmax, c);
        if (c > 0.0 && f >= (double)B_tot) bstar = fmin(bstar, c);
      }
      cand[i] = c;
      fval[i] = f;
    }
    bstar = warp_min_d(bstar);
    kmax = warp_max_d(kmax);
    if (lane == 0) { s_red[0][warp] = bstar; s_red[1][warp] = kmax; }
    __syncthreads();
    bstar = INFINITY;
#pragma unroll
    for (int i = 0; i < kAllocThreads / 32; ++i) { bstar = fmin(bstar, s_red[0][i]); kmax = fmax(kmax, s_red[1][i]); }
    __syncthreads();
    double lam = kmax;
    if (!isinf(bstar)) {
      // the largest kink a* < b* (0 counts as a kink) and f at both; equal kinks have equal f
      double astar = 0.0;
      for (int i = tid; i < 2 * L; i += kAllocThreads)
        if (cand[i] < bstar) astar = fmax(astar, cand[i]);
      astar = warp_max_d(astar);
      if (lane == 0) s_red[0][warp] = astar;
      __syncthreads();
#pragma unroll
      for (int i = 0; i < kAllocThreads / 32; ++i) astar = fmax(astar, s_red[0][i]);
      if (tid == 0) s_red[1][1] = (double)L * lo;            // f(0): L whole numbers, exact in any order
      __syncthreads();
      for (int i = tid; i < 2 * L; i += kAllocThreads) {
        if (cand[i] == bstar) s_red[1][0] = fval[i];
        if (cand[i] == astar && astar > 0.0) s_red[1][1] = fval[i];
      }
      __syncthreads();
      const double fb = s_red[1][0], fa = s_red[1][1];
      lam = (fb == fa) ? astar : astar + ((double)B_tot - fa) * (bstar - astar) / (fb - fa);
    }
    int mine = 0;
    for (int l = tid; l < L; l += kAllocThreads) {
      double q = lam * w[l];
      q = q < lo ? lo : (q > hi ? hi : q);
      const double fl = floor(q);
      frac[l] = q - fl;
      bud[l] = (int)fl;
      // the sum of the floors, low and high halves apart (it may pass 2^31)
      mine += (int)fl;
    }
    // (at most 1024 layers of at most 131072 tokens: 2^27)
    mine = __reduce_add_sync(0xffffffffu, mine);
    if (lane == 0) atomicAdd(&s_floor, mine);
    __syncthreads();
    const long long deficit = B_tot - (long long)s_floor;
    // order by (fraction descending, layer ascending)
    for (int l = tid; l < L; l += kAllocThreads) {
      int rank = 0;
      const double f = frac[l];
#pragma unroll 4
      for (int m = 0; m < L; ++m) rank += (frac[m] > f || (frac[m] == f && m < l)) ? 1 : 0;
      order[rank] = l;
    }
    __syncthreads();
    // one more token to each layer in that order that is not full, round after round: the first round in parallel,
    // further ones (only when layers are full) by one thread
    int room = 0;
    for (int l = tid; l < L; l += kAllocThreads) room += bud[l] < N ? 1 : 0;
    if (tid == 0) s_last = 0;
    __syncthreads();
    room = __reduce_add_sync(0xffffffffu, room);
    if (lane == 0) atomicAdd(&s_last, room);
    __syncthreads();
    room = s_last;
    if (deficit > 0 && deficit <= room) {
      for (int r = tid; r < L; r += kAllocThreads) {
        int before = 0;
        for (int m = 0; m < r; ++m) before += bud[order[m]] < N ? 1 : 0;
        cand[r] = (bud[order[r]] < N && before < deficit) ? 1.0 : 0.0;
      }
      __syncthreads();
      for (int r = tid; r < L; r += kAllocThreads)
        if (cand[r] > 0.0) bud[order[r]] += 1;
    } else if (deficit > 0 && tid == 0) {
      long long left = deficit;
      while (left > 0) {
        bool gave = false;
        for (int r = 0; r < L && left > 0; ++r)
          if (bud[order[r]] < N) { bud[order[r]] += 1; --left; gave = true; }
        if (!gave) break;
      }
    }
    __syncthreads();
    for (int l = tid; l < L; l += kAllocThreads) budgets[(size_t)l * B + b] = bud[l];
  }
  // the last block of the call: out_offsets[l][.] = exclusive prefix sums of budgets[l][.]
  __threadfence();
  __syncthreads();
  if (tid == 0) {
    s_last = (atomicAdd(done, 1u) + 1u == total_blocks) ? 1 : 0;
    if (s_last) *done = 0u;
    __threadfence();
  }
  __syncthreads();
  if (!s_last) return;
  for (int l = tid; l < L; l += kAllocThreads) {
    long long acc = 0;
    long long *off = out_offsets + (size_t)l * (B + 1);
    off[0] = 0;
    for (int i = 0; i < B; ++i) {
      acc += __ldcg(budgets + (size_t)l * B + i);
      off[i + 1] = acc;
    }
  }
}

// ---------------------------------------------------------------------------
// selection
// ---------------------------------------------------------------------------
// Monotone map float -> uint32: larger score, larger key.  NaN ranks with +inf, -0 with +0.
__device__ __forceinline__ unsigned score_key(float x) {
  if (x != x) return 0xFF800000u;
  if (x == 0.f) return 0x80000000u;
  const unsigned u = __float_as_uint(x);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

constexpr int kSelCluster = 8;      // blocks (one cluster) per (sequence, head) at most
constexpr int kSelKptMax = 16;      // scores per thread
constexpr int kSelMaxTokens = kSelCluster * 1024 * kSelKptMax;
constexpr int kBins = 2048;         // radix digits: 10 (sign, exponent, one mantissa bit), 11 and 11 bits
constexpr int kCandidates = 128;    // a bin of at most this many keys is finished by comparing them with one another

// Selection + compaction + row gather for one (sequence, head), by one cluster of CL blocks of NT threads.  Block r of
// the cluster owns the contiguous token range [r*chunk, (r+1)*chunk) and keeps its score keys in registers (thread t:
// tokens t, t + NT, ... of the range, so loads coalesce).  The k-th largest key is found by an MSB-first radix select
// with digits of 10, 11 and 11 bits, whose histograms are summed across the cluster through distributed shared memory; as soon as the
// chosen bin holds few keys (after two digits, i.e. 12 mantissa bits, nearly always) they are compared with one another.
// The chosen tokens are then ranked in token order (ballots per 32 tokens, one scan of the counts, cluster prefix),
// written as ascending indices, and their K/V rows are copied by the same block.
// grid (CL * sequences in chunk, heads), cluster (CL, 1, 1).
// PER_LAYER: one cluster per sequence (grid.y = 1) ranks the tokens by the sum over heads of their
// scores (the order of the head-averaged deviation), writes the same indices for every head and
// gathers the rows of all heads.  protect (may be null): a non-zero byte per token of the batch puts
// that token before every unmarked one.
template <int KPT, bool PER_LAYER, int CL, int NT>
__device__ __forceinline__ void
select_gather_body(const float *__restrict__ scores, long long T, const SeqTable &st, int b0,
                const int *__restrict__ budgets, const long long *__restrict__ out_offsets,
                int *__restrict__ out_idx, long long cap, int *__restrict__ status,
                const char *__restrict__ kin, const char *__restrict__ vin, long long stride_token_b,
                long long stride_head_b, int row_bytes, int H, char *__restrict__ out_k,
                char *__restrict__ out_v, const unsigned char *__restrict__ protect) {
  namespace cg = cooperative_groups;
  cg::cluster_group cluster = cg::this_cluster();
  constexpr int NW = NT / 32, CNT = KPT * NW;     // warps, 32-token runs of the block's range
  extern __shared__ unsigned short sel[];         // [KPT*NT] chosen tokens of the range, in order
  __shared__ int lhist[3][kBins];                 // this block's histograms, one per digit (read by the whole cluster)
  __shared__ unsigned cand[kCandidates];          // this block's keys in the chosen bin
  __shared__ unsigned all[kCandidates];           // the cluster's
  __shared__ unsigned runs[CNT];                  // (ties << 16 | greater) of every run, then their prefix sums
  __shared__ unsigned tot[CL];                    // (ties << 16 | greater) of every block of the cluster
  __shared__ unsigned wsum[32];
  __shared__ int s_ncand;
  __shared__ unsigned s_prefix;
  __shared__ int s_krem, s_count;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int r = CL == 1 ? 0 : (int)cluster.block_rank();
  const int bl = blockIdx.x / CL;
  const int b = b0 + bl, h = PER_LAYER ? 0 : blockIdx.y;
  const int s0 = st.start[bl];
  const int n = st.start[bl + 1] - s0;
  const float *sc = scores + (long long)h * T + s0;
  const int chunk = (n + CL - 1) / CL;
  const int lo = (int)r * chunk;
  const int len = (lo + chunk < n ? lo + chunk : n) - lo;         // may be <= 0

  if (n == 0) return;
  // the budget, the offset and the scores are requested together, without a branch between the loads (tokens past the
  // range read its neighbours and are not counted: with a branch 16 scores took 9.0 us)
  int k = budgets[b];
  const long long off = out_offsets[b];
  unsigned key[KPT];
  {
    float x[KPT];
    const int last = n - 1;
#pragma unroll
    for (int i = 0; i < KPT; ++i) {
      const int t = lo + tid + i * NT;
      x[i] = __ldg(sc + (t < last ? t : last));
    }
    if (PER_LAYER)
      for (int hh = 1; hh < H; ++hh) {
        const float *sh = sc + (long long)hh * T;
#pragma unroll
        for (int i = 0; i < KPT; ++i) {
          const int t = lo + tid + i * NT;
          x[i] += __ldg(sh + (t < last ? t : last));
        }
      }
#pragma unroll
    for (int i = 0; i < KPT; ++i) key[i] = score_key(x[i]);
    if (protect) {
#pragma unroll
      for (int i = 0; i < KPT; ++i) {
        const int t = lo + tid + i * NT;
        if (__ldg(protect + s0 + (t < last ? t : last))) key[i] = 0xFFFFFFFFu;
      }
    }
  }
  k = k < 0 ? 0 : (k > n ? n : k);
  if (k == 0) return;                                    // same decision in every block of the cluster
  if (off < 0 || off + k > cap) {
    if (tid == 0 && r == 0) atomicOr(status, FC_DEV_FLAG_INTERNAL);
    return;
  }
  int *dst = out_idx + (long long)h * cap + off;
  auto sync_all = [&]() { if (CL == 1) __syncthreads(); else cluster.sync(); };

  unsigned tau = 0;
  int need = 0;
  if (k < n) {
    for (int i = tid; i < 3 * kBins; i += NT) (&lhist[0][0])[i] = 0;
    if (tid == 0) s_ncand = 0;
    __syncthreads();
    unsigned prefix = 0, mask = 0;
    int krem = k;
#pragma unroll 1
    for (int pass = 0; pass < 3; ++pass) {
      const int shift = pass == 0 ? 22 : pass == 1 ? 11 : 0;
      const unsigned digits = pass == 0 ? 1023u : 2047u;
#pragma unroll
      for (int i = 0; i < KPT; ++i) {
        const bool m = (tid + i * NT < len) && ((key[i] & mask) == prefix);
        if (pass == 0) {                                 // a warp's keys share a few values of the first digit
          const unsigned act = __ballot_sync(0xffffffffu, m);
          if (m) {
            const unsigned dgt = key[i] >> shift;
            const unsigned peers = __match_any_sync(act, dgt);
            if (lane == __ffs(peers) - 1) atomicAdd(&lhist[0][dgt], __popc(peers));
          }
        } else if (m) {                                  // and are spread over the later ones
          atomicAdd(&lhist[pass][(key[i] >> shift) & digits], 1);
        }
      }
      sync_all();                                        // every block's histogram of this digit is complete
      // thread t owns the bins t*PB .. t*PB + PB - 1; find the bin where the count from the top reaches krem
      constexpr int PB = kBins / NT;
      int v[PB], mine = 0;
#pragma unroll
      for (int i = 0; i < PB; ++i) {
        v[i] = 0;
#pragma unroll
        for (int rr = 0; rr < CL; ++rr)
          v[i] += CL == 1 ? lhist[pass][tid * PB + i] : *cluster.map_shared_rank(&lhist[pass][tid * PB + i], rr);
        mine += v[i];
      }
      int above = mine;                                  // inclusive suffix sum over the lanes from this one up
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_down_sync(0xffffffffu, above, o);
        if (lane + o < 32) above += t;
      }
      if (lane == 0) wsum[warp] = (unsigned)above;
      __syncthreads();
      const int higher = __reduce_add_sync(0xffffffffu, lane < NW && lane > warp ? (int)wsum[lane] : 0);
      int cum = higher + above - mine;                   // keys strictly above this thread's bins
      if (cum < krem && krem <= cum + mine) {
#pragma unroll
        for (int i = PB - 1; i >= 0; --i) {
          if (cum < krem && krem <= cum + v[i]) {
            s_krem = krem - cum;
            s_count = v[i];
            s_prefix = prefix | ((unsigned)(tid * PB + i) << shift);
          }
          cum += v[i];
        }
      }
      __syncthreads();
      krem = s_krem;
      prefix = s_prefix;
      mask |= digits << shift;
      const int count = s_count;
      if (pass == 2) break;
      if (count <= kCandidates) {
        // the keys of the bin, from every block, then the one that krem of them (ties included) reach
#pragma unroll
        for (int i = 0; i < KPT; ++i)
          if (tid + i * NT < len && (key[i] & mask) == prefix) cand[atomicAdd(&s_ncand, 1)] = key[i];
        sync_all();
        if (CL == 1) {
          for (int i = tid; i < count; i += NT) all[i] = cand[i];
        } else {
          int at = 0;
          for (int rr = 0; rr < CL; ++rr) {
            const int c = *cluster.map_shared_rank(&s_ncand, rr);
            for (int i = tid; i < c; i += NT) all[at + i] = *cluster.map_shared_rank(&cand[i], rr);
            at += c;
          }
        }
        __syncthreads();
        for (int i = tid; i < count; i += NT) {
          const unsigned x = all[i];
          int gt = 0, eq = 0;
#pragma unroll 8
          for (int q = 0; q < count; ++q) { gt += all[q] > x ? 1 : 0; eq += all[q] == x ? 1 : 0; }
          if (gt < krem && krem <= gt + eq) { s_prefix = x; s_krem = krem - gt; }      // equal keys agree
        }
        __syncthreads();
        krem = s_krem;
        prefix = s_prefix;
        break;
      }
    }
    tau = prefix;
    need = krem;
  } else if (CL > 1) {
    cluster.sync();      // every block has started (elsewhere the digits' barriers see to it): the totals below go to all
  }

  // greater and tied keys of every run of 32 tokens, their exclusive prefix sums, the block's totals
#pragma unroll
  for (int i = 0; i < KPT; ++i) {
    const bool in = tid + i * NT < len;
    const unsigned g = __ballot_sync(0xffffffffu, in && key[i] > tau), e = __ballot_sync(0xffffffffu, in && key[i] == tau);
    if (lane == 0) runs[i * NW + warp] = (unsigned)__popc(g) | ((unsigned)__popc(e) << 16);
  }
  __syncthreads();
  {
    // CNT <= NT runs, one per thread
    const unsigned v = tid < CNT ? runs[tid] : 0u;
    unsigned incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned t = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += t;
    }
    if (lane == 31) wsum[warp] = incl;
    __syncthreads();
    const unsigned lower = __reduce_add_sync(0xffffffffu, lane < NW && lane < warp ? wsum[lane] : 0u);
    if (tid < CNT) runs[tid] = lower + incl - v;
    if (tid == NT - 1) {
      const unsigned all_runs = lower + incl;
      if (CL == 1) tot[0] = all_runs;
      else
#pragma unroll
        for (int rr = 0; rr < CL; ++rr) *cluster.map_shared_rank(&tot[r], rr) = all_runs;
    }
  }
  sync_all();                                            // also orders runs for the block
  int gt_before = 0, tie_before = 0, my_gt = 0, my_tie = 0;
#pragma unroll
  for (int rr = 0; rr < CL; ++rr) {
    const unsigned t = tot[rr];
    if (rr < r) { gt_before += (int)(t & 0xFFFFu); tie_before += (int)(t >> 16); }
    if (rr == r) { my_gt = (int)(t & 0xFFFFu); my_tie = (int)(t >> 16); }
  }
  // (a block holds at most 16384 scores, so neither 16-bit field can overflow)
  const int first = gt_before + (tie_before < need ? tie_before : need);    // rank of this block's first token
#pragma unroll
  for (int i = 0; i < KPT; ++i) {
    const bool in = tid + i * NT < len;
    const bool g = in && key[i] > tau, e = in && key[i] == tau;
    const unsigned bg = __ballot_sync(0xffffffffu, g), be = __ballot_sync(0xffffffffu, e), below = (1u << lane) - 1u;
    const unsigned base = runs[i * NW + warp];
    const int ng = gt_before + (int)(base & 0xFFFFu) + __popc(bg & below);
    const int nt = tie_before + (int)(base >> 16) + __popc(be & below);
    if (g || (e && nt < need)) {
      const int pos = ng + (nt < need ? nt : need), tok = lo + tid + i * NT;
      sel[pos - first] = (unsigned short)(tid + i * NT);
      dst[pos] = tok;
      if (PER_LAYER)
        for (int hh = 1; hh < H; ++hh) dst[(long long)hh * cap + pos] = tok;
    }
  }
  __syncthreads();                                       // this block's tokens are visible to its warps

  // gather the rows this block selected: ranks [first, first + count)
  int tie_take = need - tie_before;
  tie_take = tie_take < 0 ? 0 : (tie_take > my_tie ? my_tie : tie_take);
  const int count = my_gt + tie_take;
  const int n16 = row_bytes >> 4;
  // a warp takes kGatherRows rows at a time: their 16-byte pieces are requested together, so
  // that several independent round trips to DRAM are in flight per warp instead of one after the other
  constexpr int kGatherRows = 4;
  const int per_head = 2 * n16;
  const char *kb = kin + ((long long)s0 + lo) * stride_token_b, *vb = vin + ((long long)s0 + lo) * stride_token_b;
  for (int rr0 = warp * kGatherRows; rr0 < count; rr0 += NW * kGatherRows) {
    int tok[kGatherRows];
#pragma unroll
    for (int g = 0; g < kGatherRows; ++g) tok[g] = sel[rr0 + g < count ? rr0 + g : rr0];   // past the end: repeated, not stored
    for (int w = lane; w < (PER_LAYER ? H * per_head : per_head); w += 32) {
      const int hh = PER_LAYER ? w / per_head : h;
      const int u = PER_LAYER ? w - hh * per_head : w;
      const bool isv = u >= n16;
      const int uu = isv ? u - n16 : u;
      const char *in = (isv ? vb : kb) + (long long)hh * stride_head_b + 16ll * uu;
      char *out = (isv ? out_v : out_k) + 16ll * uu;
      uint4 val[kGatherRows];
#pragma unroll
      for (int g = 0; g < kGatherRows; ++g) val[g] = *reinterpret_cast<const uint4 *>(in + tok[g] * stride_token_b);
#pragma unroll
      for (int g = 0; g < kGatherRows; ++g)
        if (rr0 + g < count)
          *reinterpret_cast<uint4 *>(out + ((off + first + rr0 + g) * H + hh) * (long long)row_bytes) = val[g];
    }
  }
}

// The kernel: grid (CL * sequences in chunk, heads or 1, layers in chunk); blockIdx.z picks the
// layer's pointers from the table and the layer's rows of budgets [L][B] and out_offsets [L][B+1].
// overlap != 0 (launched with the programmatic-serialisation attribute): the next launch in the stream
// may start as soon as every block of this one has begun, and this grid does not finish before its
// predecessor has, so "the last launch is complete" still means "all of them are".
template <int KPT, bool PER_LAYER, int CL, int NT>
__global__ void __cluster_dims__(CL, 1, 1) __launch_bounds__(NT, 1024 / NT)
k_select_gather(const __grid_constant__ LayerTable lt, long long T, const __grid_constant__ SeqTable st, int b0, int B,
                const int *__restrict__ budgets, const long long *__restrict__ out_offsets,
                int *__restrict__ status, long long stride_token_b,
                long long stride_head_b, int row_bytes, int H, int overlap,
                const unsigned char *__restrict__ protect) {
  if (overlap) asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
  const int z = blockIdx.z;
  select_gather_body<KPT, PER_LAYER, CL, NT>(lt.scores[z], T, st, b0, budgets + (size_t)z * B,
                                         out_offsets + (size_t)z * (B + 1), lt.out_idx[z], lt.cap[z], status, lt.k[z], lt.v[z],
                                         stride_token_b, stride_head_b, row_bytes, H, lt.out_k[z], lt.out_v[z], protect);
  if (overlap) asm volatile("griddepcontrol.wait;\n" ::: "memory");
}

fc_status check_cu(const int32_t *cu, int batch) {
  if (!cu || batch < 0 || cu[0] != 0) return FC_ERR_INVALID_ARG;
  for (int b = 0; b < batch; ++b)
    if (cu[b + 1] < cu[b]) return FC_ERR_INVALID_ARG;
  return FC_OK;
}

}  // namespace

extern "C" fc_status fc_allocate_budgets(fc_handle *h, const double *energy, int32_t num_layers,
                                         int32_t batch, const int32_t *cu_seqlens_host, double rho,
                                         int32_t min_keep, int32_t *budgets, int64_t *out_offsets,
                                         fc_stream stream) {
  if (!h || !energy || !budgets || !out_offsets) return FC_ERR_INVALID_ARG;
  if (num_layers < 1 || batch < 0 || min_keep < 0) return FC_ERR_INVALID_ARG;
  if (!(rho >= 0.0) || isinf(rho)) return FC_ERR_INVALID_ARG;
  if (num_layers > 1024) return FC_ERR_UNSUPPORTED;
  fc_status s = check_cu(cu_seqlens_host, batch);
  if (s != FC_OK) return s;
  int dev = -1;
  FC_CUDA_TRY(cudaGetDevice(&dev));
  if (dev != h->device) FC_CUDA_TRY(cudaSetDevice(h->device));
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  if ((s = fc_flush_pending(h, st)) != FC_OK) return s;    // the energies may still be in flight on the internal streams
  const int L = num_layers;
  const size_t sm = (size_t)(6 * L) * sizeof(double) + (size_t)(2 * L) * sizeof(int);
  if (sm > 48 * 1024) FC_CUDA_TRY(cudaFuncSetAttribute(k_allocate, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
  for (int b0 = 0; b0 < batch || b0 == 0; b0 += kSeqChunk) {
    const int nseq = batch - b0 < kSeqChunk ? batch - b0 : kSeqChunk;
    SeqTable tab;
    for (int i = 0; i <= nseq; ++i) tab.start[i] = cu_seqlens_host[b0 + i];
    // a programmatic dependent: resident when the kernel before it ends (an empty batch still has its offsets written)
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3(nseq > 0 ? nseq : 1);
    lc.blockDim = dim3(kAllocThreads);
    lc.dynamicSmemBytes = sm;
    lc.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    lc.attrs = at;
    lc.numAttrs = 1;
    if (cudaLaunchKernelEx(&lc, k_allocate, energy, (int)L, (int)batch, b0, tab, rho, (int)min_keep, budgets,
                           reinterpret_cast<long long *>(out_offsets), h->done_counter + 2 * FC_LAYER_CHUNK,
                           (unsigned)(batch > 0 ? batch : 1)) != cudaSuccess) {
      cudaGetLastError();
      return FC_ERR_CUDA;
    }
    if ((s = fc_after_launch(h)) != FC_OK) return s;
  }
  return FC_OK;
}

extern "C" size_t fc_select_workspace_bytes(const fc_handle *h, const fc_kv_view *kv) {
  if (!h || !kv) return 0;
  return 256;   // the selection keeps its state on chip; a token amount so callers can treat both phases alike
}

extern "C" fc_status fc_select_compact(fc_handle *h, const fc_kv_view *kv, const float *scores,
                                       const int32_t *budgets, const int64_t *out_offsets,
                                       void *out_k, void *out_v, int32_t *out_idx,
                                       int64_t out_capacity_rows, void *workspace,
                                       size_t workspace_bytes, fc_stream stream) {
  return fc_select_compact_ex(h, kv, scores, budgets, out_offsets, out_k, out_v, out_idx, out_capacity_rows,
                              nullptr, workspace, workspace_bytes, stream);
}

namespace {

// Argument checks shared by the selection entry points (everything but the per-layer pointers).
fc_status check_select_shape(const fc_handle *h, const fc_kv_view *kv, const void *workspace, size_t workspace_bytes) {
  if (!h || !kv) return FC_ERR_INVALID_ARG;
  if (kv->num_heads <= 0 || kv->head_dim <= 0) return FC_ERR_INVALID_ARG;
  if (kv->dtype != FC_F32 && kv->dtype != FC_F16 && kv->dtype != FC_BF16) return FC_ERR_UNSUPPORTED;
  const int es = kv->dtype == FC_F32 ? 4 : 2;
  if ((kv->head_dim * es) % 16) return FC_ERR_UNSUPPORTED;
  fc_status s = check_cu(kv->cu_seqlens, kv->batch);
  if (s != FC_OK) return s;
  for (int b = 0; b < kv->batch; ++b)
    if (kv->cu_seqlens[b + 1] - kv->cu_seqlens[b] > kSelMaxTokens) return FC_ERR_UNSUPPORTED;
  if ((kv->stride_token * es) % 16 || (kv->stride_head * es) % 16) return FC_ERR_INVALID_ARG;
  if (!workspace || ((uintptr_t)workspace & 255) || workspace_bytes < fc_select_workspace_bytes(h, kv))
    return FC_ERR_WORKSPACE;
  return FC_OK;
}

// Dynamic shared memory beyond the default, once per kernel and device.
template <class Kern>
fc_status allow_smem(Kern kern, size_t bytes) {
  static std::mutex mu;
  static std::unordered_map<unsigned long long, size_t> done;     // (device, kernel) -> bytes already allowed
  int dev = 0;
  FC_CUDA_TRY(cudaGetDevice(&dev));
  const unsigned long long key = (unsigned long long)reinterpret_cast<uintptr_t>(reinterpret_cast<const void *>(kern)) ^
                                 ((unsigned long long)dev << 56);
  std::lock_guard<std::mutex> lock(mu);
  size_t &have = done[key];
  if (have >= bytes) return FC_OK;
  FC_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes));
  have = bytes;
  return FC_OK;
}

// Launches the selection for `nl` (<= kLayerChunk) layers whose pointers are in `lt`; budgets and
// out_offsets point at the first of these layers' rows.
fc_status launch_select(fc_handle *h, cudaStream_t st, const fc_kv_view *kv, const LayerTable &lt, int nl,
                        const int32_t *budgets, const int64_t *out_offsets, bool per_layer,
                        const unsigned char *protect) {
  const int es = kv->dtype == FC_F32 ? 4 : 2;
  const long long T = kv->cu_seqlens[kv->batch];
  fc_status s;
  for (int b0 = 0; b0 < kv->batch; b0 += kSeqChunk) {
    const int nseq = kv->batch - b0 < kSeqChunk ? kv->batch - b0 : kSeqChunk;
    SeqTable tab;
    for (int i = 0; i <= nseq; ++i) tab.start[i] = kv->cu_seqlens[b0 + i];
    int nmax = 0;
    for (int i = 0; i < nseq; ++i) nmax = tab.start[i + 1] - tab.start[i] > nmax ? tab.start[i + 1] - tab.start[i] : nmax;
    // Blocks of 1024 threads, as few per (sequence, head) as hold the longest sequence at 16 scores per thread: every
    // phase of the select waits on barriers, and one block's are a fraction of a cluster's (28 x 4 heads of 1500 tokens:
    // 22.6 us with two blocks, 12.2 with one; 8 ragged short sequences 131 -> 72 us; one layer of 1024 tokens: 10.0 us
    // with one block, 18.4 with eight).  Two where a layer keeps one index set, whose few clusters gather all heads.
    int cl = per_layer ? 2 : 1;
    while (cl < kSelCluster && nmax > cl * 1024 * kSelKptMax) cl *= 2;
    // But a block also gathers the rows it chose, so where the clusters would leave most of the SMs idle, sequences of
    // more than 2048 tokens get two blocks and of more than 4096 four (one layer of 4 heads of 4096, 8192, 16384 tokens:
    // 23.5 -> 19.5, 35.8 -> 23.4, 62.5 -> 29.6 us; 64 heads of 16384 with two: 68.6 -> 56.3).  Not with eight, whose
    // clusters run 15 at a time, and not to the last SM: 36 clusters of four do not fit at once (32768 tokens: 53 -> 68).
    const long long units = (long long)nseq * kv->num_heads * nl;
    while (!per_layer && cl < 4 && nmax > 2048 * cl && units * 2 * cl <= h->num_sms - h->num_sms / 8) cl *= 2;
    int kpt = 2;
    while (kpt < kSelKptMax && nmax > cl * 1024 * kpt) kpt *= 2;
    // Short sequences in more blocks than SMs: fewer threads with more scores each, so that several blocks share an SM
    // and some gather rows (bound by memory) while others select (bound by barriers): 28 x 32 heads of 1000 tokens
    // 62 -> 43 us, of 300 34 -> 15, 28 x 4 heads of 8 ragged sequences up to 2311 69 -> 60.  Not beyond 4096 tokens,
    // where the gather fills the time (8192: 128 -> 137, 16384: 1.12 -> 1.20 ms).
    int nt = 1024;
    if (!per_layer && kpt <= 4 && units > h->num_sms) {
      nt = nmax <= 1024 ? 256 : 512;
      kpt = nmax <= 2048 ? 4 : 8;
    }
    {
      ProfScope ps(h, FC_K_SELECT, st);
      const size_t sm = (size_t)kpt * nt * sizeof(unsigned short);
#define FC_SEL_LAUNCH(KPT, PL, CLV, NTV)                                                                \
  do {                                                                                                  \
    if ((s = allow_smem(k_select_gather<KPT, PL, CLV, NTV>, sm)) != FC_OK) return s;                    \
    cudaLaunchConfig_t lc = {};                                                                         \
    lc.gridDim = dim3(CLV * nseq, (PL) ? 1 : kv->num_heads, nl);                                        \
    lc.blockDim = dim3(NTV);                                                                             \
    lc.dynamicSmemBytes = sm;                                                                           \
    lc.stream = st;                                                                                     \
    cudaLaunchAttribute at[1];                                                                          \
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;                                      \
    at[0].val.programmaticStreamSerializationAllowed = 1;                                               \
    lc.attrs = at;                                                                                      \
    lc.numAttrs = (h->select_overlap && h->after_select) ? 1 : 0;                                       \
    launch_err = cudaLaunchKernelEx(&lc, k_select_gather<KPT, PL, CLV, NTV>, lt, (long long)T, tab, b0, (int)kv->batch, \
        budgets, reinterpret_cast<const long long *>(out_offsets),                                      \
        h->status_word, (long long)(kv->stride_token * es), (long long)(kv->stride_head * es),          \
        (int)(kv->head_dim * es), (int)kv->num_heads, (int)h->select_overlap, protect);                 \
  } while (0)
#define FC_SEL_CASE(KPT, PL, CLV) \
  else if (nt == 1024 && kpt == KPT && cl == CLV && per_layer == PL) FC_SEL_LAUNCH(KPT, PL, CLV, 1024);
#define FC_SEL_MANY(KPT, NTV) else if (nt == NTV && kpt == KPT && cl == 1) FC_SEL_LAUNCH(KPT, false, 1, NTV);
      cudaError_t launch_err = cudaErrorInvalidValue;
      if (false) {}
      FC_SEL_CASE(2, false, 1) FC_SEL_CASE(4, false, 1) FC_SEL_CASE(8, false, 1) FC_SEL_CASE(16, false, 1)
      FC_SEL_CASE(2, false, 2) FC_SEL_CASE(4, false, 2) FC_SEL_CASE(8, false, 2) FC_SEL_CASE(16, false, 2)
      FC_SEL_CASE(2, false, 4) FC_SEL_CASE(4, false, 4) FC_SEL_CASE(8, false, 4) FC_SEL_CASE(16, false, 4)
      FC_SEL_CASE(16, false, 8)
      FC_SEL_CASE(2, true, 2) FC_SEL_CASE(4, true, 2) FC_SEL_CASE(8, true, 2) FC_SEL_CASE(16, true, 2)
      FC_SEL_CASE(16, true, 4) FC_SEL_CASE(16, true, 8)
      FC_SEL_MANY(4, 256) FC_SEL_MANY(4, 512) FC_SEL_MANY(8, 512)
#undef FC_SEL_MANY
#undef FC_SEL_CASE
#undef FC_SEL_LAUNCH
      if (launch_err != cudaSuccess) { cudaGetLastError(); return FC_ERR_CUDA; }
    }
    if ((s = fc_after_launch(h)) != FC_OK) return s;
    h->after_select = true;
  }
  return FC_OK;
}

}  // namespace

extern "C" fc_status fc_select_compact_ex(fc_handle *h, const fc_kv_view *kv, const float *scores,
                                          const int32_t *budgets, const int64_t *out_offsets,
                                          void *out_k, void *out_v, int32_t *out_idx,
                                          int64_t out_capacity_rows, const fc_select_options *opt,
                                          void *workspace, size_t workspace_bytes, fc_stream stream) {
  if (!h || !kv || !kv->k || !kv->v || !scores || !budgets || !out_offsets || !out_k || !out_v || !out_idx)
    return FC_ERR_INVALID_ARG;
  if (out_capacity_rows < 0) return FC_ERR_INVALID_ARG;
  fc_status s = check_select_shape(h, kv, workspace, workspace_bytes);
  if (s != FC_OK) return s;
  if (((uintptr_t)kv->k & 15) || ((uintptr_t)kv->v & 15) || ((uintptr_t)out_k & 15) || ((uintptr_t)out_v & 15))
    return FC_ERR_INVALID_ARG;
  int dev = -1;
  FC_CUDA_TRY(cudaGetDevice(&dev));
  if (dev != h->device) FC_CUDA_TRY(cudaSetDevice(h->device));
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  if ((s = fc_flush_pending(h, st)) != FC_OK) return s;
  LayerTable lt = {};
  lt.scores[0] = scores;
  lt.k[0] = static_cast<const char *>(kv->k);
  lt.v[0] = static_cast<const char *>(kv->v);
  lt.out_k[0] = static_cast<char *>(out_k);
  lt.out_v[0] = static_cast<char *>(out_v);
  lt.out_idx[0] = out_idx;
  lt.cap[0] = out_capacity_rows;
  return launch_select(h, st, kv, lt, 1, budgets, out_offsets, opt && opt->per_layer != 0,
                       opt ? static_cast<const unsigned char *>(opt->protect) : nullptr);
}

extern "C" fc_status fc_select_compact_layers(fc_handle *h, const fc_kv_view *shape, const fc_layer_buffers *layers,
                                              int32_t num_layers, const int32_t *budgets, const int64_t *out_offsets,
                                              const fc_select_options *opt,
                                              void *workspace, size_t workspace_bytes, fc_stream stream) {
  if (!h || !shape || !layers || !budgets || !out_offsets || num_layers < 1) return FC_ERR_INVALID_ARG;
  fc_status s = check_select_shape(h, shape, workspace, workspace_bytes);
  if (s != FC_OK) return s;
  for (int l = 0; l < num_layers; ++l) {
    const fc_layer_buffers &b = layers[l];
    if (!b.k || !b.v || !b.scores || !b.out_k || !b.out_v || !b.out_idx || b.out_capacity_rows < 0) return FC_ERR_INVALID_ARG;
    if (((uintptr_t)b.k & 15) || ((uintptr_t)b.v & 15) || ((uintptr_t)b.out_k & 15) || ((uintptr_t)b.out_v & 15))
      return FC_ERR_INVALID_ARG;
  }
  int dev = -1;
  FC_CUDA_TRY(cudaGetDevice(&dev));
  if (dev != h->device) FC_CUDA_TRY(cudaSetDevice(h->device));
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  if ((s = fc_flush_pending(h, st)) != FC_OK) return s;
  const int B = shape->batch;
  for (int l0 = 0; l0 < num_layers; l0 += kLayerChunk) {
    const int nl = num_layers - l0 < kLayerChunk ? num_layers - l0 : kLayerChunk;
    LayerTable lt = {};
    for (int i = 0; i < nl; ++i) {
      const fc_layer_buffers &b = layers[l0 + i];
      lt.scores[i] = b.scores;
      lt.k[i] = static_cast<const char *>(b.k);
      lt.v[i] = static_cast<const char *>(b.v);
      lt.out_k[i] = static_cast<char *>(b.out_k);
      lt.out_v[i] = static_cast<char *>(b.out_v);
      lt.out_idx[i] = b.out_idx;
      lt.cap[i] = b.out_capacity_rows;
    }
    s = launch_select(h, st, shape, lt, nl, budgets + (size_t)l0 * B, out_offsets + (size_t)l0 * (B + 1),
                      opt && opt->per_layer != 0,
                      opt ? static_cast<const unsigned char *>(opt->protect) : nullptr);
    if (s != FC_OK) return s;
  }
  return FC_OK;
}

extern "C" int64_t fc_layer_capacity_rows(int32_t num_layers, int32_t batch, const int32_t *cu_seqlens,
                                          double rho, int32_t min_keep) {
  if (num_layers < 1 || batch < 0 || !cu_seqlens || min_keep < 0 || !(rho >= 0.0) || isinf(rho)) return -1;
  if (check_cu(cu_seqlens, batch) != FC_OK) return -1;
  long long rows = 0;
  for (int b = 0; b < batch; ++b) {
    const long long N = cu_seqlens[b + 1] - cu_seqlens[b];
    if (N == 0) continue;
    const double lo = (double)(min_keep < N ? min_keep : N), hi = (double)N, L = (double)num_layers;
    double bt = floor(rho * (double)N * L + 0.5);        // B_tot of the sequence, as k_allocate computes it
    if (bt < L * lo) bt = L * lo;
    if (bt > L * hi) bt = L * hi;
    rows += bt < hi ? (long long)bt : N;                  // one layer gets at most N and at most B_tot
  }
  return rows;
}
