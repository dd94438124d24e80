// Decoding step on the compacted cache (Sec. 3.1, Eq. 3-4): Softmax(q K^T / sqrt(d)) V over the rows the
// compressor kept plus the uncompressed tail.  The step reads every K and V row once and is bound by
// that read (or, on short caches, by the chain of latencies of one launch), so the design is about keeping HBM busy:
//
//  * the tiles (64 rows) of all sequences of all KV heads form one line, and the grid's blocks, one per SM, take equal
//    shares of it, whatever the lengths of the sequences are: a block's share is one or more runs of consecutive tiles
//    of one sequence and head each (a seventh of a step over kept rows of 1638, 205, 3277 and 820 tokens, where a grid
//    of splits sized for the longest sequence left half of the SMs without rows);
//  * a producer warp fills a four-stage shared-memory ring by tiled TMA loads (128-byte swizzle), one mbarrier pair per
//    stage; the four other warps wait for nothing but the tile they use;
//  * all query heads of a KV head (up to 16) are one 16-row operand of m16n8k16 tensor-core products,
//    so a K/V tile is read from shared memory once for the whole group; each of the 4 warps owns 16
//    rows of the tile and keeps its own running maximum, sum and 16 x 128 fp32 output;
//  * the warps' partial results are merged in shared memory; a sequence covered by one block is finished there, else a
//    second small kernel merges the blocks' shares.
// Both launches are programmatic dependents: they are set up while the kernel before them in the stream ends.
// Together: 28 layers of 65536 rows 965 -> 784 us per step, of those kept rows with tails 397 -> 310 us (from a graph 754
// and 294; the host enqueues the 28 calls in 230..370 us, behind the device).
#include <cuda.h>

#include "fc_common.cuh"
#include "fc_mbar.cuh"

namespace {

constexpr int kD = 128;                 // head_dim
constexpr int kTile = 64;               // rows per tile
constexpr int kWarps = 4;               // consumer warps; one more loads
constexpr int kConsumers = 32 * kWarps;
constexpr int kThreadsD = kConsumers + 32;
constexpr int kBoxBytes = kTile * 128;  // one TMA box: 64 rows x 64 elements of 2 bytes
constexpr int kStageBytes = 4 * kBoxBytes;   // K low/high halves, V low/high halves
constexpr int kStages = 4;
constexpr int kEarlyTiles = 2;                // tiles brought into L2 ahead

struct DecodeParams {
  const void *q;
  void *out;
  const long long *offsets;
  const int *tail_len;
  float *part_o;        // [slot][query heads of a KV head][128]
  float2 *part_ml;      // [slot][query heads of a KV head]: (running maximum in log2 units, sum)
  int2 *span;           // [H][batch]: first and last block with tiles of the sequence (first > last: none)
  int *status;
  int B, H, Hq, G, nb, tail_cap, has_tail;
  float scale_log2;     // log2(e) / sqrt(d)
  int cache_rows;
  const void *cache_k, *cache_v;
};

struct DecodeMaps {
  CUtensorMap k, v, tk, tv;
};

// Tiled loads into this block's shared memory; completion is counted in bytes on `bar`.  One destination block only.
__device__ __forceinline__ void tma_load_3d(void *dst, const CUtensorMap *map, int c0, int c1, int c2,
                                            unsigned long long *bar) {
  asm volatile("cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];\n"
               ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(reinterpret_cast<unsigned long long>(map)),
                 "r"(c0), "r"(c1), "r"(c2), "r"((unsigned)__cvta_generic_to_shared(bar)) : "memory");
}
__device__ __forceinline__ void tma_load_4d(void *dst, const CUtensorMap *map, int c0, int c1, int c2, int c3,
                                            unsigned long long *bar) {
  asm volatile("cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];\n"
               ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(reinterpret_cast<unsigned long long>(map)),
                 "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"((unsigned)__cvta_generic_to_shared(bar)) : "memory");
}

__device__ __forceinline__ void prefetch_map(const CUtensorMap *map) {
  asm volatile("prefetch.tensormap [%0];\n" ::"l"(reinterpret_cast<unsigned long long>(map)) : "memory");
}

__device__ __forceinline__ void ldmatrix_x4(unsigned addr, unsigned (&r)[4]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
__device__ __forceinline__ void ldmatrix_x4_trans(unsigned addr, unsigned (&r)[4]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}

// D += A (16x16, row) * B (16x8, col), fp32 accumulation.
template <typename T> struct Mma;
template <> struct Mma<__half> {
  __device__ static void run(float (&d)[4], const unsigned (&a)[4], unsigned b0, unsigned b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};\n"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
  }
  __device__ static unsigned pack(float x, float y) {
    const __half2 h = __floats2half2_rn(x, y);
    return *reinterpret_cast<const unsigned *>(&h);
  }
  __device__ static __half from_float(float x) { return __float2half_rn(x); }
};
template <> struct Mma<__nv_bfloat16> {
  __device__ static void run(float (&d)[4], const unsigned (&a)[4], unsigned b0, unsigned b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};\n"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
  }
  __device__ static unsigned pack(float x, float y) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(x, y);
    return *reinterpret_cast<const unsigned *>(&h);
  }
  __device__ static __nv_bfloat16 from_float(float x) { return __float2bfloat16_rn(x); }
};

// Byte offset of the 16-byte chunk `chunk` (0..15 over the 128 channels) of row `row` (0..63) inside a K or V
// half-pair as the two swizzled TMA boxes leave it: channels 0..63 in the first box, 64..127 in the second;
// inside a box a row is 128 bytes and chunk j of row r sits at position j ^ (r & 7).
__device__ __forceinline__ unsigned tile_offset(int row, int chunk) {
  return (unsigned)((chunk >> 3) * kBoxBytes + row * 128 + (((chunk & 7) ^ (row & 7)) << 4));
}

constexpr int kFoldWarps = 4;           // warps of the second kernel
constexpr int kMergeStride = kD + 4;    // floats per row of a warp's output in the merge buffer

// One sequence: its rows in the cache and in the tail, as tiles (main rows first; a tile lies in one of the two).
struct SeqRows {
  long long off0;
  int n_main, n_tail, tiles_main, tiles;
};
template <bool EARLY = false>            // before the kernels in front are done: nothing of it may stay in L1
__device__ __forceinline__ SeqRows seq_rows(const DecodeParams &P, int b) {
  SeqRows s;
  s.off0 = EARLY ? __ldcg(P.offsets + b) : P.offsets[b];
  const long long nm = (EARLY ? __ldcg(P.offsets + b + 1) : P.offsets[b + 1]) - s.off0;
  s.n_main = nm < 0 ? 0 : (int)nm;
  int nt = P.has_tail ? (EARLY ? __ldcg(P.tail_len + b) : P.tail_len[b]) : 0;
  s.n_tail = nt < 0 ? 0 : (nt > P.tail_cap ? P.tail_cap : nt);
  s.tiles_main = (s.n_main + kTile - 1) / kTile;
  s.tiles = s.tiles_main + (s.n_tail + kTile - 1) / kTile;
  return s;
}

// The line of T tiles, head after head and sequence after sequence: block i takes the tiles [i*T/nb, (i+1)*T/nb).
// (32-bit division where the product fits: a 64-bit one costs some hundred cycles before the first load.)
__device__ __forceinline__ long long muldiv(long long a, int m, long long d) {
  const unsigned long long x = (unsigned long long)a * (unsigned)m;
  return (x >> 32) == 0 && ((unsigned long long)d >> 32) == 0 ? (long long)((unsigned)x / (unsigned)d) : (long long)(x / (unsigned long long)d);
}
__device__ __forceinline__ long long share_start(int i, long long T, int nb) { return muldiv(T, i, nb); }
__device__ __forceinline__ int share_of(long long t, long long T, int nb) {
  const unsigned long long x = (unsigned long long)(t + 1) * (unsigned)nb - 1;
  return (x >> 32) == 0 && ((unsigned long long)T >> 32) == 0 ? (int)((unsigned)x / (unsigned)T) : (int)(x / (unsigned long long)T);
}

// A block's share of the line: tiles [lo, hi), the first of them in sequence b of head h, whose tiles start at `line`.
struct Share {
  long long lo, hi, line, line_len;
  int h, b, nb;                                // nb: blocks that have tiles
};
// Tiles of all sequences, 32 at a time, in every warp for itself (no barrier before the first load): the sum, then
// the sequence that holds the first tile of this block's share.
template <bool EARLY>
__device__ __forceinline__ Share find_share(const DecodeParams &P, int blk, int lane) {
  Share r;
  auto tiles_of = [&](int i) { return i < P.B ? seq_rows<EARLY>(P, i).tiles : 0; };
  const int first32 = tiles_of(lane);
  long long total = __reduce_add_sync(0xffffffffu, first32);
  for (int b0 = 32; b0 < P.B; b0 += 32) total += __reduce_add_sync(0xffffffffu, tiles_of(b0 + lane));
  r.line_len = total * P.H;                    // every head has the same tiles
  r.nb = r.line_len < P.nb ? (int)r.line_len : P.nb;
  r.lo = blk < r.nb ? share_start(blk, r.line_len, r.nb) : 0;
  r.hi = blk < r.nb ? share_start(blk + 1, r.line_len, r.nb) : 0;
  r.h = r.lo > 0 ? (int)muldiv(r.lo, 1, total) : 0;
  const long long lo_head = r.lo - r.h * total;              // within the head
  r.b = 0;
  r.line = 0;
  long long at = 0;
  for (int b0 = 0; b0 < P.B; b0 += 32) {
    const int mine = b0 == 0 ? first32 : tiles_of(b0 + lane);
    int incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += v;
    }
    const unsigned past = __ballot_sync(0xffffffffu, at + incl > lo_head);
    if (past) {
      const int first = __ffs(past) - 1;
      r.b = b0 + first;
      r.line = r.h * total + at + __shfl_sync(0xffffffffu, incl - mine, first);
      break;
    }
    at += __shfl_sync(0xffffffffu, incl, 31);
  }
  return r;
}

__device__ __forceinline__ void consumers_sync() { asm volatile("bar.sync 1, %0;\n" ::"n"(kConsumers) : "memory"); }

struct DecodeShared {
  unsigned long long full[kStages], empty[kStages];
};

__device__ __forceinline__ void fold(float4 &acc, const float4 &v, float f) {      // acc += f * v
  acc.x = fmaf(v.x, f, acc.x);
  acc.y = fmaf(v.y, f, acc.y);
  acc.z = fmaf(v.z, f, acc.z);
  acc.w = fmaf(v.w, f, acc.w);
}
template <typename T>
__device__ __forceinline__ void store_head(T *out, const float4 &o, float l) {      // four channels of o / l
  const float inv = l > 0.f ? 1.f / l : 0.f;
  uint2 pk;
  pk.x = Mma<T>::pack(o.x * inv, o.y * inv);
  pk.y = Mma<T>::pack(o.z * inv, o.w * inv);
  *reinterpret_cast<uint2 *>(out) = pk;
}

// One block: its share of the line of tiles.
template <typename T>
__global__ void __launch_bounds__(kThreadsD)
k_decode(const DecodeParams P, const __grid_constant__ DecodeMaps M) {
  extern __shared__ unsigned char smem_raw[];
  unsigned char *smem = reinterpret_cast<unsigned char *>(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  float *mbuf = reinterpret_cast<float *>(smem + kStages * kStageBytes);
  __shared__ DecodeShared sh;
  const int blk = blockIdx.x;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int g = lane >> 2, t = lane & 3;

  asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
  if (tid == 0) {
    for (int i = 0; i < kStages; ++i) { mbar::init(&sh.full[i], 1u); mbar::init(&sh.empty[i], kWarps); }
    mbar::init_done();
  }
  if (tid == kConsumers) {
    prefetch_map(&M.k);
    prefetch_map(&M.v);
    if (P.has_tail) { prefetch_map(&M.tk); prefetch_map(&M.tv); }
  }
  __syncthreads();
  if (warp < kWarps) {
    // While the kernels in front still run, the first rows of the share are brought into L2.  Nothing is read from them
    // here, so it does not matter if those kernels are still writing them, or the offsets: a wrong guess only wastes it.
    // By plain prefetches, since the tensor engine takes as long over a prefetch as over the load; two tiles are what
    // fits into the wait (four and eight lose again what two gain), and with a share of one tile the load itself is as
    // early.  3 % of a step over 65536 rows, 5 % over the short caches named above.
    const Share sr = find_share<true>(P, blk, lane);
    if (sr.hi - sr.lo > 1) {
      const SeqRows s = seq_rows<true>(P, sr.b);
      const long long first = sr.lo - sr.line, left = s.tiles_main - first;
      const int n = (int)(left < kEarlyTiles ? left : kEarlyTiles) * kTile * 4;       // four lines of 128 bytes per row
      for (int i = tid; i < n; i += kConsumers) {
        const long long row = s.off0 + first * kTile + (i >> 2);
        const char *base = static_cast<const char *>(i & 2 ? P.cache_v : P.cache_k);
        if (row >= 0 && row < P.cache_rows)
          asm volatile("prefetch.global.L2 [%0];\n" ::"l"(base + ((size_t)row * P.H + sr.h) * (kD * 2) + (i & 1) * 128) : "memory");
      }
    }
  }
  asm volatile("griddepcontrol.wait;\n" ::: "memory");       // what the kernels before this one wrote is visible from here

  const Share sr = find_share<false>(P, blk, lane);
  const long long lo = sr.lo, hi = sr.hi, line_len = sr.line_len;
  const int nb = sr.nb;
  int h = sr.h, b = sr.b;
  long long line = sr.line;
  if (blk == 0)                                // sequences without rows
    for (int i = tid; i < P.B; i += kThreadsD)
      if (seq_rows(P, i).tiles == 0) {
        for (int hh = 0; hh < P.H; ++hh) P.span[(size_t)hh * P.B + i] = make_int2(0, -1);
        for (int c = 0; c < P.Hq * kD / 8; ++c)
          reinterpret_cast<uint4 *>(static_cast<T *>(P.out) + (size_t)i * P.Hq * kD)[c] = make_uint4(0u, 0u, 0u, 0u);
      }
  if (lo >= hi) return;
  SeqRows s = seq_rows(P, b);
  auto advance = [&](long long ti) {           // on to the sequence and head that tile ti belongs to
    while (ti >= line + s.tiles) {
      line += s.tiles;
      if (++b == P.B) { b = 0; ++h; }
      s = seq_rows(P, b);
    }
  };

  if (warp == kWarps) {
    // producer
    if (lane == 0) {
      int n = 0;
      bool ok = true;
      for (long long ti = lo; ti < hi; ++ti, ++n) {
        advance(ti);
        const int st = n % kStages;
        if (n >= kStages && !mbar::wait(&sh.empty[st], (unsigned)(n / kStages - 1) & 1u)) { ok = false; break; }
        unsigned char *dst = smem + st * kStageBytes;
        mbar::expect_tx(&sh.full[st], (unsigned)kStageBytes);
        const int lt = (int)(ti - line);
        if (lt < s.tiles_main) {
          const int r = (int)(s.off0 + (long long)lt * kTile);
          tma_load_3d(dst, &M.k, 0, h, r, &sh.full[st]);
          tma_load_3d(dst + kBoxBytes, &M.k, 64, h, r, &sh.full[st]);
          tma_load_3d(dst + 2 * kBoxBytes, &M.v, 0, h, r, &sh.full[st]);
          tma_load_3d(dst + 3 * kBoxBytes, &M.v, 64, h, r, &sh.full[st]);
        } else {
          const int r = (lt - s.tiles_main) * kTile;
          tma_load_4d(dst, &M.tk, 0, h, r, b, &sh.full[st]);
          tma_load_4d(dst + kBoxBytes, &M.tk, 64, h, r, b, &sh.full[st]);
          tma_load_4d(dst + 2 * kBoxBytes, &M.tv, 0, h, r, b, &sh.full[st]);
          tma_load_4d(dst + 3 * kBoxBytes, &M.tv, 64, h, r, b, &sh.full[st]);
        }
      }
      // not before its loads have landed may the block end, also where consumers gave up (they no longer wait for them);
      // where none did, this waits for what the consumers wait for
      if (!mbar::drain(sh.full, n)) ok = false;
      if (!ok) atomicOr(P.status, FC_DEV_FLAG_TIMEOUT);
    }
    return;
  }

  // consumers
  const unsigned sbase = (unsigned)__cvta_generic_to_shared(smem);
  float *mo = mbuf;                                                            // [warp][16][kMergeStride]
  float2 *mml = reinterpret_cast<float2 *>(mo + kWarps * 16 * kMergeStride);   // [warp][16]
  bool failed = false;
  int n = 0;
  for (long long ti = lo; ti < hi;) {
    advance(ti);
    const long long seg_end = line + s.tiles < hi ? line + s.tiles : hi;
    // the query heads of this KV head as the 16 x 128 left operand (rows past the group are zero)
    unsigned qf[kD / 16][4];
    {
      const T *qb = static_cast<const T *>(P.q) + ((long long)b * P.Hq + (long long)h * P.G) * kD;
      const bool r0 = g < P.G, r1 = g + 8 < P.G;
#pragma unroll
      for (int kk = 0; kk < kD / 16; ++kk) {
        const int c = 16 * kk + 2 * t;
        qf[kk][0] = r0 ? *reinterpret_cast<const unsigned *>(qb + g * kD + c) : 0u;
        qf[kk][1] = r1 ? *reinterpret_cast<const unsigned *>(qb + (g + 8) * kD + c) : 0u;
        qf[kk][2] = r0 ? *reinterpret_cast<const unsigned *>(qb + g * kD + c + 8) : 0u;
        qf[kk][3] = r1 ? *reinterpret_cast<const unsigned *>(qb + (g + 8) * kD + c + 8) : 0u;
      }
    }
    float oacc[kD / 8][4];
#pragma unroll
    for (int j = 0; j < kD / 8; ++j) oacc[j][0] = oacc[j][1] = oacc[j][2] = oacc[j][3] = 0.f;
    float m[2] = {-INFINITY, -INFINITY}, l[2] = {0.f, 0.f};

    for (; ti < seg_end; ++ti, ++n) {
      if (failed) continue;
      const int st = n % kStages;
      if (!mbar::wait_warp(&sh.full[st], (unsigned)(n / kStages) & 1u)) {
        // a load did not arrive in time (for any lane): say so and report an empty share
        failed = true;
        if (lane == 0) atomicOr(P.status, FC_DEV_FLAG_TIMEOUT);
        continue;
      }
      const int lt = (int)(ti - line);
      int valid = lt < s.tiles_main ? s.n_main - lt * kTile : s.n_tail - (lt - s.tiles_main) * kTile;
      valid = valid > kTile ? kTile : valid;
      const int wrow = 16 * warp;
      if (wrow < valid) {
        const unsigned sb = sbase + (unsigned)(st * kStageBytes);
        float sacc[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
        const int mi = lane >> 3;
#pragma unroll
        for (int kk = 0; kk < kD / 16; ++kk) {
          unsigned r[4];
          ldmatrix_x4(sb + tile_offset(wrow + (mi >> 1) * 8 + (lane & 7), 2 * kk + (mi & 1)), r);
          Mma<T>::run(sacc[0], qf[kk], r[0], r[1]);
          Mma<T>::run(sacc[1], qf[kk], r[2], r[3]);
        }
        float mx[2] = {-INFINITY, -INFINITY};
#pragma unroll
        for (int nb = 0; nb < 2; ++nb)
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const int key = wrow + 8 * nb + 2 * t + (e & 1);
            const float sv = key < valid ? sacc[nb][e] * P.scale_log2 : -INFINITY;
            sacc[nb][e] = sv;
            mx[e >> 1] = fmaxf(mx[e >> 1], sv);
          }
        float corr[2], ms[2];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          mx[i] = fmaxf(mx[i], __shfl_xor_sync(0xffffffffu, mx[i], 1));
          mx[i] = fmaxf(mx[i], __shfl_xor_sync(0xffffffffu, mx[i], 2));
          const float mn = fmaxf(m[i], mx[i]);
          ms[i] = (mn == -INFINITY) ? 0.f : mn;
          corr[i] = exp2f(m[i] - ms[i]);
          m[i] = mn;
        }
        float ps[2] = {0.f, 0.f};
#pragma unroll
        for (int nb = 0; nb < 2; ++nb)
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const float p = exp2f(sacc[nb][e] - ms[e >> 1]);
            sacc[nb][e] = p;
            ps[e >> 1] += p;
          }
        l[0] = l[0] * corr[0] + ps[0];
        l[1] = l[1] * corr[1] + ps[1];
#pragma unroll
        for (int j = 0; j < kD / 8; ++j) {
          oacc[j][0] *= corr[0]; oacc[j][1] *= corr[0];
          oacc[j][2] *= corr[1]; oacc[j][3] *= corr[1];
        }
        // rows at or past `valid` (another sequence's rows, or memory nobody wrote) have probability 0, but
        // 0 x NaN is NaN: their value rows are cleared before the product.  k0 = first of the two rows a
        // fragment register holds (low half k0, high half k0 + 1).
        const int rem = valid - wrow;
        unsigned vm0 = 0xffffffffu, vm1 = 0xffffffffu;
        if (rem < 16) {
          vm0 = (2 * t < rem ? 0x0000ffffu : 0u) | (2 * t + 1 < rem ? 0xffff0000u : 0u);
          vm1 = (2 * t + 8 < rem ? 0x0000ffffu : 0u) | (2 * t + 9 < rem ? 0xffff0000u : 0u);
        }
        unsigned pa[4];
        pa[0] = Mma<T>::pack(sacc[0][0], sacc[0][1]);
        pa[1] = Mma<T>::pack(sacc[0][2], sacc[0][3]);
        pa[2] = Mma<T>::pack(sacc[1][0], sacc[1][1]);
        pa[3] = Mma<T>::pack(sacc[1][2], sacc[1][3]);
#pragma unroll
        for (int jj = 0; jj < kD / 16; ++jj) {
          unsigned r[4];
          ldmatrix_x4_trans(sb + 2 * kBoxBytes + tile_offset(wrow + (mi & 1) * 8 + (lane & 7), 2 * jj + (mi >> 1)), r);
          r[0] &= vm0; r[2] &= vm0;
          r[1] &= vm1; r[3] &= vm1;
          Mma<T>::run(oacc[2 * jj], pa, r[0], r[1]);
          Mma<T>::run(oacc[2 * jj + 1], pa, r[2], r[3]);
        }
      }
      __syncwarp();
      if (lane == 0) mbar::arrive(&sh.empty[st]);             // this warp is through with the stage
    }
    if (failed) {
      m[0] = m[1] = -INFINITY;
      l[0] = l[1] = 0.f;
#pragma unroll
      for (int j = 0; j < kD / 8; ++j) oacc[j][0] = oacc[j][1] = oacc[j][2] = oacc[j][3] = 0.f;
    }

    // merge the four warps (each saw a quarter of every tile)
    consumers_sync();                                        // the merge buffer is free again
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      l[i] += __shfl_xor_sync(0xffffffffu, l[i], 1);
      l[i] += __shfl_xor_sync(0xffffffffu, l[i], 2);
    }
    {
      float *w0 = mo + ((size_t)warp * 16 + g) * kMergeStride, *w1 = w0 + 8 * kMergeStride;
      if (g < P.G) {
#pragma unroll
        for (int j = 0; j < kD / 8; ++j) *reinterpret_cast<float2 *>(w0 + 8 * j + 2 * t) = make_float2(oacc[j][0], oacc[j][1]);
      }
      if (g + 8 < P.G) {
#pragma unroll
        for (int j = 0; j < kD / 8; ++j) *reinterpret_cast<float2 *>(w1 + 8 * j + 2 * t) = make_float2(oacc[j][2], oacc[j][3]);
      }
      if (t == 0) {
        mml[warp * 16 + g] = make_float2(m[0], l[0]);
        mml[warp * 16 + g + 8] = make_float2(m[1], l[1]);
      }
    }
    consumers_sync();
    const int i0 = share_of(line, line_len, nb), i1 = share_of(line + s.tiles - 1, line_len, nb);
    const size_t slot = ((size_t)blk + (size_t)h * P.B + b) * P.G;
    for (int r = warp; r < P.G; r += kWarps) {               // a warp per query head, four channels per lane
      float2 v[kWarps];
      float mm = -INFINITY, ll = 0.f;
#pragma unroll
      for (int w = 0; w < kWarps; ++w) { v[w] = mml[w * 16 + r]; mm = fmaxf(mm, v[w].x); }
      const float msafe = (mm == -INFINITY) ? 0.f : mm;
      float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int w = 0; w < kWarps; ++w) {
        const float f = exp2f(v[w].x - msafe);
        fold(o, *reinterpret_cast<const float4 *>(mo + ((size_t)w * 16 + r) * kMergeStride + 4 * lane), f);
        ll += v[w].y * f;
      }
      if (i0 == i1) {
        store_head(static_cast<T *>(P.out) + ((size_t)b * P.Hq + (size_t)h * P.G + r) * kD + 4 * lane, o, ll);
      } else {
        *reinterpret_cast<float4 *>(P.part_o + (slot + r) * kD + 4 * lane) = o;
        if (lane == 0) P.part_ml[slot + r] = make_float2(mm, ll);
      }
    }
    if (blk == i0 && tid == 0) P.span[(size_t)h * P.B + b] = make_int2(i0, i1);
  }
}

// out[b][h*G + r] = sum over the blocks i0..i1 of their shares, rescaled to the common maximum, divided by the common
// sum.  Shares sit in slot i + (h*B + b) (both only ever advance along the line, so slots do not collide).  One block per
// query head; each warp folds every fourth share, loads ahead of the arithmetic, and the warps' results meet in shared
// memory: two rounds of latency.  Launched early as a programmatic dependent, it is resident when the shares are complete
// (merging in the block that finishes last instead costs an atomic and 3..5 us on one SM: a sixth more per layer of the
// short caches named above).
template <typename T>
__global__ void __launch_bounds__(32 * kFoldWarps)
k_decode_combine(const DecodeParams P) {
  asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
  __shared__ float4 so[kFoldWarps][32];
  __shared__ float2 sml[kFoldWarps];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int b = blockIdx.x / P.Hq, hq = blockIdx.x - b * P.Hq, h = hq / P.G, r = hq - h * P.G;
  asm volatile("griddepcontrol.wait;\n" ::: "memory");
  const int2 span = __ldcg(P.span + (size_t)h * P.B + b);
  if (span.y <= span.x) return;                              // no rows, or finished by its only block
  const size_t slot0 = ((size_t)span.x + (size_t)h * P.B + b) * P.G + r;
  const int cnt = span.y - span.x + 1;
  constexpr int kAhead = 10;
  float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
  float m = -INFINITY, l = 0.f;
  for (int s0 = warp; s0 < cnt; s0 += kFoldWarps * kAhead) {
    float4 v[kAhead];
    float2 ml[kAhead];
#pragma unroll
    for (int a = 0; a < kAhead; ++a) {
      const int i = s0 + a * kFoldWarps < cnt ? s0 + a * kFoldWarps : s0;
      ml[a] = __ldcg(P.part_ml + slot0 + (size_t)i * P.G);
      v[a] = __ldcg(reinterpret_cast<const float4 *>(P.part_o + (slot0 + (size_t)i * P.G) * kD) + lane);
    }
    float mn = m;
#pragma unroll
    for (int a = 0; a < kAhead; ++a) {
      if (s0 + a * kFoldWarps >= cnt) ml[a] = make_float2(-INFINITY, 0.f);
      mn = fmaxf(mn, ml[a].x);
    }
    const float ms = mn == -INFINITY ? 0.f : mn, keep = exp2f(m - ms);
    m = mn;
    l *= keep;
    acc.x *= keep; acc.y *= keep; acc.z *= keep; acc.w *= keep;
#pragma unroll
    for (int a = 0; a < kAhead; ++a) {
      const float f = exp2f(ml[a].x - ms);
      fold(acc, v[a], f);
      l += ml[a].y * f;
    }
  }
  so[warp][lane] = acc;
  if (lane == 0) sml[warp] = make_float2(m, l);
  __syncthreads();
  if (warp != 0) return;
  float mm = -INFINITY, ll = 0.f;
#pragma unroll
  for (int w = 0; w < kFoldWarps; ++w) mm = fmaxf(mm, sml[w].x);
  const float ms = mm == -INFINITY ? 0.f : mm;
  float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
  for (int w = 0; w < kFoldWarps; ++w) {
    const float f = exp2f(sml[w].x - ms);
    fold(o, so[w][lane], f);
    ll += sml[w].y * f;
  }
  store_head(static_cast<T *>(P.out) + ((size_t)b * P.Hq + hq) * kD + 4 * lane, o, ll);
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// Looked up once; a thread that comes while another one looks waits for it (handles of several threads may call at once).
EncodeTiledFn encode_fn() {
  static const EncodeTiledFn fn = [] {
    void *p = nullptr;
    cudaDriverEntryPointQueryResult q;
    return cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
                   q == cudaDriverEntryPointSuccess
               ? reinterpret_cast<EncodeTiledFn>(p)
               : nullptr;
  }();
  return fn;
}

// Tiles of 64 rows x 64 channels of one head, rows 128 bytes wide in shared memory, 128-byte swizzle.
fc_status encode_rows(CUtensorMap *m, CUtensorMapDataType dt, int rank, const void *base, const cuuint64_t *dims,
                      const cuuint64_t *strides_b) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return FC_ERR_CUDA;
  const cuuint32_t box[4] = {64, 1, (cuuint32_t)kTile, 1};
  const cuuint32_t ones[4] = {1, 1, 1, 1};
  const CUresult r = fn(m, dt, (cuuint32_t)rank, const_cast<void *>(base), dims, strides_b, box, ones,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? FC_OK : FC_ERR_INTERNAL;
}

// ring, merge buffer (the warps' outputs, padded), slack to align the ring to 1024 bytes
constexpr size_t kDecodeSmem = (size_t)kStages * kStageBytes + kWarps * 16 * (kMergeStride + 2) * sizeof(float) + 1024;

struct DecodePlan {
  int nb;
  size_t off_ml, off_span, total;
};

fc_status check_decode(const fc_handle *h, const fc_decode_args *a) {
  if (!h || !a || !a->q || !a->cache_k || !a->cache_v || !a->offsets) return FC_ERR_INVALID_ARG;
  if (a->batch < 1 || a->num_heads < 1 || a->num_q_heads < 1 || a->cache_rows < 1 || a->max_rows < 0) return FC_ERR_INVALID_ARG;
  if (a->dtype != FC_F16 && a->dtype != FC_BF16) return FC_ERR_UNSUPPORTED;
  if (a->head_dim != kD) return FC_ERR_UNSUPPORTED;
  if (a->num_q_heads % a->num_heads != 0 || a->num_q_heads / a->num_heads > 16) return FC_ERR_UNSUPPORTED;
  if (a->cache_rows > 0x7fffffffll - 2 * kTile || a->max_rows > 0x7fffffffll - 2 * kTile || a->batch > 65535 ||
      a->num_heads > 65535)
    return FC_ERR_UNSUPPORTED;
  if (((uintptr_t)a->q & 15) || ((uintptr_t)a->cache_k & 15) || ((uintptr_t)a->cache_v & 15)) return FC_ERR_INVALID_ARG;
  const bool tail = a->tail_k || a->tail_v || a->tail_len;
  if (tail) {
    if (!a->tail_k || !a->tail_v || !a->tail_len || a->tail_capacity < 1) return FC_ERR_INVALID_ARG;
    if (((uintptr_t)a->tail_k & 15) || ((uintptr_t)a->tail_v & 15)) return FC_ERR_INVALID_ARG;
  }
  return FC_OK;
}

DecodePlan plan_decode(const fc_handle *h, const fc_decode_args *a) {
  DecodePlan p;
  // one block per SM (the ring takes most of its shared memory), or as many as there can be tiles
  const long long tiles = (long long)a->batch * a->num_heads * ((a->max_rows + kTile - 1) / kTile + (a->tail_k ? 1 : 0));
  p.nb = (int)(tiles < h->num_sms ? (tiles < 1 ? 1 : tiles) : h->num_sms);
  const size_t units = (size_t)a->batch * a->num_heads;
  const size_t slots = (p.nb + units) * (size_t)(a->num_q_heads / a->num_heads);
  p.off_ml = (slots * kD * sizeof(float) + 255) & ~(size_t)255;
  p.off_span = p.off_ml + ((slots * sizeof(float2) + 255) & ~(size_t)255);
  p.total = p.off_span + ((units * sizeof(int2) + 255) & ~(size_t)255);
  return p;
}

template <typename T>
fc_status launch_decode(fc_handle *h, const fc_decode_args *a, const DecodePlan &pl, void *out, char *ws, cudaStream_t st) {
  const CUtensorMapDataType dt = sizeof(T) == 2 && std::is_same<T, __half>::value ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16
                                                                                  : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16;
  DecodeMaps M;
  fc_status s;
  const cuuint64_t row_b = (cuuint64_t)a->num_heads * kD * 2;
  {
    const cuuint64_t dims[3] = {(cuuint64_t)kD, (cuuint64_t)a->num_heads, (cuuint64_t)a->cache_rows};
    const cuuint64_t str[2] = {(cuuint64_t)kD * 2, row_b};
    if ((s = encode_rows(&M.k, dt, 3, a->cache_k, dims, str)) != FC_OK) return s;
    if ((s = encode_rows(&M.v, dt, 3, a->cache_v, dims, str)) != FC_OK) return s;
  }
  if (a->tail_k) {
    const cuuint64_t dims[4] = {(cuuint64_t)kD, (cuuint64_t)a->num_heads, (cuuint64_t)a->tail_capacity, (cuuint64_t)a->batch};
    const cuuint64_t str[3] = {(cuuint64_t)kD * 2, row_b, row_b * (cuuint64_t)a->tail_capacity};
    if ((s = encode_rows(&M.tk, dt, 4, a->tail_k, dims, str)) != FC_OK) return s;
    if ((s = encode_rows(&M.tv, dt, 4, a->tail_v, dims, str)) != FC_OK) return s;
  } else {
    M.tk = M.k;
    M.tv = M.v;
  }
  DecodeParams P;
  P.q = a->q;
  P.out = out;
  P.offsets = reinterpret_cast<const long long *>(a->offsets);
  P.tail_len = a->tail_len;
  P.part_o = reinterpret_cast<float *>(ws);
  P.part_ml = reinterpret_cast<float2 *>(ws + pl.off_ml);
  P.span = reinterpret_cast<int2 *>(ws + pl.off_span);
  P.status = h->status_word;
  P.B = a->batch;
  P.H = a->num_heads;
  P.Hq = a->num_q_heads;
  P.G = a->num_q_heads / a->num_heads;
  P.nb = pl.nb;
  P.cache_rows = (int)a->cache_rows;
  P.cache_k = a->cache_k;
  P.cache_v = a->cache_v;
  P.tail_cap = a->tail_k ? a->tail_capacity : 0;
  P.has_tail = a->tail_k ? 1 : 0;
  P.scale_log2 = (float)(1.4426950408889634 / sqrt((double)kD));
  if (!h->decode_ready) {              // once per handle
    FC_CUDA_TRY(cudaFuncSetAttribute(k_decode<__half>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kDecodeSmem));
    FC_CUDA_TRY(cudaFuncSetAttribute(k_decode<__nv_bfloat16>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kDecodeSmem));
    h->decode_ready = true;
  }
  cudaLaunchConfig_t lc = {};
  lc.gridDim = dim3(pl.nb);
  lc.blockDim = dim3(kThreadsD);
  lc.dynamicSmemBytes = kDecodeSmem;
  lc.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  lc.attrs = at;
  lc.numAttrs = 1;
  if (cudaLaunchKernelEx(&lc, k_decode<T>, P, M) != cudaSuccess) {
    cudaGetLastError();
    return FC_ERR_CUDA;
  }
  if ((s = fc_after_launch(h)) != FC_OK) return s;
  lc.gridDim = dim3((unsigned)(a->batch * a->num_q_heads));
  lc.blockDim = dim3(32 * kFoldWarps);
  lc.dynamicSmemBytes = 0;
  if (cudaLaunchKernelEx(&lc, k_decode_combine<T>, P) != cudaSuccess) {
    cudaGetLastError();
    return FC_ERR_CUDA;
  }
  return fc_after_launch(h);
}

}  // namespace

extern "C" size_t fc_decode_workspace_bytes(const fc_handle *h, const fc_decode_args *a) {
  if (check_decode(h, a) != FC_OK) return 0;
  return plan_decode(h, a).total;
}

extern "C" fc_status fc_decode_attention(fc_handle *h, const fc_decode_args *a, void *out, void *workspace,
                                         size_t workspace_bytes, fc_stream stream) {
  fc_status s = check_decode(h, a);
  if (s != FC_OK) return s;
  if (!out || ((uintptr_t)out & 15)) return FC_ERR_INVALID_ARG;
  const DecodePlan pl = plan_decode(h, a);
  if (!workspace || ((uintptr_t)workspace & 255) || workspace_bytes < pl.total) return FC_ERR_WORKSPACE;
  // always set, not only where it differs: in a thread that has made no CUDA call yet device 0 is current but no context is,
  // and the tensor maps are encoded by the driver, which wants one
  FC_CUDA_TRY(cudaSetDevice(h->device));
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  if ((s = fc_flush_pending(h, st)) != FC_OK) return s;
  if (a->dtype == FC_F16) return launch_decode<__half>(h, a, pl, out, static_cast<char *>(workspace), st);
  return launch_decode<__nv_bfloat16>(h, a, pl, out, static_cast<char *>(workspace), st);
}
