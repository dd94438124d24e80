// Scoring in the kept band: the Base KV of Eq. 9 is a band of low frequencies, so it fits on a grid a few times coarser
// than the tokens, and only that grid is transformed.  With phi a short low-pass kernel (support W grid points), tokens
// t = 0..N-1, grid points x_j = (j + 1/2) N/M - 1/2, j = 0..M-1, both continued evenly about -1/2 and N-1/2 as the
// DCT-II of Eq. 6 does:
//   k_down   y_j = (M/N) sum_t phi((t - x_j) M/N) z_t          a banded matrix times the rows of K and V
//   k_mid    b = C^-1 diag(1 / H(m)^2, m <= omega; 0) C y      M-point DCT-II, the cutoff, inverse; H = spectrum of phi
//   k_up     base_t = sum_j phi((t - x_j) M/N) b_j             the transposed band, then |z_t - base_t|^2 per row
// phi need not be flat in the band (H is divided out exactly) nor short of the theory's length; it has to suppress what
// folds onto the band, which it does to 6e-8 of the band's own gain, i.e. to fp32 rounding.  k_down and k_up are matrix
// products on the 5th-generation tensor cores: 16-bit K and V are exact operands, phi is a sum of three bf16 or fp16 terms
// (24 and 33 bits), b a sum of two fp16 terms scaled per channel (off by at most 2^-23 of the power of two below its largest
// neighbour), every product of at least 2^-24 of the whole is formed, and sums are fp32 (what the tensor cores cut off them is
// dealt with at each kernel).  N is arbitrary.
#pragma once
#include <cuda.h>

#include <type_traits>

#include "fc_common.cuh"
#include "fc_mbar.cuh"

namespace band {

constexpr int kJ = 16;                       // grid points per step of k_down
constexpr int kSlotTok = 32;                 // tokens per ring slot of k_down and per TMA box
constexpr int kRing = 11;                    // ring slots of k_down: a window is at most seven, the rest are on their way
constexpr int kMaxSteps = 12;                // 16-token steps a window of k_down may have
constexpr int kRows = 128;                   // rows (channels of K, then of V) per tile; tokens per step of k_up
constexpr int kBoxBytes = kSlotTok * 128;    // one box: 32 tokens x 64 channels of 2 bytes
constexpr int kMaxQuads = 24;                // grid quads a window of k_up may have
constexpr int kMaxPer = 256;                 // steps a block of k_down or k_up may have
constexpr int kCheb = 28;                    // terms of the expansion of H
constexpr float kUpScale = 1024.f;           // k_up's matrix is stored times this (its low terms stay normal fp16)
constexpr float kDownScaleF16 = 4096.f;      // k_down's fp16 matrix is stored times this
constexpr float kCutOff = 5.9604644775390625e-8f;   // 2^-24 of a sum of k_down's products is put back (see there)

// One sequence's rows in every layer of the launch, as [head][64 channels][token][channel]: a box is 32 tokens of a tile's
// two 64-channel halves where both are of K or both of V (8 KB; a load costs about 80 cycles besides its bytes), else of one.
struct Maps {
  CUtensorMap k[FC_LAYER_CHUNK], v[FC_LAYER_CHUNK];
};

// How one sequence is treated; filled by the host, the same on both sides.
struct Geometry {
  int N, M, W, omega;
  int ks;                                    // 16-token steps per window of k_down
  int nq;                                    // quads per window of k_up (multiple of 8)
  int same;                                  // N/M is 2 or 4: all steps but the first and last few share their matrices
  double beta, fc;                           // phi(u) = 2 fc sinc(2 fc u) exp(beta (sqrt(1 - (2u/W)^2) - 1))
  double cheb[kCheb];                        // H(f) = sum c_i T_i(2 (f/fmax)^2 - 1), f in cycles per grid point
  double fmax;
  double up_ratio, down_ratio;               // M/N and N/M
  __host__ __device__ int down_steps() const { return M / kJ; }
  __host__ __device__ int up_steps() const { return (N + kRows - 1) / kRows; }
};

constexpr int kEdge = 2;                     // steps at either end with matrices of their own
__host__ __device__ inline int down_classes(const Geometry &g) {
  const int n = g.down_steps();
  return g.same && n > 2 * kEdge + 1 ? 2 * kEdge + 1 : n;
}
__host__ __device__ inline int up_classes(const Geometry &g) {
  const int n = g.up_steps();
  return g.same && n > 2 * kEdge + 1 ? 2 * kEdge + 1 : n;
}
// matrix of step b of n, and a step that has matrix c
__host__ __device__ inline int class_of(int b, int n, int classes) {
  return classes == n || b < kEdge ? b : b >= n - kEdge ? b - n + 2 * kEdge + 1 : kEdge;
}
__host__ __device__ inline int step_of(int c, int n, int classes) {
  return classes == n || c <= kEdge ? c : c + n - 2 * kEdge - 1;
}
__host__ __device__ inline long long floor_div(long long a, long long b) { return a >= 0 ? a / b : -((-a + b - 1) / b); }
__host__ __device__ inline long long ceil_div(long long a, long long b) { return -floor_div(-a, b); }

// First token (multiple of 16) and end of the window of step b of k_down: |t - x_j| <= W N / 2M.
__host__ __device__ inline int down_start(const Geometry &g, int b) {
  const long long t = ceil_div((2ll * kJ * b + 1 - g.W) * g.N - g.M, 2ll * g.M);
  return t <= 0 ? 0 : (int)t & ~15;
}
__host__ __device__ inline int down_end(const Geometry &g, int b) {
  const long long t = floor_div((2ll * (kJ * b + kJ - 1) + 1 + g.W) * g.N - g.M, 2ll * g.M) + 1;
  return t > g.N ? g.N : (int)t;
}
// First quad (multiple of 4) and end of the window of step b of k_up.
__host__ __device__ inline int up_quad(const Geometry &g, int b) {
  const long long j = ceil_div((2ll * kRows * b + 1) * g.M - (1ll + g.W) * g.N, 2ll * g.N);
  int q = j <= 0 ? 0 : (int)(j >> 2) & ~3;
  const int last = g.M / 4 - g.nq;
  return q > last ? last : q;
}
__host__ __device__ inline int up_quad_end(const Geometry &g, int b) {
  long long j = floor_div((2ll * (kRows * b + kRows - 1) + 1) * g.M + (g.W - 1ll) * g.N, 2ll * g.N);
  if (j > g.M - 1) j = g.M - 1;
  return (int)(j >> 2) + 1;
}

constexpr int kTerms = 3;                    // 16-bit terms of a matrix entry
__host__ __device__ inline size_t down_image(const Geometry &g) { return (size_t)g.ks * 2 * kTerms * kJ * 16; }
__host__ __device__ inline size_t up_image(const Geometry &g) { return (size_t)g.nq * kTerms * 1024; }

// ---------------------------------------------------------------------------------------------------- tables
__device__ inline double phi(const Geometry &g, double u) {
  if (!(2.0 * fabs(u) <= g.W)) return 0.0;   // most entries, and the images of all but the first and last few steps
  const double s = 2.0 * u / g.W, r = 1.0 - s * s;
  const double w = exp(g.beta * (sqrt(r) - 1.0)), a = 2.0 * g.fc * u;
  return 2.0 * g.fc * w * (fabs(a) < 1e-12 ? 1.0 : sinpi(a) / (3.14159265358979323846 * a));
}
__device__ inline double response(const Geometry &g, double f) {          // H(f) by Clenshaw's recurrence
  const double x = 2.0 * (f / g.fmax) * (f / g.fmax) - 1.0;
  double b1 = 0.0, b2 = 0.0;
  for (int i = kCheb - 1; i >= 1; --i) {
    const double b0 = 2.0 * x * b1 - b2 + g.cheb[i];
    b2 = b1;
    b1 = b0;
  }
  return x * b1 - b2 + g.cheb[0];
}

// One entry of k_down's matrix of step b, whose window starts at `start`: [8 tokens' chunk][term * 16 + j][8 tokens], rows of
// 16 bytes.
template <typename T>
__device__ __forceinline__ void down_entry(const Geometry &g, int cls, int b, int start, int i, T *__restrict__ out) {
  const int e = i & 7, j = (i >> 3) & (kJ - 1), c = i >> 7, t = start + c * 8 + e;
  T *img = out + (size_t)cls * (down_image(g) / 2);
  const double inv = g.up_ratio;
  double v = 0.0;
  if (t < g.N) {
    const double x = (b * kJ + j + 0.5) * g.down_ratio - 0.5;
    v = (phi(g, (t - x) * inv) + phi(g, (-1.0 - t - x) * inv) + phi(g, (2.0 * g.N - 1.0 - t - x) * inv)) * inv;
    if (std::is_same<T, __half>::value) v *= kDownScaleF16;
  }
#pragma unroll
  for (int k = 0; k < kTerms; ++k) {
    const T h = (T)(float)v;
    img[((size_t)c * (kTerms * kJ) + k * kJ + j) * 8 + e] = h;
    v -= (double)(float)h;
  }
}

// One entry of k_up's matrix of step b, whose window starts at quad q0: [term][8 grid values][token][8].  Values are in the order the transform keeps
// them: first (z0, z2) of ascending quads, then (z3, z1) of descending ones.  The first term is a whole number (see k_up).
__device__ __forceinline__ void up_entry(const Geometry &g, int cls, int b, int q0, int i, __half *__restrict__ out) {
  const int nk = 4 * g.nq;
  __half *img = out + (size_t)cls * (up_image(g) / 2);
  const int e = i & 7, r = (i >> 3) & (kRows - 1), c = i >> 10, k = c * 8 + e, t = b * kRows + r;
  const bool second = k >= 2 * g.nq;
  const int kk = second ? k - 2 * g.nq : k;
  const int n = second ? q0 + g.nq - 1 - (kk >> 1) : q0 + (kk >> 1);
  const int j = 4 * n + (second ? ((kk & 1) ? 1 : 3) : 2 * (kk & 1));
  double v = 0.0;
  if (t < g.N) {
    const double x = (t + 0.5) * g.up_ratio - 0.5;
    v = (phi(g, x - j) + phi(g, x + 1.0 + j) + phi(g, x - (2.0 * g.M - 1.0 - j))) * (double)kUpScale;
  }
  double part = rint(v);
#pragma unroll
  for (int k = 0; k < kTerms; ++k) {
    const __half h = __float2half_rn((float)part);
    img[((size_t)(k * (nk / 8) + c) * kRows + r) * 8 + e] = h;
    v -= (double)__half2float(h);
    part = v;
  }
}

// Everything k_mid looks up.  Stage twiddles w_L^(j p), p = 1, 2, 3, 4, 8, 12, for the stages before the last, and for
// every pair of bins (k, Mh - k) the four gains and the two rotations of its residual step (see k_mid).
struct MidTables {
  float4 *gain, *rot;                        // [Mh/2]
  float2 *tw;                                // stage after stage, [6][L / R]
};

// ---------------------------------------------------------------------------------------------------- the tensor cores
__device__ __forceinline__ unsigned smem_addr(const void *p) { return (unsigned)__cvta_generic_to_shared(p); }

// Operand descriptor in two words: start and leading byte offset, stride byte offset and layout (0 = none, 2 = 128-byte
// swizzle), in 16-byte units.  Starts move by adding to the first word.
__host__ __device__ constexpr unsigned operand_lo(unsigned lead) { return (lead >> 4) << 16; }
__host__ __device__ constexpr unsigned operand_hi(unsigned stride, unsigned layout) { return (stride >> 4) | (1u << 14) | (layout << 29); }
// fp32 sums of 16-bit products; A 128 x 16, B 16 x n, B and (unless a_by_rows) A with consecutive depth.
__host__ __device__ constexpr unsigned instruction(bool f16, bool a_by_rows, int n) {
  return (1u << 4) | ((f16 ? 0u : 1u) << 7) | ((f16 ? 0u : 1u) << 10) | ((a_by_rows ? 1u : 0u) << 15) |
         ((unsigned)(n >> 3) << 17) | ((unsigned)(128 >> 4) << 24);
}
// The warp that issues runs as a whole, and one lane of it issues: descriptors are then computed once per warp, in uniform
// registers.  (A single lane in a branch of its own took 115..134 cycles per product, several times what a product takes.)
__device__ __forceinline__ unsigned elect() {
  unsigned e;
  asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}\n" : "=r"(e));
  return e;
}
__device__ __forceinline__ void mma(unsigned lead, unsigned d, unsigned alo, unsigned ahi, unsigned blo, unsigned bhi,
                                    unsigned idesc, unsigned add) {
  asm volatile("{\n .reg .pred p, q;\n .reg .b64 a, b;\n setp.ne.u32 q, %0, 0;\n setp.ne.u32 p, %7, 0;\n"
               " mov.b64 a, {%2, %3};\n mov.b64 b, {%4, %5};\n"
               " @q tcgen05.mma.cta_group::1.kind::f16 [%1], a, b, %6, p;\n}\n"
               ::"r"(lead), "r"(d), "r"(alo), "r"(ahi), "r"(blo), "r"(bhi), "r"(idesc), "r"(add) : "memory");
}
__device__ __forceinline__ void commit(unsigned lead, unsigned long long *bar) {  // arrives once all products so far are done
  asm volatile("{\n .reg .pred q;\n setp.ne.u32 q, %0, 0;\n"
               " @q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%1];\n}\n"
               ::"r"(lead), "r"(smem_addr(bar)) : "memory");
}
__device__ __forceinline__ void tmem_alloc(unsigned *slot, unsigned cols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_addr(slot)), "r"(cols) : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
}
__device__ __forceinline__ void tmem_free(unsigned base, unsigned cols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(base), "r"(cols) : "memory");
}
__device__ __forceinline__ void before_sync() { asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory"); }
__device__ __forceinline__ void after_sync() { asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory"); }
// The wait names the registers it is for, so that nothing that uses them is moved in front of it.
__device__ __forceinline__ void tmem_wait(float (&v)[16]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;\n"
               : "+f"(v[0]), "+f"(v[1]), "+f"(v[2]), "+f"(v[3]), "+f"(v[4]), "+f"(v[5]), "+f"(v[6]), "+f"(v[7]),
                 "+f"(v[8]), "+f"(v[9]), "+f"(v[10]), "+f"(v[11]), "+f"(v[12]), "+f"(v[13]), "+f"(v[14]), "+f"(v[15])
               :: "memory");
}
// this lane's row, 16 columns
__device__ __forceinline__ void tmem_ld16(unsigned addr, float (&v)[16]) {
  unsigned *r = reinterpret_cast<unsigned *>(v);
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                 "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
               : "r"(addr));
}
__device__ __forceinline__ void load_box(void *dst, const CUtensorMap *map, int c, int h, int t, unsigned long long *bar) {
  asm volatile("cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];\n"
               ::"r"(smem_addr(dst)), "l"(reinterpret_cast<unsigned long long>(map)), "r"(c), "r"(h), "r"(t),
                 "r"(smem_addr(bar)) : "memory");
}
__device__ __forceinline__ void load_rows_box(void *dst, const CUtensorMap *map, int half, int head, int t, unsigned long long *bar) {
  asm volatile("cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];\n"
               ::"r"(smem_addr(dst)), "l"(reinterpret_cast<unsigned long long>(map)), "r"(0), "r"(t), "r"(half), "r"(head),
                 "r"(smem_addr(bar)) : "memory");
}
// 32 tokens from t of tile `tile` (rows 128 tile .. of K's channels and then V's); the second half `second` bytes on
__device__ __forceinline__ void load_tile(unsigned char *dst, unsigned second, const Maps &maps, int layer, int d64, int tile,
                                          int head, int t, unsigned long long *bar) {
  const int h = 2 * tile;
  if ((d64 & 1) == 0) {
    load_rows_box(dst, h >= d64 ? &maps.v[layer] : &maps.k[layer], h >= d64 ? h - d64 : h, head, t, bar);
  } else {
    for (int i = 0; i < 2; ++i)
      load_rows_box(dst + i * second, h + i >= d64 ? &maps.v[layer] : &maps.k[layer], h + i >= d64 ? h + i - d64 : h + i, head, t, bar);
  }
}
__device__ __forceinline__ void load_bytes(void *dst, const void *src, unsigned bytes, unsigned long long *bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n"
               ::"r"(smem_addr(dst)), "l"(__cvta_generic_to_global(src)), "r"(bytes), "r"(smem_addr(bar)) : "memory");
}

// 32 aligned bytes: a whole sector per lane where the lanes' rows are far apart
__device__ __forceinline__ void store8(float *p, float a, float b, float c, float d, float e, float f, float g, float h) {
  asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};\n"
               ::"l"(p), "f"(a), "f"(b), "f"(c), "f"(d), "f"(e), "f"(f), "f"(g), "f"(h) : "memory");
}

// ---------------------------------------------------------------------------------------------------- k_down
struct DownParams {
  const void *table;
  float *y;                                  // [unit of the launch][row][M]: (z0, z2) of quads ascending, (z3, z1) descending
  int *status;
  int H, d, u0;                              // heads, channels per head, first unit (layer * H + head) of the launch
  int per;                                   // steps per block
};
constexpr int kStepBars = 16;                // more than the steps whose windows fit the ring
struct DownShared {
  unsigned long long full[kRing], step[kStepBars], tfull[2], aempty[2];
  unsigned tmem;
  int start[kMaxPer + 1];                    // of the block's steps and the one after
};
// Loads; a warp per tile that issues products (one warp spent as long between its steps, in waits, as in them, 2100 cycles
// per step of two tiles); four warps that take the sums out.
constexpr int kDownThreads = 224;
constexpr unsigned kDownCols = 512;
constexpr unsigned kDownTable = kMaxSteps * 2 * 48 * 16;
constexpr size_t kDownSmem = 1024 + (size_t)kRing * 4 * kBoxBytes + 2 * (size_t)kDownTable;

// What bounds it: HBM and the products alike.  A step is 64 tokens of K and V at 4 tokens per grid point, ten products of
// 128 x 48 x 16 per tile (44 cycles each: the left operand's 4 KB at 128 bytes a cycle, a quarter cycle per column), 900
// cycles beside 32 KB of rows.  The rows are the left operand, so that a lane of the sums is a channel and writes whole
// sectors of its row of the grid; the three terms of the matrix are columns of one product, and sums of a window go to two
// accumulators, from the window's ends to its middle, because the tensor cores cut off, towards zero, what does not fit the
// 24 bits of a sum: half a unit of the last place at every addition of a product of depth 16.  That mean is put back, 2^-24
// of the sum for its last, largest additions; a model of these sums has 0.50e-6 of a score (rms, 10 % outlier rows) with one
// accumulator, 0.31e-6 with two, 0.11e-6 with what was cut off put back.  16 heads of 32768 tokens: 233 us with products
// issued by one lane, 75 us now (417 MB, 5.6 TB/s).
// One block: `per` steps of 16 grid points for up to two tiles (256 rows) of one unit.  grid (ranges, tile pairs, units).
template <typename T>
__global__ void __launch_bounds__(kDownThreads, 1) k_down(const __grid_constant__ Maps maps, const __grid_constant__ Geometry g,
                                                       const DownParams P) {
  constexpr int NR = kTerms * kJ;            // columns of one sum
  constexpr bool kF16 = std::is_same<T, __half>::value;
  extern __shared__ unsigned char raw[];
  unsigned char *smem = reinterpret_cast<unsigned char *>(((uintptr_t)raw + 1023) & ~(uintptr_t)1023);
  unsigned char *tab = smem + (size_t)kRing * 4 * kBoxBytes;
  __shared__ DownShared sh;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int unit = P.u0 + blockIdx.z, layer = unit / P.H, head = unit - layer * P.H;
  const int tiles = P.d / 64, tile0 = 2 * blockIdx.y, nt = tiles - tile0 < 2 ? 1 : 2;
  const int n = g.down_steps(), classes = down_classes(g);
  const int b0 = blockIdx.x * P.per, b1 = b0 + P.per < n ? b0 + P.per : n;
  const unsigned img = (unsigned)down_image(g);
  unsigned char *tab1 = tab + kDownTable;

  if (tid == 0) {
    for (int i = 0; i < kRing; ++i) mbar::init(&sh.full[i], 1u);
    for (int i = 0; i < kStepBars; ++i) mbar::init(&sh.step[i], (unsigned)nt);
    for (int i = 0; i < 2; ++i) { mbar::init(&sh.tfull[i], 1u); mbar::init(&sh.aempty[i], 4u); }
    mbar::init_done();
  }
  if (warp == 1) tmem_alloc(&sh.tmem, kDownCols);
  for (int i = tid; i <= b1 - b0; i += kDownThreads) sh.start[i] = down_start(g, b0 + i);
  before_sync();
  __syncthreads();
  after_sync();
  const unsigned tmem = sh.tmem;
  asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
  if (b0 < b1) {
    const int q0 = sh.start[0] / kSlotTok;                 // ring slots are counted from here
    if (warp == 0) {
      if (lane == 0) {
        bool ok = true;
        int q = q0, ntab = 0, cls = -1, past = 0, since[2] = {0, 0};
        // the products of every step before the `n`-th of this block are done (a step's barrier is waited for in turn, so
        // none is met a phase late)
        auto done_before = [&](int upto) {
          for (; past < upto && ok; ++past) ok = mbar::wait(&sh.step[past % kStepBars], (unsigned)(past / kStepBars) & 1u);
          return ok;
        };
        int free_to = b0;                                        // first step whose window starts past the slot wanted
        for (int b = b0; b < b1 && ok; ++b) {
          const int c = class_of(b, n, classes);
          if (c != cls) {
            cls = c;
            const int s = ntab & 1;
            since[s] = b - b0;                                   // the other buffer's matrix was used until here
            if (ntab >= 2 && !done_before(since[s ^ 1])) break;
            mbar::expect_tx(&sh.tfull[s], img);
            load_bytes(s ? tab1 : tab, static_cast<const unsigned char *>(P.table) + (size_t)c * img, img, &sh.tfull[s]);
            ++ntab;
          }
          // run ahead of this step's window as far as the ring allows without waiting for steps not yet issued
          const int last = (sh.start[b - b0] + 16 * g.ks - 1) / kSlotTok;
          for (; q <= last; ++q) {
            const int i = q - q0, s = i % kRing;
            if (i >= kRing) {
              while (free_to < b && sh.start[free_to - b0] / kSlotTok <= q - kRing) ++free_to;
              if (!done_before(free_to - b0)) break;
            }
            mbar::expect_tx(&sh.full[s], (unsigned)(2 * nt * kBoxBytes));
            for (int t = 0; t < nt; ++t)
              load_tile(smem + (size_t)(s * 4 + 2 * t) * kBoxBytes, kBoxBytes, maps, layer, tiles, tile0 + t, head, q * kSlotTok,
                        &sh.full[s]);
          }
        }
        // no load may be in flight when the block ends
        const int issued = q - q0;
        for (int i = issued > kRing ? issued - kRing : 0; i < issued; ++i)
          ok &= mbar::wait(&sh.full[i % kRing], (unsigned)(i / kRing) & 1u);
        for (int i = ntab > 2 ? ntab - 2 : 0; i < ntab; ++i) ok &= mbar::wait(&sh.tfull[i & 1], (unsigned)(i / 2) & 1u);
        if (!ok) atomicOr(P.status, FC_DEV_FLAG_TIMEOUT);
      }
    } else if (warp <= 2) {
      constexpr unsigned idesc = instruction(kF16, true, NR), ahi = operand_hi(1024, 2), bhi = operand_hi(128, 0);
      constexpr int kGroups = 2 * kRing;                         // 16-token groups in the ring
      const unsigned lead = elect();
      const int tile = warp - 1;
      const unsigned abase = ((smem_addr(smem) >> 4) | operand_lo(kBoxBytes)) + (unsigned)tile * (2 * kBoxBytes / 16), bbase = (smem_addr(tab) >> 4) | operand_lo(NR * 16);
      bool ok = true;
      int have = q0, ntab = 0, cls = -1, it = 0;
      for (int b = tile < nt ? b0 : b1; b < b1 && ok; ++b) {
        const int start = __shfl_sync(0xffffffffu, sh.start[b - b0], 0), buf = it & 1;
        const int last = (start + 16 * g.ks - 1) / kSlotTok, c = class_of(b, n, classes);
        if (c != cls) {
          cls = c;
          if (!mbar::wait_warp(&sh.tfull[ntab & 1], (unsigned)(ntab / 2) & 1u)) { ok = false; break; }
          ++ntab;
        }
        if (it >= 2 && !mbar::wait_warp(&sh.aempty[buf], (unsigned)(it / 2 - 1) & 1u)) { ok = false; break; }
        for (; have <= last && ok; ++have)
          ok = mbar::wait_warp(&sh.full[(have - q0) % kRing], (unsigned)((have - q0) / kRing) & 1u);
        if (!ok) break;
        after_sync();
        const unsigned bl = bbase + (((ntab - 1) & 1) ? kDownTable / 16 : 0u);
        const int pos = (start / 16 - 2 * q0) % kGroups;
        // steps from the window's ends to its middle, in two sums by turns: small terms first, few roundings of large sums
        for (int i = 0; i < g.ks; ++i) {
          const int k = (i & 1) ? g.ks - 1 - i / 2 : i / 2;
          int at = pos + k;
          if (at >= kGroups) at -= kGroups;
          const unsigned al = abase + (unsigned)(at >> 1) * (4 * kBoxBytes / 16) + (unsigned)(at & 1) * 128u;
          mma(lead, tmem + (unsigned)(((buf * 2 + tile) * 2 + ((i >> 1) & 1)) * NR), al, ahi, bl + (unsigned)k * (2 * NR), bhi, idesc,
              i >= 4 || (i & 1) ? 1u : 0u);
        }
        commit(lead, &sh.step[it % kStepBars]);
        ++it;
      }
      // nothing is left running when the block ends
      if (it > 0) ok &= mbar::wait_warp(&sh.step[(it - 1) % kStepBars], (unsigned)((it - 1) / kStepBars) & 1u);
      if (!ok && lane == 0) atomicOr(P.status, FC_DEV_FLAG_TIMEOUT);
    } else {
      const int quad = warp & 3, row = quad * 32 + lane, Mh = g.M / 2;
      const float scale = kF16 ? 1.f / kDownScaleF16 : 1.f;
      for (int b = b0; b < b1; ++b) {
        const int it = b - b0, buf = it & 1;
        if (!mbar::wait_warp(&sh.step[it % kStepBars], (unsigned)(it / kStepBars) & 1u)) {
          if (lane == 0) atomicOr(P.status, FC_DEV_FLAG_TIMEOUT);
          break;
        }
        after_sync();
        for (int t = 0; t < nt; ++t) {
          const unsigned at = tmem + ((unsigned)quad << 21) + (unsigned)((buf * 2 + t) * 2 * NR);
          float v[2 * kTerms][kJ];
#pragma unroll
          for (int k = 0; k < 2 * kTerms; ++k) tmem_ld16(at + k * kJ, v[k]);
#pragma unroll
          for (int k = 0; k < 2 * kTerms; ++k) tmem_wait(v[k]);
          if (t + 1 == nt) {                                      // the sums have been taken out
            before_sync();
            __syncwarp();
            if (lane == 0) mbar::arrive(&sh.aempty[buf]);
          }
          float r[kJ];
#pragma unroll
          for (int j = 0; j < kJ; ++j) {                          // low terms first, and with them what was cut off
            const float top = v[0][j] + v[kTerms][j];
            r[j] = v[2][j] + v[kTerms + 2][j];
            r[j] += v[1][j] + v[kTerms + 1][j];
            r[j] = top + fmaf(top, kCutOff, r[j]);
            if (kF16) r[j] *= scale;
          }
          float *yr = P.y + ((size_t)blockIdx.z * 2 * P.d + (tile0 + t) * kRows + row) * g.M;
          store8(yr + 8 * b, r[0], r[2], r[4], r[6], r[8], r[10], r[12], r[14]);
          store8(yr + 2 * (Mh - 4 - 4 * b), r[15], r[13], r[11], r[9], r[7], r[5], r[3], r[1]);
        }
      }
    }
  }
  before_sync();
  __syncthreads();
  if (warp == 1) tmem_free(tmem, kDownCols);
}

// ---------------------------------------------------------------------------------------------------- k_mid
// Two real rows of M grid values each as a complex transform of Mh = M/2 points, Mh = R1*R2*R3*R4, 16 points of both rows per
// thread.
template <int R1_, int R2_, int R3_, int R4_>
struct MidShape {
  static constexpr int R1 = R1_, R2 = R2_, R3 = R3_, R4 = R4_, Mh = R1 * R2 * R3 * R4, T = Mh / 16;
  static constexpr int RL = R4 > 1 ? R4 : R3 > 1 ? R3 : R2;         // radix of the last stage
  static constexpr int S = Mh / RL;                                  // bins of the stages before it
  static constexpr int PAIRS = T >= 128 ? 1 : 128 / T, NT = T * PAIRS;
  static constexpr int LEN = Mh + Mh / RL;                           // one entry of padding per RL: conflict-free in every stage
  static constexpr size_t smem = (size_t)PAIRS * LEN * sizeof(float4);
  __host__ __device__ static constexpr int sub_of(int k0) {          // position (in units of RL) of the bins k0 + S*i
    int pos = 0, rem = S, k = k0;
    const int r[3] = {R1, R4 > 1 || R3 > 1 ? R2 : 1, R4 > 1 ? R3 : 1};
#pragma unroll
    for (int s = 0; s < 3; ++s)
      if (r[s] > 1) { rem /= r[s]; pos += (k % r[s]) * rem; k /= r[s]; }
    return pos;
  }
  static constexpr int tw_len = 6 * (Mh / R1 + (R3 > 1 ? R3 * R4 : 0) + (R4 > 1 ? R4 : 0));
};

struct MidRadices {                          // of the stages (1 where there is none) and of the last one
  int r[3], last;
};
// Entry i of k_mid's tables: pair i of bins, and a stage twiddle.
__device__ __forceinline__ void mid_entry(const Geometry &g, const MidRadices &m, int i, const MidTables &t) {
  const int Mh = g.M / 2, RL = m.last, S = Mh / RL;
  if (i < Mh / 2) {
    // bins k0 + S*l and Mh minus that; the first RL pairs are the blocks that are their own partners
    const int k0 = i >= RL ? i / RL : i < RL / 2 ? 0 : S / 2;
    const int l = i >= RL ? i % RL : i % (RL / 2), k = k0 + S * l;
    auto gain = [&](int q) {
      if (q > g.omega || q >= g.M) return 0.0;
      const double h = response(g, (double)q / (2.0 * g.M));
      return 1.0 / (h * h);
    };
    const double s = 1.0 / (4.0 * Mh);
    if (k == 0) {
      t.gain[i] = make_float4((float)(gain(0) / (2.0 * Mh)), (float)(gain(Mh) / (2.0 * Mh)), (float)(gain(Mh / 2) * s),
                              (float)(gain(Mh + Mh / 2) * s));
    } else {
      t.gain[i] = make_float4((float)(gain(k) * s), (float)(gain(g.M - k) * s), (float)(gain(Mh - k) * (0.5 * s)),
                              (float)(gain(Mh + k) * (0.5 * s)));
    }
    double c, sn, c4, s4;
    const int kr = k == 0 ? Mh / 2 : k;                               // entry 0 serves the bin Mh/2
    sincospi((double)kr / (2.0 * g.M), &sn, &c);
    sincospi(2.0 * kr / (double)g.M, &s4, &c4);
    t.rot[i] = make_float4((float)c, (float)sn, (float)c4, (float)s4);
  }
  int base = 0, L = Mh;
#pragma unroll
  for (int s = 0; s < 3; ++s) {
    if (m.r[s] == 1) continue;
    const int sub = L / m.r[s], e = i - base;
    if (e >= 0 && e < 6 * sub) {
      const int w = e / sub;                                          // powers 1, 2, 3, 4, 8, 12
      double c, sn;
      sincospi(2.0 * (double)((w < 4 ? w + 1 : w == 4 ? 8 : 12) * (e % sub)) / (double)L, &sn, &c);
      t.tw[base + e] = make_float2((float)c, (float)-sn);
    }
    base += 6 * sub;
    L = sub;
  }
}

// All tables of a sequence in one launch, 256 entries at a time: `down` blocks, then `up` blocks, then those of mid_entry.  A
// block stays with one matrix for several rounds, since finding a window takes 64-bit divisions.
constexpr int kDownRounds = 2, kUpRounds = 4;
__host__ __device__ inline int down_table_blocks(const Geometry &g) { return (g.ks + kDownRounds - 1) / kDownRounds; }   // per matrix
__host__ __device__ inline int up_table_blocks(const Geometry &g) { return g.nq * 2 / kUpRounds; }
template <typename T>
__global__ void __launch_bounds__(256) k_band_tables(const __grid_constant__ Geometry g, const MidRadices m, T *down, __half *up,
                                                     MidTables mid, int down_blocks, int up_blocks) {
  int b = blockIdx.x;
  if (b < down_blocks) {                                              // a matrix: ks rounds of 16 * 16 entries
    const int per = down_table_blocks(g), cls = b / per, step = step_of(cls, g.down_steps(), down_classes(g));
    const int start = down_start(g, step), end = (b % per + 1) * kDownRounds;
    for (int k = end - kDownRounds; k < end && k < g.ks; ++k) down_entry<T>(g, cls, step, start, k * 256 + threadIdx.x, down);
    return;
  }
  b -= down_blocks;
  if (b < up_blocks) {                                                // 2 nq rounds
    const int per = up_table_blocks(g), cls = b / per, step = step_of(cls, g.up_steps(), up_classes(g)), q0 = up_quad(g, step);
#pragma unroll 1
    for (int k = 0; k < kUpRounds; ++k) up_entry(g, cls, step, q0, ((b % per) * kUpRounds + k) * 256 + threadIdx.x, up);
    return;
  }
  mid_entry(g, m, (b - up_blocks) * 256 + threadIdx.x, mid);
}

// Both rows' values side by side: every operation is a packed one, at half the issue slots.
struct C2 {
  float2 re, im;
};
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.f, -1.f), a); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 neg2(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 both(float a) { return make_float2(a, a); }
__device__ __forceinline__ C2 operator+(const C2 &a, const C2 &b) { return {add2(a.re, b.re), add2(a.im, b.im)}; }
__device__ __forceinline__ C2 operator-(const C2 &a, const C2 &b) { return {sub2(a.re, b.re), sub2(a.im, b.im)}; }
// a * w and a * conj(w), w the same for both rows or not
__device__ __forceinline__ C2 times(const C2 &a, const C2 &w) {
  return {fma2(a.re, w.re, neg2(mul2(a.im, w.im))), fma2(a.re, w.im, mul2(a.im, w.re))};
}
__device__ __forceinline__ C2 times_conj(const C2 &a, const C2 &w) {
  return {fma2(a.re, w.re, mul2(a.im, w.im)), fma2(a.im, w.re, neg2(mul2(a.re, w.im)))};
}
// a + DIR*j*b and a - DIR*j*b
template <int DIR>
__device__ __forceinline__ void sums_j(const C2 &a, const C2 &b, C2 &plus, C2 &minus) {
  const C2 p = {sub2(a.re, b.im), add2(a.im, b.re)}, m = {add2(a.re, b.im), sub2(a.im, b.re)};
  plus = DIR > 0 ? p : m;
  minus = DIR > 0 ? m : p;
}
// e + w*o and e - w*o, w = c + DIR*j*s, the rotation folded into the sums: w = c (1 + DIR*j*s/c), or s (c/s + DIR*j)
template <int DIR>
__device__ __forceinline__ void sums_w(const C2 &e, const C2 &o, float c, float s, C2 &plus, C2 &minus) {
  const bool by_c = fabsf(c) >= fabsf(s);
  const float f = by_c ? c : s, t = by_c ? DIR * s / c : DIR * c / s;
  // by_c: r = o (1 + j t);  else r = DIR * j o (1 - j t)
  const C2 r = by_c ? C2{fma2(o.im, both(-t), o.re), fma2(o.re, both(t), o.im)}
                    : DIR > 0 ? C2{fma2(o.re, both(t), neg2(o.im)), fma2(o.im, both(t), o.re)}
                              : C2{fma2(o.re, both(-t), o.im), fma2(o.im, both(-t), neg2(o.re))};
  plus = {fma2(r.re, both(f), e.re), fma2(r.im, both(f), e.im)};
  minus = {fma2(r.re, both(-f), e.re), fma2(r.im, both(-f), e.im)};
}
template <int DIR>
__device__ __forceinline__ void dft4p(C2 &x0, C2 &x1, C2 &x2, C2 &x3) {
  const C2 a = x0 + x2, b = x0 - x2, c = x1 + x3, d = x1 - x3;
  x0 = a + c;
  x2 = a - c;
  sums_j<DIR>(b, d, x1, x3);
}
template <int DIR>
__device__ __forceinline__ void dft8p(C2 (&x)[8]) {
  const float h = 0.70710678118654752440f;
  dft4p<DIR>(x[0], x[2], x[4], x[6]);
  dft4p<DIR>(x[1], x[3], x[5], x[7]);
  const C2 e0 = x[0], e1 = x[2], e2 = x[4], e3 = x[6], o0 = x[1], o1 = x[3], o2 = x[5], o3 = x[7];
  x[0] = e0 + o0;
  x[4] = e0 - o0;
  sums_w<DIR>(e1, o1, h, h, x[1], x[5]);
  sums_j<DIR>(e2, o2, x[2], x[6]);
  sums_w<DIR>(e3, o3, -h, h, x[3], x[7]);
}
template <int R, int DIR>
__device__ __forceinline__ void dftp(C2 (&x)[R]) {
  if constexpr (R == 8) {
    dft8p<DIR>(x);
  } else {
    static_assert(R == 16, "radix 8 or 16");
    const float c1 = 0.92387953251128675613f, s1 = 0.38268343236508977173f, h = 0.70710678118654752440f;
    C2 e[8], o[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) { e[i] = x[2 * i]; o[i] = x[2 * i + 1]; }
    dft8p<DIR>(e);
    dft8p<DIR>(o);
    x[0] = e[0] + o[0];
    x[8] = e[0] - o[0];
    sums_w<DIR>(e[1], o[1], c1, s1, x[1], x[9]);
    sums_w<DIR>(e[2], o[2], h, h, x[2], x[10]);
    sums_w<DIR>(e[3], o[3], s1, c1, x[3], x[11]);
    sums_j<DIR>(e[4], o[4], x[4], x[12]);
    sums_w<DIR>(e[5], o[5], -s1, c1, x[5], x[13]);
    sums_w<DIR>(e[6], o[6], -h, h, x[6], x[14]);
    sums_w<DIR>(e[7], o[7], -c1, s1, x[7], x[15]);
  }
}

// x[p] *= w^p (conjugated for the way back), w^1, 2, 3, 4, 8, 12 from the table: at most two factors each
template <int R, bool CONJ>
__device__ __forceinline__ void turn(C2 (&x)[R], const float2 *__restrict__ tw, int sub, int j) {
  C2 c[4];
#pragma unroll
  for (int p = 1; p < 4; ++p) {
    const float2 w = __ldg(tw + (p - 1) * sub + j);
    c[p] = {both(w.x), both(w.y)};
    x[p] = CONJ ? times_conj(x[p], c[p]) : times(x[p], c[p]);
  }
#pragma unroll
  for (int a = 1; a < R / 4; ++a) {
    const float2 w = __ldg(tw + (2 + a) * sub + j);
    const C2 b = {both(w.x), both(w.y)};
    x[4 * a] = CONJ ? times_conj(x[4 * a], b) : times(x[4 * a], b);
#pragma unroll
    for (int p = 1; p < 4; ++p) {
      const C2 bc = times(b, c[p]);
      x[4 * a + p] = CONJ ? times_conj(x[4 * a + p], bc) : times(x[4 * a + p], bc);
    }
  }
}

// The largest of G adjacent lanes' values, none of them negative (a NaN counts as large)
template <int G>
__device__ __forceinline__ unsigned group_max(float v) {
  unsigned u = __float_as_uint(v);
  if constexpr (G == 32) {
    u = __reduce_max_sync(0xffffffffu, u);
  } else {
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) {
      const unsigned w = __shfl_xor_sync(0xffffffffu, u, o);
      u = u > w ? u : w;
    }
  }
  return u;
}
__device__ __forceinline__ float unit_rounder(unsigned largest) { return __uint_as_float((largest & 0x7f800000u) + 0x06c00000u); }

struct MidParams {
  float *y;                                  // [row][M]; in the same place afterwards the two terms, [row][term][M]
  float *inv;                                // [row]: minus what a stored value has to be multiplied with
  MidTables t;
};

// What bounds it: shared memory (57 % of its wavefronts), the FMA pipe (half) and issue slots (42 %) at 16 warps per SM, none
// of them alone.  A row is transformed as half as many complex points, two rows per thread in packed arithmetic, which
// shares the twiddles, the gains and every address: 50 M instructions for 16 heads of 32768 tokens where one row per thread
// took 83 M; 108 us (134 us with the values stored in 16-byte pieces; one row per thread at 64 registers and 32 warps takes
// 103 us alone, but whole passes beside the other stream 1..5 % longer).
template <class S>
__global__ void __launch_bounds__(S::NT, S::NT <= 512 ? 512 / S::NT : 1) k_mid(const MidParams P) {
  constexpr int Mh = S::Mh, T = S::T, RL = S::RL;
  extern __shared__ float4 X0[];
  __shared__ float red[2][S::NT / 32];
  const int tid = threadIdx.x, t = tid % T, rl = tid / T;
  float4 *X = X0 + rl * S::LEN;
  const size_t row = 2 * ((size_t)blockIdx.x * S::PAIRS + rl);
  auto pad = [](int pos) { return pos + pos / RL; };
  auto get = [&](int pos) {
    const float4 v = X[pad(pos)];
    return C2{make_float2(v.x, v.y), make_float2(v.z, v.w)};
  };
  auto put = [&](int pos, const C2 &v) { X[pad(pos)] = make_float4(v.re.x, v.re.y, v.im.x, v.im.y); };
  const float2 *src = reinterpret_cast<const float2 *>(P.y) + row * Mh;
  constexpr int T2 = 6 * (Mh / S::R1), T3 = T2 + 6 * (Mh / S::R1 / S::R2);

  asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
  asm volatile("griddepcontrol.wait;\n" ::: "memory");
  // one stage on the points block*L + j + sub*p
  auto forward = [&](auto radix, int L, const float2 *tw, bool first, bool last) {
    constexpr int R = decltype(radix)::value;
    const int sub = L / R;
#pragma unroll
    for (int u = 0; u < 16 / R; ++u) {
      const int i = t + T * u, blk = i / sub, j = i - blk * sub, at = blk * L + j;
      C2 x[R];
#pragma unroll
      for (int p = 0; p < R; ++p) {
        if (first) {
          const float2 a = __ldcg(src + at + sub * p), b = __ldcg(src + Mh + at + sub * p);
          x[p] = {make_float2(a.x, b.x), make_float2(a.y, b.y)};
        } else {
          x[p] = get(at + sub * p);
        }
      }
      dftp<R, -1>(x);
      if (!last) turn<R, false>(x, tw, sub, j);
#pragma unroll
      for (int p = 0; p < R; ++p) put(at + sub * p, x[p]);
    }
    __syncthreads();
  };
  forward(std::integral_constant<int, S::R1>{}, Mh, P.t.tw, true, false);
  forward(std::integral_constant<int, S::R2>{}, Mh / S::R1, P.t.tw + T2, false, S::R3 == 1);
  if constexpr (S::R3 > 1) forward(std::integral_constant<int, S::R3>{}, Mh / S::R1 / S::R2, P.t.tw + T3, false, S::R4 == 1);
  if constexpr (S::R4 > 1) forward(std::integral_constant<int, S::R4>{}, S::R4, nullptr, false, true);

  // Bins in pairs.  W[k], W[M/2 - k] of the real row come from Z[k], Z[Mh - k]; C[k] and C[M - k] are the real and
  // (negated) imaginary part of e^(-j pi k / 2M) W[k], so the gains act on real and imaginary parts in that frame.
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    const int i = t + T * u;
    const int k0 = i >= RL ? i / RL : i < RL / 2 ? 0 : S::S / 2;
    const int l = i >= RL ? i % RL : i % (RL / 2);
    const int pa = S::sub_of(k0) * RL + l;
    const int pb = i == 0 ? RL / 2 : k0 == 0 ? RL - l : S::sub_of(S::S - k0) * RL + RL - 1 - l;
    C2 a = get(pa), b = get(pb);
    float4 gn = __ldg(P.t.gain + i);
    const float4 rt = __ldg(P.t.rot + i);
    if (i == 0) {                            // bins 0 and, by itself, Mh/2
      const float2 w0 = mul2(add2(a.re, a.im), both(gn.x)), wh = mul2(sub2(a.re, a.im), both(gn.y));
      put(pa, {add2(w0, wh), sub2(w0, wh)});
      a = b;
      gn = make_float4(gn.z, gn.w, 0.5f * gn.z, 0.5f * gn.w);
    }
    const C2 f = {both(rt.x), both(rt.y)}, e = {both(rt.z), both(rt.w)};     // e^(j pi k/2M), e^(2 pi j k/M)
    const C2 s = times_conj(C2{add2(a.re, b.re), sub2(a.im, b.im)}, f);
    const C2 r = times_conj(times_conj(C2{sub2(a.re, b.re), add2(a.im, b.im)}, f), e);
    const C2 p = {mul2(add2(s.re, r.im), both(gn.x)), mul2(sub2(s.im, r.re), both(gn.y))};          // r * -j
    const C2 q = {sub2(s.re, r.im), add2(s.im, r.re)};
    const float2 uu = mul2(sub2(q.re, q.im), both(gn.z)), vv = mul2(add2(q.re, q.im), both(gn.w));
    const C2 q2 = {add2(uu, vv), sub2(vv, uu)};
    const C2 gs = p + q2, gd = times(p - q2, e);
    const C2 z = times(C2{sub2(gs.re, gd.im), add2(gs.im, gd.re)}, f), y = times(C2{add2(gs.re, gd.im), sub2(gs.im, gd.re)}, f);
    if (i != 0) put(pa, z);
    put(pb, i == 0 ? z : C2{y.re, neg2(y.im)});
  }
  __syncthreads();

  auto back = [&](auto radix, int L, const float2 *tw, bool last) {
    constexpr int R = decltype(radix)::value;
    const int sub = L / R;
#pragma unroll
    for (int u = 0; u < 16 / R; ++u) {
      const int i = t + T * u, blk = i / sub, j = i - blk * sub, at = blk * L + j;
      C2 x[R];
#pragma unroll
      for (int p = 0; p < R; ++p) x[p] = get(at + sub * p);
      if (!last) turn<R, true>(x, tw, sub, j);
      dftp<R, +1>(x);
#pragma unroll
      for (int p = 0; p < R; ++p) put(at + sub * p, x[p]);
    }
    __syncthreads();
  };
  if constexpr (S::R4 > 1) back(std::integral_constant<int, S::R4>{}, S::R4, nullptr, true);
  if constexpr (S::R3 > 1) back(std::integral_constant<int, S::R3>{}, Mh / S::R1 / S::R2, P.t.tw + T3, S::R4 == 1);
  back(std::integral_constant<int, S::R2>{}, Mh / S::R1, P.t.tw + T2, S::R3 == 1);

  // the last stage stays in registers: points j + (Mh/R1)*p
  constexpr int R = S::R1, sub = Mh / R;
  C2 x[16];
  float2 m = make_float2(0.f, 0.f);
#pragma unroll
  for (int u = 0; u < 16 / R; ++u) {
    const int j = t + T * u;
    C2 y[R];
#pragma unroll
    for (int p = 0; p < R; ++p) y[p] = get(j + sub * p);
    turn<R, true>(y, P.t.tw, sub, j);
    dftp<R, +1>(y);
#pragma unroll
    for (int p = 0; p < R; ++p) {
      x[u * R + p] = y[p];
      m.x = fmaxf(m.x, fmaxf(fabsf(y[p].re.x), fabsf(y[p].im.x)));
      m.y = fmaxf(m.y, fmaxf(fabsf(y[p].re.y), fabsf(y[p].im.y)));
    }
  }
  // a row's largest value decides its power of two: values below 2^15 as two fp16 terms
  constexpr int G = T < 32 ? T : 32;
#pragma unroll
  for (int o = G / 2; o > 0; o >>= 1) {
    m.x = fmaxf(m.x, __shfl_xor_sync(0xffffffffu, m.x, o));
    m.y = fmaxf(m.y, __shfl_xor_sync(0xffffffffu, m.y, o));
  }
  if constexpr (T > 32) {
    if ((tid & 31) == 0) { red[0][tid >> 5] = m.x; red[1][tid >> 5] = m.y; }
    __syncthreads();
#pragma unroll
    for (int w = 0; w < T / 32; ++w) {
      m.x = fmaxf(m.x, red[0][rl * (T / 32) + w]);
      m.y = fmaxf(m.y, red[1][rl * (T / 32) + w]);
    }
  }
  float2 sc;
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    int ex = (int)((__float_as_uint(r ? m.y : m.x) >> 23) & 0xffu) - 127;           // largest value in [2^ex, 2^(ex+1))
    ex = ex < -100 ? -100 : ex > 126 ? 126 : ex;
    (r ? sc.y : sc.x) = __uint_as_float((unsigned)(14 - ex + 127) << 23);           // 2^(14 - ex)
    if (t == 0) P.inv[row + r] = -__uint_as_float((unsigned)(ex - 14 + 127) << 23) * (1.f / kUpScale);
  }
  // The first term of a value is a whole number of units, 2^-10 of the power of two below the largest of the 64 values
  // (2 G complex ones' worth) that lie around it, so that k_up's sums of first terms are exact; the second is what is left.
  // They go where the rows came from, which this block alone has read, before it began to compute.
  __half2 *hi = reinterpret_cast<__half2 *>(P.y) + row * 2 * Mh, *lo = hi + Mh;
#pragma unroll
  for (int u = 0; u < 16 / R; ++u)
#pragma unroll
    for (int p = 0; p < R; ++p) {
      const int n = t + T * u + sub * p;
      const float2 re = mul2(x[u * R + p].re, sc), im = mul2(x[u * R + p].im, sc);
      // 1.5 * 2^13 of that power of two: adding it rounds to whole units, subtracting it leaves them
      const float2 c = make_float2(unit_rounder(group_max<G>(fmaxf(fabsf(re.x), fabsf(im.x)))),
                                   unit_rounder(group_max<G>(fmaxf(fabsf(re.y), fabsf(im.y)))));
      const float2 hre = sub2(add2(re, c), c), him = sub2(add2(im, c), c), lre = sub2(re, hre), lim = sub2(im, him);
      hi[n] = __floats2half2_rn(hre.x, him.x);
      hi[2 * Mh + n] = __floats2half2_rn(hre.y, him.y);
      lo[n] = __floats2half2_rn(lre.x, lim.x);
      lo[2 * Mh + n] = __floats2half2_rn(lre.y, lim.y);
    }
}

// ---------------------------------------------------------------------------------------------------- k_up
// The two terms of a launch's grid values, [row][term][M]: boxes of 32 or 16 values of 128 rows of one term.
struct GridMaps {
  CUtensorMap wide, narrow;
};
struct UpParams {
  const __half *table;
  const float *inv;
  float *scores[FC_LAYER_CHUNK];
  double *part, *energy;                     // [unit of the call][step][4]; energy of the first layer
  unsigned *done;                            // [layer]
  int *status;
  long long score_stride, energy_stride;
  int H, d, u0, per, ranges;
};
constexpr int kUpBufs = 2;                   // pairs of sums of 128 x 128 in tensor memory
constexpr int x_stages(int nq) { return nq == 16 ? 3 : 2; }      // as many as fit
constexpr int kMaxX = 3;
constexpr int y_stages(int nq, int term) { return term == 0 || nq == 16 ? 2 : 1; }
// grid values and matrices, products, eight warps that take the sums out (four per 64 channels), rows, results of a step
constexpr int kUpThreads = 64 + 256 + 32 + 32;
struct UpShared {
  unsigned long long xfull[kMaxX], xempty[kMaxX], yfull[2][2], yempty[2][2], tfull[kTerms], tempty[kTerms], afull[kUpBufs],
      aempty[kUpBufs], rfull[2], rempty[2], done;                 // y: [term][stage]
  unsigned tmem;
  int last;
  float4 sums[2][2][kRows];                  // of a step's rows: |residual|^2 and |z|^2 of K, of V; per 64 channels of a tile
  int quad[kMaxPer];                         // first quad of the block's steps
};
__host__ __device__ inline size_t up_smem(int nq, int d) {
  return 1024 + (size_t)x_stages(nq) * 8 * kBoxBytes + (size_t)(y_stages(nq, 0) + y_stages(nq, 1) + kTerms) * nq * 1024 +
         (size_t)2 * d * sizeof(float);
}

__device__ __forceinline__ uint4 lds(unsigned addr) {
  uint4 v;
  asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];\n" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr) : "memory");
  return v;
}
template <typename T> __device__ __forceinline__ float2 widen(unsigned v);
template <> __device__ __forceinline__ float2 widen<__half>(unsigned v) { return __half22float2(*reinterpret_cast<const __half2 *>(&v)); }
template <> __device__ __forceinline__ float2 widen<__nv_bfloat16>(unsigned v) {
  return make_float2(__uint_as_float(v << 16), __uint_as_float(v & 0xffff0000u));
}

// What bounds it: HBM, or L2 where a launch group fits it, and shared memory.  A tile of 128 tokens and 128 channels is 64 KB
// of operands and twenty products of 128 x 128 x 16 (64 cycles each, in which they read 128 bytes a cycle, all there is); tokens are the lanes of the sums, so that a row's squares stay in one
// thread, and the grid values are the right operand as the transform left them (64- and 32-byte swizzled boxes).  Rows, and
// grid values with the matrices, have a loading warp each: with one for both, grid values waited for the rows before them.
//
// The tensor cores cut off what does not fit the 24 bits of a sum, so the sum that matters is one that always fits: the first
// terms of the matrix are whole numbers of up to 11 bits, those of the grid values of up to 11 bits and a sign in units that
// are the same for 64 values (k_mid), and a window's sum of their products stays below 2^23 such units.  All other products
// (second terms with first ones, the matrix's third with the values' first, second with second) go to a sum of their own,
// whose cut-off bits are 2^-10 of that size; both are added in fp32.  In a model of these sums, two terms of the matrix and
// one sum for everything leave 0.3..0.5e-6 of a score (rms, 10 % outlier rows), this 0.7e-7, and k_mid's fp32 0.2..0.5e-6.
//
// A matrix comes in three parts, one per term, and products are in such an order that each part is free, and the next step's
// on its way, well before it is needed again: lo x hi, mid x hi, mid x lo, hi x lo, hi x hi.
//
// One block: `per` steps of 128 tokens of one unit.  grid (ranges, units).
template <typename T, int NQ>
__global__ void __launch_bounds__(kUpThreads, 1) k_up(const __grid_constant__ Maps maps, const __grid_constant__ GridMaps grid,
                                                   const __grid_constant__ Geometry g,
                                                   const __grid_constant__ UpParams P) {
  constexpr int kXStages = x_stages(NQ), kHi = y_stages(NQ, 0), kLo = y_stages(NQ, 1);
  extern __shared__ unsigned char raw[];
  unsigned char *smem = reinterpret_cast<unsigned char *>(((uintptr_t)raw + 1023) & ~(uintptr_t)1023);
  unsigned char *ys = smem + (size_t)kXStages * 8 * kBoxBytes;                     // kHi stages of first terms, kLo of second
  constexpr unsigned ybytes = NQ * 1024u, run = NQ * 512u;                         // one term: both runs; one run
  constexpr unsigned tbytes = NQ * 1024u;                                          // one term of a matrix
  unsigned char *tab = ys + (size_t)(kHi + kLo) * ybytes;
  float *sinv = reinterpret_cast<float *>(tab + kTerms * tbytes);
  __shared__ UpShared sh;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int unit = P.u0 + blockIdx.y, layer = unit / P.H, head = unit - layer * P.H;
  const int tiles = P.d / 64, n = g.up_steps(), classes = up_classes(g);
  const int b0 = blockIdx.x * P.per, b1 = b0 + P.per < n ? b0 + P.per : n;

  if (tid == 0) {
    for (int i = 0; i < kXStages; ++i) { mbar::init(&sh.xfull[i], 1u); mbar::init(&sh.xempty[i], 8u); }
    for (int i = 0; i < 4; ++i) { mbar::init(&sh.yfull[i >> 1][i & 1], 1u); mbar::init(&sh.yempty[i >> 1][i & 1], 1u); }
    for (int i = 0; i < kTerms; ++i) { mbar::init(&sh.tfull[i], 1u); mbar::init(&sh.tempty[i], 1u); }
    for (int i = 0; i < kUpBufs; ++i) { mbar::init(&sh.afull[i], 1u); mbar::init(&sh.aempty[i], 8u); }
    for (int i = 0; i < 2; ++i) { mbar::init(&sh.rfull[i], 8u); mbar::init(&sh.rempty[i], 1u); }
    mbar::init(&sh.done, 1u);
    mbar::init_done();
  }
  if (warp == 1) tmem_alloc(&sh.tmem, 256 * kUpBufs);
  for (int i = tid; i < b1 - b0; i += kUpThreads) sh.quad[i] = up_quad(g, b0 + i);
  before_sync();
  __syncthreads();
  after_sync();
  const unsigned tmem = sh.tmem;
  if (warp == 0) {
    if (lane == 0) {
      bool ok = true;
      int ntab[kTerms] = {}, ny[2] = {}, cls = -1;
      auto matrix = [&](int term, int c) {
        if (ok && ntab[term] > 0) ok = mbar::wait(&sh.tempty[term], (unsigned)(ntab[term] - 1) & 1u);
        if (!ok) return;
        mbar::expect_tx(&sh.tfull[term], tbytes);
        load_bytes(tab + term * tbytes, reinterpret_cast<const unsigned char *>(P.table) + ((size_t)c * kTerms + term) * tbytes, tbytes,
                   &sh.tfull[term]);
        ++ntab[term];
      };
      auto values = [&](int term, int q0, int t) {
        const int stages = term == 0 ? kHi : kLo, s = ny[term] % stages;
        if (ok && ny[term] >= stages) ok = mbar::wait(&sh.yempty[term][s], (unsigned)(ny[term] / stages - 1) & 1u);
        if (!ok) return;
        mbar::expect_tx(&sh.yfull[term][s], ybytes);
        const int r0 = ((int)blockIdx.y * tiles + t) * kRows;
        unsigned char *dst = ys + (size_t)(term == 0 ? s : kHi + s) * ybytes;
        for (int rn = 0; rn < 2; ++rn, dst += run) {           // a run: a box of 32 values and, with 24 quads, one of 16
          const int x = rn == 0 ? 2 * q0 : g.M - 2 * (q0 + NQ);
          load_box(dst, &grid.wide, x, term, r0, &sh.yfull[term][s]);
          if (NQ > 16) load_box(dst + kRows * 64, &grid.narrow, x + 32, term, r0, &sh.yfull[term][s]);
        }
        ++ny[term];
      };
      const int items = (b1 - b0) * tiles;
      for (int it = 0; it < items && ok; ++it) {
        const int b = b0 + it / tiles, t = it - (b - b0) * tiles, c = class_of(b, n, classes), q0 = sh.quad[b - b0];
        const bool fresh = c != cls;
        cls = c;
        if (it == 0) {
          for (int k = kTerms - 1; k >= 0; --k) matrix(k, c);
          asm volatile("griddepcontrol.wait;\n" ::: "memory");
          asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
          values(0, q0, t);
          values(1, q0, t);
          continue;
        }
        // in the order in which the places become free
        values(0, q0, t);
        if (fresh) { matrix(2, c); matrix(1, c); }
        values(1, q0, t);
        if (fresh) matrix(0, c);
      }
      // no load may be in flight when the block ends
      for (int k = 0; k < 2; ++k) {
        const int stages = k == 0 ? kHi : kLo;
        for (int i = ny[k] > stages ? ny[k] - stages : 0; i < ny[k]; ++i)
          ok &= mbar::wait(&sh.yfull[k][i % stages], (unsigned)(i / stages) & 1u);
      }
      for (int k = 0; k < kTerms; ++k)
        if (ntab[k] > 0) ok &= mbar::wait(&sh.tfull[k], (unsigned)(ntab[k] - 1) & 1u);
      if (!ok) atomicOr(P.status, FC_DEV_FLAG_TIMEOUT);
    }
  } else if (warp == 10) {
    if (lane == 0) {
      // rows do not come from the kernel in front: they are on their way before it ends
      bool ok = true;
      const int items = (b1 - b0) * tiles;
      int nx = 0;
      for (; nx < items; ++nx) {
        const int s = nx % kXStages, b = b0 + nx / tiles, t = nx - (b - b0) * tiles;
        if (nx >= kXStages && !mbar::wait(&sh.xempty[s], (unsigned)(nx / kXStages - 1) & 1u)) { ok = false; break; }
        mbar::expect_tx(&sh.xfull[s], 8u * kBoxBytes);
        for (int i = 0; i < 4; ++i)
          load_tile(smem + (size_t)(s * 8 + 2 * i) * kBoxBytes, kBoxBytes, maps, layer, tiles, t, head, b * kRows + i * kSlotTok,
                    &sh.xfull[s]);
      }
      for (int i = nx > kXStages ? nx - kXStages : 0; i < nx; ++i) ok &= mbar::wait(&sh.xfull[i % kXStages], (unsigned)(i / kXStages) & 1u);
      if (!ok) atomicOr(P.status, FC_DEV_FLAG_TIMEOUT);
    }
  } else if (warp == 11) {
    // scores and energies of a step, beside the next step's tiles: 1700 of 5300 cycles a step went into the fp64 sums where
    // the warps that take the tiles out made them (16 heads of 32768 tokens 110 -> 97 us)
    const float inv_d = 1.f / (float)P.d;
    for (int b = b0; b < b1; ++b) {
      const int rs = (b - b0) & 1;
      if (!mbar::wait_warp(&sh.rfull[rs], (unsigned)((b - b0) / 2) & 1u)) {
        if (lane == 0) atomicOr(P.status, FC_DEV_FLAG_TIMEOUT);
        break;
      }
      float4 lo[4], hi[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) { lo[i] = sh.sums[rs][0][32 * i + lane]; hi[i] = sh.sums[rs][1][32 * i + lane]; }
      __syncwarp();
      if (lane == 0) mbar::arrive(&sh.rempty[rs]);
      double e[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int tok = b * kRows + 32 * i + lane;
        if (tok < g.N)
          P.scores[layer][(long long)head * P.score_stride + tok] = ((lo[i].x + lo[i].z) + (hi[i].x + hi[i].z)) * inv_d;
        e[0] += (double)lo[i].x + (double)hi[i].x;
        e[1] += (double)lo[i].y + (double)hi[i].y;
        e[2] += (double)lo[i].z + (double)hi[i].z;
        e[3] += (double)lo[i].w + (double)hi[i].w;
      }
      // sums of the step, so that the energies do not depend on how steps are spread over blocks: four values over the
      // lanes at once, lane 8 i ends up with value i
      const bool up = (lane & 16) != 0, up2 = (lane & 8) != 0;
      double v0 = up ? e[2] : e[0], v1 = up ? e[3] : e[1];
      v0 += __shfl_xor_sync(0xffffffffu, up ? e[0] : e[2], 16);
      v1 += __shfl_xor_sync(0xffffffffu, up ? e[1] : e[3], 16);
      double v = up2 ? v1 : v0;
      v += __shfl_xor_sync(0xffffffffu, up2 ? v0 : v1, 8);
      v += __shfl_xor_sync(0xffffffffu, v, 4);
      v += __shfl_xor_sync(0xffffffffu, v, 2);
      v += __shfl_xor_sync(0xffffffffu, v, 1);
      if ((lane & 7) == 0) P.part[((size_t)unit * n + b) * 4 + (lane >> 3)] = v;
    }
    __threadfence();
  } else if (warp == 1) {
    constexpr unsigned idesc = instruction(true, false, kRows), hi = operand_hi(128, 0);
    constexpr unsigned wide = operand_hi(512, 4), narrow = operand_hi(256, 6);     // 64- and 32-byte swizzle
    const unsigned lead = elect();
    const unsigned yb = (smem_addr(ys) >> 4) | operand_lo(16), tb = (smem_addr(tab) >> 4) | operand_lo(2048);
    bool ok = true;
    int ntab = -1, cls = -1, it = 0;
    for (int b = b0; b < b1 && ok; ++b) {
      const int c = class_of(b, n, classes);
      const bool leave = b + 1 < b1 && class_of(b + 1, n, classes) != c;           // another matrix after this step
      for (int t = 0; t < tiles; ++t, ++it) {
        const bool fresh = c != cls, last = leave && t == tiles - 1;
        if (fresh) { cls = c; ++ntab; }
        const int sh_ = it % kHi, sl = it % kLo, buf = it % kUpBufs;
        const unsigned yhi = yb + (unsigned)sh_ * (ybytes / 16), ylo = yb + (unsigned)(kHi + sl) * (ybytes / 16);
        const unsigned big = tmem + (unsigned)buf * 256u, small = big + 128u;
        auto part_here = [&](int term) { return !fresh || mbar::wait_warp(&sh.tfull[term], (unsigned)ntab & 1u); };
        auto products = [&](unsigned d, int term, unsigned y, bool start) {
#pragma unroll
          for (int k = 0; k < NQ / 4; ++k) {
            const int in = k % (NQ / 8);                                   // step within its run
            const bool w = in < 2;                                         // and its box
            const unsigned off = (k / (NQ / 8)) * run + (w ? in * 32u : kRows * 64u);
            mma(lead, d, tb + (unsigned)term * (tbytes / 16) + k * 256u, hi, y + off / 16, w ? wide : narrow, idesc,
                start && k == 0 ? 0u : 1u);
          }
        };
        if (it >= kUpBufs && !mbar::wait_warp(&sh.aempty[buf], (unsigned)(it / kUpBufs - 1) & 1u)) { ok = false; break; }
        if (!mbar::wait_warp(&sh.yfull[0][sh_], (unsigned)(it / kHi) & 1u) || !part_here(2)) { ok = false; break; }
        after_sync();
        products(small, 2, yhi, true);
        if (last) commit(lead, &sh.tempty[2]);
        if (!part_here(1)) { ok = false; break; }
        after_sync();
        products(small, 1, yhi, false);
        if (!mbar::wait_warp(&sh.yfull[1][sl], (unsigned)(it / kLo) & 1u)) { ok = false; break; }
        after_sync();
        products(small, 1, ylo, false);
        if (last) commit(lead, &sh.tempty[1]);
        if (!part_here(0)) { ok = false; break; }
        after_sync();
        products(small, 0, ylo, false);
        commit(lead, &sh.yempty[1][sl]);
        products(big, 0, yhi, true);
        commit(lead, &sh.yempty[0][sh_]);
        if (last) commit(lead, &sh.tempty[0]);
        commit(lead, &sh.afull[buf]);
      }
    }
    commit(lead, &sh.done);
    ok &= mbar::wait_warp(&sh.done, 0u);
    if (!ok && lane == 0) atomicOr(P.status, FC_DEV_FLAG_TIMEOUT);
  } else {
    const int quad = warp & 3, half = (warp - 2) >> 2, row = quad * 32 + lane;
    bool failed = false;
    int it = 0;
    asm volatile("griddepcontrol.wait;\n" ::: "memory");
    for (int i = tid - 64; i < 2 * P.d; i += 256) sinv[i] = __ldcg(P.inv + (size_t)blockIdx.y * 2 * P.d + i);
    asm volatile("bar.sync 1, 256;\n" ::: "memory");
    for (int b = b0; b < b1; ++b) {
      float2 r2[2][2], x2[2][2];             // [K, V][two chains]
#pragma unroll
      for (int i = 0; i < 4; ++i) r2[i >> 1][i & 1] = x2[i >> 1][i & 1] = make_float2(0.f, 0.f);
      for (int t = 0; t < tiles; ++t, ++it) {
        const int buf = it % kUpBufs, s = it % kXStages;
        failed = failed || !mbar::wait_warp(&sh.afull[buf], (unsigned)(it / kUpBufs) & 1u) ||
                 !mbar::wait_warp(&sh.xfull[s], (unsigned)(it / kXStages) & 1u);
        if (failed) continue;
        after_sync();
        const int kv = (2 * t + half) * 64 >= P.d;
        const unsigned xr = smem_addr(smem) + (unsigned)((s * 8 + quad * 2 + half) * kBoxBytes + lane * 128);
        const unsigned iv = smem_addr(sinv + t * kRows + half * 64);
        const unsigned at = tmem + ((unsigned)quad << 21) + (unsigned)(buf * 256 + half * 64);
        float2 rs[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)}, xs[2] = {rs[0], rs[0]};
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          float a[16], low[16];
          tmem_ld16(at + 16 * c, a);
          tmem_ld16(at + 128 + 16 * c, low);
          uint4 xv[2];
#pragma unroll
          for (int i = 0; i < 2; ++i) xv[i] = lds(xr + (((2 * c + i) ^ (lane & 7)) << 4));
          tmem_wait(a);
          tmem_wait(low);
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const uint4 sc = lds(iv + (unsigned)(4 * c + i) * 16u);
            const unsigned w0 = i & 1 ? xv[i >> 1].z : xv[i >> 1].x, w1 = i & 1 ? xv[i >> 1].w : xv[i >> 1].y;
            const float2 xa = widen<T>(w0), xb = widen<T>(w1);
            const float2 ba = add2(make_float2(a[4 * i], a[4 * i + 1]), make_float2(low[4 * i], low[4 * i + 1]));
            const float2 bb = add2(make_float2(a[4 * i + 2], a[4 * i + 3]), make_float2(low[4 * i + 2], low[4 * i + 3]));
            const float2 ra = fma2(ba, make_float2(__uint_as_float(sc.x), __uint_as_float(sc.y)), xa);
            const float2 rb = fma2(bb, make_float2(__uint_as_float(sc.z), __uint_as_float(sc.w)), xb);
            rs[0] = fma2(ra, ra, rs[0]);
            rs[1] = fma2(rb, rb, rs[1]);
            xs[0] = fma2(xa, xa, xs[0]);
            xs[1] = fma2(xb, xb, xs[1]);
          }
        }
        // reads of the rows by loads come before the tensor engine's next writes to their place
        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
        before_sync();
        __syncwarp();
        if (lane == 0) { mbar::arrive(&sh.aempty[buf]); mbar::arrive(&sh.xempty[s]); }
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          if (kv) {
            r2[1][i].x += rs[i].x; r2[1][i].y += rs[i].y; x2[1][i].x += xs[i].x; x2[1][i].y += xs[i].y;
          } else {
            r2[0][i].x += rs[i].x; r2[0][i].y += rs[i].y; x2[0][i].x += xs[i].x; x2[0][i].y += xs[i].y;
          }
        }
      }
      const int rs = (b - b0) & 1;
      if (!failed && b - b0 >= 2) failed = !mbar::wait_warp(&sh.rempty[rs], (unsigned)((b - b0) / 2 - 1) & 1u);
      if (failed) break;
      // this thread's row and channels; rows past the end count nothing
      const bool in = b * kRows + row < g.N;
      sh.sums[rs][half][row] =
          in ? make_float4((r2[0][0].x + r2[0][0].y) + (r2[0][1].x + r2[0][1].y), (x2[0][0].x + x2[0][0].y) + (x2[0][1].x + x2[0][1].y),
                           (r2[1][0].x + r2[1][0].y) + (r2[1][1].x + r2[1][1].y), (x2[1][0].x + x2[1][0].y) + (x2[1][1].x + x2[1][1].y))
             : make_float4(0.f, 0.f, 0.f, 0.f);
      __syncwarp();
      if (lane == 0) mbar::arrive(&sh.rfull[rs]);
    }
    if (failed && lane == 0) atomicOr(P.status, FC_DEV_FLAG_TIMEOUT);
  }
  before_sync();
  __syncthreads();
  if (warp == 1) tmem_free(tmem, 256 * kUpBufs);
  // energies: in the block of the layer that comes last, all steps' sums in order
  if (tid == 0) {
    __threadfence();
    const unsigned all = (unsigned)(P.H * P.ranges);
    sh.last = atomicAdd(P.done + layer, 1u) + 1u == all;
    if (sh.last) P.done[layer] = 0u;
    __threadfence();
  }
  __syncthreads();
  if (sh.last && warp < 4) {
    const double *p = P.part + (size_t)layer * P.H * n * 4;
    double v = 0.0;
    for (int i = lane; i < P.H * n; i += 32) v += __ldcg(p + 4 * (size_t)i + warp);
    v = warp_sum_d(v);
    if (lane == 0) P.energy[(long long)layer * P.energy_stride + warp] = v;
  }
}

}  // namespace band
