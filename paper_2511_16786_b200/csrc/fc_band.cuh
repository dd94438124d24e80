// Scoring in the kept band: the Base KV of Eq. 9 is a band of low frequencies, so it fits on a grid a few times coarser
// than the tokens, and only that grid is transformed.  With phi a short low-pass kernel (support W grid points), tokens
// t = 0..N-1, grid points x_j = (j + 1/2) N/M - 1/2, j = 0..M-1, both continued evenly about -1/2 and N-1/2 as the
// DCT-II of Eq. 6 does:
//   k_down   y_j = (M/N) sum_t phi((t - x_j) M/N) z_t          a banded matrix times the rows of K and V
//   k_mid    b = C^-1 diag(1 / H(m)^2, m <= omega; 0) C y      M-point DCT-II, the cutoff, inverse; H = spectrum of phi
//   k_up     base_t = sum_j phi((t - x_j) M/N) b_j             the transposed band, then |z_t - base_t|^2 per row
// phi need not be flat in the band (H is divided out exactly) nor short of the theory's length; it has to suppress what
// folds onto the band, which it does to 6e-8 of the band's own gain, i.e. to fp32 rounding.  k_down and k_up are matrix
// products on the 5th-generation tensor cores: 16-bit K and V are exact operands, phi is a sum of three bf16 or two
// fp16 terms and b a sum of two fp16 terms scaled per channel (24 bits each), and sums are fp32.  N is arbitrary.
#pragma once
#include <cuda.h>

#include "fc_common.cuh"
#include "fc_mbar.cuh"

namespace band {

constexpr int kJ = 16;                       // grid points per step of k_down
constexpr int kSlotTok = 32;                 // tokens per ring slot of k_down and per TMA box
constexpr int kRing = 11;                    // ring slots of k_down
constexpr int kMaxSteps = 12;                // 16-token steps a window of k_down may have
constexpr int kRows = 128;                   // rows (channels of K, then of V) per tile; tokens per step of k_up
constexpr int kBoxBytes = kSlotTok * 128;    // one box: 32 tokens x 64 channels of 2 bytes
constexpr int kMaxQuads = 24;                // grid quads a window of k_up may have
constexpr int kMaxPer = 256;                 // steps a block of k_down or k_up may have
constexpr int kCheb = 28;                    // terms of the expansion of H
constexpr float kUpScale = 1024.f;           // k_up's matrix is stored times this (its low terms stay normal fp16)
constexpr float kDownScaleF16 = 4096.f;      // k_down's fp16 matrix is stored times this

struct Maps {                                // one sequence's rows in every layer of the launch
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

__host__ __device__ inline int filter_terms(bool f16) { return f16 ? 2 : 3; }
__host__ __device__ inline size_t down_image(const Geometry &g, int nr) { return (size_t)g.ks * 2 * nr * 16; }
__host__ __device__ inline size_t up_image(const Geometry &g) { return (size_t)g.nq * 2048; }

// ---------------------------------------------------------------------------------------------------- tables
__device__ inline double phi(const Geometry &g, double u) {
  const double s = 2.0 * u / g.W, r = 1.0 - s * s;
  if (!(r >= 0.0)) return 0.0;
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

// The matrix of one step of k_down: [16-token step * 2][term * 16 + j][8 tokens], rows of 16 bytes.
template <typename T, int TERMS>
__global__ void k_down_table(const __grid_constant__ Geometry g, T *__restrict__ out) {
  const int classes = down_classes(g), b = step_of(blockIdx.x, g.down_steps(), classes);
  const int t0 = down_start(g, b), nt = g.ks * 16;
  T *img = out + (size_t)blockIdx.x * (down_image(g, TERMS * kJ) / 2);
  const double step = (double)g.N / g.M, inv = (double)g.M / g.N;
  const double scale = TERMS == 2 ? inv * kDownScaleF16 : inv;
  for (int i = threadIdx.x; i < nt * kJ; i += blockDim.x) {
    const int e = i & 7, j = (i >> 3) & (kJ - 1), c = i >> 7, t = t0 + c * 8 + e;
    double v = 0.0;
    if (t < g.N) {
      const double x = (b * kJ + j + 0.5) * step - 0.5;
      v = phi(g, (t - x) * inv) + phi(g, (-1.0 - t - x) * inv) + phi(g, (2.0 * g.N - 1.0 - t - x) * inv);
      v *= scale;
    }
#pragma unroll
    for (int k = 0; k < TERMS; ++k) {
      const T h = (T)(float)v;
      img[((size_t)c * (TERMS * kJ) + k * kJ + j) * 8 + e] = h;
      v -= (double)(float)h;
    }
  }
}

// The matrix of one step of k_up: [term][8 grid values][token][8].  Values are in the order the transform keeps them:
// first (z0, z2) of ascending quads, then (z3, z1) of descending ones.
static __global__ void k_up_table(const __grid_constant__ Geometry g, __half *__restrict__ out) {
  const int classes = up_classes(g), b = step_of(blockIdx.x, g.up_steps(), classes);
  const int q0 = up_quad(g, b), nk = 4 * g.nq;
  __half *img = out + (size_t)blockIdx.x * (up_image(g) / 2);
  const double inv = (double)g.M / g.N;
  for (int i = threadIdx.x; i < nk * kRows; i += blockDim.x) {
    const int e = i & 7, r = (i >> 3) & (kRows - 1), c = i >> 10, k = c * 8 + e, t = b * kRows + r;
    const bool second = k >= 2 * g.nq;
    const int kk = second ? k - 2 * g.nq : k;
    const int n = second ? q0 + g.nq - 1 - (kk >> 1) : q0 + (kk >> 1);
    const int j = 4 * n + (second ? ((kk & 1) ? 1 : 3) : 2 * (kk & 1));
    double v = 0.0;
    if (t < g.N) {
      const double x = (t + 0.5) * inv - 0.5;
      v = phi(g, x - j) + phi(g, x + 1.0 + j) + phi(g, x - (2.0 * g.M - 1.0 - j));
      v *= (double)kUpScale;
    }
    const __half h = __float2half_rn((float)v);
    const __half l = __float2half_rn((float)(v - (double)__half2float(h)));
    img[((size_t)c * kRows + r) * 8 + e] = h;
    img[((size_t)(nk / 8 + c) * kRows + r) * 8 + e] = l;
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

// Operand descriptor: start, leading and stride byte offsets in 16-byte units, layout 0 = none, 2 = 128-byte swizzle.
__device__ __forceinline__ unsigned long long operand(unsigned addr, unsigned lead, unsigned stride, unsigned layout) {
  return (unsigned long long)((addr >> 4) & 0x3fffu) | ((unsigned long long)((lead >> 4) & 0x3fffu) << 16) |
         ((unsigned long long)((stride >> 4) & 0x3fffu) << 32) | (1ull << 46) | ((unsigned long long)layout << 61);
}
// fp32 sums of 16-bit products; A 128 x 16, B 16 x n, B and (unless a_by_rows) A with consecutive depth.
__host__ __device__ constexpr unsigned instruction(bool f16, bool a_by_rows, int n) {
  return (1u << 4) | ((f16 ? 0u : 1u) << 7) | ((f16 ? 0u : 1u) << 10) | ((a_by_rows ? 1u : 0u) << 15) |
         ((unsigned)(n >> 3) << 17) | ((unsigned)(128 >> 4) << 24);
}
__device__ __forceinline__ void mma(unsigned d, unsigned long long a, unsigned long long b, unsigned idesc, bool add) {
  asm volatile("{\n .reg .pred p;\n setp.ne.u32 p, %4, 0;\n tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n"
               ::"r"(d), "l"(a), "l"(b), "r"(idesc), "r"(add ? 1u : 0u) : "memory");
}
__device__ __forceinline__ void commit(unsigned long long *bar) {          // arrives once all products issued so far are done
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(smem_addr(bar)) : "memory");
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
__device__ __forceinline__ void load_bytes(void *dst, const void *src, unsigned bytes, unsigned long long *bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n"
               ::"r"(smem_addr(dst)), "l"(__cvta_generic_to_global(src)), "r"(bytes), "r"(smem_addr(bar)) : "memory");
}

// ---------------------------------------------------------------------------------------------------- k_down
struct DownParams {
  const void *table;
  float *y;                                  // [unit of the launch][row][M]: (z0, z2) of quads ascending, (z3, z1) descending
  int *status;
  int H, d, u0;                              // heads, channels per head, first unit (layer * H + head) of the launch
  int per;                                   // steps per block
};
struct DownShared {
  unsigned long long full[kRing], empty[kRing], tfull[2], tempty[2], afull[2], aempty[2], done;
  unsigned tmem;
  int start[kMaxPer + 1];                    // of the block's steps and the one after
};
constexpr int kDownThreads = 192;            // loads, products, and four warps that take the sums out
constexpr unsigned kDownCols = 512;
constexpr size_t kDownSmem = 1024 + (size_t)kRing * 4 * kBoxBytes + 2 * (size_t)kMaxSteps * 2 * 48 * 16;

// One block: `per` steps of 16 grid points for up to two tiles (256 rows) of one unit.  grid (ranges, tile pairs, units).
template <typename T, int TERMS>
__global__ void __launch_bounds__(kDownThreads, 1) k_down(const __grid_constant__ Maps maps, const __grid_constant__ Geometry g,
                                                       const DownParams P) {
  constexpr int NR = TERMS * kJ;             // columns of one sum
  extern __shared__ unsigned char raw[];
  unsigned char *smem = reinterpret_cast<unsigned char *>(((uintptr_t)raw + 1023) & ~(uintptr_t)1023);
  unsigned char *tab = smem + (size_t)kRing * 4 * kBoxBytes;
  __shared__ DownShared sh;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int unit = P.u0 + blockIdx.z, layer = unit / P.H, head = unit - layer * P.H;
  const int tiles = P.d / 64, tile0 = 2 * blockIdx.y, nt = tiles - tile0 < 2 ? 1 : 2;
  const int n = g.down_steps(), classes = down_classes(g);
  const int b0 = blockIdx.x * P.per, b1 = b0 + P.per < n ? b0 + P.per : n;
  const unsigned img = (unsigned)down_image(g, NR);
  unsigned char *tab1 = tab + (size_t)kMaxSteps * 2 * 48 * 16;

  if (tid == 0) {
    for (int i = 0; i < kRing; ++i) { mbar::init(&sh.full[i], 1u); mbar::init(&sh.empty[i], 1u); }
    for (int i = 0; i < 2; ++i) {
      mbar::init(&sh.tfull[i], 1u); mbar::init(&sh.tempty[i], 1u);
      mbar::init(&sh.afull[i], 1u); mbar::init(&sh.aempty[i], 4u);
    }
    mbar::init(&sh.done, 1u);
    mbar::init_done();
  }
  if (warp == 1) tmem_alloc(&sh.tmem, kDownCols);
  for (int i = tid; i <= b1 - b0; i += kDownThreads) sh.start[i] = down_start(g, b0 + i);
  before_sync();
  __syncthreads();
  after_sync();
  const unsigned tmem = sh.tmem;
  if (b0 < b1) {
    const int q0 = sh.start[0] / kSlotTok;                 // ring slots are counted from here
    if (warp == 0) {
      if (lane == 0) {
        bool ok = true;
        int q = q0, ntab = 0, cls = -1;
        for (int b = b0; b < b1 && ok; ++b) {
          const int c = class_of(b, n, classes);
          if (c != cls) {
            cls = c;
            const int s = ntab & 1;
            if (ntab >= 2 && !mbar::wait(&sh.tempty[s], (unsigned)(ntab / 2 - 1) & 1u)) { ok = false; break; }
            mbar::expect_tx(&sh.tfull[s], img);
            load_bytes(s ? tab1 : tab, static_cast<const unsigned char *>(P.table) + (size_t)c * img, img, &sh.tfull[s]);
            ++ntab;
          }
          // run ahead of this step's window as far as the ring allows without waiting for steps not yet issued
          const int last = (sh.start[b - b0] + 16 * g.ks - 1) / kSlotTok;
          for (; q <= last; ++q) {
            const int i = q - q0, s = i % kRing;
            if (i >= kRing && !mbar::wait(&sh.empty[s], (unsigned)(i / kRing - 1) & 1u)) { ok = false; break; }
            mbar::expect_tx(&sh.full[s], (unsigned)(2 * nt * kBoxBytes));
            for (int hf = 0; hf < 2 * nt; ++hf) {
              const int c64 = (2 * tile0 + hf) * 64;             // K's channels, then V's
              const bool isv = c64 >= P.d;
              load_box(smem + (size_t)(s * 4 + hf) * kBoxBytes, isv ? &maps.v[layer] : &maps.k[layer], isv ? c64 - P.d : c64,
                       head, q * kSlotTok, &sh.full[s]);
            }
          }
        }
        // no load may be in flight when the block ends
        const int issued = q - q0;
        for (int i = issued > kRing ? issued - kRing : 0; i < issued; ++i)
          ok &= mbar::wait(&sh.full[i % kRing], (unsigned)(i / kRing) & 1u);
        for (int i = ntab > 2 ? ntab - 2 : 0; i < ntab; ++i) ok &= mbar::wait(&sh.tfull[i & 1], (unsigned)(i / 2) & 1u);
        if (!ok) atomicOr(P.status, FC_DEV_FLAG_TIMEOUT);
      }
    } else if (warp == 1) {
      if (lane == 0) {
        constexpr unsigned idesc = instruction(TERMS == 2, true, NR);
        bool ok = true;
        int have = q0, freed = q0, ntab = 0, cls = -1;
        for (int b = b0; b < b1 && ok; ++b) {
          const int start = sh.start[b - b0], last = (start + 16 * g.ks - 1) / kSlotTok, it = b - b0, buf = it & 1;
          const int c = class_of(b, n, classes);
          if (c != cls) {
            cls = c;
            if (ntab > 0) commit(&sh.tempty[(ntab - 1) & 1]);
            if (!mbar::wait(&sh.tfull[ntab & 1], (unsigned)(ntab / 2) & 1u)) { ok = false; break; }
            ++ntab;
          }
          if (it >= 2 && !mbar::wait(&sh.aempty[buf], (unsigned)(it / 2 - 1) & 1u)) { ok = false; break; }
          for (; have <= last && ok; ++have)
            ok = mbar::wait(&sh.full[(have - q0) % kRing], (unsigned)((have - q0) / kRing) & 1u);
          if (!ok) break;
          after_sync();
          const unsigned tb = smem_addr(((ntab - 1) & 1) ? tab1 : tab);
          // steps from the window's ends to its middle, in two sums by turns: small terms first, few roundings of large sums
          for (int i = 0; i < g.ks; ++i) {
            const int k = (i & 1) ? g.ks - 1 - i / 2 : i / 2;
            const int t16 = start / 16 + k, s = (t16 / 2 - q0) % kRing;
            const unsigned long long bd = operand(tb + (unsigned)k * (2 * NR * 16), NR * 16, 128, 0);
            for (int t = 0; t < nt; ++t) {
              const unsigned long long ad =
                  operand(smem_addr(smem + (size_t)(s * 4 + 2 * t) * kBoxBytes) + (t16 & 1) * 2048, kBoxBytes, 1024, 2);
              mma(tmem + (unsigned)(((buf * 2 + t) * 2 + ((i >> 1) & 1)) * NR), ad, bd, idesc, i >= 4 || (i & 1));
            }
          }
          commit(&sh.afull[buf]);
          const int keep = b + 1 < b1 ? sh.start[b - b0 + 1] / kSlotTok : freed;
          for (; freed < keep; ++freed) commit(&sh.empty[(freed - q0) % kRing]);
        }
        commit(&sh.done);                                        // nothing is left running when the block ends
        ok &= mbar::wait(&sh.done, 0u);
        if (!ok) atomicOr(P.status, FC_DEV_FLAG_TIMEOUT);
      }
    } else {
      const int quad = warp & 3, row = quad * 32 + lane, Mh = g.M / 2;
      const float scale = TERMS == 2 ? 1.f / kDownScaleF16 : 1.f;
      for (int b = b0; b < b1; ++b) {
        const int it = b - b0, buf = it & 1;
        if (!mbar::wait_warp(&sh.afull[buf], (unsigned)(it / 2) & 1u)) {
          if (lane == 0) atomicOr(P.status, FC_DEV_FLAG_TIMEOUT);
          break;
        }
        after_sync();
        for (int t = 0; t < nt; ++t) {
          const unsigned at = tmem + ((unsigned)quad << 21) + (unsigned)((buf * 2 + t) * 2 * NR);
          float v[16], a[16], c[16];
          tmem_ld16(at + (TERMS - 1) * kJ, v);
          tmem_ld16(at + NR + (TERMS - 1) * kJ, a);
          tmem_wait(v);
          tmem_wait(a);
#pragma unroll
          for (int j = 0; j < kJ; ++j) v[j] += a[j];
#pragma unroll
          for (int k = TERMS - 2; k >= 0; --k) {
            tmem_ld16(at + k * kJ, a);
            tmem_ld16(at + NR + k * kJ, c);
            tmem_wait(a);
            tmem_wait(c);
#pragma unroll
            for (int j = 0; j < kJ; ++j) v[j] += a[j] + c[j];
          }
          if (TERMS == 2) {
#pragma unroll
            for (int j = 0; j < kJ; ++j) v[j] *= scale;
          }
          float *yr = P.y + ((size_t)blockIdx.z * 2 * P.d + (tile0 + t) * kRows + row) * g.M;
          float4 *lo = reinterpret_cast<float4 *>(yr + 8 * b), *hi = reinterpret_cast<float4 *>(yr + 2 * (Mh - 4 - 4 * b));
          lo[0] = make_float4(v[0], v[2], v[4], v[6]);
          lo[1] = make_float4(v[8], v[10], v[12], v[14]);
          hi[0] = make_float4(v[15], v[13], v[11], v[9]);
          hi[1] = make_float4(v[7], v[5], v[3], v[1]);
        }
        before_sync();
        __syncwarp();
        if (lane == 0) mbar::arrive(&sh.aempty[buf]);
      }
    }
  }
  before_sync();
  __syncthreads();
  if (warp == 1) tmem_free(tmem, kDownCols);
}

// ---------------------------------------------------------------------------------------------------- k_mid
// One real row of M grid values as a complex transform of Mh = M/2 points, Mh = R1*R2*R3*R4, 16 points per thread.
template <int R1_, int R2_, int R3_, int R4_>
struct MidShape {
  static constexpr int R1 = R1_, R2 = R2_, R3 = R3_, R4 = R4_, Mh = R1 * R2 * R3 * R4, T = Mh / 16;
  static constexpr int RL = R4 > 1 ? R4 : R3 > 1 ? R3 : R2;         // radix of the last stage
  static constexpr int S = Mh / RL;                                  // bins of the stages before it
  static constexpr int ROWS = T >= 256 ? 1 : 256 / T, NT = T * ROWS;
  static constexpr int LEN = Mh + Mh / 16;                           // one entry of padding per 16: conflict-free in every stage
  static constexpr size_t smem = (size_t)ROWS * LEN * sizeof(float2);
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

template <class S>
__global__ void k_mid_table(const __grid_constant__ Geometry g, MidTables t) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < S::Mh / 2) {
    // pair i: bins k0 + S*l and Mh minus that; the first RL of them are the blocks that are their own partners
    const int k0 = i >= S::RL ? i / S::RL : i < S::RL / 2 ? 0 : S::S / 2;
    const int l = i >= S::RL ? i % S::RL : i % (S::RL / 2), k = k0 + S::S * l;
    auto gain = [&](int m) {
      if (m > g.omega || m >= g.M) return 0.0;
      const double h = response(g, (double)m / (2.0 * g.M));
      return 1.0 / (h * h);
    };
    const double s = 1.0 / (4.0 * S::Mh);
    if (k == 0) {
      t.gain[i] = make_float4((float)(gain(0) / (2.0 * S::Mh)), (float)(gain(S::Mh) / (2.0 * S::Mh)),
                              (float)(gain(S::Mh / 2) * s), (float)(gain(S::Mh + S::Mh / 2) * s));
    } else {
      t.gain[i] = make_float4((float)(gain(k) * s), (float)(gain(g.M - k) * s), (float)(gain(S::Mh - k) * (0.5 * s)),
                              (float)(gain(S::Mh + k) * (0.5 * s)));
    }
    double c, sn, c4, s4;
    const int kr = k == 0 ? S::Mh / 2 : k;                            // entry 0 serves the bin Mh/2
    sincospi((double)kr / (2.0 * g.M), &sn, &c);
    sincospi(2.0 * kr / (double)g.M, &s4, &c4);
    t.rot[i] = make_float4((float)c, (float)sn, (float)c4, (float)s4);
  }
  const int pw[6] = {1, 2, 3, 4, 8, 12};
  int base = 0, L = S::Mh;
  const int r[3] = {S::R1, S::R3 > 1 ? S::R2 : 1, S::R4 > 1 ? S::R3 : 1};
#pragma unroll
  for (int s = 0; s < 3; ++s) {
    if (r[s] == 1) continue;
    const int sub = L / r[s];
    for (int e = i; e < 6 * sub; e += gridDim.x * blockDim.x) {
      double c, sn;
      sincospi(2.0 * (double)(pw[e / sub] * (e % sub)) / (double)L, &sn, &c);
      t.tw[base + e] = make_float2((float)c, (float)-sn);
    }
    base += 6 * sub;
    L = sub;
  }
}

// x[p] *= w^p (conjugated for the way back), w^1, 2, 3, 4, 8, 12 from the table: at most two factors each
template <int R, bool CONJ>
__device__ __forceinline__ void turn(float2 *x, const float2 *__restrict__ tw, int sub, int j) {
  float2 c[4];
#pragma unroll
  for (int p = 1; p < (R < 4 ? R : 4); ++p) {
    c[p] = __ldg(tw + (p - 1) * sub + j);
    if (CONJ) c[p].y = -c[p].y;
    x[p] = cmul(x[p], c[p]);
  }
#pragma unroll
  for (int a = 1; a < R / 4; ++a) {
    float2 b = __ldg(tw + (2 + a) * sub + j);
    if (CONJ) b.y = -b.y;
    x[4 * a] = cmul(x[4 * a], b);
#pragma unroll
    for (int p = 1; p < 4; ++p) x[4 * a + p] = cmul(x[4 * a + p], cmul(b, c[p]));
  }
}

struct MidParams {
  const float *y;                            // [row][M]
  __half *hi, *lo;                           // [tile][quad / 4][row of the tile][8]
  float *inv;                                // [row]: minus what a stored value has to be multiplied with
  MidTables t;
};

template <class S>
__global__ void __launch_bounds__(S::NT, S::NT == 256 ? 4 : S::NT == 512 ? 2 : 1) k_mid(const MidParams P) {
  constexpr int Mh = S::Mh, T = S::T;
  extern __shared__ float2 X0[];
  __shared__ float red[S::NT / 32 > 0 ? S::NT / 32 : 1];
  const int tid = threadIdx.x, t = tid % T, rl = tid / T;
  float2 *X = X0 + rl * S::LEN;
  const size_t row = (size_t)blockIdx.x * S::ROWS + rl;
  auto pad = [](int pos) { return pos + (pos >> 4); };
  const float2 *src = reinterpret_cast<const float2 *>(P.y) + row * Mh;
  constexpr int T2 = 6 * (Mh / S::R1), T3 = T2 + 6 * (Mh / S::R1 / S::R2);

  // one stage on the points block*L + j + sub*p
  auto forward = [&](auto radix, int L, const float2 *tw, bool first, bool last) {
    constexpr int R = decltype(radix)::value;
    const int sub = L / R;
#pragma unroll
    for (int u = 0; u < 16 / R; ++u) {
      const int i = t + T * u, blk = i / sub, j = i - blk * sub, at = blk * L + j;
      float2 x[R];
#pragma unroll
      for (int p = 0; p < R; ++p) x[p] = first ? __ldcg(src + at + sub * p) : X[pad(at + sub * p)];
      dft_small<R, -1>(x);
      if (!last) turn<R, false>(x, tw, sub, j);
#pragma unroll
      for (int p = 0; p < R; ++p) X[pad(at + sub * p)] = x[p];
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
    const int k0 = i >= S::RL ? i / S::RL : i < S::RL / 2 ? 0 : S::S / 2;
    const int l = i >= S::RL ? i % S::RL : i % (S::RL / 2);
    const int pa = pad(S::sub_of(k0) * S::RL + l);
    const int pb = i == 0 ? pad(S::RL / 2) : k0 == 0 ? pad(S::RL - l) : pad(S::sub_of(S::S - k0) * S::RL + S::RL - 1 - l);
    float2 a = X[pa], b = X[pb];
    float4 gn = __ldg(P.t.gain + i);
    const float4 rt = __ldg(P.t.rot + i);
    if (i == 0) {                            // bins 0 and, by itself, Mh/2
      const float w0 = (a.x + a.y) * gn.x, wh = (a.x - a.y) * gn.y;
      X[pa] = make_float2(w0 + wh, w0 - wh);
      a = b;
      gn = make_float4(gn.z, gn.w, 0.5f * gn.z, 0.5f * gn.w);
    }
    const float2 f = make_float2(rt.x, rt.y), e = make_float2(rt.z, rt.w);   // e^(j pi k/2M), e^(2 pi j k/M)
    const float2 s = cmul_conj(make_float2(a.x + b.x, a.y - b.y), f);
    const float2 r = cmul_conj(cmul_conj(make_float2(a.x - b.x, a.y + b.y), f), e);
    const float2 p = make_float2((s.x + r.y) * gn.x, (s.y - r.x) * gn.y);    // r * -j
    const float2 q = make_float2(s.x - r.y, s.y + r.x);
    const float uu = (q.x - q.y) * gn.z, vv = (q.x + q.y) * gn.w;
    const float2 q2 = make_float2(uu + vv, vv - uu);
    const float2 gs = cadd(p, q2), gd = cmul(csub(p, q2), e);
    const float2 z = cmul(make_float2(gs.x - gd.y, gs.y + gd.x), f), y = cmul(make_float2(gs.x + gd.y, gs.y - gd.x), f);
    if (i != 0) X[pa] = z;
    X[pb] = i == 0 ? z : make_float2(y.x, -y.y);
  }
  __syncthreads();

  auto back = [&](auto radix, int L, const float2 *tw, bool last) {
    constexpr int R = decltype(radix)::value;
    const int sub = L / R;
#pragma unroll
    for (int u = 0; u < 16 / R; ++u) {
      const int i = t + T * u, blk = i / sub, j = i - blk * sub, at = blk * L + j;
      float2 x[R];
#pragma unroll
      for (int p = 0; p < R; ++p) x[p] = X[pad(at + sub * p)];
      if (!last) turn<R, true>(x, tw, sub, j);
      dft_small<R, +1>(x);
#pragma unroll
      for (int p = 0; p < R; ++p) X[pad(at + sub * p)] = x[p];
    }
    __syncthreads();
  };
  if constexpr (S::R4 > 1) back(std::integral_constant<int, S::R4>{}, S::R4, nullptr, true);
  if constexpr (S::R3 > 1) back(std::integral_constant<int, S::R3>{}, Mh / S::R1 / S::R2, P.t.tw + T3, S::R4 == 1);
  back(std::integral_constant<int, S::R2>{}, Mh / S::R1, P.t.tw + T2, S::R3 == 1);

  // the last stage stays in registers: points j + (Mh/R1)*p
  constexpr int R = S::R1, sub = Mh / R;
  float2 x[16];
  float m = 0.f;
#pragma unroll
  for (int u = 0; u < 16 / R; ++u) {
    const int j = t + T * u;
    float2 y[R];
#pragma unroll
    for (int p = 0; p < R; ++p) y[p] = X[pad(j + sub * p)];
    turn<R, true>(y, P.t.tw, sub, j);
    dft_small<R, +1>(y);
#pragma unroll
    for (int p = 0; p < R; ++p) {
      x[u * R + p] = y[p];
      m = fmaxf(m, fmaxf(fabsf(y[p].x), fabsf(y[p].y)));
    }
  }
  // the row's largest value decides its power of two: values below 2^15 as two fp16 terms
  constexpr int G = T < 32 ? T : 32;
#pragma unroll
  for (int o = G / 2; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  if constexpr (T > 32) {
    if ((tid & 31) == 0) red[tid >> 5] = m;
    __syncthreads();
#pragma unroll
    for (int w = 0; w < T / 32; ++w) m = fmaxf(m, red[rl * (T / 32) + w]);
  }
  int ex = (int)((__float_as_uint(m) >> 23) & 0xffu) - 127;            // m in [2^ex, 2^(ex+1))
  ex = ex < -100 ? -100 : ex > 126 ? 126 : ex;
  const float sc = __uint_as_float((unsigned)(14 - ex + 127) << 23);   // 2^(14 - ex)
  if (t == 0) P.inv[row] = -__uint_as_float((unsigned)(ex - 14 + 127) << 23) * (1.f / kUpScale);
  const size_t base = (row / kRows) * (size_t)(Mh / 4) * kRows + row % kRows;
  __half2 *hi = reinterpret_cast<__half2 *>(P.hi), *lo = reinterpret_cast<__half2 *>(P.lo);
#pragma unroll
  for (int u = 0; u < 16 / R; ++u)
#pragma unroll
    for (int p = 0; p < R; ++p) {
      const int n = t + T * u + sub * p;
      const float2 v = make_float2(x[u * R + p].x * sc, x[u * R + p].y * sc);
      const __half2 h = __floats2half2_rn(v.x, v.y);
      const float2 hf = __half22float2(h);
      const size_t at = (base + (size_t)(n >> 2) * kRows) * 4 + (n & 3);
      hi[at] = h;
      lo[at] = __floats2half2_rn(v.x - hf.x, v.y - hf.y);
    }
}

// ---------------------------------------------------------------------------------------------------- k_up
struct UpParams {
  const __half *table, *hi, *lo;
  const float *inv;
  float *scores[FC_LAYER_CHUNK];
  double *part, *energy;                     // [unit of the call][range][4]; energy of the first layer
  unsigned *done;                            // [layer]
  int *status;
  long long score_stride, energy_stride;
  int H, d, u0, per, ranges;
};
constexpr int kUpBufs = 4;                   // sums of 128 x 128 in tensor memory
constexpr int kXStages = 2, kYStages = 2;
constexpr int kUpThreads = 64 + 256;         // loads, products, and eight warps: four per 64 channels of a tile
struct UpShared {
  unsigned long long xfull[kXStages], xempty[kXStages], yfull[kYStages], yempty[kYStages], tfull, tempty, afull[kUpBufs],
      aempty[kUpBufs], done;
  unsigned tmem;
  int last;
  float other[2][kRows];
  double red[8][4];
  int quad[kMaxPer];                         // first quad of the block's steps
};
__host__ __device__ inline size_t up_smem(int nq, int d) {
  return 1024 + (size_t)kXStages * 8 * kBoxBytes + (size_t)(kYStages + 1) * nq * 2048 + (size_t)2 * d * sizeof(float);
}

__device__ __forceinline__ uint4 lds(unsigned addr) {
  uint4 v;
  asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];\n" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
template <typename T> __device__ __forceinline__ float2 widen(unsigned v);
template <> __device__ __forceinline__ float2 widen<__half>(unsigned v) { return __half22float2(*reinterpret_cast<const __half2 *>(&v)); }
template <> __device__ __forceinline__ float2 widen<__nv_bfloat16>(unsigned v) {
  return make_float2(__uint_as_float(v << 16), __uint_as_float(v & 0xffff0000u));
}

// One block: `per` steps of 128 tokens of one unit.  grid (ranges, units).
template <typename T>
__global__ void __launch_bounds__(kUpThreads, 1) k_up(const __grid_constant__ Maps maps, const __grid_constant__ Geometry g,
                                                   const __grid_constant__ UpParams P) {
  extern __shared__ unsigned char raw[];
  unsigned char *smem = reinterpret_cast<unsigned char *>(((uintptr_t)raw + 1023) & ~(uintptr_t)1023);
  unsigned char *ys = smem + (size_t)kXStages * 8 * kBoxBytes;
  const unsigned ybytes = (unsigned)g.nq * 2048u, run = (unsigned)g.nq * 512u;     // both terms, both runs; one run
  unsigned char *tab = ys + (size_t)kYStages * ybytes;
  float *sinv = reinterpret_cast<float *>(tab + ybytes);
  __shared__ UpShared sh;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int unit = P.u0 + blockIdx.y, layer = unit / P.H, head = unit - layer * P.H;
  const int tiles = P.d / 64, n = g.up_steps(), classes = up_classes(g);
  const int b0 = blockIdx.x * P.per, b1 = b0 + P.per < n ? b0 + P.per : n;

  if (tid == 0) {
    for (int i = 0; i < kXStages; ++i) { mbar::init(&sh.xfull[i], 1u); mbar::init(&sh.xempty[i], 8u); }
    for (int i = 0; i < kYStages; ++i) { mbar::init(&sh.yfull[i], 1u); mbar::init(&sh.yempty[i], 1u); }
    mbar::init(&sh.tfull, 1u); mbar::init(&sh.tempty, 1u);
    for (int i = 0; i < kUpBufs; ++i) { mbar::init(&sh.afull[i], 1u); mbar::init(&sh.aempty[i], 8u); }
    mbar::init(&sh.done, 1u);
    mbar::init_done();
  }
  if (warp == 1) tmem_alloc(&sh.tmem, 128 * kUpBufs);
  for (int i = tid; i < b1 - b0; i += kUpThreads) sh.quad[i] = up_quad(g, b0 + i);
  for (int i = tid; i < 2 * P.d; i += kUpThreads) sinv[i] = P.inv[(size_t)blockIdx.y * 2 * P.d + i];
  before_sync();
  __syncthreads();
  after_sync();
  const unsigned tmem = sh.tmem;
  float sum[4] = {0.f, 0.f, 0.f, 0.f};
  double en[4] = {0.0, 0.0, 0.0, 0.0};       // hiK, totK, hiV, totV
  if (warp == 0) {
    if (lane == 0) {
      bool ok = true;
      int ntab = 0, cls = -1, ny = 0, nx = 0;
      for (int b = b0; b < b1 && ok; ++b) {
        const int c = class_of(b, n, classes), q0 = sh.quad[b - b0];
        for (int t = 0; t < tiles && ok; ++t) {
          {
            const int s = ny % kYStages;
            if (ny >= kYStages && !mbar::wait(&sh.yempty[s], (unsigned)(ny / kYStages - 1) & 1u)) { ok = false; break; }
            mbar::expect_tx(&sh.yfull[s], ybytes);
            const size_t tile = ((size_t)blockIdx.y * tiles + t) * (size_t)(g.M / 8);
            const size_t r1 = (tile + q0 / 4) * (kRows * 8), r2 = (tile + (g.M / 2 - q0 - g.nq) / 4) * (kRows * 8);
            unsigned char *dst = ys + (size_t)s * ybytes;
            load_bytes(dst, P.hi + r1, run, &sh.yfull[s]);
            load_bytes(dst + run, P.hi + r2, run, &sh.yfull[s]);
            load_bytes(dst + 2 * run, P.lo + r1, run, &sh.yfull[s]);
            load_bytes(dst + 3 * run, P.lo + r2, run, &sh.yfull[s]);
            ++ny;
          }
          if (c != cls) {
            cls = c;
            if (ntab >= 1 && !mbar::wait(&sh.tempty, (unsigned)(ntab - 1) & 1u)) { ok = false; break; }
            mbar::expect_tx(&sh.tfull, ybytes);
            load_bytes(tab, reinterpret_cast<const unsigned char *>(P.table) + (size_t)c * ybytes, ybytes, &sh.tfull);
            ++ntab;
          }
          const int s = nx % kXStages;
          if (nx >= kXStages && !mbar::wait(&sh.xempty[s], (unsigned)(nx / kXStages - 1) & 1u)) { ok = false; break; }
          mbar::expect_tx(&sh.xfull[s], 8u * kBoxBytes);
          for (int hf = 0; hf < 2; ++hf) {
            const int c64 = (2 * t + hf) * 64;
            const bool isv = c64 >= P.d;
            for (int i = 0; i < 4; ++i)
              load_box(smem + (size_t)(s * 8 + hf * 4 + i) * kBoxBytes, isv ? &maps.v[layer] : &maps.k[layer],
                       isv ? c64 - P.d : c64, head, b * kRows + i * kSlotTok, &sh.xfull[s]);
          }
          ++nx;
        }
      }
      for (int i = nx > kXStages ? nx - kXStages : 0; i < nx; ++i) ok &= mbar::wait(&sh.xfull[i % kXStages], (unsigned)(i / kXStages) & 1u);
      for (int i = ny > kYStages ? ny - kYStages : 0; i < ny; ++i) ok &= mbar::wait(&sh.yfull[i % kYStages], (unsigned)(i / kYStages) & 1u);
      if (ntab > 0) ok &= mbar::wait(&sh.tfull, (unsigned)(ntab - 1) & 1u);
      if (!ok) atomicOr(P.status, FC_DEV_FLAG_TIMEOUT);
    }
  } else if (warp == 1) {
    if (lane == 0) {
      constexpr unsigned idesc = instruction(true, false, kRows);
      bool ok = true;
      int ntab = 0, cls = -1, it = 0;
      for (int b = b0; b < b1 && ok; ++b) {
        const int c = class_of(b, n, classes);
        for (int t = 0; t < tiles; ++t, ++it) {
          if (c != cls) {
            cls = c;
            if (ntab > 0) commit(&sh.tempty);
            if (!mbar::wait(&sh.tfull, (unsigned)ntab & 1u)) { ok = false; break; }
            ++ntab;
          }
          const int s = it % kYStages, buf = it % kUpBufs;
          if (it >= kUpBufs && !mbar::wait(&sh.aempty[buf], (unsigned)(it / kUpBufs - 1) & 1u)) { ok = false; break; }
          if (!mbar::wait(&sh.yfull[s], (unsigned)(it / kYStages) & 1u)) { ok = false; break; }
          after_sync();
          const unsigned ya = smem_addr(ys) + (unsigned)s * ybytes, ta = smem_addr(tab);
          // low times high, high times low, high times high: small terms first
          for (int pr = 0; pr < 3; ++pr)
            for (int k = 0; k < g.nq / 4; ++k) {
              const unsigned off = (unsigned)k * 4096u;
              mma(tmem + (unsigned)buf * 128u, operand(ta + (pr == 0 ? 2 * run : 0u) + off, 2048, 128, 0),
                  operand(ya + (pr == 1 ? 2 * run : 0u) + off, 2048, 128, 0), idesc, pr + k > 0);
            }
          commit(&sh.yempty[s]);
          commit(&sh.afull[buf]);
        }
      }
      commit(&sh.done);
      ok &= mbar::wait(&sh.done, 0u);
      if (!ok) atomicOr(P.status, FC_DEV_FLAG_TIMEOUT);
    }
  } else {
    const int quad = warp & 3, half = (warp - 2) >> 2, row = quad * 32 + lane;
    bool failed = false;
    int it = 0;
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
        const unsigned xr = smem_addr(smem) + (unsigned)((s * 8 + half * 4) * kBoxBytes + row * 128);
        const unsigned iv = smem_addr(sinv + t * kRows + half * 64);
        const unsigned at = tmem + ((unsigned)quad << 21) + (unsigned)(buf * 128 + half * 64);
        float2 rs[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)}, xs[2] = {rs[0], rs[0]};
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          float a[16];
          tmem_ld16(at + 16 * c, a);
          uint4 xv[2];
#pragma unroll
          for (int i = 0; i < 2; ++i) xv[i] = lds(xr + (((2 * c + i) ^ (row & 7)) << 4));
          tmem_wait(a);
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const uint4 sc = lds(iv + (unsigned)(4 * c + i) * 16u);
            const unsigned w0 = i & 1 ? xv[i >> 1].z : xv[i >> 1].x, w1 = i & 1 ? xv[i >> 1].w : xv[i >> 1].y;
            const float2 xa = widen<T>(w0), xb = widen<T>(w1);
            const float2 ra = fma2(make_float2(a[4 * i], a[4 * i + 1]), make_float2(__uint_as_float(sc.x), __uint_as_float(sc.y)), xa);
            const float2 rb = fma2(make_float2(a[4 * i + 2], a[4 * i + 3]), make_float2(__uint_as_float(sc.z), __uint_as_float(sc.w)), xb);
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
      const int tok = b * kRows + row;
      const bool in = tok < g.N;
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        sum[2 * i] = in ? (r2[i][0].x + r2[i][0].y) + (r2[i][1].x + r2[i][1].y) : 0.f;
        sum[2 * i + 1] = in ? (x2[i][0].x + x2[i][0].y) + (x2[i][1].x + x2[i][1].y) : 0.f;
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) en[i] += (double)sum[i];
      float &o = sh.other[(b - b0) & 1][row];
      if (half == 1) o = sum[0] + sum[2];
      asm volatile("bar.sync 1, 256;\n" ::: "memory");
      if (half == 0 && in)
        P.scores[layer][(long long)head * P.score_stride + tok] = (sum[0] + sum[2] + o) * (1.f / (float)P.d);
    }
    if (failed && lane == 0) atomicOr(P.status, FC_DEV_FLAG_TIMEOUT);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const double v = warp_sum_d(en[i]);
      if (lane == 0) sh.red[warp - 2][i] = v;
    }
  }
  before_sync();
  __syncthreads();
  if (warp == 1) tmem_free(tmem, 128 * kUpBufs);
  // energies: this block's sums, then, in the block of the layer that comes last, all of them in order
  if (tid < 4) {
    double v = 0.0;
    for (int w = 0; w < 8; ++w) v += sh.red[w][tid];
    P.part[((size_t)unit * P.ranges + blockIdx.x) * 4 + tid] = v;
    __threadfence();
  }
  __syncthreads();
  if (tid == 0) {
    __threadfence();
    const unsigned all = (unsigned)(P.H * P.ranges);
    sh.last = atomicAdd(P.done + layer, 1u) + 1u == all;
    if (sh.last) P.done[layer] = 0u;
    __threadfence();
  }
  __syncthreads();
  if (sh.last && warp < 4) {
    const double *p = P.part + (size_t)layer * P.H * P.ranges * 4;
    double v = 0.0;
    for (int i = lane; i < P.H * P.ranges; i += 32) v += __ldcg(p + 4 * (size_t)i + warp);
    v = warp_sum_d(v);
    if (lane == 0) P.energy[(long long)layer * P.energy_stride + warp] = v;
  }
}

}  // namespace band
