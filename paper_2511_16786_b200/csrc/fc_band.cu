// Host side of scoring in the kept band (fc_band.cuh).
#include "fc_band.h"
#include "fc_band.cuh"

#include <math.h>
#include <mutex>
#include <new>
#include <type_traits>
#include <utility>

namespace {

using band::Geometry;

// Kernels phi for bands up to fmax cycles per grid point: the shortest whose response folds less than 6e-8 of the band's
// own gain onto the band while that gain varies little over it (a sinc times the "exponential of semicircle" of Barnett,
// Magland and af Klinteberg, SIAM J. Sci. Comput. 41, 2019; found by scanning beta and fc; max / min, rms of max /
// gain in the band, largest folded part):
//   0.40  24  3.4  1.53  5.1e-8     0.36  20  1.8  1.15  2.5e-8     0.32  16  1.55  1.12  5.5e-8
//   0.28  14  1.3  1.06  5.3e-8     0.25  14  1.06 1.01  5.6e-8     0.20  12  1.06  1.01  2.4e-8
struct Kernel { double fmax; int W; double beta, fc; };
constexpr Kernel kKernels[] = {{0.20, 12, 16.0, 0.37}, {0.25, 14, 15.5, 0.39}, {0.28, 14, 15.5, 0.35},
                               {0.32, 16, 15.5, 0.35}, {0.36, 20, 16.0, 0.37}, {0.40, 24, 17.0, 0.37}};
constexpr int kNumKernels = sizeof(kKernels) / sizeof(kKernels[0]);

// Expansions of the kernels' responses, computed once.
const double (*responses())[band::kCheb] {
  static double cheb[kNumKernels][band::kCheb];
  static const bool ready = [] {
    const double pi = 3.14159265358979323846;
    for (int k = 0; k < kNumKernels; ++k) {
      const Kernel &q = kKernels[k];
      constexpr int per = 8;                                  // samples per grid point: phi folds nothing at that rate
      double h[band::kCheb];
      for (int i = 0; i < band::kCheb; ++i) {
        const double y = cos(pi * (i + 0.5) / band::kCheb), f = q.fmax * sqrt(0.5 * (y + 1.0));
        double s = 0.0;
        for (int n = 0; n <= q.W / 2 * per; ++n) {
          const double u = (double)n / per, r = 1.0 - (2.0 * u / q.W) * (2.0 * u / q.W), a = 2.0 * q.fc * u;
          const double p = 2.0 * q.fc * exp(q.beta * (sqrt(r > 0.0 ? r : 0.0) - 1.0)) * (n == 0 ? 1.0 : sin(pi * a) / (pi * a));
          s += (n == 0 ? 1.0 : n == q.W / 2 * per ? 1.0 : 2.0) * p * cos(2.0 * pi * f * u);
        }
        h[i] = s / per;
      }
      for (int c = 0; c < band::kCheb; ++c) {
        double s = 0.0;
        for (int i = 0; i < band::kCheb; ++i) s += h[i] * cos(pi * c * (i + 0.5) / band::kCheb);
        cheb[k][c] = s * (c == 0 ? 1.0 : 2.0) / band::kCheb;
      }
    }
    return true;
  }();
  (void)ready;
  return cheb;
}

constexpr int kMinGrid = 256, kMaxGrid = 16384;

// 16-bit rows are exact operands of the products (fp32 rows would need six of them and terms of their own).  Up to 512 tokens
// and at 1024 one kernel does it all, and a single layer of 4 heads takes 29..33 us there against 44 here when the form was new
// (28 layers: 145 and 182 against 72 and 95, but a score must not depend on how many layers share a call).  One layer of 4 heads of
// 517 / 1025 / 2048 / 4096 tokens, calls in a row: three passes 32 / 30 / 25 / 32 us, this form 23 / 29 / 29 / 31; 28 layers 150 / 277 /
// 255 / 484 against 112 / 120 / 131 / 247.  2048 is the one length where a single layer loses, and 28 layers gain twice.
bool eligible(const fc_kv_view *kv, int N) {
  return kv->dtype != FC_F32 && N > 512 && N != 1024 && N <= 65536 && kv->head_dim <= 512;
}

// The coarsest grid on which the band fits: M a power of two, N/4 <= M <= N/2 and omega <= 0.8 M (a quarter more grid than the
// band needs: the kernel's support grows without bound as that margin closes), with windows that fit the rings (N just above 2 M
// with the widest kernels has longer ones).  At powers of two that is a cutoff of up to two fifths, at others as little as 0.2;
// of lengths spread evenly over their logarithm 0.83 at cutoffs of 0.2 .. 0.25, 0.53 at 0.25 .. 0.3, 0.25 at 0.3 .. 0.35 take
// it.  Where M would pass N/2 little is saved and the passes stay.
bool make_geometry(int N, int omega, Geometry *g) {
  int M = kMinGrid;
  while (4ll * M < N || 5ll * omega > 4ll * M) M <<= 1;
  if (M > kMaxGrid || 2 * M > N) return false;
  const double edge = omega / (2.0 * M);
  int k = 0;
  while (k < kNumKernels - 1 && edge > kKernels[k].fmax) ++k;
  *g = Geometry{};
  g->N = N;
  g->M = M;
  g->W = kKernels[k].W;
  g->omega = omega;
  g->beta = kKernels[k].beta;
  g->fc = kKernels[k].fc;
  g->fmax = kKernels[k].fmax;
  g->up_ratio = (double)M / N;
  g->down_ratio = (double)N / M;
  for (int i = 0; i < band::kCheb; ++i) g->cheb[i] = responses()[k][i];
  g->same = N == 2 * M || N == 4 * M;                      // 128 tokens are whole quads of the grid
  // The longest windows, over all steps or, where most are alike, over the first and last few and one between.
  auto over = [&](int n, auto f) {
    for (int b = 0; b < n; ++b) {
      if (g->same && b == 4 && n > 8) b = n - 4;
      f(b);
    }
  };
  // floors of (a + i*d) / m for i = 0, 1, ..: one division, not one per step
  struct Line {
    long long q, r, dq, dr, m;
    Line(long long a, long long d, long long m_) : q(band::floor_div(a, m_)), r(a - q * m_), dq(d / m_), dr(d % m_), m(m_) {}
    void step() { q += dq; r += dr; if (r >= m) { r -= m; ++q; } }
  };
  int ks = 4, need = 8;
  const auto down = [&](long long lo, long long hi) {            // window [lo, hi] before it is cut to the sequence
    const int s = lo <= 0 ? 0 : (int)lo & ~15, e = hi + 1 > N ? N : (int)hi + 1, k = (e - s + 15) / 16;
    if (k > ks) ks = k;
  };
  const auto up = [&](long long lo, long long hi) {
    const int q = lo <= 0 ? 0 : (int)(lo >> 2) & ~3, e = (int)((hi > M - 1 ? M - 1 : hi) >> 2) + 1;
    if (e - q > need) need = e - q;
  };
  if (g->same) {
    over(g->down_steps(), [&](int b) {
      down(band::ceil_div((2ll * band::kJ * b + 1 - g->W) * N - M, 2ll * M),
           band::floor_div((2ll * (band::kJ * b + band::kJ - 1) + 1 + g->W) * N - M, 2ll * M));
    });
    over(g->up_steps(), [&](int b) {
      up(band::ceil_div((2ll * band::kRows * b + 1) * M - (1ll + g->W) * N, 2ll * N),
         band::floor_div((2ll * (band::kRows * b + band::kRows - 1) + 1) * M + (g->W - 1ll) * N, 2ll * N));
    });
  } else {
    Line dl((1ll - g->W) * N - M + 2ll * M - 1, 2ll * band::kJ * N, 2ll * M);
    Line dh((2ll * (band::kJ - 1) + 1 + g->W) * N - M, 2ll * band::kJ * N, 2ll * M);
    for (int b = 0; b < g->down_steps(); ++b, dl.step(), dh.step()) down(dl.q, dh.q);
    Line ul(M - (1ll + g->W) * N + 2ll * N - 1, 2ll * band::kRows * M, 2ll * N);
    Line uh((2ll * (band::kRows - 1) + 1) * M + (g->W - 1ll) * N, 2ll * band::kRows * M, 2ll * N);
    for (int b = 0; b < g->up_steps(); ++b, ul.step(), uh.step()) up(ul.q, uh.q);
  }
  g->ks = ks;
  g->nq = need <= 16 ? 16 : (need + 7) / 8 * 8;            // 16 or 24: a step of 128 tokens spans at least 44 grid points
  return g->ks <= band::kMaxSteps && g->nq <= band::kMaxQuads && g->nq <= g->M / 4;
}

// Mh and the radices of its stages
#define FC_MID_SHAPES(X)                                                                                          \
  X(128, 16, 8, 1, 1) X(256, 16, 16, 1, 1) X(512, 8, 8, 8, 1) X(1024, 16, 8, 8, 1) X(2048, 16, 16, 8, 1)          \
  X(4096, 16, 16, 16, 1) X(8192, 16, 8, 8, 8)

size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
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

// Function attributes, once per kernel and device.
template <auto kern>
fc_status allow_smem(int device, size_t bytes, int carveout) {
  static std::mutex mu;
  static size_t done[64];
  std::lock_guard<std::mutex> lock(mu);
  if (device < 64 && done[device] >= bytes) return FC_OK;
  if (bytes > 48 * 1024) FC_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes));
  FC_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, carveout));
  if (device < 64) done[device] = bytes;
  return FC_OK;
}

}  // namespace

struct FcBandJob {
  Geometry g;
  bool f16;
  int H, d;
  size_t off_up, off_mid, table_bytes;       // k_down's matrices first
  size_t y_bytes;                            // grid values of one unit
  band::Maps maps;
};

static int mid_tw_len(int Mh) {
#define X(M_, A_, B_, C_, D_) if (Mh == M_) return band::MidShape<A_, B_, C_, D_>::tw_len;
  FC_MID_SHAPES(X)
#undef X
  return 0;
}

// What the tables of a sequence take: k_down's matrices, k_up's, and what k_mid looks up.
static size_t table_bytes(const Geometry &g, size_t *off_up, size_t *off_mid) {
  *off_up = align256(band::down_classes(g) * band::down_image(g));
  *off_mid = *off_up + align256(band::up_classes(g) * band::up_image(g));
  return *off_mid + align256((size_t)g.M / 2 * 16) + align256((size_t)mid_tw_len(g.M / 2) * sizeof(float2));
}

bool fc_band_bounds(const fc_kv_view *kv, int N, FcBandSizes *s) {
  if (!eligible(kv, N)) return false;
  *s = FcBandSizes{};
  s->steps = (N + band::kRows - 1) / band::kRows;
  // the grids make_geometry may choose (two where N is a power of two, else one), with the widest kernel's windows
  for (int M = kMinGrid; M <= kMaxGrid && 2 * M <= N; M <<= 1) {
    if (4ll * M < N) continue;
    Geometry g = {};
    g.N = N;
    g.M = M;
    g.same = N == 2 * M || N == 4 * M;
    const long long span = ((band::kJ - 1ll + kKernels[kNumKernels - 1].W) * N + M - 1) / M + 16;   // tokens, from a 16th one on
    g.ks = (int)((span + 15) / 16 < band::kMaxSteps ? (span + 15) / 16 : band::kMaxSteps);
    g.nq = band::kMaxQuads;
    size_t a, b;
    const size_t tables = table_bytes(g, &a, &b), unit = (size_t)2 * kv->head_dim * M * sizeof(float) + align256((size_t)2 * kv->head_dim * 4);
    if (tables > s->tables) s->tables = tables;
    if (unit > s->unit) s->unit = unit;
  }
  return s->unit != 0;
}

int fc_band_grid(const fc_kv_view *kv, int N, int omega) {
  Geometry g;
  return eligible(kv, N) && make_geometry(N, omega, &g) ? g.M : 0;
}

FcBandJob *fc_band_plan(const fc_handle *h, const fc_kv_view *kv, int N, int omega) {
  Geometry g;
  if (h->generic_only || !eligible(kv, N) || !make_geometry(N, omega, &g)) return nullptr;
  FcBandJob *j = new (std::nothrow) FcBandJob;
  if (!j) return nullptr;
  j->g = g;
  j->f16 = kv->dtype == FC_F16;
  j->H = kv->num_heads;
  j->d = kv->head_dim;
  j->table_bytes = table_bytes(g, &j->off_up, &j->off_mid);
  j->y_bytes = (size_t)2 * j->d * g.M * sizeof(float);
  return j;
}
void fc_band_release(FcBandJob *j) { delete j; }

// grid values, in fp32 or (in the same place, after the transform) two fp16 terms, and a scale per row
static size_t unit_bytes(const FcBandJob *j) { return j->y_bytes + align256((size_t)2 * j->d * 4); }

// Launch groups.  Fuller launches beat intermediates that stay in L2, up to a point: 28 layers of 4 heads of 32768 tokens take
// 2086 / 1985 / 2015 / 1951 us with groups of up to 96 / 128 / 192 / 384 MiB, of 8192 tokens 504 / 504 / 504 / 525, 32 layers
// of 32 heads of 16384 tokens 9202 / 9050 / 9022 / 8855, and the workspace holds two of them.
// (Of the 128 MiB ones all held fifteen heads of 32768 tokens at the time, not sixteen: 2085 -> 2077 us since.)
constexpr int kGroupFactor = 4;
static size_t budget(const fc_handle *h) {
  if (h->group_bytes > ((size_t)1 << 60)) return h->group_bytes;
  const size_t values = h->group_bytes * kGroupFactor;
  return values + values / 1024;             // and the scales of the rows, so that a power of two of units fits
}

size_t fc_band_buffer_bytes(const fc_handle *h, const FcBandSizes *s, int units) {
  const size_t all = s->unit * units, most = budget(h);
  return all < most ? all : s->unit > most ? s->unit : most;
}

// Blocks a unit's n steps are spread over where a launch has so many units.
static int spread(const fc_handle *h, int n, int units) {
  int r = units < h->num_sms ? h->num_sms / units : 1;
  if (r > n) r = n;
  const int least = (n + band::kMaxPer - 1) / band::kMaxPer;
  if (r < least) r = least;
  const int per = (n + r - 1) / r;
  return (n + per - 1) / per;
}
int fc_band_ranges(const fc_handle *h, const FcBandJob *j, int units) { return spread(h, j->g.up_steps(), units); }

// Launch groups: of the unit counts that fit, the one whose steps spread most evenly over the SMs (a launch costs about
// four steps besides its own).
int fc_band_units(const fc_handle *h, const FcBandJob *j, int units, size_t buf_bytes) {
  int most = (int)(buf_bytes / unit_bytes(j)), best = 1;
  if (most > units) most = units;
  long long cost = -1;
  const int n = j->g.up_steps();
  for (int nu = 1; nu <= most; ++nu) {
    const int groups = (units + nu - 1) / nu, even = (units + groups - 1) / groups;
    if (even != nu) continue;
    const int r = fc_band_ranges(h, j, nu), per = (n + r - 1) / r, waves = (nu * r + h->num_sms - 1) / h->num_sms;
    const long long c = (long long)groups * (waves * per + 4);
    if (cost < 0 || c <= cost) { cost = c; best = nu; }
  }
  return best;
}

long long fc_band_table_key(const FcBandJob *j) { return (long long)j->g.N + ((long long)(j->g.omega + 1) << 20) + (j->f16 ? 1ll << 40 : 0); }

int fc_band_kept(fc_handle *h, const FcBandJob *j) {
  for (int i = 0; i < FC_BAND_KEPT; ++i)
    if (h->band_kept[i].key == fc_band_table_key(j)) {
      h->band_kept[i].used = ++h->band_clock;
      return i;
    }
  return -1;
}

int fc_band_place(fc_handle *h, const FcBandJob *j, const bool (&used)[FC_BAND_KEPT]) {
  auto &kept = h->band_kept;
  const size_t bytes = j->table_bytes;
  size_t held = 0;
  for (int i = 0; i < FC_BAND_KEPT; ++i)
    if (used[i]) held += kept[i].bytes;
  if (held + bytes > h->band_pool_bytes) return -1;
  for (;;) {
    int free_entry = -1, oldest = -1;
    for (int i = 0; i < FC_BAND_KEPT; ++i) {
      if (kept[i].key == 0 && !used[i]) free_entry = i;
      else if (!used[i] && (oldest < 0 || (int)(kept[i].used - kept[oldest].used) < 0)) oldest = i;
    }
    // behind one of the tables (or first) and in nobody's way
    for (int c = -1; free_entry >= 0 && c < FC_BAND_KEPT; ++c) {
      if (c >= 0 && kept[c].key == 0 && !used[c]) continue;
      const size_t off = c < 0 ? 0 : kept[c].off + kept[c].bytes;
      bool fits = off + bytes <= h->band_pool_bytes;
      for (int i = 0; i < FC_BAND_KEPT && fits; ++i)
        if (kept[i].key != 0 || used[i]) fits = off + bytes <= kept[i].off || off >= kept[i].off + kept[i].bytes;
      if (fits) {
        kept[free_entry] = {0, off, bytes, ++h->band_clock};
        return free_entry;
      }
    }
    if (oldest < 0) return -1;
    kept[oldest].key = 0;
  }
}

static band::MidTables mid_tables(const FcBandJob *j, const char *tables) {
  const int Mh = j->g.M / 2;
  char *m = const_cast<char *>(tables) + j->off_mid;
  return {reinterpret_cast<float4 *>(m), reinterpret_cast<float4 *>(m) + Mh / 2,
          reinterpret_cast<float2 *>(m + align256((size_t)Mh * 16))};
}

fc_status fc_band_tables(fc_handle *h, cudaStream_t st, const FcBandJob *j, char *tables) {
  const Geometry &g = j->g;
  const int Mh = g.M / 2, down = band::down_classes(g) * band::down_table_blocks(g), up = band::up_classes(g) * band::up_table_blocks(g);
  band::MidRadices r = {};
#define X(M_, A_, B_, C_, D_) \
  if (Mh == M_) r = band::MidRadices{{A_, C_ > 1 ? B_ : 1, D_ > 1 ? C_ : 1}, D_ > 1 ? D_ : C_ > 1 ? C_ : B_};
  FC_MID_SHAPES(X)
#undef X
  const int tw = mid_tw_len(Mh), mid = ((tw > Mh / 2 ? tw : Mh / 2) + 255) / 256;
  __half *um = reinterpret_cast<__half *>(tables + j->off_up);
  if (j->f16)
    band::k_band_tables<__half><<<down + up + mid, 256, 0, st>>>(g, r, reinterpret_cast<__half *>(tables), um,
                                                                  mid_tables(j, tables), down, up);
  else
    band::k_band_tables<__nv_bfloat16><<<down + up + mid, 256, 0, st>>>(g, r, reinterpret_cast<__nv_bfloat16 *>(tables), um,
                                                                         mid_tables(j, tables), down, up);
  return fc_after_launch(h);
}

fc_status fc_band_bind(fc_handle *h, FcBandJob *j, const fc_kv_view *kv, const FcBandLaunch &l) {
  (void)h;
  EncodeTiledFn fn = encode_fn();
  if (!fn) return FC_ERR_CUDA;
  const CUtensorMapDataType dt = j->f16 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16;
  const cuuint64_t dims[4] = {64, (cuuint64_t)j->g.N, (cuuint64_t)j->d / 64, (cuuint64_t)j->H};
  const cuuint64_t str[3] = {(cuuint64_t)kv->stride_token * 2, 128, (cuuint64_t)kv->stride_head * 2};
  const cuuint32_t box[4] = {64, (cuuint32_t)band::kSlotTok, j->d / 64 % 2 ? 1u : 2u, 1}, ones[4] = {1, 1, 1, 1};
  for (int i = 0; i < l.layers; ++i)
    for (int v = 0; v < 2; ++v) {
      const CUresult r = fn(v ? &j->maps.v[i] : &j->maps.k[i], dt, 4, const_cast<void *>(v ? l.v[i] : l.k[i]), dims, str, box,
                            ones, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                            CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
      if (r != CUDA_SUCCESS) return FC_ERR_INTERNAL;
    }
  return FC_OK;
}

// A launch that may start before the kernel in front of it has ended (`early`); the kernels wait for it where they need to.
template <class... A, class... B>
static fc_status launch(fc_handle *h, cudaStream_t st, bool early, void (*kern)(A...), dim3 grid, int threads, size_t smem, B &&...args) {
  cudaLaunchConfig_t lc = {};
  lc.gridDim = grid;
  lc.blockDim = dim3((unsigned)threads);
  lc.dynamicSmemBytes = smem;
  lc.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  lc.attrs = at;
  lc.numAttrs = early ? 1 : 0;
  if (cudaLaunchKernelEx(&lc, kern, std::forward<B>(args)...) != cudaSuccess) {
    cudaGetLastError();
    return FC_ERR_CUDA;
  }
  return fc_after_launch(h);
}

template <class S>
static fc_status launch_mid(fc_handle *h, cudaStream_t st, bool early, int rows, const band::MidParams &P) {
  fc_status s = allow_smem<band::k_mid<S>>(h->device, S::smem, 70);
  if (s != FC_OK) return s;
  ProfScope ps(h, FC_K_PASS2, st);
  return launch(h, st, early, band::k_mid<S>, dim3((unsigned)(rows / (2 * S::PAIRS))), S::NT, S::smem, P);
}

template <typename T, int NQ>
static fc_status launch_up(fc_handle *h, cudaStream_t st, bool early, const band::Maps &maps, const band::GridMaps &grid, const Geometry &g, const band::UpParams &P, int nu) {
  const size_t sm = band::up_smem(NQ, P.d);
  const fc_status s = allow_smem<band::k_up<T, NQ>>(h->device, sm, cudaSharedmemCarveoutMaxShared);
  if (s != FC_OK) return s;
  ProfScope ps(h, FC_K_PASS3, st);
  return launch(h, st, early, band::k_up<T, NQ>, dim3(P.ranges, nu), band::kUpThreads, sm, maps, grid, g, P);
}

static fc_status encode_grid(band::GridMaps *m, const void *values, int rows, int M) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return FC_ERR_CUDA;
  const cuuint64_t dims[3] = {(cuuint64_t)M, 2, (cuuint64_t)rows}, str[2] = {(cuuint64_t)M * 2, (cuuint64_t)M * 4};
  const cuuint32_t ones[3] = {1, 1, 1};
  for (int w = 0; w < 2; ++w) {
    const cuuint32_t box[3] = {w ? 32u : 16u, 1, (cuuint32_t)band::kRows};
    if (fn(w ? &m->wide : &m->narrow, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 3, const_cast<void *>(values), dims, str, box, ones,
           CU_TENSOR_MAP_INTERLEAVE_NONE, w ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_32B,
           CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
      return FC_ERR_INTERNAL;
  }
  return FC_OK;
}

template <typename T>
static fc_status run_group(fc_handle *h, cudaStream_t st, const FcBandJob *j, const FcBandLaunch &l, int u0, int nu, int cap,
                           int ranges, bool early, char *buf) {
  const Geometry &g = j->g;
  fc_status s;
  float *y = reinterpret_cast<float *>(buf);
  // the same place for every launch of a sequence, also where the last one has fewer units
  float *inv = reinterpret_cast<float *>(buf + cap * j->y_bytes);
  const int tiles = j->d / 64, pairs = (tiles + 1) / 2, n = g.down_steps();
  {
    band::DownParams P = {l.tables, y, h->status_word, j->H, j->d, u0, 0};
    const int r = spread(h, n, nu * pairs);
    P.per = (n + r - 1) / r;
    if ((s = allow_smem<band::k_down<T>>(h->device, band::kDownSmem, cudaSharedmemCarveoutMaxShared)) != FC_OK) return s;
    ProfScope ps(h, FC_K_PASS1, st);
    // never early: the caller may have put a wait for an event in front of it, and its rows may be on their way until then
    s = launch(h, st, false, band::k_down<T>, dim3(r, pairs, nu), band::kDownThreads, band::kDownSmem,
               j->maps, g, P);
    if (s != FC_OK) return s;
  }
  {
    const int Mh = g.M / 2;
    const band::MidParams P = {y, inv, mid_tables(j, l.tables)};
    s = FC_ERR_INTERNAL;
#define X(M_, A_, B_, C_, D_) if (Mh == M_) s = launch_mid<band::MidShape<A_, B_, C_, D_>>(h, st, early, nu * 2 * j->d, P);
    FC_MID_SHAPES(X)
#undef X
    if (s != FC_OK) return s;
  }
  {
    band::UpParams P = {};
    P.table = reinterpret_cast<const __half *>(l.tables + j->off_up);
    P.inv = inv;
    for (int i = 0; i < l.layers; ++i) P.scores[i] = l.scores[i];
    P.part = l.part;
    P.energy = l.energy;
    P.done = l.done;
    P.status = h->status_word;
    P.score_stride = l.score_stride;
    P.energy_stride = l.energy_stride;
    P.H = j->H;
    P.d = j->d;
    P.u0 = u0;
    P.ranges = ranges;
    P.per = (g.up_steps() + ranges - 1) / ranges;
    band::GridMaps grid;
    if ((s = encode_grid(&grid, y, nu * 2 * j->d, g.M)) != FC_OK) return s;
    return g.nq == 16 ? launch_up<T, 16>(h, st, early, j->maps, grid, g, P, nu)
                      : launch_up<T, 24>(h, st, early, j->maps, grid, g, P, nu);
  }
}

fc_status fc_band_group(fc_handle *h, cudaStream_t st, const FcBandJob *j, const FcBandLaunch &l, int u0, int nu, int cap, int ranges,
                        bool early, char *buf) {
  return j->f16 ? run_group<__half>(h, st, j, l, u0, nu, cap, ranges, early, buf)
                : run_group<__nv_bfloat16>(h, st, j, l, u0, nu, cap, ranges, early, buf);
}
