// Host side of scoring in the kept band (fc_band.cuh).
#include "fc_band.h"
#include "fc_band.cuh"

#include <math.h>
#include <mutex>
#include <new>
#include <type_traits>

namespace {

using band::Geometry;

// Kernels phi for bands up to fmax cycles per grid point: the shortest whose response folds less than 6e-8 of the band's
// own gain onto the band while that gain varies little over it (found by scanning beta and fc; max / min, rms of max /
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

bool eligible(const fc_kv_view *kv, int N) {
  return kv->dtype != FC_F32 && N >= 1024 && N <= 65536 && kv->head_dim <= 512;
}

// The coarsest grid on which the band fits: N/4 <= M <= N/2 and omega <= 0.8 M.
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
  for (int i = 0; i < band::kCheb; ++i) g->cheb[i] = responses()[k][i];
  g->same = N == 2 * M || N == 4 * M;                      // 128 tokens are whole quads of the grid
  g->ks = 0;
  for (int b = 0; b < g->down_steps(); ++b) {
    const int s = (band::down_end(*g, b) - band::down_start(*g, b) + 15) / 16;
    if (s > g->ks) g->ks = s;
  }
  if (g->ks < 4) g->ks = 4;
  g->nq = g->M / 4;                                        // no clamping at the end while the extent is measured
  int need = 8;
  for (int b = 0; b < g->up_steps(); ++b) {
    const long long j = band::ceil_div((2ll * band::kRows * b + 1) * M - (1ll + g->W) * N, 2ll * N);
    const int q = j <= 0 ? 0 : (int)(j >> 2) & ~3;
    const int e = band::up_quad_end(*g, b) - q;
    if (e > need) need = e;
  }
  g->nq = (need + 7) / 8 * 8;
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
  size_t y_bytes, plane_bytes;               // of one unit
  band::Maps maps;
};

static int mid_tw_len(int Mh) {
#define X(M_, A_, B_, C_, D_) if (Mh == M_) return band::MidShape<A_, B_, C_, D_>::tw_len;
  FC_MID_SHAPES(X)
#undef X
  return 0;
}

bool fc_band_bounds(const fc_kv_view *kv, int N, FcBandSizes *s) {
  if (!eligible(kv, N)) return false;
  // M <= N/2, windows at their largest, every step with matrices of its own
  const int M = N / 2 < kMaxGrid ? N / 2 : kMaxGrid;
  s->tables = align256((size_t)(M / band::kJ) * band::kMaxSteps * 2 * 48 * 16) +
              align256((size_t)((N + band::kRows - 1) / band::kRows) * band::kMaxQuads * 2048) + align256((size_t)M * 32) +
              align256((size_t)M * 6 * sizeof(float2));
  s->unit = (size_t)2 * kv->head_dim * M * 8 + align256((size_t)2 * kv->head_dim * 4) + 1024;
  s->steps = (N + band::kRows - 1) / band::kRows;
  return true;
}

bool fc_band_takes(const fc_kv_view *kv, int N, int omega) {
  Geometry g;
  return eligible(kv, N) && make_geometry(N, omega, &g);
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
  const int nr = band::filter_terms(j->f16) * band::kJ;
  j->off_up = align256(band::down_classes(g) * band::down_image(g, nr));
  j->off_mid = j->off_up + align256(band::up_classes(g) * band::up_image(g));
  j->table_bytes = j->off_mid + align256((size_t)g.M / 2 * 16) + align256((size_t)mid_tw_len(g.M / 2) * sizeof(float2));
  j->y_bytes = (size_t)2 * j->d * g.M * sizeof(float);
  j->plane_bytes = (size_t)2 * j->d * g.M * sizeof(__half);
  return j;
}
void fc_band_release(FcBandJob *j) { delete j; }

// values before the transform, two planes after it, a scale per row
static size_t unit_bytes(const FcBandJob *j) { return j->y_bytes + 2 * j->plane_bytes + align256((size_t)2 * j->d * 4); }

static size_t budget(const fc_handle *h) { return h->group_bytes > ((size_t)1 << 60) ? h->group_bytes : h->group_bytes / 2 * 3; }

size_t fc_band_buffer_bytes(const fc_handle *h, const FcBandSizes *s, int units) {
  const size_t all = s->unit * units, most = budget(h);
  return all < most ? all : s->unit > most ? s->unit : most;
}

int fc_band_units(const fc_handle *h, const FcBandJob *j, int units, size_t buf_bytes) {
  int nu = (int)(buf_bytes / unit_bytes(j));
  if (nu > units) nu = units;
  if (nu < 1) nu = 1;
  int groups = (units + nu - 1) / nu;
  if (groups < h->num_aux && units >= h->num_aux) groups = h->num_aux;
  return (units + groups - 1) / groups;
}

int fc_band_ranges(const FcBandJob *j, int units) {
  const int n = j->g.up_steps();
  int r = (148 + units - 1) / units;
  if (r > n) r = n;
  const int floor_r = (n + band::kMaxPer - 1) / band::kMaxPer;
  if (r < floor_r) r = floor_r;
  const int per = (n + r - 1) / r;
  return (n + per - 1) / per;
}

fc_status fc_band_tables(fc_handle *h, cudaStream_t st, const FcBandJob *j, char *tables) {
  const Geometry &g = j->g;
  fc_status s;
  if (j->f16) band::k_down_table<__half, 2><<<band::down_classes(g), 256, 0, st>>>(g, reinterpret_cast<__half *>(tables));
  else band::k_down_table<__nv_bfloat16, 3><<<band::down_classes(g), 256, 0, st>>>(g, reinterpret_cast<__nv_bfloat16 *>(tables));
  if ((s = fc_after_launch(h)) != FC_OK) return s;
  band::k_up_table<<<band::up_classes(g), 256, 0, st>>>(g, reinterpret_cast<__half *>(tables + j->off_up));
  if ((s = fc_after_launch(h)) != FC_OK) return s;
  const int Mh = g.M / 2;
  char *m = tables + j->off_mid;
  const band::MidTables t = {reinterpret_cast<float4 *>(m), reinterpret_cast<float4 *>(m) + Mh / 2,
                             reinterpret_cast<float2 *>(m + align256((size_t)Mh * 16))};
#define X(M_, A_, B_, C_, D_) \
  if (Mh == M_) band::k_mid_table<band::MidShape<A_, B_, C_, D_>><<<(Mh / 2 + 63) / 64, 64, 0, st>>>(g, t);
  FC_MID_SHAPES(X)
#undef X
  return fc_after_launch(h);
}

fc_status fc_band_bind(fc_handle *h, FcBandJob *j, const fc_kv_view *kv, const FcBandLaunch &l) {
  (void)h;
  EncodeTiledFn fn = encode_fn();
  if (!fn) return FC_ERR_CUDA;
  const CUtensorMapDataType dt = j->f16 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16;
  const cuuint64_t dims[3] = {(cuuint64_t)j->d, (cuuint64_t)j->H, (cuuint64_t)j->g.N};
  const cuuint64_t str[2] = {(cuuint64_t)kv->stride_head * 2, (cuuint64_t)kv->stride_token * 2};
  const cuuint32_t box[3] = {64, 1, (cuuint32_t)band::kSlotTok}, ones[3] = {1, 1, 1};
  for (int i = 0; i < l.layers; ++i)
    for (int v = 0; v < 2; ++v) {
      const CUresult r = fn(v ? &j->maps.v[i] : &j->maps.k[i], dt, 3, const_cast<void *>(v ? l.v[i] : l.k[i]), dims, str, box,
                            ones, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                            CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
      if (r != CUDA_SUCCESS) return FC_ERR_INTERNAL;
    }
  return FC_OK;
}

template <class S>
static fc_status launch_mid(fc_handle *h, cudaStream_t st, int rows, const band::MidParams &P) {
  fc_status s = allow_smem<band::k_mid<S>>(h->device, S::smem, 70);
  if (s != FC_OK) return s;
  ProfScope ps(h, FC_K_PASS2, st);
  band::k_mid<S><<<rows / S::ROWS, S::NT, S::smem, st>>>(P);
  return fc_after_launch(h);
}

template <typename T>
static fc_status run_group(fc_handle *h, cudaStream_t st, const FcBandJob *j, const FcBandLaunch &l, int u0, int nu, int ranges,
                           char *buf) {
  const Geometry &g = j->g;
  constexpr int TERMS = std::is_same<T, __half>::value ? 2 : 3;
  fc_status s;
  float *y = reinterpret_cast<float *>(buf);
  __half *hi = reinterpret_cast<__half *>(buf + nu * j->y_bytes), *lo = hi + nu * (j->plane_bytes / 2);
  float *inv = reinterpret_cast<float *>(buf + nu * (j->y_bytes + 2 * j->plane_bytes));
  const int tiles = j->d / 64, pairs = (tiles + 1) / 2, n = g.down_steps();
  {
    band::DownParams P = {l.tables, y, h->status_word, j->H, j->d, u0, 0};
    int r = (148 + nu * pairs - 1) / (nu * pairs);
    if (r > n) r = n;
    P.per = (n + r - 1) / r;
    if (P.per > band::kMaxPer) P.per = band::kMaxPer;
    if ((s = allow_smem<band::k_down<T, TERMS>>(h->device, band::kDownSmem, cudaSharedmemCarveoutMaxShared)) != FC_OK) return s;
    ProfScope ps(h, FC_K_PASS1, st);
    band::k_down<T, TERMS><<<dim3((n + P.per - 1) / P.per, pairs, nu), band::kDownThreads, band::kDownSmem, st>>>(j->maps, g, P);
    if ((s = fc_after_launch(h)) != FC_OK) return s;
  }
  {
    const int Mh = g.M / 2;
    char *m = const_cast<char *>(l.tables) + j->off_mid;
    const band::MidParams P = {y, hi, lo, inv, {reinterpret_cast<float4 *>(m), reinterpret_cast<float4 *>(m) + Mh / 2,
                               reinterpret_cast<float2 *>(m + align256((size_t)Mh * 16))}};
    s = FC_ERR_INTERNAL;
#define X(M_, A_, B_, C_, D_) if (Mh == M_) s = launch_mid<band::MidShape<A_, B_, C_, D_>>(h, st, nu * 2 * j->d, P);
    FC_MID_SHAPES(X)
#undef X
    if (s != FC_OK) return s;
  }
  {
    band::UpParams P = {};
    P.table = reinterpret_cast<const __half *>(l.tables + j->off_up);
    P.hi = hi;
    P.lo = lo;
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
    const size_t sm = band::up_smem(g.nq, j->d);
    if ((s = allow_smem<band::k_up<T>>(h->device, sm, cudaSharedmemCarveoutMaxShared)) != FC_OK) return s;
    ProfScope ps(h, FC_K_PASS3, st);
    band::k_up<T><<<dim3(ranges, nu), band::kUpThreads, sm, st>>>(j->maps, g, P);
    return fc_after_launch(h);
  }
}

fc_status fc_band_group(fc_handle *h, cudaStream_t st, const FcBandJob *j, const FcBandLaunch &l, int u0, int nu, int ranges, char *buf) {
  return j->f16 ? run_group<__half>(h, st, j, l, u0, nu, ranges, buf) : run_group<__nv_bfloat16>(h, st, j, l, u0, nu, ranges, buf);
}
