// Scoring in the kept band (fc_band.cuh): what the scoring calls use of it.
#pragma once
#include "fc_common.cuh"

struct FcBandSizes {
  size_t tables, unit;     // bytes: one sequence's tables, one unit's (layer, head) intermediates
  int steps;               // 128-token steps of a sequence
};
// Upper bounds over all cutoffs for a sequence of N tokens; false: no cutoff takes this form.
bool fc_band_bounds(const fc_kv_view *kv, int N, FcBandSizes *s);
// Intermediates of one launch group, one copy per internal stream, of a call with so many units.
size_t fc_band_buffer_bytes(const fc_handle *h, const FcBandSizes *s, int units);

// The grid's points where a cutoff takes this form, 0 where it does not.
int fc_band_grid(const fc_kv_view *kv, int N, int omega);

// One sequence of a chunk of layers.
struct FcBandJob;
// nullptr where the other forms are used.  Freed with fc_band_release.
FcBandJob *fc_band_plan(const fc_handle *h, const fc_kv_view *kv, int N, int omega);
void fc_band_release(FcBandJob *j);
int fc_band_units(const fc_handle *h, const FcBandJob *j, int units, size_t buf_bytes);   // units per launch
int fc_band_ranges(const fc_handle *h, const FcBandJob *j, int units);      // blocks a unit's rows are spread over where a launch has so many units
// The sequence's tables: their size, what they depend on (the dtype, the length and the cutoff), and the launch that builds
// them on `st`.
long long fc_band_table_key(const FcBandJob *j);
// Tables the handle keeps: the place of the sequence's (-1: none), and a place for new ones, for which the longest unused
// that are not in `used` make room (-1: there is none).  The caller sets the place's key once the tables are on their way.
int fc_band_kept(fc_handle *h, const FcBandJob *j);
int fc_band_place(fc_handle *h, const FcBandJob *j, const bool (&used)[FC_BAND_KEPT]);
fc_status fc_band_tables(fc_handle *h, cudaStream_t st, const FcBandJob *j, char *tables);
struct FcBandLaunch {
  const void *const *k, *const *v;     // first token of the sequence, layer by layer
  float *const *scores;
  int layers;
  const char *tables;
  double *part, *energy;
  unsigned *done;
  long long score_stride, energy_stride;
};
// Tensor maps of the layers' rows; the launches of fc_band_group use them until the next call.
fc_status fc_band_bind(fc_handle *h, FcBandJob *j, const fc_kv_view *kv, const FcBandLaunch &l);
// Units [u0, u0 + nu) on `st`, intermediates at `buf`, laid out for `cap` units.  `early`: kernels are
// set up while the one in front ends (where the launch group has its stream to itself).
fc_status fc_band_group(fc_handle *h, cudaStream_t st, const FcBandJob *j, const FcBandLaunch &l, int u0, int nu, int cap, int ranges,
                        bool early, char *buf);
