// Host/device shared structures of the propagation library.
//
// Every launch receives its parameters by value (a PassParams of a few KB in the
// kernel parameter space), so a call needs no host-to-device copies and stays
// capturable in a CUDA graph once its tables exist.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <string>

#include "../../include/top.h"

namespace top {

constexpr int kMaxSets = 24;      // distinct (lambda, z) parameter sets per launch
constexpr int kMaxFields = 2048;  // fields per launch (larger batches run in chunks)

// One (lambda, z) parameter set: the transfer function and the lens factors, computed in
// float64 and rounded to float32. H depends on the frequencies only through fx^2 and fy^2, so
// one quadrant is stored: hq[|kx| (My + 2) + j] = H(|kx|, |ky|) / (Py Px) for |kx| <= Px / 2,
// with the even |ky| = 2 k (k <= My/2) in the first My/2 + 1 entries, the odd |ky| = 2 k + 1
// (k < My/2) after them and one zero entry (one row per |kx|; a column half reads the even or the
// odd part of its row). Within a part, k sits where the column plan's lanes hold the bin: k =
// kbase(b) + S j at b + S j (S = My / RL; the identity for two-stage plans).
struct FieldSet {
  const float2* hq;      // [Px/2 + 1][My + 2]
  const float2* src_lx;  // lens factor tables of the source-side modulation: [nx], [ny]
  const float2* src_ly;
  const float2* epi_lx;  // lens factor tables of the epilogue-side modulation
  const float2* epi_ly;
};

// Element modulation (Eq. 1) applied in a prologue or epilogue.
struct ModDev {
  uint32_t flags;          // TOP_MOD_*
  int conj;                // apply conj(M)
  const float2* cmask;     // complex mask
  const float* amp;        // amplitude
  const float* phase;      // phase
  long long stride;        // elements between consecutive fields' masks (0 = shared)
  const int2* circ;        // [ny] inclusive x range inside the aperture per row (x > y: empty)
};

enum SrcKind : int {
  SRC_FIELD = 0,      // v = modsrc * in[f]
  SRC_INTENSITY = 1,  // v = modsrc * 2 w_f gI[f / group] psi[f]
};

enum EpiKind : int {
  EPI_FIELD = 0,      // out[f] = modepi * v
  EPI_INTENSITY = 1,  // I[g] += w_f |modepi * v|^2 over the group; optional out[f] = modepi * v
  EPI_MODGRAD = 2,    // gradient of a modulation y = M x: grad_in = conj(M) v, grads of M (partials)
  EPI_OVERLAP = 3,    // per row tile: sums of psi conj(phi) and |psi|^2, psi = modepi * v (Eq. 7); optional out[f]
};

struct PassParams {
  // geometry of the padded problem
  int ny, nx;      // field samples
  int Py, Px;      // padded sizes (even; each handled as two interleaved halves)
  int My, Mx;      // Py / 2, Px / 2
  int oy, ox;      // offset of the field in the padded grid
  int ci;          // workspace lines interleaved (1 or 2, of the row plan)
  int xr0, xr1, xstep;  // row plan: line b + xstep j of a half holds bin b / xr1 + (b % xr1) xr0 + xstep j
  int nfields;     // fields in this launch
  int group;       // fields per epilogue group (R2 grid.y = ceil(nfields / group))
  int src_group;   // fields sharing one intensity-gradient plane (SRC_INTENSITY)
  int in_repeat;   // SRC_FIELD: output field f reads input field f / in_repeat
  int method;      // top_method
  int adjoint;     // use conj(H)
  int src_kind;
  int epi_kind;
  int l2_ahead;    // blocks ahead whose input a block prefetches into L2 (0: none)
  uint32_t tune_rows;  // TOP_TUNE_* choices for the row passes (of Mx) and the column pass (of My)
  uint32_t tune_cols;

  // buffers (element strides per field)
  const float2* in;   long long in_stride;
  // ragged batches: per-field device pointers (device arrays of nfields entries) that replace
  // in + f * in_stride and out + f * out_stride when non-null
  const float2* const* in_list;
  float2* const* out_list;
  // per-field transfer-function tables (device array of nfields entries) that replace
  // sets[set_of[f]].hq in the column pass when non-null (ragged batches: no limit on the sets)
  const float2* const* hq_list;
  float2* ws;         long long ws_stride;   // pass workspace [field][Px][ny]
  float2* out;        long long out_stride;
  float* outf;        long long outf_stride; // intensity output per group / partial sums per group
  const float2* psi;  long long psi_stride;  // saved output field (SRC_INTENSITY)
  const float2* xs;   long long xs_stride;   // saved input x of the modulation (EPI_MODGRAD, modulate backward)
  const float* gI;    long long gI_stride;   // intensity gradient per group (SRC_INTENSITY)
  const float* weights;                      // per field or null
  float* part_phase;  float* part_amp;  float2* part_mask;  long long part_stride;  // EPI_MODGRAD partials per group
  int part_accumulate;                       // add to the partials instead of overwriting (later chunks)

  // engine tables
  const float2* twx;  // stage twiddles of the x engine
  const float2* twy;
  const float2* wpx;  // exp(-2 pi i p / Px), p < Mx
  const float2* wpy;

  // EPI_OVERLAP: target phi (+ f * target_stride) and float64 partial sums [field][row tile][3]
  // (re and im of sum psi conj(phi), sum |psi|^2)
  const float2* target; long long target_stride;
  double* ov_part;
  // shared sources (input_repeat): the column pass stores the forward spectrum of every column in
  // its register order (spec_out, one spectrum per launch field), or starts from the spectrum of
  // field f / in_repeat (spec_in) instead of loading, folding and transforming its columns.
  // Spectrum of field s, column kpos, half r, slot e, lane t at ((s Px + kpos) 2 + r) M + e G + t.
  float2* spec_out;
  const float2* spec_in;
  // column pass as the second half of a forward 2-D transform: bins of columns kx <= Px/2 go to
  // this quadrant table (FieldSet::hq layout) times hq_scale, nothing else is written
  float2* hq_out;
  float hq_scale;

  ModDev msrc;  // modulation applied to the R1 source
  ModDev mepi;  // modulation applied in the R2 epilogue

  int* fault;  // host-mapped word set when a bounded wait of a kernel runs out (may be null)

  int nsets;
  FieldSet sets[kMaxSets];
  unsigned char set_of[kMaxFields];
};

// Line transforms of any length P by Bluestein's chirp-z method (padded sizes without a plan of
// their own): with c[n] = exp(-i pi n^2 / P), the DFT is X[k] = c[k] sum_n (x[n] c[n]) conj(c[k - n]),
// a convolution done as an L-point FFT (L >= 2P - 1), a product with the transform of the chirp
// (in bins) and an inverse L-point FFT; the inverse DFT uses the conjugate chirps.
enum CztMode : int {
  CZT_FWD = 0,     // forward DFT of the zero-padded line
  CZT_INV = 1,     // inverse DFT (unnormalised), then the output window
  CZT_FILTER = 2,  // forward DFT, times the transfer function (conjugated for the adjoint), inverse DFT, window
};

constexpr int kFewTables = 16;

struct CztParams {
  const float2* in;      // line i of field f at in + (f / in_repeat) in_fstride + i in_lstride
  long long in_fstride;
  long long in_lstride;
  int in_repeat;
  float2* out;           // window sample k - k0 of line i of field f at out + f out_fstride + i out_lstride
  long long out_fstride;
  long long out_lstride;
  int nlines, nfields;
  int P;                 // DFT length
  int n_in, off_in;      // the line's samples sit at [off_in, off_in + n_in) of the zero-padded line
  int k0, n_out;         // output window
  int mode;              // CztMode
  int adjoint;
  float inv_l;           // 1 / L, L the convolution length
  const float2* chirp;   // c[n], n < P
  // L-point transforms of conj(c) (forward) and c (inverse) on the lags (-P, P), entry e G + t = the
  // bin lane t of the transforming engine holds in slot e; for L = 8192 split by parity (half r,
  // bins 2k + r, at r L/2, on the 4096-point engine)
  const float2* bh_fwd;
  const float2* bh_inv;
  const float2* tw;      // stage twiddles of the transforming engine
  const float2* wsplit;  // L = 8192: exp(-2 pi i p / L), p < L/2
  // CZT_FILTER: rows [line][P] of H / (Py Px) in natural order, field f's at h[f], or without a list in device
  // memory at h_few[f h_step] (h_step 0: one table for all). The list is written by a launch of its own, which
  // the calls with one table, or with few fields, go without (one field of 1021 x 1021: 2 us less; 2048 of
  // 16 x 16: 8 us).
  const float2* const* h;
  int h_step;
  const float2* h_few[kFewTables];
};

// The workspace as a tensor for tile copies: [fields][lines][samples] of complex64, in boxes of
// box_lines lines x 4 samples (a tile) and x 16 samples (four tiles, 128 bytes a line, for prefetches).
// Strides in samples; a line is a whole number of 16-byte units.
struct TileMap {
  CUtensorMap tile;
  CUtensorMap wide;
};
cudaError_t encode_tile_map(TileMap* map, const void* ws, long long samples, long long lines, int nfields,
                            long long field_stride, int box_lines, bool with_wide);

// The autotune table (top_tune.cu): TOP_TUNE_* flags per line length M (0: the defaults).
uint32_t tune_flags(int M);
bool tune_flags_valid(uint32_t flags);
void tune_set(int M, uint32_t flags);
void tune_clear();
bool tune_save(const char* path, std::string* err);
bool tune_load(const char* path, std::string* err);
// Kernel launch timing kinds (instrumentation)
enum KernelKind : int { KK_ROWS_FWD = 0, KK_COLS, KK_ROWS_INV, KK_AUX, KK_ROWS_CHAIN, KK_ONCHIP, KK_COUNT };

}  // namespace top
