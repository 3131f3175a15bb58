// Whole propagations of 64 x 64 fields at padding 2 (128 x 128 transforms, Eq. 4 with H of Eq. 5)
// in one kernel, every intermediate in shared memory: one block of 256 threads per field, the
// fields of a launch taken in turn by a grid of two blocks per SM.
//
// A field crosses HBM twice (read once, written once: 16 n^2 bytes) instead of the 80 n^2 of the
// three passes, and each line's 128 frequencies are four threads' 32-point DFTs in registers (no
// exchanges inside a transform): quarter r holds the frequencies 4 k + r, and with the field at the
// start of the padded line (the result does not depend on where it sits)
//   X[4 k + r] = DFT32(w^(r m) (x[m] + (-i)^r x[m + 32]))[k],  w = exp(-2 pi i / 128),  m < 32,
//   y[m] = sum_r E_r[m],  y[m + 32] = sum_r i^r E_r[m],  E_r[m] = w^(-r m) IDFT32(Y_r)[m].
//   1. rows:    thread (r, y) folds row y, transforms it and stores its bins in a tile [kx][y];
//   2. columns: two rounds of 64; thread (r, kx) folds the column from the tile, transforms it,
//               multiplies by H / (Py Px) (conjugated for the adjoint) from the quadrant table staged
//               in shared memory, inverse transforms; the quarters add up through the tile;
//   3. rows:    thread (r, y) inverse transforms the bins of row y; the quarters add up into the row,
//               staged for a coalesced store.
// Bound by the FMA pipe and the shared-memory wavefronts, which 16 warps an SM (128 registers: 32
// samples a thread) overlap better than the 8 that 64 samples a thread allowed. Results agree with
// the three passes to rounding, not bit for bit.
#include "top_aux.h"
#include "top_passes.cuh"

namespace top {

namespace {

constexpr int kN = 64;                   // field side
constexpr int kP = 128;                  // padded side
constexpr int kQ = 32;                   // points of a quarter line
constexpr int kLT = kN + 1;              // tile stride (float2): [kx][y] and the [y][x] staging
constexpr int kHS = kN + 2;              // quadrant-table row (the FieldSet::hq layout)
constexpr int kLH = kHS + 1;             // staged row stride: an odd number of samples
constexpr int kHRows = kP / 2 + 1;       // |kx| = 0 .. 64
constexpr int kThreads = 4 * kN;
constexpr int kTile = kP * kLT;          // float2
constexpr size_t kSmem = sizeof(float2) * (size_t(kTile) + size_t(kHRows) * kLH);
static_assert(2 * kN * kLT <= kTile, "two [y][x] staging planes fit the tile");

// w^(r m) for the quarters' twiddles, read by whole warps at one r. One copy of the code serves all quarters:
// a copy for each, with its twiddles as constants, did not fit the instruction cache (85 ns a field against 62).
struct QuarterTable {
  float2 w[4][kQ];
};
constexpr QuarterTable quarter_table() {
  QuarterTable t{};
  for (int r = 0; r < 4; ++r)
    for (int m = 0; m < kQ; ++m) {
      t.w[r][m].x = float(cx_cos2pi(r * m, kP));
      t.w[r][m].y = float(-cx_sin2pi(r * m, kP));
    }
  return t;
}
__constant__ QuarterTable kQuarter = quarter_table();

// Quarter r of the line whose sample s is at line[s]: folded and transformed.
__device__ __forceinline__ void forward(float2 (&v)[kQ], const float2* line, int r) {
  auto fold = [&](auto rot) {
#pragma unroll
    for (int m = 0; m < kQ; ++m) v[m] = s_add(line[m], tw_const<-1, long(decltype(rot)::value), 4L>(line[m + kQ]));
  };
  if (r == 0) fold(std::integral_constant<int, 0>{});
  else if (r == 1) fold(std::integral_constant<int, 1>{});
  else if (r == 2) fold(std::integral_constant<int, 2>{});
  else fold(std::integral_constant<int, 3>{});
  if (r) {
#pragma unroll
    for (int m = 1; m < kQ; ++m) v[m] = c_mul(v[m], kQuarter.w[r][m]);
  }
  dft<kQ, 1, -1>(v);
}
// Bins k of quarter r (ky = 4 k + r) times the row of |kx|: |ky| = ky below the middle, 128 - ky above;
// even ones at |ky| / 2 of the row, odd ones at 33 + (|ky| - 1) / 2.
__device__ __forceinline__ void filter(float2 (&v)[kQ], const float2* row, int r, bool adjoint) {
  const float sg = adjoint ? -1.f : 1.f;
  const float2* up = row + (r >> 1) + (r & 1) * (kP / 4 + 1);
  const float2* down = row + kP / 2 - (r >> 1) + (r & 1) * (kP / 4);
#pragma unroll
  for (int k = 0; k < kQ; ++k) {
    float2 h = k < kQ / 2 ? up[2 * k] : down[-2 * k];
    h.y *= sg;
    v[k] = c_mul(v[k], h);
  }
}
__device__ __forceinline__ void inverse(float2 (&v)[kQ], int r) {
  dft<kQ, 1, +1>(v);
  if (r) {
#pragma unroll
    for (int m = 1; m < kQ; ++m) v[m] = c_mulc(v[m], kQuarter.w[r][m]);
  }
}
// The sum over the quarters, through the line's 64 places: first r with r ^ 2 (each keeps the sums and
// differences of half of the m), then r with r ^ 1. Leaves in o the samples y[out0 + m], m < 16, with
// out0 = 16 (r >> 1) + 32 (r & 1). `sync` is the barrier of the lines' threads; on entry every one of
// them is past its reads of the line, on return past those of the differences.
template <class Sync>
__device__ __forceinline__ void add_quarters(float2 (&v)[kQ], float2* line, int r, float2 (&o)[kQ / 2], Sync&& sync) {
  constexpr int H = kQ / 2;
  float2* mine = line + r * H;
  const float2* across = line + (r ^ 2) * H;
  const float2* beside = line + (r ^ 1) * H;
  float2 d[H];
  if (r < 2) {
#pragma unroll
    for (int m = 0; m < H; ++m) mine[m] = v[H + m];
    sync();
#pragma unroll
    for (int m = 0; m < H; ++m) {
      const float2 q = across[m];
      o[m] = c_add(v[m], q);  // E_r + E_(r + 2)
      d[m] = c_sub(v[m], q);
    }
  } else {
#pragma unroll
    for (int m = 0; m < H; ++m) mine[m] = v[m];
    sync();
#pragma unroll
    for (int m = 0; m < H; ++m) {
      const float2 q = across[m];
      o[m] = c_add(q, v[H + m]);
      d[m] = c_sub(q, v[H + m]);
    }
  }
  sync();
  // y[m] = (E0 + E2) + (E1 + E3), y[m + 32] = (E0 - E2) + i (E1 - E3)
  if (r & 1) {
#pragma unroll
    for (int m = 0; m < H; ++m) mine[m] = o[m];
    sync();
#pragma unroll
    for (int m = 0; m < H; ++m) o[m] = s_add(beside[m], c_mul_i(d[m]));
  } else {
#pragma unroll
    for (int m = 0; m < H; ++m) mine[m] = d[m];
    sync();
#pragma unroll
    for (int m = 0; m < H; ++m) o[m] = c_add(o[m], beside[m]);
  }
}

__global__ void __launch_bounds__(kThreads, 2) k_onchip64(const __grid_constant__ PassParams p) {
  TOP_DYN_SMEM(float2, smem);
  float2* tile = smem;           // [kx][y] bins, or a [y][x] plane
  float2* hs = smem + kTile;     // staged quadrant rows [|kx|][kLH]
  const int tid = threadIdx.x;
  const int c = tid & 63;        // row y (phases 1, 3) or column of the round (phase 2)
  const int r = tid >> 6;        // quarter: two warps each
  const int out0 = 16 * (r >> 1) + 32 * (r & 1);
  // the four quarters of 32 consecutive lines
  const auto lines_sync = [&] { top_named_barrier(1 + (c >> 5), 128); };
  const float2* staged = nullptr;  // the quadrant table in shared memory

  for (int f = blockIdx.x; f < p.nfields; f += gridDim.x) {
    // ---- stage the field rows [y][x] (stride kLT) and, when the set changes, its quadrant rows
    const float2* src = field_in(p, f);
#pragma unroll 4
    for (int i = tid; i < kN * kN; i += kThreads) top_cp_async8(tile + (i >> 6) * kLT + (i & 63), src + i);
    const float2* hq = p.hq_list ? p.hq_list[f] : p.sets[p.set_of[f]].hq;
    if (hq != staged) {
      for (int i = tid; i < kHRows * kHS; i += kThreads) {
        const int row = i / kHS, e = i - row * kHS;
        top_cp_async8(hs + row * kLH + e, hq + i);
      }
      staged = hq;
    }
    top_cp_async_wait_all();
    __syncthreads();
    float2 v[kQ], o[kQ / 2];

    // ---- 1. rows
    forward(v, tile + c * kLT, r);
    __syncthreads();  // every row is read before the bins overwrite it
#pragma unroll
    for (int k = 0; k < kQ; ++k) tile[(4 * k + r) * kLT + c] = v[k];
    __syncthreads();

    // ---- 2. columns
#pragma unroll 1
    for (int it = 0; it < 2; ++it) {
      const int kx = it * kN + c, akx = kx <= kP / 2 ? kx : kP - kx;
      float2* col = tile + kx * kLT;
      forward(v, col, r);
      filter(v, hs + akx * kLH, r, p.adjoint);
      inverse(v, r);
      lines_sync();  // all quarters have read the column
      add_quarters(v, col, r, o, lines_sync);
      lines_sync();
#pragma unroll
      for (int m = 0; m < kQ / 2; ++m) col[out0 + m] = o[m];
    }
    __syncthreads();

    // ---- 3. rows
#pragma unroll
    for (int k = 0; k < kQ; ++k) v[k] = tile[(4 * k + r) * kLT + c];
    inverse(v, r);
    __syncthreads();  // every bin is read: the tile becomes a [y][x] plane
    float2* row = tile + c * kLT;
    add_quarters(v, row, r, o, lines_sync);
    lines_sync();
#pragma unroll
    for (int m = 0; m < kQ / 2; ++m) row[out0 + m] = o[m];
    __syncthreads();
    float2* dst = field_out(p, f);
#pragma unroll 4
    for (int i = tid; i < kN * kN; i += kThreads) dst[i] = tile[(i >> 6) * kLT + (i & 63)];
    __syncthreads();  // the plane is read before the next field's copies land in it
  }
}

}  // namespace

bool onchip_supported(const PassParams& p) {
  return p.Py == kP && p.Px == kP && p.ny == kN && p.nx == kN && p.src_kind == SRC_FIELD && p.msrc.flags == 0 &&
         p.epi_kind == EPI_FIELD && p.mepi.flags == 0 && p.in_repeat >= 1 && !p.spec_in && !p.spec_out && !p.hq_out;
}

cudaError_t launch_onchip(const PassParams& p, cudaStream_t s) {
  // two blocks fit an SM; the fields are taken in turn
  static KernelOnDevices setup;
  int resident = 0;
  const cudaError_t ready = setup.ready(k_onchip64, kThreads, kSmem, &resident);
  if (ready != cudaSuccess) return ready;
  if (resident == 0) resident = 2;  // not known: any number of blocks does
  const int grid = p.nfields < resident ? p.nfields : resident;
  if (grid <= 0) return cudaSuccess;
  TOP_LAUNCH(k_onchip64, grid, kThreads, kSmem, s, p);
  return cudaGetLastError();
}

}  // namespace top
