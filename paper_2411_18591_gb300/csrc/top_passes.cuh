// The three passes of one batched propagation, Eq. 4 with H_z of Eq. 5:
//
//   R1  rows:    modulate (Eq. 1), zero-pad along x, forward DFT along x,
//                store transposed:  ws[field][line][y]
//   C   columns: zero-pad along y, forward DFT along y, multiply by H(kx, ky) / (Py Px)
//                (a float64-built table), inverse DFT along y, crop, in place
//   R2  rows:    inverse DFT along x, crop, epilogue (modulation, |psi|^2,
//                incoherent sums of Eq. 14, or modulation gradients)
//
// Each padded line of even length P = 2M is handled as its two interleaved halves (even and odd
// frequencies), transformed by two thread groups side by side. With a field of n <= P samples at
// offset o, the even half is the M-point DFT of the folded sequence v[q] = sum_{p = q mod M} x[p - o]
// and the odd half that of sum_{p = q mod M} x[p - o] w^p, w = exp(-2 pi i / P); the inverse yields
// x[p] = E[p mod M] + w^-p O[p mod M]. With padding exactly 2 (n = M and o = M/2, "X2") every slot has
// one sample, x(q) = q + M/2 below the middle (where w^p = -w^q) and q - M/2 above it. Zero samples of
// the padding are never loaded or transformed and the inverse only produces the cropped window.
//
// Slots of the two halves. Lane t holds the same positions in both groups of a line, so each half
// "owns" half of the register slots (the even half the first E/2, the odd half the others): the
// groups trade the other E/2 through shared memory once per direction, each combines its own slots,
// and every sample is loaded, modulated and stored once.
//
// Layout of the workspace between passes: for each field Px lines of ny samples. Line r Mx + b + S j
// (S = Mx / RL) holds the bin kbase(b) + j S of half r, the order in which lanes hold bins after the
// last stage, so plain lane-consecutive accesses touch consecutive lines. A line's samples are
// contiguous (lines interleaved in pairs for the plans whose row tiles hold two rows, CI = 2), so the
// column pass moves its samples straight between registers and memory, one column per two thread
// groups with no barrier beyond theirs. The row passes get whole 32-byte sectors without a tile
// transpose: the rows of a tile (four, or two with CI = 2) regroup in the last exchange of the row
// transform, whose reader lanes take the same bins of all rows of the tile instead of more bins of
// one row.
#pragma once

#include <type_traits>
#include <utility>

#include "top_device.h"
#include "top_engine.cuh"
#include "top_internal.h"
#include "top_launch.h"

namespace top {

// A row tile: ROWS rows by both halves.
template <class EN>
struct RowShape {
  static constexpr int M = EN::M;
  static constexpr int GW = EN::GW;
  static constexpr int ROWS = GW <= 32 ? 4 : 2;  // rows of a tile (groups wider than a warp: fewer threads a barrier)
  static constexpr int HALF = ROWS * GW;         // threads of one half of a tile
  static constexpr int TILE = 2 * HALF;
  // Stride of the line buffers: the reader lanes of the last exchange (rows fastest) fall on
  // distinct banks (checked by simulation; exact for the power-of-two plans).
  static constexpr int RES = ROWS == 4 || EN::RL == 8 ? 4 : 8;
  static constexpr int LS = EN::BUF + ((RES - EN::BUF) % 16 + 16) % 16;
  static constexpr int XH = (ROWS * LS + 15) / 16 * 16;  // float2 of one half's line buffers
  // Lines interleaved in the workspace: pairs with two rows a tile and for the short plans, whose row
  // tiles go straight between registers and memory (64 contiguous bytes a tile halve the wavefronts of
  // their accesses; the column pass then reads half of every sector twice: at 1024 points 14.7 us a
  // field against 13.3).
  static constexpr bool LONG = M >= 250 && M <= 2048;
  static constexpr int CI = ROWS == 2 || !LONG ? 2 : 1;
  // Tile copies (COPY): a tile is a box of four 8-byte samples (ROWS rows x CI lines) by HL lines a half,
  // moved by the copy engine in boxes of LB lines.
  static constexpr int HL = M / CI;
  static constexpr int box_lines() {
    if (HL <= 256) return HL;
    for (int l = 256; l > 4; l -= 4)
      if (HL % l == 0) return l;
    return 4;
  }
  static constexpr int LB = box_lines();
  static constexpr int TH = (HL * 4 + 15) / 16 * 16;  // float2 of one half of a copied tile
  static constexpr unsigned TILE_BYTES = unsigned(2 * HL * 4 * sizeof(float2));
  static constexpr size_t SMEM_DUO = sizeof(float2) * size_t(4 * XH + 2 * TH) + 128;
  static constexpr bool COPY = LONG && EN::E >= 16 && SMEM_DUO <= 226 * 1024;
  // registers a thread: 128 for plans of 24 or more samples a thread, 80 for 16 to 20, else 64
  static constexpr int REGS = EN::E >= 24 ? 128 : EN::E >= 16 ? 80 : 64;
  static_assert(TH <= XH, "a half's bins fit its line buffers");
  static_assert(EN::M % 2 == 0 && EN::E % 2 == 0, "slots split between the halves");
  static_assert(CI == 1 || (EN::G % 2 == 0 && EN::SL % 2 == 0), "line pairs stay whole");
};

// A block of T tiles.
template <class EN, int T_>
struct RowBlock : RowShape<EN> {
  using SH = RowShape<EN>;
  static constexpr int T = T_;
  static constexpr int THREADS = SH::TILE * T;
  static constexpr int BLOCK_ROWS = SH::ROWS * T;
  static constexpr size_t SMEM_X = sizeof(float2) * size_t(T) * 2 * SH::XH + 64;
  static constexpr int MINB = 65536 / (THREADS * SH::REGS) > 0 ? 65536 / (THREADS * SH::REGS) : 1;
  static_assert(THREADS <= 1024, "row block too large");
  static_assert(THREADS % 32 == 0 && SMEM_X >= 3 * sizeof(double) * (THREADS / 32), "room for the overlap reduction");
};
// Tiles per block: enough for 128 threads; two sharing one copied tile in the passes that load bins by copy.
template <class EN>
constexpr int row_tiles() {
  return RowShape<EN>::TILE >= 128 ? 1 : 128 / RowShape<EN>::TILE;
}

// Columns per block of the column pass; two thread groups (the two halves) per column, one exchange
// buffer each.
template <class EN>
struct ColShape {
  static constexpr int GW = EN::GW;
  static constexpr int COLS = 2 * GW * 2 >= 128 ? 2 : 128 / (2 * GW);
  static constexpr int THREADS = 2 * GW * COLS;
  static constexpr int LS = RowShape<EN>::LS;
  static constexpr size_t SMEM = sizeof(float2) * size_t(COLS) * 2 * LS;
  static constexpr int REGS = EN::E >= 24 ? 128 : EN::E >= 16 ? 80 : 64;
  static constexpr int MINB = 65536 / (THREADS * REGS) > 0 ? 65536 / (THREADS * REGS) : 1;
  static_assert(GW <= 32 || 2 * COLS + COLS <= 15, "group and column barriers have ids of their own");
};

__device__ __forceinline__ float2 ldg2(const float2* p) { return __ldg(p); }

// exp(i a) for a float32 phase: two-constant Cody-Waite reduction of a to [-pi, pi]
// (2 pi = 6.28125 + 1.9353071795864769e-3, the first part exact in a few bits) and the
// fast sin/cos there; large arguments take the library path.
__device__ __forceinline__ float2 cis(float a) {
  float s, c;
  if (fabsf(a) < 1.0e5f) {
    const float n = rintf(a * 0.15915494309189535f);
    float r = fmaf(-n, 6.28125f, a);
    r = fmaf(-n, 1.9353071795864769e-3f, r);
    __sincosf(r, &s, &c);
  } else {
    sincosf(a, &s, &c);
  }
  return make_float2(c, s);
}

// Modulation flags a kernel is compiled for; TOP_MOD_DYNAMIC reads them at run time.
constexpr uint32_t TOP_MOD_DYNAMIC = 0xffffffffu;

template <uint32_t MF>
__device__ __forceinline__ uint32_t mod_flags(const ModDev& m) {
  return MF == TOP_MOD_DYNAMIC ? m.flags : MF;
}

// M(x, y) of Eq. 1 for field f at sample (y, x)
__device__ __forceinline__ float2 mod_value(const ModDev& m, uint32_t flags, int conj, const float2* lx,
                                            const float2* ly, int f, int y, int x, int nx) {
  if (flags & TOP_MOD_CIRC) {
    const int2 rg = __ldg(m.circ + y);
    if (x < rg.x || x > rg.y) return make_float2(0.f, 0.f);
  }
  float2 r = make_float2(1.f, 0.f);
  const long long idx = (long long)f * m.stride + (long long)y * nx + x;
  if (flags & TOP_MOD_COMPLEX) r = ldg2(m.cmask + idx);
  if (flags & TOP_MOD_AMPLITUDE) r = c_scale(r, __ldg(m.amp + idx));
  if (flags & TOP_MOD_PHASE) r = c_mul(r, cis(__ldg(m.phase + idx)));
  if (flags & TOP_MOD_LENS) r = c_mul(r, c_mul(ldg2(lx + x), ldg2(ly + y)));
  return conj ? c_conj(r) : r;
}

// Source field f of R1 and output field f of R2 (per-field pointers for ragged batches).
__device__ __forceinline__ const float2* field_in(const PassParams& p, int f) {
  return p.in_list ? p.in_list[f] : p.in + (long long)(f / p.in_repeat) * p.in_stride;
}
__device__ __forceinline__ float2* field_out(const PassParams& p, int f) {
  return p.out_list ? p.out_list[f] : p.out + (long long)f * p.out_stride;
}

// The place of a thread in a block of T row tiles: half r, row and lane of its line, and the row and
// lane it takes in the frequency layout, where the lanes of one half hold the rows fastest.
template <class EX, int T>
struct RowLane {
  using SH = RowShape<EX>;
  float2* smem;

  __device__ __forceinline__ explicit RowLane(float2* s) : smem(s) {}
  __device__ __forceinline__ static int tid() { return int(threadIdx.x); }
  __device__ __forceinline__ static int in_tile(int v) { return T == 1 ? v : v % SH::TILE; }
  __device__ __forceinline__ static int spare(int l) { return SH::GW == EX::G ? l : min(l, EX::G - 1); }
  __device__ __forceinline__ static int half_of(int v) { return in_tile(v) / SH::HALF; }
  __device__ __forceinline__ static int tile_of(int v) { return T == 1 ? 0 : v / SH::TILE; }
  __device__ __forceinline__ static int row_of(int v) { return in_tile(v) % SH::HALF / SH::GW; }
  __device__ __forceinline__ static int qrow_of(int v) { return v % SH::ROWS; }
  __device__ __forceinline__ static int tile() { return tile_of(tid()); }
  __device__ __forceinline__ static int r() { return half_of(tid()); }
  __device__ __forceinline__ static int row() { return row_of(tid()); }
  __device__ __forceinline__ static int t() { return spare(tid() % SH::GW); }
  __device__ __forceinline__ static int qrow() { return qrow_of(tid()); }
  __device__ __forceinline__ static int qt() { return spare(in_tile(tid()) % SH::HALF / SH::ROWS); }
  // not one of the spare threads of a padded group
  __device__ __forceinline__ static bool act() { return SH::GW == EX::G || tid() % SH::GW < EX::G; }
  __device__ __forceinline__ static bool lead() { return in_tile(tid()) == 0; }             // of the tile
  __device__ __forceinline__ static bool hlead() { return in_tile(tid()) % SH::HALF == 0; }  // of the tile's half
  // this half's line buffers, this line's, the other half's line's, the one of (half, qrow)
  __device__ __forceinline__ float2* half(int v) const { return smem + (tile_of(v) * 2 + half_of(v)) * SH::XH; }
  __device__ __forceinline__ float2* half() const { return half(tid()); }
  __device__ __forceinline__ float2* buf() const {
    const int v = tid();
    return half(v) + row_of(v) * SH::LS;
  }
  __device__ __forceinline__ const float2* peer() const {
    const int v = tid();
    return smem + (tile_of(v) * 2 + (half_of(v) ^ 1)) * SH::XH + row_of(v) * SH::LS;
  }
  __device__ __forceinline__ float2* qbuf() const {
    const int v = tid();
    return half(v) + qrow_of(v) * SH::LS;
  }
  // Barrier ids: tiles 1.., halves, rows; line groups wider than a warp count down from 15 (EX::sync_group).
  // all threads of the tile
  __device__ __forceinline__ void tile_sync() const {
    if constexpr (T == 1) __syncthreads();
    else if constexpr (SH::TILE <= 32) __syncwarp();
    else top_named_barrier(1 + tile(), SH::TILE);
  }
  // the rows of this half (the last exchange regroups them)
  __device__ __forceinline__ void quad_sync() const {
    if constexpr (SH::HALF <= 32) __syncwarp();
    else if constexpr (T <= 2) top_named_barrier(3 + tid() / SH::HALF, SH::HALF);
    else tile_sync();
  }
  // the two halves of this row
  __device__ __forceinline__ void pair_sync() const {
    if constexpr (SH::GW == 32) top_named_barrier(7 + SH::ROWS * tile() + row(), 2 * SH::GW);
    else tile_sync();
  }
  static_assert(SH::GW <= 32 || (T <= 2 && 15 - T * 2 * SH::ROWS >= 6), "group barriers clear of the others");
  static_assert(SH::GW != 32 || T <= 2, "row barriers have ids of their own");
};

// First workspace sample of lane qt of half r, row y of field f; slot (q, j) sits (G q + S j) ny on.
template <class EX>
__device__ __forceinline__ float2* ws_lane(const PassParams& p, int f, int r, int qt, int y) {
  float2* ws = p.ws + (long long)f * p.ws_stride;
  const int line = r * EX::M + qt;
  if constexpr (RowShape<EX>::CI == 1) return ws + (long long)line * p.ny + y;
  else return ws + ((long long)(line >> 1) * p.ny + y) * 2 + (line & 1);
}
// The same in one half of a copied tile, [HL][4]; slot (q, j) sits (G q + S j) / CI lines on.
template <class EX>
__device__ __forceinline__ int tile_lane(int qt, int qrow) {
  if constexpr (RowShape<EX>::CI == 1) return qt * 4 + qrow;
  else return (qt >> 1) * 4 + qrow * 2 + (qt & 1);
}

template <class EX, class Lane>
__device__ __forceinline__ void load_bins(const PassParams& p, int f, const Lane& c, int y, float2 (&v)[EX::E]) {
  const float2* w = ws_lane<EX>(p, f, c.r(), c.qt(), y);
  const bool live = y < p.ny;
#pragma unroll
  for (int e = 0; e < EX::E; ++e) {
    const int q = e / EX::RL, j = e % EX::RL;
    v[e] = live ? w[(EX::G * q + EX::SL * j) * p.ny] : make_float2(0.f, 0.f);
  }
}
template <class EX, class Lane>
__device__ __forceinline__ void store_bins(const PassParams& p, int f, const Lane& c, int y, const float2 (&v)[EX::E]) {
  float2* w = ws_lane<EX>(p, f, c.r(), c.qt(), y);
  if (y < p.ny) {
#pragma unroll
    for (int e = 0; e < EX::E; ++e) {
      const int q = e / EX::RL, j = e % EX::RL;
      w[(EX::G * q + EX::SL * j) * p.ny] = v[e];
    }
  }
}
template <class EX, class Lane>
__device__ __forceinline__ void read_tile(const float2* tile, const Lane& c, float2 (&v)[EX::E]) {
  const float2* w = tile + c.r() * RowShape<EX>::TH + tile_lane<EX>(c.qt(), c.qrow());
#pragma unroll
  for (int e = 0; e < EX::E; ++e) {
    const int q = e / EX::RL, j = e % EX::RL;
    v[e] = w[(EX::G * q + EX::SL * j) * (4 / RowShape<EX>::CI)];
  }
}
// The bins of a tile to the workspace through the half's line buffers, by copy. Returns with the copy
// in flight: the half's leading thread waits for it (top_bulk_wait_read) before the buffers are written
// again.
template <class EX, class Lane>
__device__ __forceinline__ void copy_bins_out(const TileMap& map, int f, const Lane& c, int y0, const float2 (&v)[EX::E]) {
  using SH = RowShape<EX>;
  c.quad_sync();  // the half's last exchange reads are done
  float2* w = c.half() + tile_lane<EX>(c.qt(), c.qrow());
#pragma unroll
  for (int e = 0; e < EX::E; ++e) {
    const int q = e / EX::RL, j = e % EX::RL;
    w[(EX::G * q + EX::SL * j) * (4 / SH::CI)] = v[e];
  }
  top_async_fence();
  c.quad_sync();
  if (c.hlead()) {
#pragma unroll 1
    for (int l = 0; l < SH::HL; l += SH::LB) top_tma_store3(&map.tile, y0 * SH::CI, c.r() * SH::HL + l, f, c.half() + l * 4);
    top_bulk_commit();
  }
}
// The half's buffers are free of outgoing copies.
template <class Lane>
__device__ __forceinline__ void copy_out_done(const Lane& c) {
  if (c.hlead()) top_bulk_wait_read();
  c.quad_sync();
}

// Bound of the waits on copies and tickets, in clock cycles (about two seconds).
constexpr long long kWaitCycles = 4000000000ll;

// The work items a block runs: its own index, then those of blocks that have not started. Items are handed
// out in order, so the tiles in flight stay neighbours and the sectors of a line meet in L2: fixed shares
// of the items per block drifted apart over a long launch (the 384-field step's fused rows took 11.1 us
// a field with 24 fields and 16.4 with 384).
struct Tickets {
  struct Shared {
    alignas(16) unsigned answer[4];
    unsigned long long bar;
    int parity, open;
  };
  Shared* s;

  __device__ __forceinline__ explicit Tickets(void* mem) : s(static_cast<Shared*>(mem)) {}
  // one thread, before the block's first barrier
  __device__ __forceinline__ void init() const {
    top_mbar_init(&s->bar, 1);
    top_mbar_fence();
    s->parity = 0;
    s->open = 1;
  }
  __device__ __forceinline__ void ask() const {
    top_mbar_expect(&s->bar, 16);
    top_ask_ticket(s->answer, &s->bar);
  }
  // The asked item, or -1; asks for the next one. One thread at a time, in an order that barriers give.
  __device__ __forceinline__ int take(int* fault) const {
    if (!s->open) return -1;
    int item = -1;
    if (top_mbar_wait(&s->bar, s->parity, kWaitCycles)) {
      item = top_ticket(s->answer);
    } else {
      if (fault) *fault = 1;
      top_mbar_wait(&s->bar, s->parity, kWaitCycles);  // the answer may still come: not into another block's memory
    }
    s->parity ^= 1;
    if (item < 0) {
      s->open = 0;
    } else {
      top_async_fence();  // the answer has been read
      ask();
    }
    return item;
  }
};

// Rows by tile copies. The scattered accesses of a row tile (2 x 1024 lines, 32 bytes each at 1024
// points) took half of the row passes' L1 wavefronts and left their latency exposed; the copy engine
// moves the same boxes at 5.4 TB/s read and 2 x 2.5 TB/s in place, without either. Per field at 1024
// points (64-field launches, direct with its own best layout -> copies): forward rows 4.6 -> 4.2 us,
// fused rows 10.4 -> 9.7, inverse rows 5.8 -> 5.3, with the phase gradient 12.9 -> 10.4, and the column
// pass, whose lines no longer need to be interleaved for the rows' sake, 14.2 -> 12.7.
//
// Two tiles of a block (groups 0 and 1, 256 threads each at 1024 points) work in antiphase on one copied
// tile of shared memory: while a group transforms its rows in registers and its own line buffers, the
// copy engine brings the other group's next tile. Tiles are brought for group 0, 1, 0, 1, ... (a group
// that has run out is skipped); the group that has read a tile starts the next copy. An item is a row
// tile of the fields of one group.
template <class EX>
struct TileFeed {
  using SH = RowShape<EX>;
  struct Shared {
    Tickets::Shared tickets;
    unsigned long long full[2];
    int item[2], f[2], x[2];    // the tile each group is to take next (item < 0: there is none), its box's x
    int cur_item[2][2], cur_f[2][2];  // [turn][group]: the tile each group has in hand (a group's threads
                                      // are at most one take apart)
    int alive[2];  // not yet told that there are no more tiles
    int ok[2];
  };
  static_assert(sizeof(Shared) <= 128, "reserved after the tiles");
  float2* tile;
  Shared* s;
  int ntiles, group, nfields, ahead;
  unsigned turn;  // of this group's next take: the parity of its copy

  __device__ __forceinline__ TileFeed(float2* smem, int ny, int nfields_, int group_, int ahead_)
      : tile(smem + 4 * SH::XH), s(reinterpret_cast<Shared*>(smem + 4 * SH::XH + 2 * SH::TH)), group(group_),
        nfields(nfields_), ahead(ahead_), turn(0) {
    ntiles = (ny + SH::ROWS - 1) / SH::ROWS;
    if (threadIdx.x == 0) {
      const Tickets tickets(&s->tickets);
      tickets.init();
      top_mbar_init(s->full, 1);
      top_mbar_init(s->full + 1, 1);
      top_mbar_fence();
      s->item[1] = -1;
      s->alive[0] = s->alive[1] = 1;
      tickets.ask();
    }
    __syncthreads();
  }
  // group 0's first tile, the block's own item (one thread)
  __device__ __forceinline__ void start(const TileMap& map) const {
    plan(0, blockIdx.x, first_field(blockIdx.x));
    bring(map, 0);
  }
  __device__ __forceinline__ int first_field(int it) const { return it / ntiles * group; }
  __device__ __forceinline__ int end_field(int it) const { return min(first_field(it) + group, nfields); }
  // the tile in hand (after take, until the group's next)
  __device__ __forceinline__ int item() const { return s->cur_item[turn ^ 1][RowLane<EX, 2>::tile()]; }
  __device__ __forceinline__ int field() const { return s->cur_f[turn ^ 1][RowLane<EX, 2>::tile()]; }
  __device__ __forceinline__ int y0() const {
    const int it = item();
    return (it - it / ntiles * ntiles) * SH::ROWS;
  }

  __device__ __forceinline__ void plan(int g, int it, int ff) const {
    s->item[g] = it;
    s->f[g] = ff;
    s->x[g] = (it - it / ntiles * ntiles) * SH::ROWS * SH::CI;
    s->alive[g] = it >= 0;
  }
  // Copy in the planned tile of group g, or tell it that there is none.
  __device__ __forceinline__ void bring(const TileMap& map, int g) const {
    if (s->item[g] < 0) {
      top_mbar_arrive(s->full + g);
      return;
    }
    top_mbar_expect(s->full + g, SH::TILE_BYTES);
    const int x = s->x[g], f = s->f[g];
#pragma unroll 1
    for (int l = 0; l < 2 * SH::HL; l += SH::LB)
      top_tma_load3(tile + (l < SH::HL ? l * 4 : SH::TH + (l - SH::HL) * 4), &map.tile, x, l, f, s->full + g);
    if (ahead > 0 && (x & 15) == 0) {
      // the first of four tiles side by side: the four's next field, or the four tiles one wave of
      // resident groups later, go to L2
      int it = s->item[g], nf = f + 1;
      if (nf >= end_field(it)) {
        it += ahead;
        nf = first_field(it);
        if (nf >= nfields) return;
      }
      const int nx = (it - it / ntiles * ntiles) * SH::ROWS * SH::CI & ~15;
#pragma unroll 1
      for (int l = 0; l < 2 * SH::HL; l += SH::LB) top_tma_prefetch3(&map.wide, nx, l, nf);
    }
  }
  // the item and field after (it, ff), from the tickets at the end of an item; it < 0: none
  __device__ __forceinline__ void following(int& it, int& ff, int* fault) const {
    if (it >= 0 && ff + 1 < end_field(it)) {
      ++ff;
    } else {
      it = Tickets(&s->tickets).take(fault);
      ff = it >= 0 ? first_field(it) : 0;
    }
  }
  // Wait for this group's tile, take its bins, start the next copy. False (for the whole group) when there
  // is none, or if the copy has not come within the bound (the fault word is then set).
  template <class Lane>
  __device__ __forceinline__ bool take(const TileMap& map, const Lane& c, int* fault, float2 (&v)[EX::E]) {
    int calls = 0;  // groups to bring tiles for: bit g
    if (c.lead()) {
      const int g = c.tile(), o = g ^ 1;
      const bool ok = top_mbar_wait(s->full + g, turn, kWaitCycles);
      if (!ok) {
        if (fault) *fault = 1;
        // what is still in flight lands before the block leaves its memory to another
        top_mbar_wait(s->full + g, turn, kWaitCycles);
        if (s->tickets.open) top_mbar_wait(&s->tickets.bar, s->tickets.parity, kWaitCycles);
      }
      const int it = s->item[g], ff = s->f[g];
      s->ok[g] = ok && it >= 0;
      s->cur_item[turn][g] = it;
      s->cur_f[turn][g] = ff;
      if (ok && it >= 0) {
        int ni = -1, nf = 0;
        if (s->alive[o]) {
          ni = s->item[o];
          nf = s->f[o];
          following(ni, nf, fault);
          plan(o, ni, nf);
          calls |= 1 << o;
        }
        if (ni < 0) {  // the other group has run out: this one goes on alone
          ni = it;
          nf = ff;
          following(ni, nf, fault);
          plan(g, ni, nf);
          calls |= 1 << g;
        }
      }
    }
    c.tile_sync();
    const int g = c.tile();
    if (!s->ok[g]) return false;
    top_mbar_try(s->full + g, turn);  // complete: orders the copied tile before this thread's reads
    read_tile<EX>(tile, c, v);
    c.tile_sync();
    if (calls & 1) bring(map, 0);
    if (calls & 2) bring(map, 1);
    turn ^= 1;
    return true;
  }
};

// Position of own slot k of half r (slot k or E/2 + k: a constant step between the two).
template <class EN>
__device__ __forceinline__ int own_pos(int r, int t, int k) {
  constexpr int R0 = EN::radix(0), Q = EN::E / R0;
  static_assert(Q % 2 == 0 || (Q == 1 && R0 % 2 == 0), "slots split at a constant step");
  return EN::in_pos(t, k) + (r ? (Q % 2 == 0 ? EN::G * Q / 2 : EN::span(0) * R0 / 2) : 0);
}

// Field sample of position pos: with LO, the one of x[pos - o] (X2: the position's only sample), else
// of x[pos + M - o].
template <class EN, bool X2>
__device__ __forceinline__ int sample_lo(int pos, int o) {
  if constexpr (X2) return pos < EN::M / 2 ? pos + EN::M / 2 : pos - EN::M / 2;
  else return pos - o;
}
template <class EN>
__device__ __forceinline__ int sample_hi(int pos, int o) {
  return pos + EN::M - o;
}
// whether sample x exists
template <bool X2>
__device__ __forceinline__ bool in_line(int x, int n) {
  return X2 || (unsigned)x < (unsigned)n;
}

// Samples of the own slots: lo or hi (a constant once inlined).
template <class EX, bool X2>
struct OwnSamples {
  int r, t, o;
  bool hi;
  __device__ __forceinline__ int operator()(int k) const {
    const int pos = own_pos<EX>(r, t, k);
    return hi ? sample_hi<EX>(pos, o) : sample_lo<EX, X2>(pos, o);
  }
};

// Calls f(std::integral_constant<int, e>) for every register slot e, so slot positions are constants.
template <class F, int... Es>
__device__ __forceinline__ void for_slots(F&& f, std::integer_sequence<int, Es...>) {
  (f(std::integral_constant<int, Es>{}), ...);
}

// exp(-2 pi i pos / 2M) for the stage-0 position pos = t + G q + SP0 j of slot e, as the lane's
// exp(-2 pi i t / 2M) times a compile-time constant.
template <class EN, int e>
__device__ __forceinline__ float2 slot_split_twiddle(float2 wt) {
  constexpr int R0 = EN::radix(0), SP0 = EN::span(0);
  return tw_const<-1, long(EN::G * (e / R0) + SP0 * (e % R0)), long(2 * EN::M)>(wt);
}

// The odd half's fold twiddles on the slots of v (X2: w^p of the slot's sample; else w^pos).
template <class EN, bool X2>
__device__ __forceinline__ void fold_odd(float2 (&v)[EN::E], const float2* __restrict__ wp, int t) {
  if constexpr (X2) {
    const float2 wt = ldg2(wp + t);
    for_slots(
        [&](auto ec) {
          constexpr int e = decltype(ec)::value;
          const float2 w = slot_split_twiddle<EN, e>(wt);
          v[e] = c_mul(v[e], EN::in_pos(t, e) < EN::M / 2 ? c_neg(w) : w);
        },
        std::make_integer_sequence<int, EN::E>{});
  } else {
#pragma unroll
    for (int e = 0; e < EN::E; ++e) v[e] = c_mul(v[e], ldg2(wp + EN::in_pos(t, e)));
  }
}
// The odd half's unfold twiddles: O'[pos] = w^-pos O[pos].
template <class EN, bool X2>
__device__ __forceinline__ void unfold_odd(float2 (&v)[EN::E], const float2* __restrict__ wp, int t) {
  if constexpr (X2) {
    const float2 wt = ldg2(wp + t);
    for_slots(
        [&](auto ec) {
          constexpr int e = decltype(ec)::value;
          v[e] = c_mulc(v[e], slot_split_twiddle<EN, e>(wt));
        },
        std::make_integer_sequence<int, EN::E>{});
  } else {
#pragma unroll
    for (int e = 0; e < EN::E; ++e) v[e] = c_mulc(v[e], ldg2(wp + EN::in_pos(t, e)));
  }
}

// After the inverse transforms (v = E in the even half, O' in the odd one): trade and return the own
// slots' samples: lo, x[pos - o] = E + O' (X2: E - O' below the middle), and, unless X2, hi, x[pos + M - o]
// = E - O'. Each half writes the slots it does not own to its buffer, lane-consecutively.
template <class EX, bool X2, class Own, class Sync>
__device__ __forceinline__ void trade_combine(const float2 (&v)[EX::E], float2 (&lo)[EX::E / 2], float2 (&hi)[EX::E / 2],
                                              float2* buf, const float2* peer, int r, int t, Own&& own_sync,
                                              Sync&& pair) {
  constexpr int H = EX::E / 2;
  own_sync();  // the own group's last exchange reads are done
#pragma unroll
  for (int k = 0; k < H; ++k) buf[k * EX::G + t] = r ? v[k] : v[H + k];
  pair();
#pragma unroll
  for (int k = 0; k < H; ++k) {
    const float2 o = peer[k * EX::G + t];
    const float2 mine = r ? v[H + k] : v[k];
    const float2 ev = r ? o : mine, od = r ? mine : o;
    if constexpr (X2) {
      lo[k] = own_pos<EX>(r, t, k) < EX::M / 2 ? c_sub(ev, od) : c_add(ev, od);
    } else {
      lo[k] = c_add(ev, od);
      hi[k] = c_sub(ev, od);
    }
  }
}

// Own slots' samples lo (and hi) to the folded input of both halves, before the odd half's twiddles;
// the trade goes through the upper part of the buffers, which trade_combine and the exchanges before it
// do not read.
template <class EX, bool X2, class Sync>
__device__ __forceinline__ void trade_fold(float2 (&v)[EX::E], const float2 (&lo)[EX::E / 2], const float2 (&hi)[EX::E / 2],
                                           float2* buf, const float2* peer, int r, int t, Sync&& pair) {
  constexpr int H = EX::E / 2;
  float2* mine = buf + H * EX::G + t;
  const float2* theirs = peer + H * EX::G + t;
#pragma unroll
  for (int k = 0; k < H; ++k) {
    if constexpr (X2) mine[k * EX::G] = lo[k];
    else mine[k * EX::G] = r ? c_add(lo[k], hi[k]) : c_sub(lo[k], hi[k]);
  }
  pair();
#pragma unroll
  for (int k = 0; k < H; ++k) {
    float2 w = lo[k];
    if constexpr (!X2) w = r ? c_sub(lo[k], hi[k]) : c_add(lo[k], hi[k]);
    const float2 o = theirs[k * EX::G];
    v[k] = r ? o : w;
    v[H + k] = r ? w : o;
  }
}

// The row's modulation operands that do not change along it.
struct ModRow {
  int2 rg;          // aperture range
  float2 ly;        // lens factor of the row
  const float2* lx;
  long long base;   // first element of the row in per-sample planes
};
__device__ __forceinline__ ModRow mod_row(const ModDev& m, uint32_t flags, const float2* lx, const float2* ly, int f,
                                          int y, int nx) {
  ModRow mr;
  mr.rg = (flags & TOP_MOD_CIRC) ? __ldg(m.circ + y) : make_int2(0, nx - 1);
  mr.ly = (flags & TOP_MOD_LENS) ? ldg2(ly + y) : make_float2(1.f, 0.f);
  mr.lx = lx;
  mr.base = (long long)f * m.stride + (long long)y * nx;
  return mr;
}
// M(x, y) of Eq. 1 in the order of mod_value
__device__ __forceinline__ float2 mod_at(const ModDev& m, uint32_t flags, int conj, const ModRow& mr, int x) {
  float2 r = make_float2(1.f, 0.f);
  if (flags & TOP_MOD_COMPLEX) r = ldg2(m.cmask + mr.base + x);
  if (flags & TOP_MOD_AMPLITUDE) r = c_scale(r, __ldg(m.amp + mr.base + x));
  if (flags & TOP_MOD_PHASE) r = c_mul(r, cis(__ldg(m.phase + mr.base + x)));
  if (flags & TOP_MOD_LENS) r = c_mul(r, c_mul(ldg2(mr.lx + x), mr.ly));
  if ((flags & TOP_MOD_CIRC) && (x < mr.rg.x || x > mr.rg.y)) r = make_float2(0.f, 0.f);
  return conj ? c_conj(r) : r;
}

// M (Eq. 1) at samples sample(k) of a row, in the order of mod_value (any value where the sample is
// outside the row). Each factor's operands are
// loaded for all slots before any is used: the branches of a factor (its flag, the range test of the
// sine and cosine) would otherwise put every load behind the one before it.
template <int N, class At>
__device__ __forceinline__ void mod_values(const ModDev& m, uint32_t flags, int conj, const ModRow& mr, int nx,
                                           At&& sample, float2 (&mv)[N]) {
  auto at = [&](int k) { return max(0, min(sample(k), nx - 1)); };
  float op[N];
  if (flags & TOP_MOD_COMPLEX) {
#pragma unroll
    for (int k = 0; k < N; ++k) mv[k] = ldg2(m.cmask + mr.base + at(k));
  } else {
#pragma unroll
    for (int k = 0; k < N; ++k) mv[k] = make_float2(1.f, 0.f);
  }
  if (flags & TOP_MOD_AMPLITUDE) {
#pragma unroll
    for (int k = 0; k < N; ++k) op[k] = __ldg(m.amp + mr.base + at(k));
#pragma unroll
    for (int k = 0; k < N; ++k) mv[k] = c_scale(mv[k], op[k]);
  }
  if (flags & TOP_MOD_PHASE) {
#pragma unroll
    for (int k = 0; k < N; ++k) op[k] = __ldg(m.phase + mr.base + at(k));
#pragma unroll
    for (int k = 0; k < N; ++k) mv[k] = c_mul(mv[k], cis(op[k]));
  }
  if (flags & TOP_MOD_LENS) {
#pragma unroll
    for (int k = 0; k < N; ++k) mv[k] = c_mul(mv[k], c_mul(ldg2(mr.lx + at(k)), mr.ly));
  }
  if (flags & TOP_MOD_CIRC) {
#pragma unroll
    for (int k = 0; k < N; ++k) {
      const int x = at(k);
      if (x < mr.rg.x || x > mr.rg.y) mv[k] = make_float2(0.f, 0.f);
    }
  }
  if (conj) {
#pragma unroll
    for (int k = 0; k < N; ++k) mv[k] = c_conj(mv[k]);
  }
}

// ----------------------------------------------------------------------------- R1

// Source of field f in row y before its modulation: the field, or 2 w g_I psi of the intensity backward.
struct SrcRow {
  const float2* x;
  const float* gi;
  float w2;
};
__device__ __forceinline__ SrcRow src_row(const PassParams& p, int f, int y) {
  SrcRow s;
  const long long row = (long long)y * p.nx;
  if (p.src_kind == SRC_INTENSITY) {
    s.x = p.psi + (long long)f * p.psi_stride + row;
    s.gi = p.gI + (long long)(f / p.src_group) * p.gI_stride + row;
    s.w2 = 2.f * (p.weights ? __ldg(p.weights + f) : 1.f);
  } else {
    s.x = field_in(p, f) + row;
    s.gi = nullptr;
    s.w2 = 1.f;
  }
  return s;
}
// N source samples at(i) (zero outside [0, n)), all loads in flight at once
template <int N, class At>
__device__ __forceinline__ void src_samples(const SrcRow& s, int n, At&& at, float2 (&v)[N]) {
#pragma unroll
  for (int i = 0; i < N; ++i) v[i] = (unsigned)at(i) < (unsigned)n ? ldg2(s.x + at(i)) : make_float2(0.f, 0.f);
  if (s.gi) {
    float g[N];
#pragma unroll
    for (int i = 0; i < N; ++i) g[i] = (unsigned)at(i) < (unsigned)n ? __ldg(s.gi + at(i)) : 0.f;
#pragma unroll
    for (int i = 0; i < N; ++i) v[i] = c_scale(v[i], s.w2 * g[i]);
  }
}

// Without a source modulation (MF = 0) both halves load the whole row (the second read hits L1) and
// nothing is traded; with one, each half modulates its own slots and the halves trade. With COPY the
// bins leave through the copy engine, and a block goes on to the next tile while they do.
template <class EX, bool X2, uint32_t MF, bool COPY>
__global__ void __launch_bounds__(RowBlock<EX, row_tiles<EX>()>::THREADS, RowBlock<EX, row_tiles<EX>()>::MINB)
    k_rows_fwd(const __grid_constant__ PassParams p, const __grid_constant__ TileMap map) {
  constexpr int T = row_tiles<EX>();
  using SH = RowBlock<EX, T>;
  constexpr int E = EX::E, H = E / 2;
  TOP_DYN_SMEM(float2, smem);
  const RowLane<EX, T> c(smem);
  const int nx = p.nx, o = p.ox;
  const int ntiles = (p.ny + SH::BLOCK_ROWS - 1) / SH::BLOCK_ROWS;
  const int total = ntiles * p.nfields;
  struct Next {
    Tickets::Shared tickets;
    int item[2];
  };
  static_assert(sizeof(Next) <= 64, "reserved after the line buffers");
  Next* next = reinterpret_cast<Next*>(smem + T * 2 * SH::XH);
  const Tickets tickets(&next->tickets);
  if constexpr (COPY) {
    if (threadIdx.x == 0) {
      tickets.init();
      tickets.ask();
    }
  }
  int turn = 0;
#pragma unroll 1
  for (int i = blockIdx.x; i >= 0; turn ^= 1) {
    const int f = COPY ? i / ntiles : blockIdx.y;
    const int tile0 = (COPY ? i - f * ntiles : i) * SH::BLOCK_ROWS + c.tile() * SH::ROWS;
    const int y = tile0 + c.row();
    const bool live = y < p.ny;
    const int next_wave = (COPY ? i : blockIdx.y * ntiles + i) + p.l2_ahead;
    if (threadIdx.x == 0 && p.l2_ahead > 0 && next_wave < total) {
      // the rows of the tile one wave of resident blocks later go to L2 while this one works
      const int fa = next_wave / ntiles, ya = (next_wave - fa * ntiles) * SH::BLOCK_ROWS;
      const int na = min(SH::BLOCK_ROWS, p.ny - ya);
      const long long rowa = (long long)ya * nx;
      const float2* src = p.src_kind == SRC_INTENSITY ? p.psi + (long long)fa * p.psi_stride + rowa : field_in(p, fa) + rowa;
      top_prefetch_l2(src, unsigned(na) * nx * 8u);
    }
    const SrcRow s = src_row(p, f, live ? y : 0);
    const int n = live ? nx : 0;  // rows past the field are zero
    float2 v[E];
    if constexpr (MF == 0) {
      src_samples<E>(s, n, [&](int e) { return sample_lo<EX, X2>(EX::in_pos(c.t(), e), o); }, v);
      if constexpr (!X2) {
#pragma unroll
        for (int e0 = 0; e0 < E; e0 += H) {
          float2 b[H];
          src_samples<H>(s, n, [&](int e) { return sample_hi<EX>(EX::in_pos(c.t(), e0 + e), o); }, b);
#pragma unroll
          for (int e = 0; e < H; ++e) v[e0 + e] = c.r() ? c_sub(v[e0 + e], b[e]) : c_add(v[e0 + e], b[e]);
        }
      }
    } else {
      const ModDev& m = p.msrc;
      const uint32_t flags = mod_flags<MF>(m);
      const FieldSet& fs = p.sets[p.set_of[f]];
      const ModRow mr = mod_row(m, flags, fs.src_lx, fs.src_ly, f, live ? y : 0, nx);
      float2 lo[H], hi[H], mv[H];
      const OwnSamples<EX, X2> at_lo{c.r(), c.t(), o, false};
      src_samples<H>(s, n, at_lo, lo);
      mod_values(m, flags, m.conj, mr, nx, at_lo, mv);
#pragma unroll
      for (int k = 0; k < H; ++k) lo[k] = c_mul(lo[k], mv[k]);
      if constexpr (!X2) {
        const OwnSamples<EX, X2> at_hi{c.r(), c.t(), o, true};
        src_samples<H>(s, n, at_hi, hi);
        mod_values(m, flags, m.conj, mr, nx, at_hi, mv);
#pragma unroll
        for (int k = 0; k < H; ++k) hi[k] = c_mul(hi[k], mv[k]);
      }
      if constexpr (COPY) copy_out_done(c);
      trade_fold<EX, X2>(v, lo, hi, c.buf(), c.peer(), c.r(), c.t(), [&] { c.pair_sync(); });
    }
    if (c.r()) fold_odd<EX, X2>(v, p.wpx, c.t());
    EX::template fwd_to<false>(
        v, c.buf(), c.t(), p.twx,
        [&] {
          if constexpr (MF != 0) c.pair_sync();  // the other half has read the traded slots
          else if constexpr (COPY) copy_out_done(c);
        },
        c.qbuf(), c.qt(), [&] { c.quad_sync(); });
    if constexpr (COPY) {
      copy_bins_out<EX>(map, f, c, tile0, v);
      if (threadIdx.x == 0) next->item[turn] = tickets.take(p.fault);
      __syncthreads();
      i = next->item[turn];
    } else {
      store_bins<EX>(p, f, c, tile0 + c.qrow(), v);
      i = -1;
    }
  }
  if constexpr (COPY) {
    if (c.hlead()) top_bulk_wait();
  }
}

// ----------------------------------------------------------------------------- C

// Multiply the bins of half r of column kx by H(kx, ky) / (Py Px), conjugated for the adjoint, from
// the quadrant row of |kx|: bin k of the half holds ky = 2k + r, whose |signed ky| is 2k + r below
// the middle and Py - 2k - r above it, so the even half reads entries k or M - k of the row's even
// part and the odd half entries k or M - 1 - k of its odd part. Entry k = kbase(b) + S j of a part is
// stored at b + S j (the frequency layout), so a warp's loads are consecutive, and bins above the
// middle (j >= RL/2) read entry (RL - 1 - j) S + (S - r - kbase(b)).
template <class EY>
__device__ __forceinline__ void apply_transfer(float2 (&v)[EY::E], const float2* row, int r, bool adjoint, int t) {
  constexpr int M = EY::M, S = EY::SL, RL = EY::RL;
  static_assert(RL % 2 == 0, "the middle falls between slots");
  const float2* part = row + r * (M / 2 + 1);
  const float sg = adjoint ? -1.f : 1.f;
#pragma unroll
  for (int q = 0; q < EY::E / RL; ++q) {
    const int b = t + EY::G * q;
    const int rest = EY::kbase(b) + r;
    const float2* up = part + b;
    const float2* down = part + (rest == 0 ? S : EY::kbase_inv(S - rest));
    // eight loads at a time: the compiler barrier keeps it from hoisting all of them at once
    constexpr int CH = RL % 8 == 0 ? 8 : RL;
#pragma unroll
    for (int j0 = 0; j0 < RL; j0 += CH) {
#pragma unroll
      for (int j = j0; j < j0 + CH; ++j) {
        float2 h = ldg2(j < RL / 2 ? up + j * S : down + (RL - 1 - j) * S);
        h.y *= sg;
        v[q * RL + j] = c_mul(v[q * RL + j], h);
      }
      asm volatile("" ::: "memory");
    }
  }
}

// |signed kx| of a workspace line
__device__ __forceinline__ int line_abs_kx(const PassParams& p, int line) {
  const int r = line >= p.Mx ? 1 : 0;
  const int s = line - r * p.Mx;
  const int j = s / p.xstep, b = s - j * p.xstep;
  const int d0 = b / p.xr1;  // digits of the row plan's first two stages (xr1 = 1: two-stage plans)
  const int k = d0 + (b - d0 * p.xr1) * p.xr0 + j * p.xstep;
  const int kx = 2 * k + r;
  return kx <= p.Px / 2 ? kx : p.Px - kx;
}

// One column per two thread groups, straight between registers and the workspace: the two groups
// share nothing but the trade before the store, so a block has no barrier of its own. Bound by the FMA
// pipe and the L1 data path together (60 and 62 % of their peaks at 1024 points: the exchanges, the
// column's two reads, the H row). Against blocks that staged four-line columns through shared memory: 1024
// points 15.7 -> 12.7 us a field, 4096 points 483 -> 373, 1000 points 38 -> 23.8.
template <class EY, bool X2, int CI>
__global__ void __launch_bounds__(ColShape<EY>::THREADS, ColShape<EY>::MINB) k_cols(const __grid_constant__ PassParams p) {
  using SH = ColShape<EY>;
  constexpr int G = EY::G, E = EY::E, M = EY::M, H = E / 2, COLS = SH::COLS;
  TOP_DYN_SMEM(float2, smem);
  const int grp = int(threadIdx.x) / SH::GW;
  const int t = SH::GW == G ? int(threadIdx.x) % SH::GW : min(int(threadIdx.x) % SH::GW, G - 1);
  const int cl = grp >> 1, r = grp & 1;
  const int ny = p.ny;
  const int line = blockIdx.x * COLS + cl;
  const bool live = line < p.Px;
  const int ln = live ? line : p.Px - 1;
  const int f = blockIdx.y;
  float2* buf = smem + grp * SH::LS;
  const float2* peer = smem + (grp ^ 1) * SH::LS;
  float2* col = p.ws + (long long)f * p.ws_stride +
                (CI == 1 ? (long long)ln * ny : (long long)(ln >> 1) * ny * 2 + (ln & 1));
  auto column_sync = [&] {
    if constexpr (2 * SH::GW <= 32) __syncwarp();
    else top_named_barrier(1 + cl, 2 * SH::GW);
  };
  // the columns of the block one wave of resident blocks later go to L2 while this one works
  if (threadIdx.x == 0 && p.l2_ahead > 0 && !p.spec_in) {
    const long long nb = (long long)gridDim.x * gridDim.y;
    const long long lb = (long long)blockIdx.y * gridDim.x + blockIdx.x + p.l2_ahead;
    if (lb < nb) {
      const int l0 = int(lb % gridDim.x) * COLS, l1 = min(l0 + COLS, p.Px);
      const float2* a = p.ws + (lb / gridDim.x) * p.ws_stride + (long long)l0 * ny;
      if (((unsigned)(l1 - l0) * ny) % 2 == 0 && ((long long)l0 * ny) % 2 == 0) top_prefetch_l2(a, unsigned(l1 - l0) * ny * 8u);
    }
  }
  float2 v[E];
  // spectrum slot of this thread's column and half (spec_in / spec_out)
  const long long spec_at = ((long long)ln * 2 + r) * M + t;
  if (p.spec_in) {
    const float2* sp = p.spec_in + (long long)(f / p.in_repeat) * p.Px * (2 * M) + spec_at;
#pragma unroll
    for (int e = 0; e < E; ++e) v[e] = ldg2(sp + e * G);
  } else {
#pragma unroll
    for (int e = 0; e < E; ++e) {
      const int pos = EY::in_pos(t, e), x0 = sample_lo<EY, X2>(pos, p.oy);
      if constexpr (X2) {
        v[e] = col[x0 * CI];
      } else {
        const int x1 = sample_hi<EY>(pos, p.oy);
        const float2 a = in_line<false>(x0, ny) ? col[x0 * CI] : make_float2(0.f, 0.f);
        const float2 b = in_line<false>(x1, ny) ? col[x1 * CI] : make_float2(0.f, 0.f);
        v[e] = r ? c_sub(a, b) : c_add(a, b);
      }
    }
    if (r) fold_odd<EY, X2>(v, p.wpy, t);
    EY::template fwd_to<false>(v, buf, t, p.twy, [] {}, buf, t, [] { EY::sync_group(); });
  }
  if (p.spec_out) {
    // forward transform only: the spectrum, for the fields that share this source
    if (live) {
      float2* sp = p.spec_out + (long long)f * p.Px * (2 * M) + spec_at;
#pragma unroll
      for (int e = 0; e < E; ++e) sp[e * G] = v[e];
    }
    return;
  }
  const int akx = line_abs_kx(p, ln);
  if (p.hq_out) {
    // forward transform only (a transfer-function table from sampled kernels): half r holds
    // ky = 2k + r, kept where |ky| <= Py/2, i.e. k <= M/2 (even) and k < M/2 (odd), plus the
    // zero that pads each row
    const int rx = ln >= p.Mx ? 1 : 0;
    const int s = ln - rx * p.Mx;
    const bool lower = s < p.Mx / 2 || (s == p.Mx / 2 && rx == 0);  // kx <= Px/2
    if (live && lower) {
      float2* row = p.hq_out + (long long)akx * (M + 2) + r * (M / 2 + 1);
#pragma unroll
      for (int e = 0; e < E; ++e) {
        const int q = e / EY::RL, j = e % EY::RL, b = t + G * q;
        if (j < EY::RL / 2) {
          row[b + EY::SL * j] = c_scale(v[e], p.hq_scale);
        } else if (j == EY::RL / 2 && b == 0) {
          row[M / 2] = r ? make_float2(0.f, 0.f) : c_scale(v[e], p.hq_scale);
        }
      }
    }
    return;
  }
  const float2* hq = p.hq_list ? p.hq_list[f] : p.sets[p.set_of[f]].hq;
  apply_transfer<EY>(v, hq + (long long)akx * (M + 2), r, p.adjoint, t);
  EY::template inv_from<false>(v, buf, t, [] { EY::sync_group(); }, buf, t, [] { EY::sync_group(); }, p.twy);
  if (r) unfold_odd<EY, X2>(v, p.wpy, t);
  float2 lo[H], hi[H];
  trade_combine<EY, X2>(v, lo, hi, buf, peer, r, t, [] { EY::sync_group(); }, column_sync);
  if (live) {
#pragma unroll
    for (int k = 0; k < H; ++k) {
      const int pos = own_pos<EY>(r, t, k), x0 = sample_lo<EY, X2>(pos, p.oy), x1 = sample_hi<EY>(pos, p.oy);
      if (in_line<X2>(x0, ny)) col[x0 * CI] = lo[k];
      if constexpr (!X2) {
        if (in_line<false>(x1, ny)) col[x1 * CI] = hi[k];
      }
    }
  }
}

// ----------------------------------------------------------------------------- R2

// Per-thread float64 sums of the overlap epilogue: psi conj(phi) and |psi|^2.
struct OvAcc {
  double re, im, pw;
};

__device__ __forceinline__ void overlap_add(OvAcc& acc, float2 val, float2 phi) {
  const double vx = val.x, vy = val.y, px = phi.x, py = phi.y;
  acc.re = fma(vx, px, fma(vy, py, acc.re));
  acc.im = fma(vy, px, fma(-vx, py, acc.im));
  acc.pw = fma(vx, vx, fma(vy, vy, acc.pw));
}

// A tile's rows of p.group consecutive fields. At padding 2 the group's intensity and phase partials are
// summed in registers (each own slot stands for one sample of the row), otherwise and for the amplitude
// and mask partials the owner thread adds to the planes in memory; both in field order.
template <class EX, bool X2, int KIND>
struct RowEpilogue {
  static constexpr int H = EX::E / 2;
  static constexpr bool REG_ACC = X2 && (KIND == EPI_INTENSITY || KIND == EPI_MODGRAD);
  static constexpr bool FEW = EX::E < 16;  // samples a thread
  float acc[REG_ACC ? H : 1];
  OvAcc ov;

  // first field of a group: the partials so far
  template <class Lane>
  __device__ __forceinline__ void open(const PassParams& p, const Lane& c, int g, int y) {
    if constexpr (REG_ACC) {
#pragma unroll
      for (int k = 0; k < H; ++k) acc[k] = 0.f;
      if (KIND == EPI_MODGRAD && p.part_phase && p.part_accumulate && c.act() && y < p.ny) {
        const float* src = p.part_phase + (long long)g * p.part_stride + (long long)y * p.nx;
#pragma unroll
        for (int k = 0; k < H; ++k) acc[k] = src[sample_lo<EX, X2>(own_pos<EX>(c.r(), c.t(), k), 0)];
      }
    }
  }
  // last field done
  template <class Lane>
  __device__ __forceinline__ void close(const PassParams& p, const Lane& c, int g, int y) {
    if constexpr (REG_ACC) {
      const long long row0 = (long long)y * p.nx;
      float* dst = KIND == EPI_INTENSITY ? p.outf + (long long)g * p.outf_stride + row0
                                         : (p.part_phase ? p.part_phase + (long long)g * p.part_stride + row0 : nullptr);
      if (c.act() && y < p.ny && dst) {
#pragma unroll
        for (int k = 0; k < H; ++k) dst[sample_lo<EX, X2>(own_pos<EX>(c.r(), c.t(), k), 0)] = acc[k];
      }
    }
  }
  // a round's partials in memory (read only when they are added to)
  template <class V, int N, class At>
  __device__ __forceinline__ static void partials_so_far(const V* part, bool fresh, int nx, At&& of, V (&v)[N]) {
    if (!part || fresh) return;
#pragma unroll
    for (int k = 0; k < N; ++k) v[k] = part[max(0, min(of(k), nx - 1))];
  }
  // the own slots' samples of row y of field f in group g
  template <uint32_t MF, class Lane>
  __device__ __forceinline__ void field(const PassParams& p, const Lane& c, int f, int g, bool first, int y,
                                        const float2 (&lo)[H], const float2 (&hi)[H]) {
    const int nx = p.nx;
    const bool live = y < p.ny && c.act();
    const ModDev& m = p.mepi;
    const uint32_t flags = mod_flags<MF>(m);
    const long long row0 = (long long)y * nx;
    const bool grads = KIND == EPI_MODGRAD && (p.part_phase || p.part_amp || p.part_mask);
    const long long part0 = (long long)g * p.part_stride + row0;
    const FieldSet& fs = p.sets[p.set_of[f]];
    const ModRow mr = mod_row(m, flags, fs.epi_lx, fs.epi_ly, f, live ? y : 0, nx);
    const float w = KIND == EPI_INTENSITY && p.weights ? __ldg(p.weights + f) : 1.f;
    float2* out = KIND == EPI_FIELD ? field_out(p, f) + row0 : (p.out ? p.out + (long long)f * p.out_stride + row0 : nullptr);
    const float2* xs = grads ? p.xs + (long long)f * p.xs_stride + row0 : nullptr;
    const bool fresh = first && !p.part_accumulate;
    // a kernel compiled for a modulation without an amplitude plane and a mask has no gradients of theirs
    constexpr bool PHASE_ONLY = MF != TOP_MOD_DYNAMIC && !(MF & (TOP_MOD_AMPLITUDE | TOP_MOD_COMPLEX));
    ov = OvAcc{0.0, 0.0, 0.0};
    // own slots' samples val0
    auto samples = [&](const float2 (&val0)[H], bool hi_part) {
      const OwnSamples<EX, X2> at{c.r(), c.t(), p.ox, hi_part};
      if constexpr (KIND == EPI_MODGRAD) {
        // val = dL/dy with y = M x (M without conjugation), in rounds of slots. A round has what it reads in
        // flight (saved samples, the mask's operands, the partials so far) before it stores anything: loads
        // do not pass stores, and with a partial loaded, added to and stored slot by slot the pass took 226 us
        // for eight unpadded fields of 1024 x 1024, now 96. Rounds of four keep the three gradients' operands in
        // registers at 16 and more samples a thread; fewer samples, and the phase's gradient alone, go in two.
        constexpr int ROUNDS = PHASE_ONLY || FEW ? (H % 2 == 0 ? 2 : 1) : (H + 3) / 4;
        constexpr int N = (H + ROUNDS - 1) / ROUNDS;
#pragma unroll
        for (int k0 = 0; k0 < H; k0 += N) {
          const auto of = [&](int k) { return k0 + k < H ? at(k0 + k) : -1; };
          float2 mv[N], xv[N];
#pragma unroll
          for (int k = 0; k < N; ++k) xv[k] = grads && k0 + k < H && in_line<X2>(of(k), nx) ? ldg2(xs + of(k)) : make_float2(0.f, 0.f);
          float so_far[N];
          if constexpr (!REG_ACC) partials_so_far(p.part_phase ? p.part_phase + part0 : nullptr, fresh, nx, of, so_far);
          mod_values(m, flags, 0, mr, nx, of, mv);
#pragma unroll
          for (int k = 0; k < N; ++k) {
            const int x = of(k);
            if (k0 + k >= H || !in_line<X2>(x, nx)) continue;
            const float2 val = val0[k0 + k];
            if (out) out[x] = c_mulc(val, mv[k]);  // conj(M) dL/dy
            if (p.part_phase) {
              const float2 ys = c_mul(mv[k], xv[k]);
              const float gp = fmaf(val.y, ys.x, -__fmul_rn(val.x, ys.y));  // Im(val conj(y))
              if constexpr (REG_ACC) acc[k0 + k] = __fadd_rn(acc[k0 + k], gp);
              else p.part_phase[part0 + x] = fresh ? gp : __fadd_rn(so_far[k], gp);
            }
          }
          if (!PHASE_ONLY && p.part_amp) {
            // dM/dA = M without its amplitude factor
            float* part = p.part_amp + part0;
            partials_so_far(part, fresh, nx, of, so_far);
            mod_values(m, flags & ~TOP_MOD_AMPLITUDE, 0, mr, nx, of, mv);
#pragma unroll
            for (int k = 0; k < N; ++k) {
              if (k0 + k >= H || !in_line<X2>(of(k), nx)) continue;
              const float2 val = val0[k0 + k], d = c_mul(mv[k], xv[k]);
              const float ga = fmaf(val.x, d.x, __fmul_rn(val.y, d.y));  // Re(conj(val) d)
              part[of(k)] = fresh ? ga : __fadd_rn(so_far[k], ga);
            }
          }
          if (!PHASE_ONLY && p.part_mask) {
            float2* part = p.part_mask + part0;
            float2 mask_so_far[N];
            partials_so_far(part, fresh, nx, of, mask_so_far);
            mod_values(m, flags & ~TOP_MOD_COMPLEX, 0, mr, nx, of, mv);
#pragma unroll
            for (int k = 0; k < N; ++k) {
              if (k0 + k >= H || !in_line<X2>(of(k), nx)) continue;
              const float2 gm = c_mulc(val0[k0 + k], c_mul(mv[k], xv[k]));  // val conj(M_rest x)
              part[of(k)] = fresh ? gm : c_add(mask_so_far[k], gm);
            }
          }
        }
      } else {
        float2 mv[H];
        if (MF != 0) mod_values(m, flags, m.conj, mr, nx, at, mv);
#pragma unroll
        for (int k = 0; k < H; ++k) {
          const int x = at(k);
          if (!in_line<X2>(x, nx)) continue;
          const float2 val = MF != 0 && flags ? c_mul(val0[k], mv[k]) : val0[k];
          if (KIND == EPI_FIELD || out) out[x] = val;
          if constexpr (KIND == EPI_INTENSITY) {
            const float i = fmaf(val.x, val.x, __fmul_rn(val.y, val.y));
            if constexpr (REG_ACC) {
              // the weight and the sum in one rounding for the 32 x 32 plan, in two for the others: results
              // of either keep the bits they have always had
              acc[k] = EX::NS == 2 && EX::G == 32 ? fmaf(w, i, acc[k]) : __fadd_rn(acc[k], __fmul_rn(w, i));
            } else {
              float* dst = p.outf + (long long)g * p.outf_stride + row0 + x;
              *dst = first ? __fmul_rn(w, i) : __fadd_rn(*dst, __fmul_rn(w, i));
            }
          }
          if constexpr (KIND == EPI_OVERLAP) overlap_add(ov, val, ldg2(p.target + (long long)f * p.target_stride + row0 + x));
        }
      }
    };
    if (live) {
      if constexpr (X2) {
        samples(lo, false);
      } else if constexpr (KIND == EPI_MODGRAD && !FEW) {
        // one copy of the code for both ends of the line: two spilled 250 bytes and more
        float2 val[H];
#pragma unroll 1
        for (int part = 0; part < 2; ++part) {
#pragma unroll
          for (int k = 0; k < H; ++k) val[k] = part ? hi[k] : lo[k];
          samples(val, part != 0);
        }
      } else {
        samples(lo, false);
        samples(hi, true);
      }
    }
  }
};

// Blocks an SM. The gradients of any set of planes take the next larger number of registers a thread, 128
// instead of 80 and 80 instead of 64 (64 unpadded fields of 256 x 256: 118 us a backward at 80, 87 at 128).
template <class SH, int KIND, uint32_t MF>
constexpr int inv_min_blocks() {
  constexpr int wider = 65536 / (SH::THREADS * (SH::REGS == 64 ? 80 : 128));
  return KIND == EPI_MODGRAD && MF == TOP_MOD_DYNAMIC && wider > 0 ? wider : SH::MINB;
}

// Inverse rows. Without COPY a block holds its tiles for the fields of one group and reads bins straight
// from the workspace; with it two tiles share a TileFeed.
template <class EX, bool X2, int KIND, uint32_t MF, bool COPY>
__global__ void __launch_bounds__(RowBlock<EX, COPY ? 2 : row_tiles<EX>()>::THREADS,
                                  inv_min_blocks<RowBlock<EX, COPY ? 2 : row_tiles<EX>()>, KIND, MF>())
    k_rows_inv(const __grid_constant__ PassParams p, const __grid_constant__ TileMap map) {
  constexpr int T = COPY ? 2 : row_tiles<EX>();
  using SH = RowBlock<EX, T>;
  constexpr int E = EX::E, H = E / 2;
  static_assert(!COPY || KIND != EPI_OVERLAP, "the overlap sums are taken by whole blocks");
  TOP_DYN_SMEM(float2, smem);
  const RowLane<EX, T> c(smem);
  RowEpilogue<EX, X2, KIND> epi;
  float2 v[E];
  float2 lo[H], hi[H];
  if constexpr (COPY) {
    TileFeed<EX> feed(smem, p.ny, p.nfields, p.group, p.l2_ahead);
    if (threadIdx.x == 0) feed.start(map);
#pragma unroll 1
    while (feed.take(map, c, p.fault, v)) {
      EX::template inv_from<false>(v, c.qbuf(), c.qt(), [] {}, c.buf(), c.t(), [&] { c.quad_sync(); }, p.twx);
      if (c.r()) unfold_odd<EX, X2>(v, p.wpx, c.t());
      trade_combine<EX, X2>(v, lo, hi, c.buf(), c.peer(), c.r(), c.t(), [] { EX::sync_group(); }, [&] { c.pair_sync(); });
      const int f = feed.field(), g = feed.item() / feed.ntiles, y = feed.y0() + c.row();
      const bool first = f == g * p.group;
      if (first) epi.open(p, c, g, y);
      epi.template field<MF>(p, c, f, g, first, y, lo, hi);
      if (f + 1 == feed.end_field(feed.item())) epi.close(p, c, g, y);
    }
  } else {
    const int tile0 = (blockIdx.x * SH::T + c.tile()) * SH::ROWS;
    const int y = tile0 + c.row();
    const int g = blockIdx.y;
    const int f0 = g * p.group, f1 = min(f0 + p.group, p.nfields);
    epi.open(p, c, g, y);
#pragma unroll 1
    for (int f = f0; f < f1; ++f) {
      load_bins<EX>(p, f, c, tile0 + c.qrow(), v);
      EX::template inv_from<KIND != EPI_MODGRAD || !X2>(
          v, c.qbuf(), c.qt(),
          [&] {
            if (f > f0) c.tile_sync();  // the previous field's trade has been read
          },
          c.buf(), c.t(), [&] { c.quad_sync(); }, p.twx);
      if (c.r()) unfold_odd<EX, X2>(v, p.wpx, c.t());
      trade_combine<EX, X2>(v, lo, hi, c.buf(), c.peer(), c.r(), c.t(), [] { EX::sync_group(); }, [&] { c.pair_sync(); });
      epi.template field<MF>(p, c, f, g, f == f0, y, lo, hi);
      if constexpr (KIND == EPI_OVERLAP) {
        // the block's sums in a fixed order: over the lanes of each warp, then over the warps (one thread that adds
        // every thread's three values held the pass at 379 us for eight fields of 1024 x 1024, now 193)
        double sum[3] = {epi.ov.re, epi.ov.im, epi.ov.pw};
#pragma unroll
        for (int d = 16; d > 0; d >>= 1)
#pragma unroll
          for (int q = 0; q < 3; ++q) sum[q] += __shfl_xor_sync(0xffffffffu, sum[q], d);
        __syncthreads();
        double* red = reinterpret_cast<double*>(smem);
        if (threadIdx.x % 32 == 0) {
#pragma unroll
          for (int q = 0; q < 3; ++q) red[threadIdx.x / 32 * 3 + q] = sum[q];
        }
        __syncthreads();
        if (threadIdx.x < 3) {
          double total = 0.0;
          for (int i = 0; i < SH::THREADS / 32; ++i) total += red[3 * i + threadIdx.x];
          p.ov_part[((long long)f * gridDim.x + blockIdx.x) * 3 + threadIdx.x] = total;
        }
        __syncthreads();
      }
    }
    epi.close(p, c, g, y);
  }
}

// ----------------------------------------------------------------------------- R2 + R1 fused

// The inverse row pass of one propagation (pa) fused with the forward row pass of the next (pb) in a
// system chain (Eq. 1 and Eq. 4 in turn): the field between them stays in registers and reaches
// global memory only when it is kept (pa.out). pb's bins replace pa's in the workspace, tile by tile,
// each tile read before it is written. With COPY tiles come by TileFeed and leave by copy.
template <class EX, bool X2, uint32_t MF, bool COPY>
__global__ void __launch_bounds__(RowBlock<EX, COPY ? 2 : row_tiles<EX>()>::THREADS, RowBlock<EX, COPY ? 2 : row_tiles<EX>()>::MINB)
    k_rows_chain(const __grid_constant__ PassParams pa, const __grid_constant__ PassParams pb,
                 const __grid_constant__ TileMap map) {
  constexpr int T = COPY ? 2 : row_tiles<EX>();
  using SH = RowBlock<EX, T>;
  constexpr int E = EX::E, H = E / 2;
  TOP_DYN_SMEM(float2, smem);
  const RowLane<EX, T> c(smem);
  const int nx = pa.nx;
  const ModDev& m = pb.msrc;
  const uint32_t flags = mod_flags<MF>(m);
  float2 v[E];
  // bins of (f, rows from tile0) in v to the next propagation's bins in v
  auto tile = [&](int f, int tile0) {
    const int y = tile0 + c.row();
    const bool live = y < pa.ny;
    EX::template inv_from<!COPY>(
        v, c.qbuf(), c.qt(),
        [&] {
          if constexpr (COPY) copy_out_done(c);
        },
        c.buf(), c.t(), [&] { c.quad_sync(); }, pa.twx);
    if (c.r()) unfold_odd<EX, X2>(v, pa.wpx, c.t());
    float2 lo[H], hi[H];
    trade_combine<EX, X2>(v, lo, hi, c.buf(), c.peer(), c.r(), c.t(), [] { EX::sync_group(); }, [&] { c.pair_sync(); });
    const FieldSet& fsb = pb.sets[pb.set_of[f]];
    const ModRow mr = mod_row(m, flags, fsb.src_lx, fsb.src_ly, f, live ? y : 0, nx);
    float2* kept = pa.out ? pa.out + (long long)f * pa.out_stride + (long long)y * nx : nullptr;
    const int n = live ? nx : 0;
    auto samples = [&](float2 (&val)[H], bool hi_part) {
      const OwnSamples<EX, X2> at{c.r(), c.t(), pa.ox, hi_part};
      if (kept) {
#pragma unroll
        for (int k = 0; k < H; ++k)
          if ((unsigned)at(k) < (unsigned)n) kept[at(k)] = val[k];
      }
      if (MF != 0) {
        float2 mv[H];
        mod_values(m, flags, m.conj, mr, nx, at, mv);
#pragma unroll
        for (int k = 0; k < H; ++k) val[k] = c_mul(val[k], mv[k]);
      }
#pragma unroll
      for (int k = 0; k < H; ++k)
        if ((unsigned)at(k) >= (unsigned)n) val[k] = make_float2(0.f, 0.f);
    };
    samples(lo, false);
    if constexpr (!X2) samples(hi, true);
    trade_fold<EX, X2>(v, lo, hi, c.buf(), c.peer(), c.r(), c.t(), [&] { c.pair_sync(); });
    if (c.r()) fold_odd<EX, X2>(v, pb.wpx, c.t());
    EX::template fwd_to<true>(v, c.buf(), c.t(), pb.twx, [&] { c.pair_sync(); }, c.qbuf(), c.qt(), [&] { c.quad_sync(); });
  };
  if constexpr (COPY) {
    TileFeed<EX> feed(smem, pa.ny, pa.nfields, 1, pa.l2_ahead);
    if (threadIdx.x == 0) feed.start(map);
#pragma unroll 1
    while (feed.take(map, c, pa.fault, v)) {
      tile(feed.field(), feed.y0());
      copy_bins_out<EX>(map, feed.field(), c, feed.y0(), v);
    }
    if (c.hlead()) top_bulk_wait();
  } else {
    const int tile0 = (blockIdx.x * SH::T + c.tile()) * SH::ROWS;
    const int f = blockIdx.y;
    load_bins<EX>(pa, f, c, tile0 + c.qrow(), v);
    tile(f, tile0);
    store_bins<EX>(pb, f, c, tile0 + c.qrow(), v);
  }
}

// ----------------------------------------------------------------------------- launchers

// The kernels are compiled for the modulation flag sets of common elements (none, a phase mask, a lens
// or a phase mask behind an aperture) and for flags read at run time.
constexpr uint32_t kPhase = TOP_MOD_PHASE;
constexpr uint32_t kLensCirc = TOP_MOD_LENS | TOP_MOD_CIRC;
constexpr uint32_t kPhaseCirc = TOP_MOD_PHASE | TOP_MOD_CIRC;

// Whether lines start on 16-byte boundaries, as tile copies need.
template <class EX>
inline bool copies(const PassParams& p) {
  using SH = RowShape<EX>;
  return SH::COPY && (p.ny * SH::CI) % 2 == 0;
}
// The passes that also load tiles by copy want three tiles or more for each resident group of a launch:
// one tile each, the pipeline only adds its start (one 1024 x 1024 field: inverse rows 13.5 us direct,
// 14.7 by copy; four fields: 35.1 and 31.2; 16 fields at 512: 27.4 and 26.9).
template <class EX>
inline bool copies_in(const PassParams& p, int resident) {
  return copies<EX>(p) && (long long)p.ny * p.nfields >= 6LL * RowShape<EX>::ROWS * resident;
}
template <class EX>
inline cudaError_t tile_map(const PassParams& p, TileMap* map, bool with_wide) {
  using SH = RowShape<EX>;
  return encode_tile_map(map, p.ws, p.ny * SH::CI, p.Px / SH::CI, p.nfields, p.ws_stride, SH::LB, with_wide);
}

template <class EX, bool X2, uint32_t MF, bool COPY>
cudaError_t launch_rows_fwd_k(const PassParams& p, cudaStream_t s) {
  using SH = RowBlock<EX, row_tiles<EX>()>;
  static KernelOnDevices setup;
  int resident = 0;
  const cudaError_t ready = setup.ready(k_rows_fwd<EX, X2, MF, COPY>, SH::THREADS, SH::SMEM_X, &resident);
  if (ready != cudaSuccess) return ready;
  PassParams q = p;
  // bulk prefetches move whole 16-byte units
  q.l2_ahead = p.nx % 2 == 0 && !(p.tune_rows & TOP_TUNE_NO_L2_FWD) ? resident : 0;
  const int tiles = (p.ny + SH::BLOCK_ROWS - 1) / SH::BLOCK_ROWS;
  const dim3 grid(COPY ? tiles * p.nfields : tiles, COPY ? 1 : p.nfields);
  TileMap map{};
  if (COPY) {
    const cudaError_t e = tile_map<EX>(p, &map, false);
    if (e != cudaSuccess) return e;
  }
  TOP_LAUNCH((k_rows_fwd<EX, X2, MF, COPY>), grid, SH::THREADS, SH::SMEM_X, s, q, map);
  return cudaGetLastError();
}
template <class EX, bool X2, uint32_t MF>
cudaError_t launch_rows_fwd_m(const PassParams& p, cudaStream_t s) {
  if constexpr (RowShape<EX>::COPY) {
    if (copies<EX>(p)) return launch_rows_fwd_k<EX, X2, MF, true>(p, s);
  }
  return launch_rows_fwd_k<EX, X2, MF, false>(p, s);
}

template <class EX, bool X2>
cudaError_t launch_rows_fwd_t(const PassParams& p, cudaStream_t s) {
  const uint32_t fl = p.msrc.flags;
  if (fl == 0) return launch_rows_fwd_m<EX, X2, 0>(p, s);
  if constexpr (X2) {
    if (fl == kPhase) return launch_rows_fwd_m<EX, X2, kPhase>(p, s);
  }
  return launch_rows_fwd_m<EX, X2, TOP_MOD_DYNAMIC>(p, s);
}

template <class EY, bool X2, int CI>
cudaError_t launch_cols_k(const PassParams& p, cudaStream_t s) {
  using SH = ColShape<EY>;
  static KernelOnDevices setup;
  int resident = 0;
  const cudaError_t ready = setup.ready(k_cols<EY, X2, CI>, SH::THREADS, SH::SMEM, &resident);
  if (ready != cudaSuccess) return ready;
  PassParams q = p;
  q.l2_ahead = !(p.tune_cols & TOP_TUNE_NO_L2_COLS) ? resident : 0;
  dim3 grid((p.Px + SH::COLS - 1) / SH::COLS, p.nfields);
  TOP_LAUNCH((k_cols<EY, X2, CI>), grid, SH::THREADS, SH::SMEM, s, q);
  return cudaGetLastError();
}

template <class EX, bool X2, int KIND, uint32_t MF>
cudaError_t launch_rows_inv_k(const PassParams& p, cudaStream_t s) {
  PassParams q = p;
  if (KIND == EPI_FIELD) q.group = 1;  // no sums: one field at a time
  const int groups = (q.nfields + q.group - 1) / q.group;
  if constexpr (RowShape<EX>::COPY && KIND != EPI_OVERLAP) {
    using SH = RowBlock<EX, 2>;
    static KernelOnDevices setup;
    int resident = 0;
    const cudaError_t ready = setup.ready(k_rows_inv<EX, X2, KIND, MF, true>, SH::THREADS, SH::SMEM_DUO, &resident);
    if (ready != cudaSuccess) return ready;
    if (copies_in<EX>(p, resident)) {
      TileMap map{};
      const cudaError_t e = tile_map<EX>(p, &map, true);
      if (e != cudaSuccess) return e;
      const int items = (p.ny + SH::ROWS - 1) / SH::ROWS * groups;
      q.l2_ahead = 2 * resident;  // both groups of every resident block
      TOP_LAUNCH((k_rows_inv<EX, X2, KIND, MF, true>), items, SH::THREADS, SH::SMEM_DUO, s, q, map);
      return cudaGetLastError();
    }
  }
  using SH = RowBlock<EX, row_tiles<EX>()>;
  static KernelOnDevices setup;
  int resident = 0;
  const cudaError_t ready = setup.ready(k_rows_inv<EX, X2, KIND, MF, false>, SH::THREADS, SH::SMEM_X, &resident);
  if (ready != cudaSuccess) return ready;
  dim3 grid((q.ny + SH::BLOCK_ROWS - 1) / SH::BLOCK_ROWS, groups);
  TOP_LAUNCH((k_rows_inv<EX, X2, KIND, MF, false>), grid, SH::THREADS, SH::SMEM_X, s, q, TileMap{});
  return cudaGetLastError();
}

template <class EX, bool X2>
cudaError_t launch_rows_inv_t(const PassParams& p, cudaStream_t s) {
  const uint32_t fl = p.mepi.flags;
  switch (p.epi_kind) {
    case EPI_FIELD:
      return fl == 0 ? launch_rows_inv_k<EX, X2, EPI_FIELD, 0>(p, s) : launch_rows_inv_k<EX, X2, EPI_FIELD, TOP_MOD_DYNAMIC>(p, s);
    case EPI_INTENSITY:
      return fl == 0 ? launch_rows_inv_k<EX, X2, EPI_INTENSITY, 0>(p, s)
                     : launch_rows_inv_k<EX, X2, EPI_INTENSITY, TOP_MOD_DYNAMIC>(p, s);
    case EPI_MODGRAD:
      if constexpr (X2) {
        if (fl == kPhase) return launch_rows_inv_k<EX, X2, EPI_MODGRAD, kPhase>(p, s);
        if (fl == kPhaseCirc) return launch_rows_inv_k<EX, X2, EPI_MODGRAD, kPhaseCirc>(p, s);
      }
      return launch_rows_inv_k<EX, X2, EPI_MODGRAD, TOP_MOD_DYNAMIC>(p, s);
    default:
      return launch_rows_inv_k<EX, X2, EPI_OVERLAP, TOP_MOD_DYNAMIC>(p, s);
  }
}

template <class EX, bool X2, uint32_t MF>
cudaError_t launch_rows_chain_k(const PassParams& pa, const PassParams& pb, cudaStream_t s) {
  if constexpr (RowShape<EX>::COPY) {
    using SH = RowBlock<EX, 2>;
    static KernelOnDevices setup;
    int resident = 0;
    const cudaError_t ready = setup.ready(k_rows_chain<EX, X2, MF, true>, SH::THREADS, SH::SMEM_DUO, &resident);
    if (ready != cudaSuccess) return ready;
    if (copies_in<EX>(pa, resident)) {
      TileMap map{};
      const cudaError_t e = tile_map<EX>(pa, &map, false);
      if (e != cudaSuccess) return e;
      const int items = (pa.ny + SH::ROWS - 1) / SH::ROWS * pa.nfields;
      PassParams qa = pa;
      qa.l2_ahead = 0;  // its tiles are a while in coming; prefetches measured slower (9.7 -> 10.0 us a field)
      TOP_LAUNCH((k_rows_chain<EX, X2, MF, true>), items, SH::THREADS, SH::SMEM_DUO, s, qa, pb, map);
      return cudaGetLastError();
    }
  }
  using SH = RowBlock<EX, row_tiles<EX>()>;
  static KernelOnDevices setup;
  int resident = 0;
  const cudaError_t ready = setup.ready(k_rows_chain<EX, X2, MF, false>, SH::THREADS, SH::SMEM_X, &resident);
  if (ready != cudaSuccess) return ready;
  dim3 grid((pa.ny + SH::BLOCK_ROWS - 1) / SH::BLOCK_ROWS, pa.nfields);
  TOP_LAUNCH((k_rows_chain<EX, X2, MF, false>), grid, SH::THREADS, SH::SMEM_X, s, pa, pb, TileMap{});
  return cudaGetLastError();
}

template <class EX, bool X2>
cudaError_t launch_rows_chain_t(const PassParams& pa, const PassParams& pb, cudaStream_t s) {
  const uint32_t fl = pb.msrc.flags;
  if constexpr (X2) {
    if (fl == 0) return launch_rows_chain_k<EX, X2, 0>(pa, pb, s);
    if (fl == kPhase) return launch_rows_chain_k<EX, X2, kPhase>(pa, pb, s);
    if (fl == kLensCirc) return launch_rows_chain_k<EX, X2, kLensCirc>(pa, pb, s);
    if (fl == kPhaseCirc) return launch_rows_chain_k<EX, X2, kPhaseCirc>(pa, pb, s);
  }
  return launch_rows_chain_k<EX, X2, TOP_MOD_DYNAMIC>(pa, pb, s);
}

// padding exactly 2 along an axis: n = M and the field sits at M/2
inline bool exact2(int n, int M, int o) { return n == M && o == M / 2; }

template <class EX>
cudaError_t launch_rows_fwd(const PassParams& p, cudaStream_t s) {
  return exact2(p.nx, p.Mx, p.ox) ? launch_rows_fwd_t<EX, true>(p, s) : launch_rows_fwd_t<EX, false>(p, s);
}
template <class EY>
cudaError_t launch_cols(const PassParams& p, cudaStream_t s) {
  if (p.ci == 2) return exact2(p.ny, p.My, p.oy) ? launch_cols_k<EY, true, 2>(p, s) : launch_cols_k<EY, false, 2>(p, s);
  return exact2(p.ny, p.My, p.oy) ? launch_cols_k<EY, true, 1>(p, s) : launch_cols_k<EY, false, 1>(p, s);
}
template <class EX>
cudaError_t launch_rows_chain(const PassParams& pa, const PassParams& pb, cudaStream_t s) {
  return exact2(pa.nx, pa.Mx, pa.ox) ? launch_rows_chain_t<EX, true>(pa, pb, s) : launch_rows_chain_t<EX, false>(pa, pb, s);
}
template <class EX>
cudaError_t launch_rows_inv(const PassParams& p, cudaStream_t s) {
  return exact2(p.nx, p.Mx, p.ox) ? launch_rows_inv_t<EX, true>(p, s) : launch_rows_inv_t<EX, false>(p, s);
}

}  // namespace top
