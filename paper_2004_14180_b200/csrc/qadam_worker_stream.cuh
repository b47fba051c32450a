// The worker side of pairs too large for the chip: two pipelined passes over memory.
//
//   worker_sweep_kernel    moments on the server, ternary and five-level codes: forms u and finishes
//                          whatever a lower bound of the scale settles
//   worker_form_kernel     everything else: folds max |u|; with the moments on the workers u, formed
//                          after the moment updates, is left in e's place
//   worker_settle_kernel   codes and e', once the scales are final: of every row, or of what the sweep
//                          left; u out of e's place, or of g and e again
// (Leaving u in e's place in every case moves the same bytes, but a first pass that only reads is
// faster than one that writes: 1.2 x 10^8 dense elements, n = 2, both passes 792 us with u written.)
//
// One CTA per SM.  A producer thread brings tiles of 4096 elements into a ring of shared-memory
// stages with bulk copies that complete on an mbarrier; consumer warps work from the stages and
// store their results from registers.  Tiles are handed out by a counter, in the order of memory.
// That order is what the rate depends on: CTAs that take every G-th tile drift apart, and DRAM then
// serves a wide set of open rows for reads and writes at once.  The traffic of the sweep (read g, e,
// write e and codes, 2^28 elements): 6.2 TB/s with static strides and 128 KB of loads in flight per SM,
// 6.9 with 64 KB in flight, 6.9 .. 7.0 with tiles in order, whatever is in flight.
//
// Every wait on an mbarrier is bounded as in the server pass.
#pragma once

#include "qadam_server_pipe.cuh"

namespace qadam {

constexpr int kStreamWarps = 16;                      // consumer warps
constexpr int kStreamGroups = 2;                      // of 8 warps, which take alternate tiles (sweep, settle)
constexpr int kStreamThreads = kStreamWarps * 32 + 64;// and a warp each for the producer and the exchange of bounds
constexpr int kStreamMaxStages = 8;
constexpr int kStreamHeadBytes = 1024;
constexpr unsigned kNoTile = ~0u;
constexpr int kChunkRows = 4;                         // rows of 128 elements with a byte of flags
constexpr int kChunkElems = kChunkRows * 128;
constexpr int kTileChunks = kTileElems / kChunkElems; // 8

// Words of the workspace the two passes count in; zero between launches (a launch's last CTA clears its own,
// which spares the step a clear).
struct StreamCounters {
  unsigned form_tickets, form_left;      // tiles handed out beyond each CTA's first ones; CTAs that have left
  unsigned settle_tickets, settle_left;
  unsigned rows;                         // rows of 128 elements the sweep flagged
};

struct StreamHeader {
  long long off;            // first element of the tile
  unsigned long long flags; // settle pass after a sweep: byte c, bit i: row 4 c + i is to be settled
  int count;                // elements of the tile
  unsigned t;               // its number in the call, kNoTile: no more tiles
  int worker;
  unsigned pair;            // worker * S + segment
  unsigned scale_bits;      // settle pass: the pair's final scale
};
struct StreamSmem {
  unsigned long long full[kStreamMaxStages];
  unsigned long long empty[kStreamMaxStages];
  // sweep: {pair, bits of a maximum}, what the block knows of its pair, and what is known to be in the
  // pair's word.  Pairs grow along the block's tiles, so a 64-bit maximum lets a newer pair replace an
  // older one.
  unsigned long long known, published;
  StreamHeader hd[kStreamMaxStages];
  unsigned pair;            // sweep: of the tile issued last, kNoTile: there are no more; settle pass: rows flagged
  int abort_flag;
};
static_assert(sizeof(StreamSmem) <= kStreamHeadBytes, "head of the shared-memory layout");

// A stage: [g][e][m][v][held weights of the l2 term], or u alone in the settle pass after one with m, v
__host__ __device__ constexpr int form_stage_bytes(bool worker_moments, int held_bytes) {
  return (worker_moments ? 4 : 2) * kTileElems * 4 + held_bytes;
}
__host__ __device__ constexpr int settle_stage_bytes(bool worker_moments, int held_bytes) {
  return worker_moments ? kTileElems * 4 : form_stage_bytes(false, held_bytes);
}
inline int stream_stages(int max_smem, int stage_bytes) {
  const int stages = (max_smem - kStreamHeadBytes) / stage_bytes;
  return stages < kStreamMaxStages ? stages : kStreamMaxStages;
}
inline size_t stream_smem_bytes(int stages, int stage_bytes) { return kStreamHeadBytes + (size_t)stages * stage_bytes; }

__device__ __forceinline__ void stream_init(StreamSmem* ps, int stages, int readers, unsigned pair) {
  if (threadIdx.x == 0) {
    for (int s = 0; s < stages; ++s) {
      mbar_init(&ps->full[s], 1);
      mbar_init(&ps->empty[s], readers);
    }
    ps->known = ps->published = 0ull;
    ps->pair = pair;
    ps->abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
}

// By the producer thread, once it draws no more: the last CTA's clears the launch's counters for the next.  Every
// CTA's draws, and whatever of the counters it has read, come before its count (release), all counts before the
// clearing (acquire).
__device__ __forceinline__ void stream_leave(unsigned* tickets, unsigned* left, unsigned* also) {
  unsigned gone;
  asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], 1;" : "=r"(gone) : "l"(left) : "memory");
  if (gone == gridDim.x - 1u) {
    *tickets = 0u;
    *left = 0u;
    if (also) *also = 0u;
  }
}

// The producer thread.  look(t): what has to be known of a tile, besides its descriptor, before it is
// issued (both are asked for two rounds ahead); issue(tile, worker, t, look, stage, header): header and
// copies of a tile, false if it needs no stage; `ends` marks for the consumers close the ring.
template <typename Look, typename Issue>
__device__ __forceinline__ void produce_tiles(const StreamParams& p, StreamSmem* ps, unsigned* tickets,
                                              bool backwards, int ends, Look&& look, Issue&& issue) {
  volatile int* abort_flag = &ps->abort_flag;
  const int stages = p.stages;
  const unsigned total = (unsigned)p.total_tiles, tpw = (unsigned)p.tiles_per_worker;
  int s = 0;
  unsigned ph = 0, armed = 0, armed_par = 0;
  constexpr int kAhead = 8;
  const auto draw = [&]() { return kAhead * gridDim.x + atomicAdd(tickets, 1u); };
  const auto place = [&](unsigned at) { return backwards ? total - 1u - at : at; };
  const auto descriptor = [&](unsigned at) { return at < total ? p.tiles[place(at) % tpw] : Tile{0, 0, 0}; };
  const auto looked = [&](unsigned at) { return at < total ? look(place(at)) : 0ull; };
  // (a fresh barrier passes a wait on the parity opposite to its first phase)
  const auto stage_free = [&]() {
    return mbar_wait_bounded(&ps->empty[s], ph ^ 1u, abort_flag, p.status, p.spin_limit);
  };
  // Numbers are drawn kAhead tiles before their turn (the first kAhead are every G-th tile, so that
  // nothing waits at the start), descriptors asked for two tiles before it: a trip to L2 takes as long as
  // a tile or two, an atomic on one address for all SMs the longest (drawn three ahead: 1.2 x 10^8
  // dense elements, n = 2, second pass 388 -> 371 us with eight).  Slots are named by unrolling, not
  // moved along: a move would wait for what is on its way.
  unsigned nt[kAhead];
#pragma unroll
  for (int k = 0; k < kAhead; ++k) nt[k] = blockIdx.x + k * gridDim.x;
  Tile tile[4] = {descriptor(nt[0]), descriptor(nt[1]), {0, 0, 0}, {0, 0, 0}};
  unsigned long long seen[4] = {looked(nt[0]), looked(nt[1]), 0ull, 0ull};
  bool more = true;
  while (more) {
#pragma unroll
    for (int k = 0; k < kAhead; ++k) {
      tile[(k + 2) & 3] = descriptor(nt[(k + 2) % kAhead]);
      seen[(k + 2) & 3] = looked(nt[(k + 2) % kAhead]);
      if (nt[k] >= total || !stage_free()) {
        more = false;
        break;
      }
      const unsigned at = place(nt[k]);
      if (issue(tile[k & 3], at / tpw, at, seen[k & 3], s, &ps->hd[s])) {
        armed |= 1u << s;
        armed_par = (armed_par & ~(1u << s)) | (ph << s);
        if (++s == stages) { s = 0; ph ^= 1u; }
      }
      nt[k] = draw();
    }
  }
  for (int i = 0; i < ends && !*abort_flag && stage_free(); ++i) {
    ps->hd[s].t = kNoTile;
    mbar_arrive(&ps->full[s]);
    if (++s == stages) { s = 0; ph ^= 1u; }
  }
  *reinterpret_cast<volatile unsigned*>(&ps->pair) = kNoTile;
  // drain after an abort: nothing may still be landing in shared memory when the CTA exits
  if (*abort_flag) {
    for (int ds = 0; ds < stages; ++ds) {
      if (!((armed >> ds) & 1u)) continue;
      for (unsigned it = 0; it < kSpinLimit; ++it) {
        if (mbar_try_wait(&ps->full[ds], (armed_par >> ds) & 1u)) break;
        __nanosleep(100);
      }
    }
  }
}

// g, e (m, v, the held weights) of a tile into its stage
template <bool WM, bool L2>
__device__ __forceinline__ void issue_inputs(const WorkerParams& p, unsigned char* st, const Tile& tile, unsigned wl,
                                             unsigned long long* full) {
  const unsigned bytes = (unsigned)tile.count * 4u;
  const int hbits = p.kx < 0 ? 32 : p.xbits;
  const unsigned hbytes = L2 ? (unsigned)(tile.count / 8 * hbits) : 0u;
  const long long so = (long long)(p.worker_begin + (int)wl) * p.D + tile.off;
  mbar_arrive_expect_tx(full, (WM ? 4u : 2u) * bytes + hbytes);
  bulk_load(st, p.g + (long long)wl * p.D + tile.off, bytes, full);
  bulk_load(st + kTileElems * 4, p.e + so, bytes, full);
  if constexpr (WM) {
    bulk_load(st + 2 * kTileElems * 4, p.m + so, bytes, full);
    bulk_load(st + 3 * kTileElems * 4, p.v + so, bytes, full);
  }
  if constexpr (L2)       // tile starts are multiples of 128 elements: 16-byte aligned at any width
    bulk_load(st + form_stage_bytes(WM, 0),
              (p.kx < 0 ? reinterpret_cast<const unsigned char*>(p.x) : p.wcodes) + tile.off / 8 * hbits, hbytes, full);
}
__device__ __forceinline__ void fill_header(const WorkerParams& p, StreamHeader* hd, const Tile& tile, unsigned wl,
                                            unsigned t) {
  hd->off = tile.off;
  hd->count = tile.count;
  hd->t = t;
  hd->worker = p.worker_begin + (int)wl;
  hd->pair = (unsigned)hd->worker * (unsigned)p.S + (unsigned)tile.seg;
}

// ---------------------------------------------------------------------------
// Moments on the server, ternary and five-level codes.
//
// A coordinate has level 0 whenever |u| <= t s, t = 2^-(k+1) the lowest midpoint of the grid,
// and then its code is L and e' = u: the scale itself does not enter.  Any maximum seen so far
// bounds s from below, so a row of 128 elements whose largest |u| is at most t times that bound is
// finished in the sweep: 12 + b/8 bytes per element, the least there is.  Of a row with few open
// elements (at most kListedPerRow) level 0 is written for all, and the open ones are listed with their u:
// when the scale is known the settle pass goes over the list and mends those whose level turns out not
// to be 0 (a 4-byte store of e' and an exclusive-or of the code each).  Every other row is left untouched
// and flagged, and the settle pass reads its g and e again: 20 + b/8 bytes in all, as in two full passes.  The error
// feedback keeps the codes of heavy-tailed gradients
// sparse (2^28 elements of the benchmark's mixture after 18 steps: 10 % of the rows hold a code
// other than level 0, as a rule one or two).  Flagging all of these, the second pass took 1.53 ms there
// (n = 16), with the list 0.41.  A listed element costs some 33 ps (its entry written and read, two
// scattered accesses of 4 bytes), a row left 150 ps (1 KB more): with up to 8 listed per row in
// place of 4, 1.2 x 10^8 Gaussian elements, n = 2, of which one in twenty is open, took 5 % longer.
//
// Two groups of 8 warps take alternate tiles; a warp owns 512 consecutive elements (4 rows, so that
// its ternary codes are one 128-byte line).  The block keeps the bound of its current pair in shared
// memory; a warp of its own exchanges it with the pair's word of the scales, about once a tile, so
// that no tile waits for it.  The first tiles of a pair find a low bound and are mostly left: a few per
// mille of a pair of 10^8 elements.
// ---------------------------------------------------------------------------
constexpr unsigned kListedPerRow = 4;                 // open elements of a row, at most, that are listed
constexpr unsigned kListParts = 3;                    // warps a region is dealt out to (4 x 10^8 elements: 43.8 -> 41.7 us; few: 0.5 more)
constexpr int kListBatch = 4;

// BITS: code width, 2 (ternary) or 3 (five levels).
template <int BITS, bool L2>
__global__ void __launch_bounds__(kStreamThreads, 1)
worker_sweep_kernel(const StreamParams p) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  StreamSmem* ps = reinterpret_cast<StreamSmem*>(smem_raw);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int stages = p.stages;
  const int stage_bytes = form_stage_bytes(false, L2 ? held_tile_bytes(p.kx, p.xbits) : 0);
  unsigned char* ring = smem_raw + kStreamHeadBytes;
  volatile unsigned long long* known = &ps->known;
  volatile int* abort_flag = &ps->abort_flag;
  stream_init(ps, stages, kStreamWarps / kStreamGroups + p.missing_readers, (unsigned)p.worker_begin * (unsigned)p.S);

  if (warp == kStreamWarps) {
    if (lane == 0) {
      produce_tiles(
          p, ps, &p.counters->form_tickets, false, kStreamGroups, [&](unsigned) { return 0ull; },
          [&](const Tile& tile, unsigned wl, unsigned t, unsigned long long, int s, StreamHeader* hd) {
            fill_header(p, hd, tile, wl, t);
            *reinterpret_cast<volatile unsigned*>(&ps->pair) = hd->pair;
            issue_inputs<false, L2>(p, ring + (size_t)s * stage_bytes, tile, wl, &ps->full[s]);
            return true;
          });
      stream_leave(&p.counters->form_tickets, &p.counters->form_left, nullptr);
    }
  } else if (warp == kStreamWarps + 1) {
    // ------------------------------------------------------------------ exchange of bounds
    // (ends when the producer has issued its last tile, which its bounded waits see to)
    unsigned pair;
    while (lane == 0 && (pair = *reinterpret_cast<volatile unsigned*>(&ps->pair)) != kNoTile) {
      const unsigned long long tag = (unsigned long long)pair << 32;
      const unsigned word = *reinterpret_cast<volatile const unsigned*>(p.scale_bits + pair);
      const unsigned long long kn = *known;
      const unsigned mine = (unsigned)(kn >> 32) == pair ? (unsigned)kn : 0u;
      if (mine > word) atomicMax(p.scale_bits + pair, mine);
      else if (word > mine) atomicMax(&ps->known, tag | word);
      atomicMax(&ps->published, tag | max(mine, word));
      __nanosleep(400);
    }
  } else {
    // ------------------------------------------------------------------ consumers
    // words of the level-0 pattern: code L in fields of BITS bits, from bit 32 j of a row on
    unsigned long long rep = (unsigned long long)p.L;
#pragma unroll
    for (int width = BITS; width < 64; width *= 2) rep |= rep << width;
    constexpr int kRowWords = 4 * BITS;                 // 32-bit words of one row of codes
    const float mid = exp2i(-p.k - 1);                  // the lowest midpoint
    const HeldLane hl = held_lane(p, lane);
    const int chunk = warp % kTileChunks;               // of the tiles of its group
    const int first = chunk * kChunkElems;
    unsigned run = 0;                                   // maximum of this warp's rows of the pair
    unsigned cur_pair = ~0u;                            // n * S and the tiles fit 31 bits (their data would not fit a GPU)
    // what this warp knows of a pair it leaves goes into the pair's word unless it is there
    auto leave = [&]() {
      if (lane == 0 && run != 0u) {
        const unsigned long long pub = *reinterpret_cast<volatile unsigned long long*>(&ps->published);
        if ((unsigned)(pub >> 32) != cur_pair || (unsigned)pub < run) atomicMax(p.scale_bits + cur_pair, run);
      }
    };
    unsigned flagged = 0;
    unsigned long long* const list = p.open_list + (size_t)(blockIdx.x * kStreamWarps + warp) * p.open_stride;
    unsigned listed = 0;                                // entries of this warp's region
    int s = warp / kTileChunks;                         // (the ring holds a multiple of the groups, see pipe_legal_stages)
    unsigned ph = 0;
    while (true) {
      if (!__all_sync(0xffffffffu, mbar_wait_bounded(&ps->full[s], ph, abort_flag, p.status, p.spin_limit))) break;
      const StreamHeader hd = ps->hd[s];
      if (hd.t == kNoTile) break;
      if (hd.pair != cur_pair) {
        leave();
        run = 0;
        cur_pair = hd.pair;
      }
      const unsigned char* st = ring + (size_t)s * stage_bytes;
      const float* sg = reinterpret_cast<const float*>(st) + first + lane * 4;
      float4 u4[kChunkRows];
      unsigned row_max[kChunkRows], mx = 0;
#pragma unroll
      for (int r = 0; r < kChunkRows; ++r) {
        row_max[r] = 0;
        if (first + r * 128 >= hd.count) continue;
        const float4 g4 = *reinterpret_cast<const float4*>(sg + r * 128);
        const float4 e4 = *reinterpret_cast<const float4*>(sg + kTileElems + r * 128);
        float gg[4] = {g4.x, g4.y, g4.z, g4.w};
        if constexpr (L2) add_l2_term_staged(p, hl, st + form_stage_bytes(false, 0), first + r * 128, lane, gg);
        u4[r] = make_float4(__fadd_rn(gg[0], e4.x), __fadd_rn(gg[1], e4.y), __fadd_rn(gg[2], e4.z),
                            __fadd_rn(gg[3], e4.w));
        row_max[r] = max(max(__float_as_uint(fabsf(u4[r].x)), __float_as_uint(fabsf(u4[r].y))),
                         max(__float_as_uint(fabsf(u4[r].z)), __float_as_uint(fabsf(u4[r].w))));
        mx = max(mx, row_max[r]);
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&ps->empty[s]);        // the stage has been read: it can be refilled
      if ((s += kStreamGroups) >= stages) { s -= stages; ph ^= 1u; }
      if (first >= hd.count) {                          // a short tile: nothing of this warp's
        if (lane == 0) p.deferred[(long long)hd.t * kTileChunks + chunk] = 0;
        continue;
      }
      const unsigned wm = warp_max(mx);
      run = max(run, wm);
      const unsigned long long kn = *known;
      const unsigned in_block = (unsigned)(kn >> 32) == hd.pair ? (unsigned)kn : 0u;
      const unsigned best = max(run, in_block);
      if (lane == 0) {
        if (wm >= 0x7f800000u) atomicOr(p.status, 1u);
        if (best > in_block) atomicMax(&ps->known, (unsigned long long)hd.pair << 32 | best);
      }
      // mid * bound is exact for bounds of ordinary size; below that only zeros are sure of level 0
      const float bound = __uint_as_float(best);
      const unsigned thr = bound >= 1e-30f ? __float_as_uint(__fmul_rn(bound, mid)) : 0u;
      float* ep = p.e + (long long)hd.worker * p.D + hd.off + first + lane * 4;
      unsigned flags = 0;
#pragma unroll
      for (int r = 0; r < kChunkRows; ++r) {
        if (first + r * 128 >= hd.count) continue;
        const unsigned lanes = __ballot_sync(0xffffffffu, row_max[r] > thr);
        if (lanes == 0u) {
          st_f4(ep + r * 128, u4[r]);
          continue;
        }
        const float uu[4] = {u4[r].x, u4[r].y, u4[r].z, u4[r].w};
        unsigned open[4], count = kListedPerRow + 1u;
        if (__popc(lanes) <= kListedPerRow) {
          count = 0u;
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            open[c] = __ballot_sync(0xffffffffu, __float_as_uint(fabsf(uu[c])) > thr);
            count += __popc(open[c]);
          }
        }
        if (count > kListedPerRow || listed + count >= p.open_stride) {
          flags |= 1u << r;
          continue;
        }
        st_f4(ep + r * 128, u4[r]);
        unsigned at = listed + 1u;
        listed += count;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          if ((open[c] >> lane) & 1u)
            list[at + __popc(open[c] & ((1u << lane) - 1u))] =
                (unsigned long long)__float_as_uint(uu[c]) << 32 | (hd.t << 9 | (unsigned)(r * 128 + lane * 4 + c));
          at += __popc(open[c]);
        }
      }
      unsigned* cw = reinterpret_cast<unsigned*>(p.gcodes + (long long)hd.worker * p.gcode_bytes +
                                                 (hd.off + first) * BITS / 8);
      const int words = min(kChunkRows, (hd.count - first) >> 7) * kRowWords;
#pragma unroll
      for (int j0 = 0; j0 < kChunkRows * kRowWords; j0 += 32) {
        const int j = j0 + lane, r = j / kRowWords;
        if (j < words && !((flags >> r) & 1u)) cw[j] = (unsigned)(rep >> ((32 * (j - r * kRowWords)) % BITS));
      }
      if (lane == 0) p.deferred[(long long)hd.t * kTileChunks + chunk] = (unsigned char)flags;
      flagged += __popc(flags);
    }
    leave();
    if (lane == 0 && flagged) atomicAdd(&p.counters->rows, flagged);
    if (lane == 0 && p.open_stride != 0u) list[0] = listed;
  }
}

// ---------------------------------------------------------------------------
// Everything the sweep does not serve: max |u| of every (worker, segment) pair; with the moments on the
// workers the moment updates of Algorithm 3, and u into e's place.  The maximum is taken on the bit
// patterns of |u| (monotone for non-negative floats, exact, order-free; a NaN or Inf ends up as the
// maximum and is reported by the settle pass).  All 16 warps work on one tile: rows row0, row0 + 2
// of 1024 elements.
// ---------------------------------------------------------------------------
template <bool WM, bool L2>
__global__ void __launch_bounds__(kStreamThreads, 1)
worker_form_kernel(const StreamParams p) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  StreamSmem* ps = reinterpret_cast<StreamSmem*>(smem_raw);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int stages = p.stages;
  const int stage_bytes = form_stage_bytes(WM, L2 ? held_tile_bytes(p.kx, p.xbits) : 0);
  unsigned char* ring = smem_raw + kStreamHeadBytes;
  volatile int* abort_flag = &ps->abort_flag;
  stream_init(ps, stages, kStreamWarps + p.missing_readers, 0u);

  if (warp == kStreamWarps) {
    if (lane == 0) {
      produce_tiles(
          p, ps, &p.counters->form_tickets, false, 1, [&](unsigned) { return 0ull; },
          [&](const Tile& tile, unsigned wl, unsigned t, unsigned long long, int s, StreamHeader* hd) {
            fill_header(p, hd, tile, wl, t);
            issue_inputs<WM, L2>(p, ring + (size_t)s * stage_bytes, tile, wl, &ps->full[s]);
            return true;
          });
      stream_leave(&p.counters->form_tickets, &p.counters->form_left, nullptr);
    }
  } else if (warp < kStreamWarps) {
    const int gt = threadIdx.x & (kThreads - 1), row0 = threadIdx.x / kThreads;
    const HeldLane hl = held_lane(p, lane);
    unsigned mx = 0, cur_pair = ~0u;
    auto leave = [&]() {
      const unsigned r = warp_max(mx);
      if (lane == 0 && r) atomicMax(p.scale_bits + cur_pair, r);
    };
    int s = 0;
    unsigned ph = 0;
    while (true) {
      if (!__all_sync(0xffffffffu, mbar_wait_bounded(&ps->full[s], ph, abort_flag, p.status, p.spin_limit))) break;
      const StreamHeader hd = ps->hd[s];
      if (hd.t == kNoTile) break;
      if (hd.pair != cur_pair) {
        if (cur_pair != ~0u) leave();
        mx = 0;
        cur_pair = hd.pair;
      }
      const unsigned char* st = ring + (size_t)s * stage_bytes;
      const float* sg = reinterpret_cast<const float*>(st) + gt * 4;
      float4 g4[2], e4[2], m4[2], v4[2];
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        const int q = (row0 + 2 * r) * kRowElems;
        if (q + gt * 4 >= hd.count) continue;                       // warp-uniform
        g4[r] = *reinterpret_cast<const float4*>(sg + q);
        e4[r] = *reinterpret_cast<const float4*>(sg + kTileElems + q);
        if constexpr (WM) {
          m4[r] = *reinterpret_cast<const float4*>(sg + 2 * kTileElems + q);
          v4[r] = *reinterpret_cast<const float4*>(sg + 3 * kTileElems + q);
        }
        if constexpr (L2) {
          float gg[4] = {g4[r].x, g4[r].y, g4[r].z, g4[r].w};
          add_l2_term_staged(p, hl, st + form_stage_bytes(WM, 0), q + (gt >> 5) * 128, lane, gg);
          g4[r] = make_float4(gg[0], gg[1], gg[2], gg[3]);
        }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&ps->empty[s]);                    // the stage has been read: it can be refilled
      if (++s == stages) { s = 0; ph ^= 1u; }
      const long long so = (long long)hd.worker * p.D + hd.off + gt * 4;
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        const int q = (row0 + 2 * r) * kRowElems;
        if (q + gt * 4 >= hd.count) continue;
        const float gg[4] = {g4[r].x, g4[r].y, g4[r].z, g4[r].w};
        const float ee[4] = {e4[r].x, e4[r].y, e4[r].z, e4[r].w};
        float uu[4];
        if constexpr (WM) {
          float mm[4] = {m4[r].x, m4[r].y, m4[r].z, m4[r].w};
          float vs[4] = {v4[r].x, v4[r].y, v4[r].z, v4[r].w};
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            moments(p.h, gg[c], mm[c], vs[c]);
            uu[c] = __fadd_rn(adam_step(p.h, mm[c], vs[c], p.alpha), ee[c]);
          }
          st_f4(p.m + so + q, make_float4(mm[0], mm[1], mm[2], mm[3]));
          st_f4(p.v + so + q, make_float4(vs[0], vs[1], vs[2], vs[3]));
        } else {
#pragma unroll
          for (int c = 0; c < 4; ++c) uu[c] = __fadd_rn(gg[c], ee[c]);
        }
        if constexpr (WM) st_f4(p.e + so + q, make_float4(uu[0], uu[1], uu[2], uu[3]));
#pragma unroll
        for (int c = 0; c < 4; ++c) mx = max(mx, __float_as_uint(fabsf(uu[c])));
      }
    }
    if (cur_pair != ~0u) leave();
  }
}

// The open elements the sweep listed, now that their scales are final: the code of a listed element
// that has one other than level 0 goes over the level 0 the sweep wrote (as the bits in which the two
// differ: several elements share a word), and its e' over u.
template <int MODE>
__device__ __forceinline__ void close_listed(const StreamParams& p) {
  constexpr int kBits = MODE == G_TERNARY ? 2 : 3;
  const unsigned lane = threadIdx.x & 31, warps = gridDim.x * kStreamWarps;
  const unsigned tpw = (unsigned)p.tiles_per_worker;
  const unsigned regions = p.open_regions;
  for (unsigned unit = blockIdx.x * kStreamWarps + (threadIdx.x >> 5); unit < regions * kListParts; unit += warps) {
    const unsigned region = unit / kListParts;
    const unsigned long long* list = p.open_list + (size_t)region * p.open_stride;
    const unsigned listed = (unsigned)list[0];
    // four entries per lane at a time: what they lead to (tile, scale) is two more trips to L2
    for (unsigned i0 = unit % kListParts * (32u * kListBatch) + lane; i0 < listed; i0 += 32u * kListBatch * kListParts) {
      unsigned long long entry[kListBatch];
      long long elem[kListBatch], w[kListBatch];
      float s[kListBatch];
#pragma unroll
      for (int a = 0; a < kListBatch; ++a) entry[a] = i0 + 32u * a < listed ? list[i0 + 32u * a + 1u] : 0ull;
#pragma unroll
      for (int a = 0; a < kListBatch; ++a) {
        if (i0 + 32u * a >= listed) continue;
        const unsigned t = (unsigned)entry[a] >> 9, wl = t / tpw;
        const Tile tile = p.tiles[t - wl * tpw];
        w[a] = p.worker_begin + (long long)wl;
        elem[a] = tile.off + (region % kTileChunks) * kChunkElems + ((unsigned)entry[a] & (kChunkElems - 1));
        s[a] = __uint_as_float(p.scale_bits[w[a] * p.S + tile.seg]);
      }
#pragma unroll
      for (int a = 0; a < kListBatch; ++a) {
        if (i0 + 32u * a >= listed) continue;
        const float u = __uint_as_float((unsigned)(entry[a] >> 32));
        const float y = __fdiv_rn(fabsf(u), s[a]);
        int c;                                            // level index; the value is s * value
        float value;
        if constexpr (MODE == G_TERNARY) {
          c = y > 0.5f ? 1 : 0;
          value = 1.0f;
        } else {
          c = (y > 0.25f ? 1 : 0) + (y > 0.75f ? 1 : 0);
          value = c == 2 ? 1.0f : 0.5f;
        }
        if (c == 0) continue;
        const float mag = __fmul_rn(s[a], value);
        p.e[w[a] * p.D + elem[a]] = __fsub_rn(u, u < 0.0f ? -mag : mag);
        const unsigned change = (unsigned)(u < 0.0f ? p.L - c : p.L + c) ^ (unsigned)p.L;
        const long long bit = elem[a] * kBits;
        unsigned* word = reinterpret_cast<unsigned*>(p.gcodes + w[a] * p.gcode_bytes) + (bit >> 5);
        const unsigned at = (unsigned)bit & 31u;
        atomicXor(word, change << at);
        if (kBits == 3 && at > 29u) atomicXor(word + 1, change >> (32u - at));
      }
    }
  }
}

// One row of 128 elements out of u: codes and e'.  elem: the lane's first element (padded layout).
template <int MODE>
__device__ __forceinline__ void settle_row(const WorkerParams& p, const float4& u4, const GradScale& gs, int w,
                                           long long elem, int lane) {
  const float uu[4] = {u4.x, u4.y, u4.z, u4.w};
  float en[4];
  const long long row_elem = elem - lane * 4;
  void* dst = p.gcodes + (long long)w * p.gcode_bytes + row_elem * p.bits / 8;
  if constexpr (MODE == G_STOCHASTIC) {
    // the four coordinates of this thread are one block of the stream: counter
    // (element / 4, worker, step), key = seed
    const unsigned long long block = (unsigned long long)elem >> 2;
    const uint4 rnd = philox4x32_10(make_uint4((unsigned)block, (unsigned)(block >> 32), (unsigned)w, p.step),
                                    make_uint2(p.seed_lo, p.seed_hi));
    store_row_of_code_bytes(quantize_stochastic4(uu, gs, rnd, en), dst, lane);
  } else if constexpr (MODE == G_TERNARY) {
    store_row_of_code_bytes(quantize_ternary4(uu, gs, en), dst, lane);
  } else if constexpr (MODE == G_FIVE) {
    pack_row_store_fields<3>(quantize_five4(uu, gs, en), dst, lane);
  } else if constexpr (MODE == G_UNIFORM) {
    pack_row_store_fields_rt(p.bits, quantize_uniform4(uu, gs, p.k, p.L, p.bits, en), dst, lane);
  } else {
    unsigned code[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) code[c] = quantize_grad<MODE>(uu[c], gs, p.k, p.L, en[c]);
    pack_row_store_rt(p.bits, code[0], code[1], code[2], code[3], dst, lane);
  }
  st_f4(p.e + (long long)w * p.D + elem, make_float4(en[0], en[1], en[2], en[3]));
}

// The few rows a sweep has flagged: a warp takes 32 chunks (4 tiles) at a time, one byte of flags per
// lane, and settles their rows four at a time, so that it keeps as many loads in flight as with full
// tiles; the flags and descriptors of its next 32 are fetched meanwhile.  The rows left crowd where a pair
// begins and its bound is low, so a warp takes 16, 8, ... 1 chunks at a time where it would have fewer than eight
// turns (Student-t gradients, 1.2 x 10^7 elements, n = 4, a fifth of the rows left, this pass: one turn 110 us, four
// 48, eight 43; hardly a row left: 12.9, 14.6, 16.9).  The held weights of the l2 term are asked for with g and e
// (the same with the term: one turn 183 us, four 58, eight 52).
template <int MODE, bool L2>
__device__ __forceinline__ void settle_few(const StreamParams& p) {
  constexpr int kBatch = 4;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const unsigned total = (unsigned)p.total_tiles, tpw = (unsigned)p.tiles_per_worker;
  const unsigned warps = gridDim.x * kStreamWarps, chunks = total * kTileChunks;   // below 2^32: 512 elements each
  unsigned span = 32u;
  while (span > 1u && chunks < 8u * span * warps) span >>= 1;
  unsigned c_next = (blockIdx.x * kStreamWarps + warp) * span + (unsigned)lane;
  unsigned fl_next = 0, wl_next = 0;
  Tile tile_next = Tile{0, 0, 0};
  bool more = false;                                      // this lane has a chunk in the span
  auto fetch = [&]() {
    fl_next = 0;
    more = (unsigned)lane < span && c_next < chunks;
    if (more) {
      const unsigned t = c_next / kTileChunks;
      wl_next = t / tpw;
      tile_next = p.tiles[t - wl_next * tpw];
      // (only rows the tile has: a sweep that gave up has left bytes of the workspace as they were)
      const int rows = (tile_next.count >> 7) - (int)(c_next & (kTileChunks - 1)) * kChunkRows;
      fl_next = p.deferred[c_next] & ((1u << min(max(rows, 0), kChunkRows)) - 1u);
    }
  };
  fetch();
  while (__any_sync(0xffffffffu, more)) {
    const unsigned fl = fl_next, wl = wl_next;
    const long long elem = tile_next.off + (int)(c_next & (kTileChunks - 1)) * kChunkElems;
    unsigned sb = 0;                                      // asked for now, looked at after the first rows' loads
    if (fl != 0u) sb = p.scale_bits[(long long)(p.worker_begin + (int)wl) * p.S + tile_next.seg];
    c_next += warps * span;
    fetch();
    unsigned pending = __ballot_sync(0xffffffffu, fl != 0u);
    unsigned rows = 0;                                    // flagged rows left of the chunk of lane `cur`
    int cur = 0;
    while (pending | rows) {
      float4 gv[kBatch], ev[kBatch];
      HeldRaw hw[L2 ? kBatch : 1];
      long long at[kBatch];
      int row_w[kBatch], src[kBatch];
      bool have[kBatch];
#pragma unroll
      for (int a = 0; a < kBatch; ++a) {
        if (rows == 0u && pending != 0u) {
          cur = __ffs((int)pending) - 1;
          pending &= pending - 1u;
          rows = __shfl_sync(0xffffffffu, fl, cur);
        }
        have[a] = rows != 0u;                             // warp-uniform
        if (!have[a]) continue;
        const int r = __ffs((int)rows) - 1;
        rows &= rows - 1u;
        src[a] = cur;
        at[a] = __shfl_sync(0xffffffffu, elem, cur) + r * 128 + lane * 4;
        row_w[a] = (int)__shfl_sync(0xffffffffu, wl, cur);
        gv[a] = ld_f4_stream(p.g + (long long)row_w[a] * p.D + at[a]);
        row_w[a] += p.worker_begin;
        ev[a] = ld_f4(p.e + (long long)row_w[a] * p.D + at[a]);
        if constexpr (L2) hw[a] = held_fetch(p, at[a] - lane * 4, lane);
      }
#pragma unroll
      for (int a = 0; a < kBatch; ++a) {
        if (!have[a]) continue;
        const GradScale gs = grad_scale<MODE>(__uint_as_float(__shfl_sync(0xffffffffu, sb, src[a])), p.k);
        float gg[4] = {gv[a].x, gv[a].y, gv[a].z, gv[a].w};
        if constexpr (L2) add_l2_term_fetched(p, at[a] - lane * 4, lane, hw[a], gg);
        settle_row<MODE>(p, make_float4(__fadd_rn(gg[0], ev[a].x), __fadd_rn(gg[1], ev[a].y), __fadd_rn(gg[2], ev[a].z),
                                        __fadd_rn(gg[3], ev[a].w)), gs, row_w[a], at[a], lane);
      }
    }
  }
}

// ---------------------------------------------------------------------------
// Codes and e'.  SWEPT: of the elements the sweep listed and the rows it flagged,
// the latter tile by tile where they are half of all rows or more, else row by row.  Tiles are gone
// through from the last to the first: the u written last is still in L2.
// ---------------------------------------------------------------------------
template <int MODE, bool SWEPT, bool WM, bool L2>
__global__ void __launch_bounds__(kStreamThreads, 1)
worker_settle_kernel(const StreamParams p) {
  static_assert(!WM || (!SWEPT && !L2), "with the moments on the workers u is in e's place");
  static_assert(!SWEPT || MODE == G_TERNARY || MODE == G_FIVE, "grids the sweep serves");
  extern __shared__ __align__(128) unsigned char smem_raw[];
  StreamSmem* ps = reinterpret_cast<StreamSmem*>(smem_raw);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int stages = p.stages;
  unsigned char* ring = smem_raw + kStreamHeadBytes;
  volatile int* abort_flag = &ps->abort_flag;
  // (the count of rows goes through shared memory: read by every CTA before any of them can clear it)
  stream_init(ps, stages, kStreamWarps / kStreamGroups + p.missing_readers,
              SWEPT && threadIdx.x == 0 ? __ldcg(&p.counters->rows) : 0u);
  const unsigned left = *reinterpret_cast<volatile unsigned*>(&ps->pair);
  const bool tiles = !SWEPT || left / 16u >= (unsigned)p.total_tiles;
  const int stage_bytes = settle_stage_bytes(WM, L2 ? held_tile_bytes(p.kx, p.xbits) : 0);
  __syncthreads();

  if (warp == kStreamWarps) {
    unsigned scale_bits = 0u, scale_pair = ~0u;         // read where the pair changes
    if (lane == 0) {
      if (tiles) produce_tiles(
          p, ps, &p.counters->settle_tickets, true, kStreamGroups,
          [&](unsigned t) { return SWEPT ? reinterpret_cast<const unsigned long long*>(p.deferred)[t] : ~0ull; },
          [&](const Tile& tile, unsigned wl, unsigned t, unsigned long long flags, int s, StreamHeader* hd) {
            if (SWEPT && flags == 0ull) return false;
            fill_header(p, hd, tile, wl, t);
            if (hd->pair != scale_pair) {
              scale_pair = hd->pair;
              scale_bits = p.scale_bits[scale_pair];
            }
            hd->scale_bits = scale_bits;
            hd->flags = flags;
            unsigned char* st = ring + (size_t)s * stage_bytes;
            if constexpr (WM) {
              const unsigned bytes = (unsigned)tile.count * 4u;
              mbar_arrive_expect_tx(&ps->full[s], bytes);
              bulk_load(st, p.e + (long long)hd->worker * p.D + tile.off, bytes, &ps->full[s]);
            } else {
              issue_inputs<false, L2>(p, st, tile, wl, &ps->full[s]);
            }
            return true;
          });
      stream_leave(&p.counters->settle_tickets, &p.counters->settle_left, SWEPT ? &p.counters->rows : nullptr);
    }
  } else if (warp < kStreamWarps) {
    if constexpr (SWEPT) {
      if (p.open_stride != 0u) close_listed<MODE>(p);
      if (!tiles && left != 0u) settle_few<MODE, L2>(p);
    }
    const HeldLane hl = held_lane(p, lane);
    const int gt = threadIdx.x & (kThreads - 1);
    int s = threadIdx.x / kThreads;                                 // group g takes stages g, g + groups, ...
    unsigned ph = 0;
    while (tiles) {
      if (!__all_sync(0xffffffffu, mbar_wait_bounded(&ps->full[s], ph, abort_flag, p.status, p.spin_limit))) break;
      const StreamHeader hd = ps->hd[s];
      if (hd.t == kNoTile) break;
      const unsigned char* st = ring + (size_t)s * stage_bytes;
      const float* su = reinterpret_cast<const float*>(st) + gt * 4;
      float4 u4[kRows];
#pragma unroll
      for (int r = 0; r < kRows; ++r) {
        u4[r] = *reinterpret_cast<const float4*>(su + r * kRowElems);
        if constexpr (!WM) {
          const float4 e4 = *reinterpret_cast<const float4*>(su + kTileElems + r * kRowElems);
          float gg[4] = {u4[r].x, u4[r].y, u4[r].z, u4[r].w};
          if constexpr (L2) add_l2_term_staged(p, hl, st + form_stage_bytes(false, 0), r * kRowElems + (gt >> 5) * 128, lane, gg);
          u4[r] = make_float4(__fadd_rn(gg[0], e4.x), __fadd_rn(gg[1], e4.y), __fadd_rn(gg[2], e4.z), __fadd_rn(gg[3], e4.w));
        }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&ps->empty[s]);
      if ((s += kStreamGroups) >= stages) { s -= stages; ph ^= 1u; }
      if (gt == 0 && hd.scale_bits >= 0x7f800000u) atomicOr(p.status, 1u);
      const GradScale gs = grad_scale<MODE>(__uint_as_float(hd.scale_bits), p.k);
#pragma unroll
      for (int r = 0; r < kRows; ++r) {
        const int q = r * kRowElems + gt * 4;
        const int row = q >> 7;                                     // of 128 elements, 0 .. 31
        if (q >= hd.count) continue;                                // warp-uniform: counts are multiples of 128
        if (SWEPT && !((unsigned)(hd.flags >> (8 * (row >> 2) + (row & 3))) & 1u)) continue;
        settle_row<MODE>(p, u4[r], gs, hd.worker, hd.off + q, lane);
      }
    }
  }
}

}  // namespace qadam
