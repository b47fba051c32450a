// The plain step kernels: the identity worker, the stochastic operator in calls of few tiles, the server pass for the
// streams the pipelined one does not take and the stand-alone weight broadcast, grid-stride loops over a tile table; and
// what the pipelined kernels share with them.
//
// Thread/tile mapping (all kernels here): a CTA of 256 threads owns a tile of up to
// 4096 consecutive padded elements as 4 CTA-wide rows of 1024; in row r thread t
// owns the 4 consecutive elements starting at r*1024 + 4*t, so every global
// access of fp32 state is one coalesced 128-bit access per thread, and one warp
// in one row owns 128 elements = one aligned run of the packed code stream.
#pragma once

#include "qadam_device.cuh"

namespace qadam {

struct StreamCounters;          // see the streaming passes

struct WorkerParams {
  const float* g;        // [worker_count][D] gradients of the workers of this call
  float* m;              // [n][D] worker moments (PLACE_WORKER) or nullptr
  float* v;
  float* e;              // [n][D]
  unsigned* scale_bits;  // [n][S] the scales buffer, seen as bit patterns
  unsigned char* gcodes; // [n][gcode_bytes]
  const Tile* tiles;     // [tiles_per_worker]
  unsigned* status;
  long long D;
  long long gcode_bytes;
  long long total_tiles; // worker_count * tiles_per_worker
  int tiles_per_worker;
  int S;
  int worker_begin;
  int k, L, bits;        // level parameter, positive levels, code width
  float alpha;
  Hyper h;
  // l2 term (kernels instantiated with L2 = true): lambda * (held weights) is added to g
  const float* x;               // [D] master copy (held as is when kx < 0)
  const unsigned char* wcodes;  // packed Q_x(x) (kx >= 0)
  int kx, xbits;
  float lambda;
  unsigned spin_limit;          // persistent kernels: polls of one wait before it gives up
  // stochastic operator: key of the random stream and the step number
  unsigned seed_lo, seed_hi, step;
};
// What the streaming passes alone read.  The other worker kernels go without: parameters are fetched anew in every
// launch, and with these 40 bytes among its own the on-chip kernel cost a step of 2^20 elements, n = 4, 0.5 us
// (24.1 against 23.6 us).
struct StreamParams : WorkerParams {
  // sweep: the rows it leaves, one byte per 512-element chunk of a tile, [total_tiles][8] ...
  unsigned char* deferred;
  // ... and the open elements it listed instead: a region of open_stride entries per warp of the sweep,
  // {entry 0: how many follow} {u : 32, tile : 23, element of the chunk : 9} ...
  unsigned long long* open_list;
  unsigned open_stride;         // 0: no list
  unsigned open_regions;
  int stages;                   // of the streaming passes' rings
  int missing_readers;          // TESTING: 1: a stage waits for a reader that does not exist (test_missing_tiles)
  StreamCounters* counters;
};

// Packed weight codes of at most 8 bits: the two 32-bit words that hold this lane's 4 codes
// of a 128-element row (row_elem: first element of the row).  Split from the decode so
// that a kernel can issue the loads a tile ahead of their use.
__device__ __forceinline__ void held_fetch8(const WorkerParams& p, long long row_elem, int lane,
                                            unsigned& lo, unsigned& hi) {
  const unsigned* words = reinterpret_cast<const unsigned*>(p.wcodes + row_elem * p.xbits / 8);
  const int F = 4 * p.xbits;                            // bits per lane = words per row
  const int w = (F * lane) >> 5;
  lo = __ldg(words + w);
  // the lane's field runs into the next word only for widths that do not divide 32
  hi = ((F * lane) & 31) + F > 32 ? __ldg(words + w + 1) : 0u;
}
// ... and their values: (code - 2^kx) times the grid step, exact.
__device__ __forceinline__ void held_decode8(const WorkerParams& p, int lane, unsigned lo, unsigned hi,
                                             float out[4]) {
  const int F = 4 * p.xbits;
  const unsigned v = __funnelshift_r(lo, hi, (F * lane) & 31);
  const unsigned f = F == 32 ? v : (v & ((1u << F) - 1u));
  const unsigned mask = (1u << p.xbits) - 1u;
  const float step = exp2i(-(p.kx + 1));
  // code -> float without a conversion: 2^23 + code as a bit pattern, minus 2^23 + 2^kx
  const float bias = -(8388608.0f + (float)(1 << p.kx));
#pragma unroll
  for (int c = 0; c < 4; ++c)
    out[c] = __fmul_rn(__fadd_rn(__uint_as_float(0x4b000000u | ((f >> (c * p.xbits)) & mask)), bias), step);
}

// The weights a worker holds for this lane's 4 elements of a 128-element row: the broadcast
// Q_x(x) decoded from its packed codes (code - 2^kx times the grid step, exact), or x itself
// when the weights are not quantized.  row_elem: first element of the row.
__device__ __forceinline__ void held_weights4(const WorkerParams& p, long long row_elem, int lane,
                                              float out[4]) {
  if (p.kx < 0) {
    const float4 v = *reinterpret_cast<const float4*>(p.x + row_elem + lane * 4);
    out[0] = v.x; out[1] = v.y; out[2] = v.z; out[3] = v.w;
    return;
  }
  if (p.xbits <= 8) {
    unsigned lo, hi;
    held_fetch8(p, row_elem, lane, lo, hi);
    held_decode8(p, lane, lo, hi, out);
    return;
  }
  const unsigned char* row = p.wcodes + row_elem * p.xbits / 8;
  const unsigned mask = (1u << p.xbits) - 1u;
  const float step = exp2i(-(p.kx + 1));
  const float bias = -(8388608.0f + (float)(1 << p.kx));
  auto value = [&](unsigned code) {
    return __fmul_rn(__fadd_rn(__uint_as_float(0x4b000000u | code), bias), step);
  };
  const unsigned* words = reinterpret_cast<const unsigned*>(row);
  const int row_words = 4 * p.xbits;                    // 128 codes
  const int half = 2 * p.xbits;                         // two codes, at most 32 bits
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int bit = 2 * half * lane + h * half;
    const int w = bit >> 5;
    const unsigned lo = __ldg(words + w);
    const unsigned hi = __ldg(words + (w + 1 < row_words ? w + 1 : w));
    const unsigned f = __funnelshift_r(lo, hi, bit & 31);
    out[2 * h] = value(f & mask);
    out[2 * h + 1] = value((f >> p.xbits) & mask);
  }
}
// g + lambda * (held weights), each operation rounded once (Section 5.1's l2 term)
__device__ __forceinline__ void add_l2_term(const WorkerParams& p, long long row_elem, int lane,
                                            float gg[4]) {
  float w[4];
  held_weights4(p, row_elem, lane, w);
#pragma unroll
  for (int c = 0; c < 4; ++c) gg[c] = __fadd_rn(gg[c], __fmul_rn(p.lambda, w[c]));
}

// The same in two halves, for kernels that ask for all they need before the first use: codes of at most 8 bits are
// fetched raw, other weights (and x itself) read where they are added.
struct HeldRaw {
  unsigned lo, hi;
};
__device__ __forceinline__ HeldRaw held_fetch(const WorkerParams& p, long long row_elem, int lane) {
  HeldRaw h = {0u, 0u};
  if (p.kx >= 0 && p.xbits <= 8) held_fetch8(p, row_elem, lane, h.lo, h.hi);
  return h;
}
__device__ __forceinline__ void add_l2_term_fetched(const WorkerParams& p, long long row_elem, int lane,
                                                    const HeldRaw& h, float gg[4]) {
  if (p.kx < 0 || p.xbits > 8) {
    add_l2_term(p, row_elem, lane, gg);
    return;
  }
  float w[4];
  held_decode8(p, lane, h.lo, h.hi, w);
#pragma unroll
  for (int c = 0; c < 4; ++c) gg[c] = __fadd_rn(gg[c], __fmul_rn(p.lambda, w[c]));
}

// With the l2 term a pipeline stage also carries its tile's held weights: b_x bits (x: 32) per element.
__host__ __device__ constexpr int held_tile_bytes(int kx, int xbits) { return kTileElems / 8 * (kx < 0 ? 32 : xbits); }

// The same from a copy of the tile's held weights in shared memory (packed codes, or x itself).  What a
// thread needs for it is prepared once: a pair of codes moves into the mantissas of two floats whose
// exponents give them the weight 1; less 2^E + 2^kx these are the weights in grid steps, exactly, and
// lambda times the step, exact too, times that is fl(lambda w): the same product, rounded once.
// 3 instructions per element where the fields were shifted, masked, converted and scaled one by one (7).
struct HeldLane {
  unsigned m0, m1, g1;     // masks of the two codes, exponent of the second
  float2 k;                // -(2^E + 2^kx)
  float unit;              // lambda 2^-(kx+1); 0: one by one (unquantized weights, wide codes, tiny lambda)
  int word, shift, next;   // the lane's field: first word, bit in it, whether it runs on
};
__device__ __forceinline__ HeldLane held_lane(const WorkerParams& p, int lane) {
  HeldLane h;
  const int b = p.xbits & 15, bit = 4 * p.xbits * lane;
  h.unit = p.kx >= 0 && p.xbits <= 8 && p.lambda >= 1e-30f ? __fmul_rn(p.lambda, exp2i(-(p.kx + 1))) : 0.0f;
  h.m0 = (1u << b) - 1u;
  h.m1 = h.m0 << b;
  h.g1 = (unsigned)(150 - b) << 23;
  const float zero = exp2i(p.kx < 0 ? 0 : p.kx);
  h.k = make_float2(-(8388608.0f + zero), -(exp2i(23 - b) + zero));
  h.word = bit >> 5;
  h.shift = bit & 31;
  h.next = h.shift + 4 * p.xbits > 32 ? 1 : 0;
  return h;
}
// row: the row's first element in the tile.  PREPARED = false: field by field in any case, for the on-chip kernel with the
// moments on the workers, which has no registers for the masks (they made it spill: weights of 16 bits, ResNet-18-shaped
// set, n = 8, 501 us a step against 496; BERT-shaped set, n = 16, 9.32 ms against 9.22; of at most 8 bits the same).
// Its five-level kernel keeps the masks (weights of 3 bits 487 us against 491).
template <bool PREPARED = true>
__device__ __forceinline__ void add_l2_term_staged(const WorkerParams& p, const HeldLane& h, const unsigned char* held,
                                                   int row, int lane, float gg[4]) {
  if (PREPARED && h.unit != 0.0f) {
    const unsigned* words = reinterpret_cast<const unsigned*>(held + row / 8 * p.xbits) + h.word;
    const unsigned f = __funnelshift_r(words[0], words[h.next], h.shift);
    const float2 unit = make_float2(h.unit, h.unit);
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      const unsigned pair = c == 0 ? f : f >> (2 * p.xbits);
      const float2 w = add2_rn(make_float2(__uint_as_float((pair & h.m0) | 0x4b000000u),
                                           __uint_as_float((pair & h.m1) | h.g1)), h.k);
      const float2 term = mul2_rn(w, unit);
      gg[2 * c] = __fadd_rn(gg[2 * c], term.x);
      gg[2 * c + 1] = __fadd_rn(gg[2 * c + 1], term.y);
    }
    return;
  }
  float w[4];
  if (p.kx < 0) {
    const float4 v = *reinterpret_cast<const float4*>(held + (row + lane * 4) * 4);
    w[0] = v.x; w[1] = v.y; w[2] = v.z; w[3] = v.w;
  } else if (!PREPARED && p.xbits <= 8) {
    const unsigned* words = reinterpret_cast<const unsigned*>(held + row / 8 * p.xbits);
    const int bit = 4 * p.xbits * lane, at = bit >> 5;
    held_decode8(p, lane, words[at], (bit & 31) + 4 * p.xbits > 32 ? words[at + 1] : 0u, w);
  } else {
    const unsigned* words = reinterpret_cast<const unsigned*>(held + row / 8 * p.xbits);
    const int half = 2 * p.xbits;                     // two codes, at most 32 bits
    const unsigned mask = (1u << p.xbits) - 1u;
    const float step = exp2i(-(p.kx + 1));
    const float bias = -(8388608.0f + (float)(1 << p.kx));
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int bit = (2 * lane + i) * half, at = bit >> 5;
      const unsigned hi = (bit & 31) + half > 32 ? words[at + 1] : 0u;
      const unsigned f = __funnelshift_r(words[at], hi, bit & 31);
      w[2 * i] = __fmul_rn(__fadd_rn(__uint_as_float(0x4b000000u | (f & mask)), bias), step);
      w[2 * i + 1] = __fmul_rn(__fadd_rn(__uint_as_float(0x4b000000u | ((f >> p.xbits) & mask)), bias), step);
    }
  }
#pragma unroll
  for (int c = 0; c < 4; ++c) gg[c] = __fadd_rn(gg[c], __fmul_rn(p.lambda, w[c]));
}

struct ServerParams {
  float* x;              // [D]
  float* m;              // [D] (PLACE_SERVER) or nullptr
  float* v;
  const float* scales;   // [n][S]
  const unsigned char* gcodes;  // [n][gcode_bytes]
  unsigned char* wcodes; // [wcode_bytes] or nullptr
  float* wresid;         // [D] or nullptr
  float* wfeedback;      // [D] or nullptr: error buffer of the broadcast (Q_x is applied to x + wfeedback)
  const Tile* tiles;
  long long D;
  long long gcode_bytes;
  int tiles_per_worker;
  int S;
  int n;
  int k, L, gbits;       // gradient level parameter / levels / code width
  int gmode;             // GMode of the gradient grid
  int kx, xbits;         // weight level parameter (-1: none) / code width
  float alpha;
  float nf;              // (float)n
  float inv_nf;          // 1/n, exact when n is a power of two
  unsigned* status;
  Hyper h;
  unsigned spin_limit;   // pipelined pass: polls of one wait before it gives up
};

__device__ __forceinline__ float4 ld_f4(const float* p) {
  return *reinterpret_cast<const float4*>(p);
}
__device__ __forceinline__ float4 ld_f4_stream(const float* p) {
  return __ldcs(reinterpret_cast<const float4*>(p));
}
__device__ __forceinline__ void st_f4(float* p, const float4& v) {
  *reinterpret_cast<float4*>(p) = v;
}

// CTA-wide max of a 32-bit pattern; result valid in thread 0.
__device__ __forceinline__ unsigned block_max(unsigned v, unsigned* smem8) {
  v = warp_max(v);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (lane == 0) smem8[warp] = v;
  __syncthreads();
  unsigned r = 0;
  if (threadIdx.x == 0) {
#pragma unroll
    for (int w = 0; w < kThreads / 32; ++w) r = max(r, smem8[w]);
  }
  __syncthreads();
  return r;
}

// ---------------------------------------------------------------------------
// The two streaming launches as plain kernels, for calls of few tiles under the stochastic operator (see
// kPlainTiles; the rings of the streaming passes take their place above).  First max |u| of every (worker, segment)
// pair; with the moments on the workers the moment updates too, and u into e's place.  The maximum is taken on the bit
// patterns (exact, order-free).  Internal linkage: this header is included by more than one source file.
// ---------------------------------------------------------------------------
template <bool WORKER_MOMENTS, bool L2>
static __global__ void __launch_bounds__(kThreads, WORKER_MOMENTS ? 2 : (L2 ? 3 : 4))
worker_absmax_kernel(const WorkerParams p) {
  __shared__ unsigned red[kThreads / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned mx = 0;
  long long cur_pair = -1;
  auto leave = [&]() {
    const unsigned r = block_max(mx, red);
    if (threadIdx.x == 0 && r) atomicMax(p.scale_bits + cur_pair, r);
  };
  for (long long t = blockIdx.x; t < p.total_tiles; t += gridDim.x) {
    const int wl = (int)(t / p.tiles_per_worker);
    const Tile tile = p.tiles[(int)(t - (long long)wl * p.tiles_per_worker)];
    const int w = p.worker_begin + wl;
    const long long pair = (long long)w * p.S + tile.seg;
    if (pair != cur_pair) {
      if (cur_pair >= 0) leave();
      mx = 0;
      cur_pair = pair;
    }
    const float* gp = p.g + (long long)wl * p.D + tile.off;
    const long long so = (long long)w * p.D + tile.off;
    float4 gv[kRows], ev[kRows], mv[kRows], vv[kRows];
    HeldRaw hw[L2 ? kRows : 1];
#pragma unroll
    for (int r = 0; r < kRows; ++r) {
      const int idx = r * kRowElems + threadIdx.x * 4;
      if (idx >= tile.count) continue;
      gv[r] = ld_f4_stream(gp + idx);
      ev[r] = ld_f4(p.e + so + idx);
      if constexpr (WORKER_MOMENTS) {
        mv[r] = ld_f4(p.m + so + idx);
        vv[r] = ld_f4(p.v + so + idx);
      }
      if constexpr (L2) hw[r] = held_fetch(p, tile.off + r * kRowElems + warp * 128, lane);
    }
#pragma unroll
    for (int r = 0; r < kRows; ++r) {
      const int idx = r * kRowElems + threadIdx.x * 4;
      if (idx >= tile.count) continue;
      float gg[4] = {gv[r].x, gv[r].y, gv[r].z, gv[r].w};
      const float ee[4] = {ev[r].x, ev[r].y, ev[r].z, ev[r].w};
      float uu[4];
      if constexpr (L2) add_l2_term_fetched(p, tile.off + r * kRowElems + warp * 128, lane, hw[r], gg);
      if constexpr (WORKER_MOMENTS) {
        float mm[4] = {mv[r].x, mv[r].y, mv[r].z, mv[r].w};
        float vs[4] = {vv[r].x, vv[r].y, vv[r].z, vv[r].w};
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          moments(p.h, gg[c], mm[c], vs[c]);
          uu[c] = __fadd_rn(adam_step(p.h, mm[c], vs[c], p.alpha), ee[c]);
        }
        st_f4(p.m + so + idx, make_float4(mm[0], mm[1], mm[2], mm[3]));
        st_f4(p.v + so + idx, make_float4(vs[0], vs[1], vs[2], vs[3]));
        st_f4(p.e + so + idx, make_float4(uu[0], uu[1], uu[2], uu[3]));
      } else {
#pragma unroll
        for (int c = 0; c < 4; ++c) uu[c] = __fadd_rn(gg[c], ee[c]);
      }
#pragma unroll
      for (int c = 0; c < 4; ++c) mx = max(mx, __float_as_uint(fabsf(uu[c])));
    }
  }
  if (cur_pair >= 0) leave();
}

// Then codes and e' of the stochastic operator; WORKER_MOMENTS: u is in e's place.  The four coordinates of a thread
// are one block of the stream: counter (element / 4, worker, step), key = seed.  Three blocks per SM: left to itself
// the compiler takes 97 registers, which are two (8 x 10^6 elements, n = 4: 45.1 us a step against 43.0).
template <bool WORKER_MOMENTS, bool L2>
static __global__ void __launch_bounds__(kThreads, 3)
worker_toss_kernel(const WorkerParams p) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (long long t = blockIdx.x; t < p.total_tiles; t += gridDim.x) {
    const int wl = (int)(t / p.tiles_per_worker);
    const Tile tile = p.tiles[(int)(t - (long long)wl * p.tiles_per_worker)];
    const int w = p.worker_begin + wl;
    const float* gp = p.g + (long long)wl * p.D + tile.off;
    const long long so = (long long)w * p.D + tile.off;
    float4 gv[kRows], ev[kRows];
    HeldRaw hw[L2 ? kRows : 1];
#pragma unroll
    for (int r = 0; r < kRows; ++r) {
      const int idx = r * kRowElems + threadIdx.x * 4;
      if (idx >= tile.count) continue;
      if constexpr (!WORKER_MOMENTS) gv[r] = ld_f4_stream(gp + idx);
      ev[r] = ld_f4(p.e + so + idx);
      if constexpr (L2) hw[r] = held_fetch(p, tile.off + r * kRowElems + warp * 128, lane);
    }
    const unsigned sb = p.scale_bits[(long long)w * p.S + tile.seg];
    const GradScale gs = grad_scale<G_STOCHASTIC>(__uint_as_float(sb), p.k);
    if (sb >= 0x7f800000u && threadIdx.x == 0) atomicOr(p.status, 1u);
#pragma unroll
    for (int r = 0; r < kRows; ++r) {
      const int idx = r * kRowElems + threadIdx.x * 4;
      if (idx >= tile.count) continue;                  // warp-uniform: counts are multiples of 128
      float uu[4] = {ev[r].x, ev[r].y, ev[r].z, ev[r].w};
      if constexpr (!WORKER_MOMENTS) {
        float gg[4] = {gv[r].x, gv[r].y, gv[r].z, gv[r].w};
        if constexpr (L2) add_l2_term_fetched(p, tile.off + r * kRowElems + warp * 128, lane, hw[r], gg);
#pragma unroll
        for (int c = 0; c < 4; ++c) uu[c] = __fadd_rn(gg[c], uu[c]);
      }
      const unsigned long long block = (unsigned long long)(tile.off + idx) >> 2;
      const uint4 rnd = philox4x32_10(make_uint4((unsigned)block, (unsigned)(block >> 32), (unsigned)w, p.step),
                                      make_uint2(p.seed_lo, p.seed_hi));
      float en[4];
      const unsigned code = quantize_stochastic4(uu, gs, rnd, en);      // the lane's byte of four codes
      st_f4(p.e + so + idx, make_float4(en[0], en[1], en[2], en[3]));
      store_row_of_code_bytes(code, p.gcodes + (long long)w * p.gcode_bytes +
                                        (tile.off + r * kRowElems + warp * 128) * p.bits / 8, lane);
    }
  }
}

// ---------------------------------------------------------------------------
// Identity Q_g: the stream is u itself, the scale is 1, e <- u - u.
// ---------------------------------------------------------------------------
template <bool WORKER_MOMENTS, bool L2 = false>
__global__ void __launch_bounds__(kThreads)
worker_identity_kernel(const WorkerParams p) {
  for (long long t = blockIdx.x; t < p.total_tiles; t += gridDim.x) {
    const int wl = (int)(t / p.tiles_per_worker);
    const int tl = (int)(t - (long long)wl * p.tiles_per_worker);
    const Tile tile = p.tiles[tl];
    const int w = p.worker_begin + wl;
    if (tl == 0 && threadIdx.x < p.S) {
      for (int s = threadIdx.x; s < p.S; s += kThreads)
        p.scale_bits[(long long)w * p.S + s] = __float_as_uint(1.0f);
    }
    const float* gp = p.g + (long long)wl * p.D + tile.off;
    const long long so = (long long)w * p.D + tile.off;
    float* out = reinterpret_cast<float*>(p.gcodes + (long long)w * p.gcode_bytes) + tile.off;
#pragma unroll
    for (int r = 0; r < kRows; ++r) {
      const int idx = r * kRowElems + threadIdx.x * 4;
      if (idx >= tile.count) continue;
      const float4 g4 = ld_f4_stream(gp + idx);
      const float4 e4 = ld_f4(p.e + so + idx);
      float gg[4] = {g4.x, g4.y, g4.z, g4.w};
      float ee[4] = {e4.x, e4.y, e4.z, e4.w};
      float uu[4], en[4];
      if constexpr (L2)
        add_l2_term(p, tile.off + r * kRowElems + (threadIdx.x >> 5) * 128, threadIdx.x & 31, gg);
      if constexpr (WORKER_MOMENTS) {
        const float4 m4 = ld_f4(p.m + so + idx);
        const float4 v4 = ld_f4(p.v + so + idx);
        float mm[4] = {m4.x, m4.y, m4.z, m4.w};
        float vs[4] = {v4.x, v4.y, v4.z, v4.w};
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          moments(p.h, gg[c], mm[c], vs[c]);
          uu[c] = __fadd_rn(adam_step(p.h, mm[c], vs[c], p.alpha), ee[c]);
        }
        st_f4(p.m + so + idx, make_float4(mm[0], mm[1], mm[2], mm[3]));
        st_f4(p.v + so + idx, make_float4(vs[0], vs[1], vs[2], vs[3]));
      } else {
#pragma unroll
        for (int c = 0; c < 4; ++c) uu[c] = __fadd_rn(gg[c], ee[c]);
      }
#pragma unroll
      for (int c = 0; c < 4; ++c) en[c] = __fsub_rn(uu[c], uu[c]);
      st_f4(out + idx, make_float4(uu[0], uu[1], uu[2], uu[3]));
      st_f4(p.e + so + idx, make_float4(en[0], en[1], en[2], en[3]));
    }
  }
}

// ---------------------------------------------------------------------------
// Q_x of 4 consecutive weights of one lane, packed row store, optional residual.
// ---------------------------------------------------------------------------
// With an error buffer for the broadcast (wfeedback, not in the paper) the quantized value is
// y = x + wfeedback and the buffer becomes y - Q_x(y).
__device__ __forceinline__ void broadcast_row(const float xin[4], int kx, int xbits,
                                              unsigned char* wcodes, float* wresid, float* wfeedback,
                                              long long elem, long long row_elem, int lane) {
  unsigned code[4];
  float xx[4] = {xin[0], xin[1], xin[2], xin[3]};
  float xq[4];
  if (wfeedback) {
    const float4 ew = ld_f4(wfeedback + elem);
    xx[0] = __fadd_rn(xx[0], ew.x); xx[1] = __fadd_rn(xx[1], ew.y);
    xx[2] = __fadd_rn(xx[2], ew.z); xx[3] = __fadd_rn(xx[3], ew.w);
  }
#pragma unroll
  for (int c = 0; c < 4; ++c) code[c] = quantize_weight(xx[c], kx, xq[c]);
  if (wresid || wfeedback) {
    const float4 r = make_float4(__fsub_rn(xx[0], xq[0]), __fsub_rn(xx[1], xq[1]),
                                 __fsub_rn(xx[2], xq[2]), __fsub_rn(xx[3], xq[3]));
    if (wresid) st_f4(wresid + elem, r);
    if (wfeedback) st_f4(wfeedback + elem, r);
  }
  void* dst = wcodes + row_elem * xbits / 8;
  switch (xbits) {
    case 2: pack_row_store<2>(code[0], code[1], code[2], code[3], dst, lane); break;
    case 3: pack_row_store<3>(code[0], code[1], code[2], code[3], dst, lane); break;
    case 8: pack_row_store<8>(code[0], code[1], code[2], code[3], dst, lane); break;
    default: pack_row_store_rt(xbits, code[0], code[1], code[2], code[3], dst, lane); break;
  }
}

// Stand-alone Q_x(x) (the broadcast of x_1 before the first step).  Internal linkage:
// this header is included by more than one source file of the library.
static __global__ void __launch_bounds__(kThreads)
weight_broadcast_kernel(const ServerParams p) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int t = blockIdx.x; t < p.tiles_per_worker; t += gridDim.x) {
    const Tile tile = p.tiles[t];
#pragma unroll
    for (int r = 0; r < kRows; ++r) {
      const int idx = r * kRowElems + threadIdx.x * 4;
      if (idx >= tile.count) continue;
      const float4 x4 = ld_f4(p.x + tile.off + idx);
      const float xx[4] = {x4.x, x4.y, x4.z, x4.w};
      broadcast_row(xx, p.kx, p.xbits, p.wcodes, p.wresid, p.wfeedback, tile.off + idx,
                    tile.off + r * kRowElems + warp * 128, lane);
    }
  }
}

// ---------------------------------------------------------------------------
// The fused server pass (Algorithm 2's gather/average/update and the next
// broadcast): for every element, decode the n workers' codes and sum them in
// worker order, divide by n, update x (and m, v when they live here), quantize
// the new x for the broadcast.
//
// GDEC selects how a gradient code becomes a value:
//   G_TERNARY  2-bit codes {0,1,2} <-> {-s, 0, +s}.  The code is moved into the
//              mantissa of a float whose exponent gives its bit position the
//              weight 1 (value 2^E + code); subtracting 2^E + 1 leaves the level
//              index q as a float, and fma(q, s, acc) = fl(acc + q*s) is the same
//              rounding as adding the decoded value because q*s is exact.
//   G_IDENTITY the streams are binary32 values.
//   otherwise  a per-CTA table value[worker][code] = +-fl(s * level) in shared
//              memory, rebuilt when the segment changes.
// ---------------------------------------------------------------------------
constexpr int kMaxLutCodes = 256;

template <bool SERVER_MOMENTS, int GDEC>
__global__ void __launch_bounds__(kThreads)
server_step_kernel(const ServerParams p) {
  extern __shared__ float smem[];
  float* s_scale = smem;                 // [n]
  float* s_lut = smem + p.n;             // [n][1 << gbits]   (table decode only)
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int cur_seg = -1;
  for (int t = blockIdx.x; t < p.tiles_per_worker; t += gridDim.x) {
    const Tile tile = p.tiles[t];
    if (tile.seg != cur_seg) {
      __syncthreads();
      cur_seg = tile.seg;
      for (int i = threadIdx.x; i < p.n; i += kThreads)
        s_scale[i] = p.scales[(long long)i * p.S + cur_seg];
      if constexpr (GDEC != G_TERNARY && GDEC != G_IDENTITY) {
        const int ncodes = 1 << p.gbits;
        for (int idx = threadIdx.x; idx < p.n * ncodes; idx += kThreads) {
          const int i = idx / ncodes, code = idx - i * ncodes;
          const float s = p.scales[(long long)i * p.S + cur_seg];
          int q = code - p.L;
          const int c = q < 0 ? -q : q;
          float val = 0.0f;
          if (c != 0 && c <= p.L) {
            float lv;
            if (GDEC == G_FIVE) lv = level_value<G_FIVE>(c, p.k);
            else if (GDEC == G_POW2) lv = level_value<G_POW2>(c, p.k);
            else lv = level_value<G_UNIFORM>(c, p.k);
            const float mag = __fmul_rn(s, lv);
            val = q < 0 ? -mag : mag;
          }
          s_lut[idx] = val;
        }
      }
      __syncthreads();
    }

    bool act[kRows];
    float4 xv[kRows], mv[kRows], vv[kRows];
#pragma unroll
    for (int r = 0; r < kRows; ++r) {
      const int idx = r * kRowElems + threadIdx.x * 4;
      act[r] = idx < tile.count;
      if (act[r]) {
        xv[r] = ld_f4(p.x + tile.off + idx);
        if constexpr (SERVER_MOMENTS) {
          mv[r] = ld_f4(p.m + tile.off + idx);
          vv[r] = ld_f4(p.v + tile.off + idx);
        }
      }
    }

    float acc[kRows][4];
#pragma unroll
    for (int r = 0; r < kRows; ++r)
#pragma unroll
      for (int c = 0; c < 4; ++c) acc[r][c] = 0.0f;

    if constexpr (GDEC == G_TERNARY) {
      // one byte = this thread's 4 codes of a row
      const unsigned char* cb = p.gcodes + (tile.off >> 2) + threadIdx.x;
#pragma unroll 4
      for (int i = 0; i < p.n; ++i) {
        const float s = s_scale[i];
        const unsigned char* ci = cb + (long long)i * p.gcode_bytes;
        unsigned b[kRows];
#pragma unroll
        for (int r = 0; r < kRows; ++r) b[r] = act[r] ? (unsigned)__ldg(ci + r * (kRowElems / 4)) : 0x55u;
#pragma unroll
        for (int r = 0; r < kRows; ++r) {
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            const unsigned bits = (b[r] & (3u << (2 * c))) | ((unsigned)(150 - 2 * c) << 23);
            const float q = __fadd_rn(__uint_as_float(bits), -(exp2i(23 - 2 * c) + 1.0f));
            acc[r][c] = __fmaf_rn(q, s, acc[r][c]);
          }
        }
      }
    } else if constexpr (GDEC == G_IDENTITY) {
      for (int i = 0; i < p.n; ++i) {
        const float* ui = reinterpret_cast<const float*>(p.gcodes + (long long)i * p.gcode_bytes) + tile.off;
#pragma unroll
        for (int r = 0; r < kRows; ++r) {
          if (!act[r]) continue;
          const float4 u4 = ld_f4_stream(ui + r * kRowElems + threadIdx.x * 4);
          acc[r][0] = __fadd_rn(acc[r][0], u4.x);
          acc[r][1] = __fadd_rn(acc[r][1], u4.y);
          acc[r][2] = __fadd_rn(acc[r][2], u4.z);
          acc[r][3] = __fadd_rn(acc[r][3], u4.w);
        }
      }
    } else {
      const int ncodes = 1 << p.gbits;
      const unsigned cmask = (unsigned)ncodes - 1u;
      for (int i = 0; i < p.n; ++i) {
        const unsigned char* ci = p.gcodes + (long long)i * p.gcode_bytes;
        const float* lut = s_lut + i * ncodes;
#pragma unroll
        for (int r = 0; r < kRows; ++r) {
          if (!act[r]) continue;
          const long long row_elem = tile.off + r * kRowElems + warp * 128;
          const unsigned f = unpack_row_field(ci + row_elem * p.gbits / 8, p.gbits, lane);
#pragma unroll
          for (int c = 0; c < 4; ++c)
            acc[r][c] = __fadd_rn(acc[r][c], lut[(f >> (c * p.gbits)) & cmask]);
        }
      }
    }

#pragma unroll
    for (int r = 0; r < kRows; ++r) {
      if (!act[r]) continue;
      const int idx = r * kRowElems + threadIdx.x * 4;
      float xx[4] = {xv[r].x, xv[r].y, xv[r].z, xv[r].w};
      if constexpr (SERVER_MOMENTS) {
        float mm[4] = {mv[r].x, mv[r].y, mv[r].z, mv[r].w};
        float vs[4] = {vv[r].x, vv[r].y, vv[r].z, vv[r].w};
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const float dhat = __fdiv_rn(acc[r][c], p.nf);
          moments(p.h, dhat, mm[c], vs[c]);
          xx[c] = __fsub_rn(xx[c], adam_step(p.h, mm[c], vs[c], p.alpha));
        }
        st_f4(p.m + tile.off + idx, make_float4(mm[0], mm[1], mm[2], mm[3]));
        st_f4(p.v + tile.off + idx, make_float4(vs[0], vs[1], vs[2], vs[3]));
      } else {
#pragma unroll
        for (int c = 0; c < 4; ++c) xx[c] = __fsub_rn(xx[c], __fdiv_rn(acc[r][c], p.nf));
      }
      st_f4(p.x + tile.off + idx, make_float4(xx[0], xx[1], xx[2], xx[3]));
      if (p.kx >= 0) {
        broadcast_row(xx, p.kx, p.xbits, p.wcodes, p.wresid, p.wfeedback, tile.off + idx,
                      tile.off + r * kRowElems + warp * 128, lane);
      }
    }
  }
}

}  // namespace qadam
