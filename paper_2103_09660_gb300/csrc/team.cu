// Small graphs: whole V-cycles (or the sweeps of one level) in one launch.
//
// A half-sweep of a small level takes a few microseconds of device time, and
// a launch per row class, fork, join and reduction costs several times that.
// Here a team of thread blocks (a cooperative launch, one block per SM) runs
// every step of a V-cycle, with a barrier among the team's blocks between
// the steps: copy in, then per level project, and per sweep the hyperedge
// rows, then the node rows. One graph takes one team of the whole grid; a
// batch of graphs is dealt over several teams, so that the graphs in work
// together fit L2 and a barrier spans few SMs.
//
// What bounds a step is a chain of dependent loads (descriptor, neighbour
// index, row), not bandwidth, so the split of the work keeps chains short:
//   - a long row or chunk goes to one warp per 32 words of the row, a lane per
//     32-bit word, which keeps 32 row loads in flight per lane in 32 registers
//     (a 16-byte vector per lane would need 128): a chunk of 128 incidences is
//     4 rounds of loads instead of 16;
//   - rows of at most 16 incidences take a lane per 16-byte vector, 8 loads in
//     flight (rows of at most 4: two vectors, so that a warp has twice the rows),
//     descriptors two passes ahead and neighbours one pass ahead;
//   - the descriptors and neighbours of a step's first pass are loaded before
//     the barrier that starts it (they do not change);
//   - a split row of at most 32 chunks is summed by one block, its partials in
//     shared memory, where there are few such rows; only rows with more chunks
//     (or many split rows) go through global partials and a step of their own.
//
// The items and split rows are the level's plans (SplitPlan) and every row is
// summed in the order of the per-launch kernels (refine.cu, batch.cu): the
// results are the same bits. Which levels take it: team_pays, team_fits, and for a
// batch the estimates below.
//
// Measured (GB300, same bits): the V-cycle of a 2,000-node graph (d = 32, 7
// levels x 10 sweeps) 2.25 -> 0.70 ms, of a 41K-node graph (d = 100, 33 levels
// x 20 sweeps) 31.2 -> 13.0 ms, of a batch of 64 graphs of 1K-100K nodes
// (d = 64) 91 -> 71 ms. What is left of a sweep of the 41K-node graph (20 us)
// is 3-6 us of dependent loads a half-sweep, 1.4 us a barrier (2 or 3 a
// sweep) and 4 us for a hub row's reduction. On larger levels the per-launch
// kernels, with twice the warps per SM, are faster (a level of 150K nodes, 2.1M
// incidences, d = 100: 2.0 against 3.9 ms for 10 sweeps).
//
// Rows written in one step are read in the next by other blocks, so row and
// partial loads are plain (never the read-only path); the barrier's
// acquire/release pair orders them. Every wait is bounded: a block that gives
// up records ERRBIT_TIMEOUT and returns, and so does the rest of its team. It
// goes to the graph's error word (read by hnv_sync_status), or, with the
// stopping rule, to the launch's own result, which that call reads anyway.
#include <algorithm>
#include <cmath>
#include <cstring>

#include "refine_device.cuh"

namespace hnv {

namespace {

using dev::VecT;

constexpr int kTeamThreads = 512;
constexpr int kTeamWarps = kTeamThreads / 32;
constexpr int kFinSlots = 1024;   // (slice, vector) pairs of a split row's reduction, as in
                                  // finalize_kernel's 1,024-thread blocks

__device__ __forceinline__ uint64_t global_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// A barrier among the `blocks` blocks that share `counter` (0 at launch).
// False once a wait gave up (the whole block sees the same answer). A wait is
// limited to g->wait_ns; the barrier at target *stop waits for one arrival
// more than comes (TeamGraph::stop_at). (A timeout is recorded here rather than
// where the kernel's body returns: with that body in a function of its own the
// batch of 64 graphs took 76.2 ms instead of 72.2, with no more spills.)
struct TeamBarrier {
  uint32_t* counter;
  uint32_t blocks;
  uint32_t target;
  const TeamGraph* graphs;   // a batch's, of which [q, q1) are still to be run
  int32_t q, q1;
  int32_t* result;           // the stopping rule's word for a timeout, or null
  int* dead;             // shared memory, as g and stop
  const TeamGraph* g;
  const uint32_t* stop;

  __device__ __forceinline__ bool wait() {
    __syncthreads();
    if (threadIdx.x == 0) {
      target += blocks;
      const uint32_t want = target == *stop ? target + 1 : target;
      asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(counter) : "memory");
      uint64_t t0 = 0;
      int spins = 0;
      for (;;) {
        uint32_t v;
        asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(counter) : "memory");
        if ((int32_t)(v - want) >= 0) break;
        if ((++spins & 1023) == 0) {
          const uint64_t now = global_ns();
          if (t0 == 0) {
            t0 = now;
          } else if (now - t0 > g->wait_ns) {
            *dead = 1;
            if (result) {
              atomicOr(result, (int32_t)ERRBIT_TIMEOUT);
            } else if (!graphs) {
              atomicOr(g->err, (int32_t)ERRBIT_TIMEOUT);
            } else {   // the team's later graphs are not run
              for (int32_t r = q; r < q1; ++r) atomicOr(graphs[r].err, (int32_t)ERRBIT_TIMEOUT);
            }
            break;
          }
        }
      }
      asm volatile("fence.acq_rel.gpu;" ::: "memory");
    }
    __syncthreads();
    return *dead == 0;
  }
};

// What a warp's first pass of a step needs: a descriptor and this lane's
// neighbour (and weight) in the first round.
struct Head {
  int4 it;
  int32_t i0;
  float w0;
};

template <bool W>
__device__ __forceinline__ void load_neighbour(const TeamSide& sd, int lane, Head& h) {
  h.i0 = 0;
  h.w0 = 0.f;
  if (lane < h.it.z) {
    h.i0 = __ldg(sd.idx + h.it.y + lane);
    if (W) h.w0 = __ldg(sd.inc_w + h.it.y + lane);
  }
}

// Words of a row per warp: `slices` equal shares of the row's words, at most 32.
struct Slices {
  int words, slices, per;
  __device__ __forceinline__ explicit Slices(int dv)
      : words(4 * dv), slices((words + 31) / 32), per((words + slices - 1) / slices) {}
};

// The running maximum of |change| of one block into *slot.
__device__ __forceinline__ void team_diff_out(float diff, unsigned* slot) {
  for (int o = 16; o > 0; o >>= 1) diff = fmaxf(diff, __shfl_xor_sync(dev::kFull, diff, o));
  if ((threadIdx.x & 31) == 0 && diff > 0.f) atomicMax(slot, __float_as_uint(diff));
}

// A 32-bit word of a row: one float32 or two bfloat16 (the lower-indexed in
// the low half).
template <typename T>
struct Word;
template <>
struct Word<float> {
  static constexpr int N = 1;
  __device__ __forceinline__ static void unpack(uint32_t w, float* f) { f[0] = __uint_as_float(w); }
  __device__ __forceinline__ static uint32_t pack(const float* f) { return __float_as_uint(f[0]); }
};
template <>
struct Word<__nv_bfloat16> {
  static constexpr int N = 2;
  __device__ __forceinline__ static void unpack(uint32_t w, float* f) {
    f[0] = __uint_as_float(w << 16);
    f[1] = __uint_as_float(w & 0xffff0000u);
  }
  __device__ __forceinline__ static uint32_t pack(const float* f) {
    return VecT<__nv_bfloat16>::pair(f[0], f[1]);
  }
};

__device__ __forceinline__ uint32_t load_word(const uint32_t* p) {
  uint32_t v;
  asm volatile("ld.global.u32 %0, [%1];" : "=r"(v) : "l"(p));
  return v;
}

// One warp's share (word `word` of the row per lane, if `on`) of a long row
// (out row written) or of a chunk (its sums to `part`), h.it's first 32
// neighbours in h. Incidences are added in order.
template <typename T, bool W, bool DIFF>
__device__ __forceinline__ void team_long(const TeamSide& sd, const Head& h, int word, bool on,
                                          const uint32_t* src, const uint32_t* self_in,
                                          uint32_t* out, float* part, int words, float keep,
                                          float omega, float& diff) {
  using WT = Word<T>;
  constexpr int N = WT::N;
  const int lane = threadIdx.x & 31;
  const int32_t beg = h.it.y, len = h.it.z;
  const bool is_row = h.it.w < 0;
  const float norm = is_row ? __ldg(sd.inv_norm + h.it.x) : 0.f;
  uint32_t self = 0u;
  if (is_row && on && (DIFF || keep != 0.f)) self = load_word(self_in + (size_t)h.it.x * words + word);
  float acc[N];
#pragma unroll
  for (int e = 0; e < N; ++e) acc[e] = 0.f;
  const uint32_t* base = src + (on ? word : 0);   // lanes past the share load its first word
  int32_t my = h.i0;
  float mw = h.w0;
#pragma unroll 1
  for (int32_t off = 0; off < len; off += 32) {
    const int32_t ahead = off + 32 + lane;
    int32_t nx = 0;
    float nw = 0.f;
    if (ahead < len) {
      nx = __ldg(sd.idx + beg + ahead);
      if (W) nw = __ldg(sd.inc_w + beg + ahead);
    }
    const int32_t cnt = len - off < 32 ? len - off : 32;
    // slots past the end load the round's first row again and are not added
    const int32_t nb0 = __shfl_sync(dev::kFull, my, 0);
    const int32_t own_nb = lane < cnt ? my : nb0;
    uint32_t x[32];
    auto load = [&](int u) {
      x[u] = load_word(base + (size_t)__shfl_sync(dev::kFull, own_nb, u) * words);
    };
    auto add = [&](int u) {
      float f[N];
      WT::unpack(x[u], f);
      const float w = W ? __shfl_sync(dev::kFull, mw, u) : 1.f;
#pragma unroll
      for (int e = 0; e < N; ++e) {
        const float t = W ? fmaf(w, f[e], acc[e]) : acc[e] + f[e];
        acc[e] = u < cnt ? t : acc[e];
      }
    };
#pragma unroll
    for (int u = 0; u < 16; ++u) load(u);
    if (cnt > 16) {
#pragma unroll
      for (int u = 16; u < 32; ++u) load(u);
#pragma unroll
      for (int u = 0; u < 32; ++u) add(u);
    } else {
#pragma unroll
      for (int u = 0; u < 16; ++u) add(u);
    }
    my = nx;
    mw = nw;
  }
  if (!on) return;
  if (is_row) {
    float sf[N], r[N];
    WT::unpack(self, sf);
    const float sc = omega * norm;
#pragma unroll
    for (int e = 0; e < N; ++e) r[e] = fmaf(keep, dev::own<DIFF>(keep, sf[e]), sc * acc[e]);
    const uint32_t res = WT::pack(r);
    out[(size_t)h.it.x * words + word] = res;
    if (DIFF) {
      float nf[N];
      WT::unpack(res, nf);
#pragma unroll
      for (int e = 0; e < N; ++e) diff = fmaxf(diff, fabsf(nf[e] - sf[e]));
    }
  } else {
#pragma unroll
    for (int e = 0; e < N; ++e) part[word * N + e] = acc[e];
  }
}

// The first passes of one side's step for one warp. Long tasks (item, slice)
// are numbered from the last item down, short passes likewise; the warps take
// the two lists from opposite ends.
struct StepHeads {
  Head lng, a, b;
};

// Lanes per row of the rows of 1-4 incidences: half of a long row's, two
// vectors each, so that a warp has twice as many rows in flight and still all
// of a row's loads.
template <int G>
__host__ __device__ constexpr int lanes_a() { return G > 4 ? G / 2 : G; }
template <int G, int VPL>
__host__ __device__ constexpr int vectors_a() { return VPL * G / lanes_a<G>(); }

// Split rows are summed inside a block where that saves the reduction's step
// (no row needs it anyway), a block has one row, and no row's chunks take its
// warps more than two rounds. (A row of 32 chunks on one block took 20 us, a
// reduction step with its barrier takes 4.)
template <typename T>
__device__ __forceinline__ bool block_mid(const TeamSide& sd, int blocks, int dv) {
  const int32_t most = sd.n_mid_chunks - 2 * (sd.n_mid - 1);   // a split row has >= 2 chunks
  return sd.n_mid > 0 && sd.n_huge == 0 && sd.n_mid <= blocks && kMidChunks * dv <= kFinSlots &&
         most * Slices(dv).slices <= 2 * kTeamWarps;
}

// Items [lo, hi) of the long list of a step.
template <typename T>
__device__ __forceinline__ int32_t long_count(const TeamSide& sd, int blocks, int dv) {
  // without the chunks of split rows that a block sums by itself
  return sd.n_items - sd.n_short - (block_mid<T>(sd, blocks, dv) ? sd.n_mid_chunks : 0);
}
// Item of position q of that list, from the last down: chunks, then the
// longest rows.
template <typename T>
__device__ __forceinline__ int32_t long_item(const TeamSide& sd, int32_t q, int blocks, int dv) {
  return (block_mid<T>(sd, blocks, dv) ? sd.n_rows : sd.n_items) - 1 - q;
}

template <typename T, int G, bool W>
__device__ __forceinline__ StepHeads load_heads(const TeamSide& sd, int dv, int block, int blocks) {
  const int lane = threadIdx.x & 31;
  const int warp = (threadIdx.x >> 5) * blocks + block, warps = kTeamWarps * blocks;
  const Slices sl(dv);
  StepHeads h;
  h.lng.it = make_int4(-1, 0, 0, -1);
  h.a.it = h.b.it = make_int4(-1, 0, 0, -1);
  if (warp < (int64_t)long_count<T>(sd, blocks, dv) * sl.slices)
    h.lng.it = __ldg(sd.items + long_item<T>(sd, warp / sl.slices, blocks, dv));
  const int back = warps - 1 - warp;
  constexpr int GA = lanes_a<G>();
  const int32_t ib = back * (32 / G) + lane / G, ia = back * (32 / GA) + lane / GA;
  if (ib < sd.n_short - sd.n_a) h.b.it = __ldg(sd.items + (sd.n_short - 1 - ib));
  if (ia < sd.n_a) h.a.it = __ldg(sd.items + (sd.n_a - 1 - ia));
  load_neighbour<W>(sd, lane, h.lng);
  load_neighbour<W>(sd, lane & (G - 1), h.b);
  load_neighbour<W>(sd, lane & (GA - 1), h.a);
  return h;
}

// The short rows [lo, hi) of a step, R = 32/G per pass, from the last down.
template <typename T, int G, int VPL, int U, bool W, bool DIFF>
__device__ __forceinline__ void team_short(const TeamSide& sd, int32_t lo, int32_t hi, Head cur,
                                           const uint4* src, const uint4* self_in, uint4* out,
                                           int dv, float keep, float omega, int warp, int warps,
                                           float& diff) {
  constexpr int R = 32 / G;
  const int lane = threadIdx.x & 31;
  const int lg = lane & (G - 1), grp = lane / G;
  const int32_t n = hi - lo, step = warps * R;
  auto load_item = [&](int32_t i) -> int4 {
    return i < n ? __ldg(sd.items + (hi - 1 - i)) : make_int4(-1, 0, 0, -1);
  };
  if (warp * R >= n) return;
  Head nxt;
  nxt.it = load_item(warp * R + grp + step);
  for (int32_t base = warp * R; base < n; base += step) {
    load_neighbour<W>(sd, lg, nxt);
    const int4 nn = load_item(base + grp + 2 * step);
    dev::gather_item<T, G, VPL, W, true, false, true, U, DIFF>(
        cur.it, lg, sd.idx, sd.inc_w, sd.inv_norm, src, self_in, out, dv, keep, omega, nullptr,
        cur.i0, cur.w0, &diff);
    cur = nxt;
    nxt.it = nn;
  }
}

// One half-sweep by the team, up to but without its last barrier. False: a
// wait gave up.
template <typename T, int G, int VPL, bool W, bool DIFF>
__device__ __forceinline__ bool team_half(const TeamSide& sd, const StepHeads& hd,
                                          const uint4* src, const uint4* self_in, uint4* out,
                                          float* partials, int dv, float keep, float omega,
                                          int block, int blocks, float* sm, unsigned* slot,
                                          TeamBarrier& bar) {
  constexpr int N = VecT<T>::N;
  constexpr int U = VPL == 2 ? 4 : (G < 8 ? G : 8);
  const int lane = threadIdx.x & 31;
  // block-fastest numbering: consecutive tasks go to different SMs
  const int warp = (threadIdx.x >> 5) * blocks + block;
  const int warps = kTeamWarps * blocks;
  const Slices sl(dv);
  const uint32_t* src32 = reinterpret_cast<const uint32_t*>(src);
  const uint32_t* self32 = reinterpret_cast<const uint32_t*>(self_in);
  uint32_t* out32 = reinterpret_cast<uint32_t*>(out);
  const int d = dv * N;
  float diff = 0.f;
  const bool bmid = block_mid<T>(sd, blocks, dv);
  // long rows and chunks
  {
    const int64_t tasks = (int64_t)long_count<T>(sd, blocks, dv) * sl.slices;
    Head cur = hd.lng;
    for (int64_t t = warp; t < tasks; t += warps) {
      Head nxt;
      nxt.it = make_int4(-1, 0, 0, -1);
      if (t + warps < tasks)
        nxt.it = __ldg(sd.items + long_item<T>(sd, (int32_t)((t + warps) / sl.slices), blocks, dv));
      const int word = (int)(t % sl.slices) * sl.per + lane;
      const bool on = lane < sl.per && word < sl.words;
      float* part = cur.it.w < 0 ? nullptr : partials + (size_t)cur.it.w * d;
      team_long<T, W, DIFF>(sd, cur, word, on, src32, self32, out32, part, sl.words, keep, omega,
                            diff);
      load_neighbour<W>(sd, lane, nxt);
      cur = nxt;
    }
  }
  constexpr int GA = lanes_a<G>(), VA = vectors_a<G, VPL>();
  team_short<T, G, VPL, U, W, DIFF>(sd, sd.n_a, sd.n_short, hd.b, src, self_in, out, dv, keep,
                                    omega, warps - 1 - warp, warps, diff);
  team_short<T, GA, VA, VA == 4 ? 2 : 4, W, DIFF>(sd, 0, sd.n_a, hd.a, src, self_in, out, dv, keep,
                                                  omega, warps - 1 - warp, warps, diff);
  // split rows of few chunks, a block each
  if (bmid) {
    for (int32_t k = blocks - 1 - block; k < sd.n_mid; k += blocks) {
      const int4 ds = __ldg(sd.long_desc + k);
      for (int t = threadIdx.x >> 5; t < ds.z * sl.slices; t += kTeamWarps) {
        const int c = t / sl.slices;
        Head h;
        h.it = __ldg(sd.items + sd.n_rows + ds.y + c);
        load_neighbour<W>(sd, lane, h);
        const int word = (t - c * sl.slices) * sl.per + lane;
        team_long<T, W, DIFF>(sd, h, word, lane < sl.per && word < sl.words, src32, self32, out32,
                              sm + (size_t)c * d, sl.words, keep, omega, diff);
      }
      __syncthreads();
      if (threadIdx.x < 32)
        dev::finalize_mid<T, true, DIFF, true>(make_int4(ds.x, 0, ds.z, 0), lane, sm, sd.inv_norm,
                                               self_in, out, dv, keep, omega, &diff);
      __syncthreads();
    }
  }
  if (sd.n_huge > 0 || (sd.n_mid > 0 && !bmid)) {
    if (!bar.wait()) return false;
    for (int32_t k = block; k < sd.n_huge; k += blocks) {
      dev::finalize_huge<T, 8, true, DIFF>(__ldg(sd.long_desc + sd.n_mid + k), sm, partials,
                                           sd.inv_norm, self_in, out, dv, keep, omega,
                                           kFinSlots / dv, &diff);
      __syncthreads();
    }
    if (!bmid)
      for (int32_t k = warps - 1 - warp; k < sd.n_mid; k += warps)
        dev::finalize_mid<T, true, DIFF>(__ldg(sd.long_desc + k), lane, partials, sd.inv_norm,
                                         self_in, out, dv, keep, omega, &diff);
  }
  if (DIFF) team_diff_out(diff, slot);
  return true;
}

// dst[i] = src[i], i < count, by the team (rows of an earlier step: plain loads).
__device__ __forceinline__ void team_copy(uint4* dst, const uint4* src, int64_t count, int64_t t,
                                          int64_t threads) {
  for (int64_t i = t; i < count; i += threads) dst[i] = dev::load_row<true>(src + i);
}

// Fine rows from coarse rows through the level's rep maps, and a second copy
// into `ckpt` where that is given.
template <int G, int VPL>
__device__ __forceinline__ void team_project(const TeamLevel& f, const uint4* zc_v,
                                             const uint4* zc_e, uint4* zf_v, uint4* zf_e,
                                             uint4* ckpt, int dv, int warp, int warps) {
  constexpr int R = 32 / G;
  const int lg = threadIdx.x & (G - 1), grp = (threadIdx.x & 31) / G;
  const int64_t rows = (int64_t)f.n + f.m, step = (int64_t)warps * R;
  constexpr int U = 4;
  for (int64_t r0 = (int64_t)warp * R + grp; r0 < rows; r0 += U * step) {
    const uint4* s[U];
    uint4* o[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int64_t r = r0 + u * step;
      s[u] = nullptr;
      o[u] = nullptr;
      if (r < f.n) {
        s[u] = zc_v + (size_t)__ldg(f.rep_v + r) * dv;
        o[u] = zf_v + (size_t)r * dv;
      } else if (r < rows) {
        const int32_t q = __ldg(f.rep_e + (r - f.n));
        s[u] = q >= 0 ? zc_e + (size_t)q * dv : zc_v + (size_t)(-1 - q) * dv;
        o[u] = zf_e + (size_t)(r - f.n) * dv;
      }
    }
#pragma unroll
    for (int j = 0; j < VPL; ++j) {
      const int col = lg + j * G;
      uint4 x[U];
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (s[u] && col < dv) x[u] = dev::load_row<true>(s[u] + col);
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (s[u] && col < dv) {
          o[u][col] = x[u];
          if (ckpt) ckpt[(size_t)(r0 + u * step) * dv + col] = x[u];
        }
    }
  }
}

template <typename T, int G, int VPL, bool DIFF>
__global__ void __launch_bounds__(kTeamThreads, 1) team_kernel(const TeamArgs a) {
  __shared__ __align__(16) float sm[kFinSlots * VecT<T>::N];
  __shared__ int dead;
  __shared__ uint32_t stop;
  __shared__ TeamGraph g;
  if (threadIdx.x == 0) dead = 0;
  const int team = blockIdx.x / a.blocks, block = blockIdx.x - team * a.blocks;
  const int warp = (threadIdx.x >> 5) * a.blocks + block, warps = kTeamWarps * a.blocks;
  const int64_t thread = (int64_t)warp * 32 + (threadIdx.x & 31), threads = (int64_t)warps * 32;
  TeamBarrier bar{a.barriers + 32 * team, (uint32_t)a.blocks, 0u,    a.graphs, 0, 0,
                  DIFF ? a.result + 2 : nullptr,          &dead, &g,       &stop};
  const int32_t q0 = a.graphs ? a.team_first[team] : 0, q1 = a.graphs ? a.team_first[team + 1] : 1;
  const int dv = a.dv;
  for (int32_t q = q0; q < q1; ++q) {
    __syncthreads();
    if (threadIdx.x == 0) {
      g = a.graphs ? a.graphs[q] : a.one;
      stop = g.stop_at > 0 ? bar.target + (uint32_t)g.stop_at * bar.blocks : 0u;
    }
    __syncthreads();
    bar.q = q;
    bar.q1 = q1;
    for (int l = g.top; l >= g.bottom; --l) {
      const TeamLevel& lv = g.levels[l];
      uint4* zv = l == g.bottom ? g.zv0 : g.buf[l & 1];
      uint4* ze = l == g.bottom ? g.ze0 : zv + (size_t)lv.n * dv;
      uint4* ck = g.ckpt ? g.ckpt + (size_t)lv.row0 * dv : nullptr;
      if (l == g.top) {
        if (g.zc) {
          team_copy(zv, g.zc, (int64_t)lv.n * dv, thread, threads);
          team_copy(ze, g.zc + (size_t)lv.n * dv, (int64_t)lv.m * dv, thread, threads);
          if (ck) team_copy(ck, g.zc, ((int64_t)lv.n + lv.m) * dv, thread, threads);
        }
      } else {
        const uint4* cv = g.buf[(l + 1) & 1];
        team_project<G, VPL>(lv, cv, cv + (size_t)g.levels[l + 1].n * dv, zv, ze, ck, dv, warp,
                            warps);
      }
      uint4* e_in = ze;
      StepHeads he = load_heads<T, G, false>(lv.side[0], dv, block, a.blocks);
      if (!bar.wait()) return;
      for (int it = 0; it < a.sweeps; ++it) {
        // Jacobi: the new hyperedge rows go to a second buffer, the nodes
        // read the old ones, and the buffers change places
        uint4* e_out = a.jacobi ? (e_in == ze ? g.jtmp : ze) : ze;
        unsigned* slot = DIFF ? a.delta + it % 3 : nullptr;
        // the slot of the next sweep was last read two barriers ago
        if (DIFF && blockIdx.x == 0 && threadIdx.x == 0) a.delta[(it + 1) % 3] = 0u;
        if (!team_half<T, G, VPL, false, DIFF>(lv.side[0], he, zv, e_in, e_out, g.partials, dv,
                                               a.keep, a.omega, block, a.blocks, sm, slot, bar))
          return;
        const StepHeads hv = load_heads<T, G, true>(lv.side[1], dv, block, a.blocks);
        if (!bar.wait()) return;
        if (!team_half<T, G, VPL, true, DIFF>(lv.side[1], hv, a.jacobi ? e_in : e_out, zv, zv,
                                              g.partials, dv, a.keep, a.omega, block, a.blocks,
                                              sm, slot, bar))
          return;
        he = load_heads<T, G, false>(lv.side[0], dv, block, a.blocks);
        if (!bar.wait()) return;
        e_in = e_out;
        if (DIFF) {
          const float delta = __uint_as_float(load_word(slot));
          if (blockIdx.x == 0 && threadIdx.x == 0) {
            a.result[0] = it + 1;
            a.result[1] = __float_as_int(delta);
          }
          if (delta <= a.eps) break;
        }
      }
      if (e_in != ze) {
        team_copy(ze, e_in, (int64_t)lv.m * dv, thread, threads);
        if (!bar.wait()) return;
      }
    }
  }
}

template <typename T, int G, int VPL, bool DIFF>
int launch_team(const TeamArgs& a, int teams, cudaStream_t s) {
  void* kern = reinterpret_cast<void*>(team_kernel<T, G, VPL, DIFF>);
  TeamArgs args = a;
  void* params[] = {&args};
  const cudaError_t e = cudaLaunchCooperativeKernel(kern, dim3((unsigned)(teams * a.blocks)),
                                                    dim3(kTeamThreads), params, 0, s);
  if (e != cudaSuccess) {
    cudaGetLastError();
    if (team_refused(e)) return kTeamRefused;
    return cuda_status(e, "team_kernel");
  }
  note_launch();
  return HNV_OK;
}

template <typename T, bool DIFF>
int launch_team_dispatch(const TeamArgs& a, int teams, cudaStream_t s) {
  if (a.dv <= 4) return launch_team<T, 4, 1, DIFF>(a, teams, s);
  if (a.dv <= 8) return launch_team<T, 8, 1, DIFF>(a, teams, s);
  if (a.dv <= 16) return launch_team<T, 16, 1, DIFF>(a, teams, s);
  if (a.dv <= 32) return launch_team<T, 32, 1, DIFF>(a, teams, s);
  return launch_team<T, 32, 2, DIFF>(a, teams, s);
}

}  // namespace

bool team_refused(cudaError_t e) {
  return e == cudaErrorCooperativeLaunchTooLarge || e == cudaErrorNotSupported;
}

void team_level(const Level& lv, int64_t row0, TeamLevel* out) {
  *out = TeamLevel();
  out->n = lv.n;
  out->m = lv.m;
  out->row0 = row0;
  out->rep_v = lv.rep_v;
  out->rep_e = lv.rep_e;
  for (int side = 0; side < 2; ++side) {
    const SplitPlan& p = side == 0 ? lv.planE : lv.planV;
    TeamSide& t = out->side[side];
    t.items = p.items;
    t.long_desc = p.long_desc;
    t.idx = side == 0 ? lv.e_nodes : lv.v_edges;
    t.inc_w = side == 0 ? nullptr : lv.v_w;
    t.inv_norm = side == 0 ? lv.inv_size_e : lv.inv_deg_v;
    t.n_a = p.n_a;
    t.n_short = p.n_a + p.n_b;
    t.n_rows = p.n_a + p.n_b + p.n_c + p.n_d;
    t.n_mid_chunks = p.n_mid_chunks;
    t.n_items = p.n_a + p.n_b + p.n_c + p.n_d + p.n_chunks;
    t.n_mid = p.n_mid;
    t.n_huge = p.n_huge;
  }
}

bool team_fits(const Level& lv, int dtype, int d) {
  const int64_t rb = (int64_t)(dtype == HNV_BF16 ? 2 : 4) * d;
  return rb <= kTeamMaxRowBytes && lv.nnz * rb <= kTeamMaxGather &&
         ((int64_t)lv.n + lv.m) * rb <= kTeamMaxRows;
}

// The line between the two paths, measured on 36 levels of graphs of 5K-600K
// nodes (members of 2-3,000, coarse levels with hub nodes of up to thousands of
// incidences) at 17 row sizes, us a sweep, this path against a launch per row
// class (whose time differs by up to 20% between runs):
//   - it costs about 35 us per million incidences however narrow the rows are,
//     where the launches' floor is 50 us: of 32 bytes 1.36M 59 against 81-85,
//     1.74M 65 against 69-75, 1.87M 68 against 50, 2.14M 82 against 52 (the
//     launches are slower for bfloat16 rows of one vector: 1.87M 70 against 87,
//     2.14M 84 against 59);
//   - beyond 100 MB of gathered rows its 16 warps per SM keep too few loads in
//     flight: 256-byte float32 rows 115 MB 51 against 56, 400-byte ones 131 MB 66
//     against 52, 162 MB 79 against 56-60. The launches need more time for rows of
//     at most 128 bytes (174 MB: float32 74 against 88-105, bfloat16 77 against
//     75-94), for bfloat16, whose conversions they spend issue slots on (256 bytes:
//     167 MB 69 against 83, 215 MB 80 against 73), and for rows of two vectors per
//     lane (151 MB 50 against 60).
bool team_pays(const Level& lv, int dtype, int d) {
  const int64_t rb = (int64_t)(dtype == HNV_BF16 ? 2 : 4) * d;
  int64_t gather = 125000000;
  if (rb > 512) gather = 160000000;
  else if (rb <= 128) gather = kTeamMaxGather;
  else if (dtype == HNV_BF16 && rb <= 256) gather = 170000000;
  const int64_t most = dtype == HNV_BF16 && rb == 16 ? 2000000 : 1800000;
  return team_fits(lv, dtype, d) && lv.nnz <= most && lv.nnz * rb <= gather;
}

int team_blocks_for(const Level& lv, int dtype, int d) {
  // warps of one pass over the larger side: a short row takes a lane per
  // vector, a long row or chunk a lane per word
  const int dv = (dtype == HNV_BF16 ? 2 : 4) * d / 16;
  int g = 4;
  while (g < 32 && g < dv) g <<= 1;
  int64_t warps = 1;
  for (const SplitPlan* p : {&lv.planE, &lv.planV})
    warps = std::max<int64_t>(warps, ((int64_t)p->n_a + p->n_b) * g / 32 +
                                         ((int64_t)p->n_c + p->n_d + p->n_chunks) *
                                             ((4 * dv + 31) / 32));
  const int64_t want = (warps + kTeamWarps - 1) / kTeamWarps;
  return (int)std::max<int64_t>(1, std::min<int64_t>(want, num_sms()));
}

double team_sweep_us(const Level& lv, int dtype, int d, int blocks) {
  // fitted to a batch of 64 graphs of 1K-100K nodes (d = 64, 9 blocks a
  // team): 12 us of dependent loads and barriers a sweep, 52 GB/s of rows per
  // SM beyond it
  const double bytes = (double)(dtype == HNV_BF16 ? 2 : 4) * d *
                       (2.0 * lv.nnz + 3.0 * ((double)lv.n + lv.m));
  return 12.0 + bytes / (52e3 * blocks);
}

namespace {

// Nanoseconds per incidence of a sweep (both sides) on the whole device, at rows
// of 16 << i bytes; between them by the logarithm. From batches of 2-300 graphs
// of 2K-600K nodes with the whole device at work (float32, bfloat16).
constexpr double kTeamNs[2][7] = {{.034, .034, .037, .055, .112, .23, .42},
                                  {.039, .040, .045, .062, .112, .21, .415}};
constexpr double kStepNs[2][7] = {{.020, .020, .034, .054, .118, .182, .34},
                                  {.026, .023, .040, .070, .137, .27, .53}};

double per_incidence_us(const double* ns, double row_bytes) {
  const double x = std::max(0.0, std::log2(row_bytes / 16.0));
  const int i = std::min((int)x, 5);
  return 1e-3 * (ns[i] + (x - i) * (ns[i + 1] - ns[i]));
}

}  // namespace

double team_batch_us(const Level& lv, int dtype, int d, int blocks) {
  const int k = dtype == HNV_BF16 ? 1 : 0;
  return 8.0 + (double)lv.nnz * per_incidence_us(kTeamNs[k], (k ? 2.0 : 4.0) * d) * num_sms() /
                   blocks;
}

double step_batch_us(int steps, int64_t nnz, int dtype, int d) {
  const int k = dtype == HNV_BF16 ? 1 : 0;
  return 50.0 * steps + (double)nnz * per_incidence_us(kStepNs[k], (k ? 2.0 : 4.0) * d);
}

int team_launch(TeamArgs a, int teams, int dtype, int d, cudaStream_t s) {
  a.dv = (dtype == HNV_BF16 ? 2 : 4) * d / 16;
  const bool diff = a.result != nullptr;
  if (dtype == HNV_BF16)
    return diff ? launch_team_dispatch<__nv_bfloat16, true>(a, teams, s)
                : launch_team_dispatch<__nv_bfloat16, false>(a, teams, s);
  return diff ? launch_team_dispatch<float, true>(a, teams, s)
              : launch_team_dispatch<float, false>(a, teams, s);
}

}  // namespace hnv
