// One coarsening step (Algorithm 1, Section 3.1), integer only and
// bit-exact: every node picks a hyperedge, nodes that picked the same
// hyperedge merge into one coarse node, hyperedges whose members all merged
// into one coarse node are removed, the rest connect the coarse nodes of
// their members.
#include <cmath>

#include "hnv_internal.cuh"

namespace hnv {

namespace {

constexpr unsigned FULL = 0xffffffffu;
constexpr uint64_t kGamma = 0x9E3779B97F4A7C15ull;  // SplitMix64 increment

// SplitMix64 finaliser (Steele, Lea & Flood, OOPSLA 2014).
__host__ __device__ inline uint64_t mix64(uint64_t z) {
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

// prio_l(e) for the policies of hnv_assign (see hnv.h).
__global__ void priority_kernel(int32_t m, int32_t policy, uint64_t salt,
                                const int32_t* __restrict__ e_ptr, const float* __restrict__ w,
                                const int32_t* __restrict__ orig_e,
                                const uint64_t* __restrict__ explicit_tab,
                                uint64_t* __restrict__ prio) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < m;
       e += (int64_t)gridDim.x * blockDim.x) {
    const uint64_t h = mix64((uint64_t)e ^ salt);
    uint64_t p = h;
    if (policy == HNV_ASSIGN_LOW_DEGREE) {
      uint64_t sz = (uint64_t)(e_ptr[e + 1] - e_ptr[e]);
      if (sz > 0xFFFFFFull) sz = 0xFFFFFFull;
      p = (sz << 40) | (h >> 24);
    } else if (policy == HNV_ASSIGN_HIGH_WEIGHT) {
      const uint64_t bits = (uint64_t)__float_as_uint(w[e]);
      p = ((0xFFFFFFFFull - bits) << 32) | (h >> 32);
    } else if (policy == HNV_ASSIGN_EXPLICIT) {
      p = explicit_tab[orig_e[e]];
    }
    prio[e] = p;
  }
}

// c(v) = argmin_{e in N(v)} (-score(v, e), prio(e), e), or -1; a group of
// lanes per node (8 where nodes have at most 24 incidences on average, so that
// a warp has four nodes' dependent loads in flight and three shuffle rounds
// instead of five; 32 otherwise), lanes stride the CSC row, then a
// lexicographic min over the group. score is the cosine of the feature rule
// (per CSC entry), or absent (all equal: the featureless rules). Long rows go
// to `long_rows` for assign_long_kernel (a block per row or part).
// Rows longer than kHubRow are cut into kHubParts parts, a block each: one
// block took 331 us of the 1M-node workload's coarsening on hub nodes of up
// to 810,823 incidences.
constexpr int32_t kHubRow = 16384;
constexpr int kHubParts = 64;
constexpr int kLongThreads = 512;

__device__ __forceinline__ void lex_min(float& bs, uint64_t& bp, int32_t& be, float sc, uint64_t p,
                                        int32_t e) {
  if (sc > bs || (sc == bs && (p < bp || (p == bp && e < be)))) {
    bs = sc;
    bp = p;
    be = e;
  }
}

// ---------------------------------------------------------------------------
// Feature rule (Section 3.1, nodes with features). The cosine decides an
// argmax, so every float step is an explicitly rounded float32 operation
// (no fused multiply-add) in a fixed order; the oracle takes the same steps.
// ---------------------------------------------------------------------------

// out[r] = mean of X rows idx[ptr[r] .. ptr[r+1]) (one thread per (r, dim),
// added in list order, 8 loads in flight, then divided by the count; an empty
// list gives 0). Rows longer than kMeanLong go to long_rows, for
// segment_mean_long_kernel.
constexpr int32_t kMeanLong = 64;
constexpr int kMeanTile = 128;      // members per shared-memory tile
constexpr int kMeanThreads = 256;

__global__ void segment_mean_kernel(int32_t rows, int32_t k, const int32_t* __restrict__ ptr,
                                    const int32_t* __restrict__ idx, const float* __restrict__ X,
                                    float* __restrict__ out, int32_t* __restrict__ long_rows,
                                    int32_t* __restrict__ n_long) {
  const int64_t total = (int64_t)rows * k;
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < total;
       t += (int64_t)gridDim.x * blockDim.x) {
    const int64_t r = t / k;
    const int32_t i = (int32_t)(t - r * k);
    const int32_t b = ptr[r], e = ptr[r + 1];
    if (e - b > kMeanLong) {
      if (i == 0) long_rows[atomicAdd(n_long, 1)] = (int32_t)r;
      continue;
    }
    float acc = 0.f;
    for (int32_t j = b; j < e; j += 8) {
      float x[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) x[u] = j + u < e ? X[(size_t)idx[j + u] * k + i] : 0.f;
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (j + u < e) acc = __fadd_rn(acc, x[u]);
    }
    out[t] = (e > b) ? __fdiv_rn(acc, (float)(e - b)) : 0.f;
  }
}

// The listed rows, 32 dimensions a task: the block copies kMeanTile members'
// values at a time into shared memory, kMeanStages - 1 tiles ahead of the
// warp that adds them in list order (cp.async; the member IDs of a tile are
// loaded one tile before its copies). A thread walking a 5,000-member list
// alone, one dependent load after the other, took 660 us; tiles loaded through
// registers, the loads of a tile exposed, 268 us.
constexpr int kMeanStages = 3;

__global__ void __launch_bounds__(kMeanThreads)
segment_mean_long_kernel(int32_t k, const int32_t* __restrict__ ptr,
                         const int32_t* __restrict__ idx, const float* __restrict__ X,
                         float* __restrict__ out, const int32_t* __restrict__ long_rows,
                         const int32_t* __restrict__ n_long) {
  constexpr int W = kMeanThreads / 32, PER = kMeanTile / W;   // copies per thread and tile
  __shared__ float tile[kMeanStages][kMeanTile][32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int32_t slabs = (k + 31) / 32;
  const int64_t tasks = (int64_t)*n_long * slabs;
  for (int64_t q = blockIdx.x; q < tasks; q += gridDim.x) {
    const int32_t r = long_rows[q / slabs];
    const int32_t col = (int32_t)(q % slabs) * 32 + lane;
    const int32_t b = ptr[r], e = ptr[r + 1];
    const int32_t tiles = (e - b + kMeanTile - 1) / kMeanTile;
    int32_t id[PER];
    auto ids = [&](int32_t t) {
#pragma unroll
      for (int u = 0; u < PER; ++u) {
        const int32_t j = b + t * kMeanTile + w + u * W;
        id[u] = j < e ? idx[j] : -1;
      }
    };
    // copies tile t (its IDs in id) and loads the IDs of tile t + 1
    auto copy = [&](int32_t t) {
#pragma unroll
      for (int u = 0; u < PER; ++u) {
        const uint32_t dst =
            (uint32_t)__cvta_generic_to_shared(&tile[t % kMeanStages][w + u * W][lane]);
        if (id[u] >= 0 && col < k)
          asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst),
                       "l"(X + (size_t)id[u] * k + col)
                       : "memory");
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
      ids(t + 1);
    };
    ids(0);
    __syncthreads();   // the adder is done with the row before
#pragma unroll
    for (int t = 0; t < kMeanStages - 1; ++t) copy(t);   // (empty past the row's end)
    float acc = 0.f;
    for (int32_t t = 0; t < tiles; ++t) {
      asm volatile("cp.async.wait_group %0;" ::"n"(kMeanStages - 2) : "memory");
      __syncthreads();   // tile t is there, tile t - 1 has been added
      copy(t + kMeanStages - 1);
      if (w == 0) {
        const float (*x)[32] = tile[t % kMeanStages];
        const int32_t cnt = min(kMeanTile, e - b - t * kMeanTile);
        int32_t j = 0;
        for (; j + 16 <= cnt; j += 16) {
          float y[16];
#pragma unroll
          for (int u = 0; u < 16; ++u) y[u] = x[j + u][lane];
#pragma unroll
          for (int u = 0; u < 16; ++u) acc = __fadd_rn(acc, y[u]);
        }
        for (; j < cnt; ++j) acc = __fadd_rn(acc, x[j][lane]);
      }
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    if (w == 0 && col < k) out[(size_t)r * k + col] = __fdiv_rn(acc, (float)(e - b));
  }
}

// A warp's 32 rows, 32 dimensions at a time through shared memory: lane l of
// row r's load reads dimension t + l (one 128-byte access per row), then lane
// r has row r's dimensions to itself, in order. A lane reading its own row in
// global memory touches 32 lines per load: the cosines of 2.6M incidences
// (k = 32) took 305 us so.
constexpr int kTileWarps = 8;

__device__ __forceinline__ void load_row_tile(float (*tile)[33], const float* __restrict__ F,
                                              int32_t row, int32_t k, int32_t t) {
  const int lane = threadIdx.x & 31;
  __syncwarp();
#pragma unroll 8
  for (int r = 0; r < 32; ++r) {
    const int32_t x = __shfl_sync(FULL, row, r);
    tile[r][lane] = (x >= 0 && t + lane < k) ? F[(size_t)x * k + t + lane] : 0.f;
  }
  __syncwarp();
}

// |F[r]| = sqrt(sum_i F[r,i] * F[r,i]), squares added in dimension order.
__global__ void __launch_bounds__(32 * kTileWarps)
row_norm_kernel(int32_t rows, int32_t k, const float* __restrict__ F, float* __restrict__ out) {
  __shared__ float tiles[kTileWarps][32][33];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int64_t warps = (int64_t)gridDim.x * kTileWarps;
  for (int64_t r0 = ((int64_t)blockIdx.x * kTileWarps + w) * 32; r0 < rows; r0 += warps * 32) {
    const int32_t r = r0 + lane < rows ? (int32_t)(r0 + lane) : -1;
    float acc = 0.f;
    for (int32_t t = 0; t < k; t += 32) {
      load_row_tile(tiles[w], F, r, k, t);
      const int32_t cnt = min(32, k - t);
      for (int32_t i = 0; i < cnt; ++i) {
        const float x = tiles[w][lane][i];
        acc = __fadd_rn(acc, __fmul_rn(x, x));
      }
    }
    if (r >= 0) out[r] = __fsqrt_rn(acc);
  }
}

// node_of[j] = the node of CSC entry j.
__global__ void __launch_bounds__(kEntryThreads)
node_of_kernel(int32_t n, int64_t nnz, const int32_t* __restrict__ v_ptr,
               int32_t* __restrict__ node_of) {
  csr_entries_visit(n, v_ptr, nnz, [&](int64_t v, int64_t j) { node_of[j] = (int32_t)v; });
}

// score[j] = cos(f(e), f(v)) for CSC entry j = (v, e): f(e).f(v) with the
// products added in dimension order, over |f(e)| |f(v)|; 0 where that
// product is 0 (an undefined cosine). (Neighbouring entries mostly share v,
// so its values come as broadcasts.)
__global__ void __launch_bounds__(32 * kTileWarps)
cosine_score_kernel(int64_t nnz, int32_t k, const int32_t* __restrict__ node_of,
                    const int32_t* __restrict__ v_edges, const float* __restrict__ X,
                    const float* __restrict__ FE, const float* __restrict__ nv,
                    const float* __restrict__ ne, float* __restrict__ score) {
  __shared__ float tiles[kTileWarps][32][33];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int64_t warps = (int64_t)gridDim.x * kTileWarps;
  for (int64_t j0 = ((int64_t)blockIdx.x * kTileWarps + w) * 32; j0 < nnz; j0 += warps * 32) {
    const int64_t j = j0 + lane;
    const bool on = j < nnz;
    const int32_t v = on ? node_of[j] : 0, e = on ? v_edges[j] : -1;
    const float* fv = X + (size_t)v * k;
    const float den = on ? __fmul_rn(ne[e], nv[v]) : 0.f;
    float dot = 0.f;
    for (int32_t t = 0; t < k; t += 32) {
      load_row_tile(tiles[w], FE, e, k, t);
      const int32_t cnt = min(32, k - t);
      int32_t i = 0;
      for (; i + 8 <= cnt; i += 8) {
        float y[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) y[u] = fv[t + i + u];
#pragma unroll
        for (int u = 0; u < 8; ++u)
          dot = __fadd_rn(dot, __fmul_rn(tiles[w][lane][i + u], y[u]));
      }
      for (; i < cnt; ++i) dot = __fadd_rn(dot, __fmul_rn(tiles[w][lane][i], fv[t + i]));
    }
    if (on) score[j] = (den > 0.f) ? __fdiv_rn(dot, den) : 0.f;
  }
}

// Means of the listed rows of X (both kernels).
int segment_means(int32_t rows, int64_t entries, int32_t k, const int32_t* ptr, const int32_t* idx,
                  const float* X, float* out, TempPool& pool, cudaStream_t s) {
  int32_t *long_rows = nullptr, *n_long = nullptr;
  HNV_CHECK(pool.get(&long_rows, (size_t)(entries / kMeanLong + 1)));
  HNV_CHECK(pool.get(&n_long, 1));
  HNV_CUDA(cudaMemsetAsync(n_long, 0, sizeof(int32_t), s));
  HNV_CHECK(launch("segment_mean", segment_mean_kernel, grid_for((int64_t)rows * k, 256, 16), 256,
                   0, s, rows, k, ptr, idx, X, out, long_rows, n_long));
  if (entries <= kMeanLong) return HNV_OK;
  return launch("segment_mean_long", segment_mean_long_kernel, (unsigned)(6 * num_sms()),
                kMeanThreads, 0, s, k, ptr, idx, X, out, (const int32_t*)long_rows,
                (const int32_t*)n_long);
}

// G lanes per node. long_rows: [0, cap) the rows longer than G * 32, from the
// front; [cap, 2 cap) those longer than kHubRow; counts in n_long[0], n_long[1].
template <int G>
__global__ void assign_kernel(int32_t n, const int32_t* __restrict__ v_ptr,
                              const int32_t* __restrict__ v_edges,
                              const uint64_t* __restrict__ prio, const float* __restrict__ score,
                              int32_t* __restrict__ c, int32_t* __restrict__ long_rows, int64_t cap,
                              int32_t* __restrict__ n_long) {
  const int lg = threadIdx.x & (G - 1);
  const unsigned mask = G == 32 ? FULL : ((1u << (G & 31)) - 1u) << (threadIdx.x & 31 & ~(G - 1));
  const int64_t groups = (int64_t)gridDim.x * (blockDim.x / G);
  for (int64_t v = (int64_t)blockIdx.x * (blockDim.x / G) + threadIdx.x / G; v < n; v += groups) {
    const int64_t b = v_ptr[v], end = v_ptr[v + 1];
    if (end - b > G * 32) {
      const int hub = end - b > kHubRow ? 1 : 0;
      if (lg == 0) long_rows[hub * cap + atomicAdd(n_long + hub, 1)] = (int32_t)v;
      continue;
    }
    float bs = -INFINITY;
    uint64_t bp = ~0ull;
    int32_t be = 0x7fffffff;
    for (int64_t k = b + lg; k < end; k += G) {
      const int32_t e = v_edges[k];
      lex_min(bs, bp, be, score ? score[k] : 0.f, prio[e], e);
    }
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) {
      const float os = score ? __shfl_xor_sync(mask, bs, o) : bs;
      const uint64_t op = __shfl_xor_sync(mask, bp, o);
      const int32_t oe = __shfl_xor_sync(mask, be, o);
      lex_min(bs, bp, be, score ? os : bs, op, oe);
    }
    if (lg == 0) c[v] = (end > b) ? be : -1;
  }
}

struct Best {
  float s;
  int32_t e;
  uint64_t p;
};

// Tasks of PARTS parts per listed row; a part's best goes to c (PARTS = 1) or
// to parts.
template <int PARTS>
__global__ void __launch_bounds__(kLongThreads)
assign_long_kernel(const int32_t* __restrict__ long_rows, const int32_t* __restrict__ n_long,
                   const int32_t* __restrict__ v_ptr, const int32_t* __restrict__ v_edges,
                   const uint64_t* __restrict__ prio, const float* __restrict__ score,
                   int32_t* __restrict__ c, Best* __restrict__ parts) {
  __shared__ float ss[kLongThreads / 32];
  __shared__ uint64_t sp[kLongThreads / 32];
  __shared__ int32_t se[kLongThreads / 32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int64_t count = (int64_t)*n_long * PARTS;
  for (int64_t i = blockIdx.x; i < count; i += gridDim.x) {
    const int32_t v = long_rows[i / PARTS];
    const int64_t rb = v_ptr[v], len = v_ptr[v + 1] - rb;
    const int64_t b = rb + len * (i % PARTS) / PARTS, end = rb + len * (i % PARTS + 1) / PARTS;
    float bs = -INFINITY;
    uint64_t bp = ~0ull;
    int32_t be = 0x7fffffff;
    // four incidences per step keep four independent load chains in flight
    // (the minimum of a total order does not depend on the visiting order)
    int64_t k = b + threadIdx.x;
    for (; k + 3 * kLongThreads < end; k += 4 * kLongThreads) {
      int32_t e[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) e[u] = v_edges[k + u * kLongThreads];
      uint64_t pr[4];
      float sc[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        pr[u] = prio[e[u]];
        sc[u] = score ? score[k + u * kLongThreads] : 0.f;
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) lex_min(bs, bp, be, sc[u], pr[u], e[u]);
    }
    for (; k < end; k += kLongThreads) {
      const int32_t e = v_edges[k];
      lex_min(bs, bp, be, score ? score[k] : 0.f, prio[e], e);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const float os = __shfl_xor_sync(FULL, bs, o);
      const uint64_t op = __shfl_xor_sync(FULL, bp, o);
      const int32_t oe = __shfl_xor_sync(FULL, be, o);
      lex_min(bs, bp, be, os, op, oe);
    }
    if (lane == 0) {
      ss[w] = bs;
      sp[w] = bp;
      se[w] = be;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      for (int q = 1; q < kLongThreads / 32; ++q) lex_min(bs, bp, be, ss[q], sp[q], se[q]);
      if (PARTS == 1) c[v] = be;
      else parts[i] = Best{bs, be, bp};
    }
    __syncthreads();
  }
}

// The best of every hub row's parts (a warp per row).
__global__ void assign_hub_kernel(const int32_t* __restrict__ hub_rows,
                                  const int32_t* __restrict__ n_hub,
                                  const Best* __restrict__ parts, int32_t* __restrict__ c) {
  const int lane = threadIdx.x & 31;
  const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
  for (int64_t i = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); i < *n_hub;
       i += warps) {
    float bs = -INFINITY;
    uint64_t bp = ~0ull;
    int32_t be = 0x7fffffff;
    for (int q = lane; q < kHubParts; q += 32) {
      const Best x = parts[i * kHubParts + q];
      lex_min(bs, bp, be, x.s, x.p, x.e);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const float os = __shfl_xor_sync(FULL, bs, o);
      const uint64_t op = __shfl_xor_sync(FULL, bp, o);
      const int32_t oe = __shfl_xor_sync(FULL, be, o);
      lex_min(bs, bp, be, os, op, oe);
    }
    if (lane == 0) c[hub_rows[i]] = be;
  }
}

__global__ void iota_kernel(int64_t n, int32_t* __restrict__ out) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    out[i] = (int32_t)i;
}

// key(v) = c(v) or m + v; flags[key] = 1 (all writers store the same value).
__global__ void mark_keys_kernel(int32_t n, int32_t m, const int32_t* __restrict__ c,
                                 int32_t* __restrict__ flags) {
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n;
       v += (int64_t)gridDim.x * blockDim.x) {
    const int32_t cv = c[v];
    flags[cv >= 0 ? (int64_t)cv : (int64_t)m + v] = 1;
  }
}

__global__ void rep_v_kernel(int32_t n, int32_t m, const int32_t* __restrict__ c,
                             const int32_t* __restrict__ rank, int32_t* __restrict__ rep_v) {
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n;
       v += (int64_t)gridDim.x * blockDim.x) {
    const int32_t cv = c[v];
    rep_v[v] = rank[cv >= 0 ? (int64_t)cv : (int64_t)m + v];
  }
}

// key = (e << 32) | rep_v[member].
__global__ void __launch_bounds__(kEntryThreads)
pack_image_keys(int32_t m, int64_t nnz, const int32_t* __restrict__ e_ptr,
                const int32_t* __restrict__ e_nodes, const int32_t* __restrict__ rep_v,
                uint64_t* __restrict__ keys) {
  csr_entries_visit(m, e_ptr, nnz, [&](int64_t e, int64_t k) {
    keys[k] = ((uint64_t)(uint32_t)e << 32) | (uint32_t)rep_v[e_nodes[k]];
  });
}

__global__ void max_row_len(int32_t rows, const int32_t* __restrict__ ptr, int32_t* __restrict__ out) {
  int32_t mx = 0;
  for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < rows;
       r += (int64_t)gridDim.x * blockDim.x)
    mx = max(mx, ptr[r + 1] - ptr[r]);
  for (int o = 16; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(FULL, mx, o));
  if ((threadIdx.x & 31) == 0 && mx) atomicMax(out, mx);
}

// keep[e] = 1 if e's image has at least 2 coarse nodes.
__global__ void keep_kernel(int32_t m, const int32_t* __restrict__ img_ptr,
                            int32_t* __restrict__ keep) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < m;
       e += (int64_t)gridDim.x * blockDim.x)
    keep[e] = img_ptr[e + 1] - img_ptr[e] >= 2 ? 1 : 0;
}

// Per fine hyperedge: survivors get their new ID in rep_e and carry their
// weight and level-0 ID to the coarse level; removed ones (images of one
// node c) record -1 - c. A removed hyperedge has one image entry, so a
// survivor's entries move down by the number of removed ones before it.
__global__ void survivor_rows(int32_t m, int32_t m2, int32_t nnz2,
                              const int32_t* __restrict__ img_ptr,
                              const int32_t* __restrict__ img_nodes,
                              const int32_t* __restrict__ new_id, const float* __restrict__ w,
                              const int32_t* __restrict__ orig_e, int32_t* __restrict__ rep_e,
                              int32_t* __restrict__ e_ptr2, float* __restrict__ w2,
                              int32_t* __restrict__ orig2) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < m;
       e += (int64_t)gridDim.x * blockDim.x) {
    if (e == 0) e_ptr2[m2] = nnz2;
    const int32_t b = img_ptr[e];
    if (img_ptr[e + 1] - b < 2) {
      rep_e[e] = -1 - img_nodes[b];
      continue;
    }
    const int32_t r = new_id[e];
    rep_e[e] = r;
    e_ptr2[r] = b - ((int32_t)e - r);
    w2[r] = w[e];
    orig2[r] = orig_e[e];
  }
}

__global__ void __launch_bounds__(kEntryThreads)
survivor_nodes(int32_t m, int64_t nnz_img, const int32_t* __restrict__ img_ptr,
               const int32_t* __restrict__ img_nodes, const int32_t* __restrict__ rep_e,
               int32_t* __restrict__ e_nodes2) {
  csr_entries_visit(m, img_ptr, nnz_img, [&](int64_t e, int64_t k) {
    const int32_t r = rep_e[e];
    if (r >= 0) e_nodes2[k - (e - r)] = img_nodes[k];
  });
}

}  // namespace

int coarsen_step(hnv_graph* g, int level, const hnv_coarsen_params* p,
                 const uint64_t* d_explicit, Level* fine, Level* coarse) {
  NvtxRange nvtx("hnv coarsen level %d", level);
  cudaStream_t s = g->stream;
  const int32_t n = fine->n, m = fine->m;
  const int64_t nnz = fine->nnz;
  TempPool pool(s);

  // 1. AssignHyperedge for every node
  uint64_t* prio = nullptr;
  int32_t* c = nullptr;
  HNV_CHECK(pool.get(&prio, (size_t)m));
  HNV_CHECK(pool.get(&c, (size_t)n));
  const uint64_t salt = mix64(p->seed + (uint64_t)level * kGamma);
  HNV_CHECK(launch("priority", priority_kernel, grid_for(m, 256), 256, 0, s, m, p->policy, salt,
                   (const int32_t*)fine->e_ptr, (const float*)fine->w,
                   (const int32_t*)fine->orig_e, d_explicit, prio));
  // the feature rule: a cosine per CSC entry
  float* score = nullptr;
  const int32_t k = fine->feat_k;
  if (p->policy == HNV_ASSIGN_COSINE) {
    if (!fine->feat || k < 1) HNV_FAIL(HNV_ERR_STATE, "level %d has no node features", level);
    float *fe = nullptr, *nv = nullptr, *ne = nullptr;
    int32_t* node_of = nullptr;
    HNV_CHECK(pool.get(&fe, (size_t)m * k));
    HNV_CHECK(pool.get(&nv, (size_t)n));
    HNV_CHECK(pool.get(&ne, (size_t)m));
    HNV_CHECK(pool.get(&node_of, (size_t)nnz));
    HNV_CHECK(pool.get(&score, (size_t)nnz));
    HNV_CHECK(segment_means(m, nnz, k, fine->e_ptr, fine->e_nodes, fine->feat, fe, pool, s));
    HNV_CHECK(launch("node_norms", row_norm_kernel, grid_for(n, 32 * kTileWarps), 32 * kTileWarps,
                     0, s, n, k, (const float*)fine->feat, nv));
    HNV_CHECK(launch("edge_norms", row_norm_kernel, grid_for(m, 32 * kTileWarps), 32 * kTileWarps,
                     0, s, m, k, (const float*)fe, ne));
    HNV_CHECK(launch("node_of", node_of_kernel, entry_grid(nnz), kEntryThreads, 0, s, n, nnz,
                     (const int32_t*)fine->v_ptr, node_of));
    HNV_CHECK(launch("cosine_score", cosine_score_kernel, grid_for(nnz, 32 * kTileWarps, 32),
                     32 * kTileWarps, 0, s, nnz, k, (const int32_t*)node_of,
                     (const int32_t*)fine->v_edges, (const float*)fine->feat, (const float*)fe,
                     (const float*)nv, (const float*)ne, score));
  }
  int32_t *long_rows = nullptr, *n_long = nullptr;
  const bool few = nnz <= 24 * (int64_t)n;
  const int64_t cap = nnz / (few ? 256 : 1024) + 1;
  HNV_CHECK(pool.get(&long_rows, 2 * (size_t)cap));
  HNV_CHECK(pool.get(&n_long, 2));
  HNV_CUDA(cudaMemsetAsync(n_long, 0, 2 * sizeof(int32_t), s));
  HNV_CHECK(launch("assign", few ? assign_kernel<8> : assign_kernel<32>,
                   grid_for((int64_t)n * (few ? 8 : 32), 256, 16), 256, 0, s, n,
                   (const int32_t*)fine->v_ptr, (const int32_t*)fine->v_edges,
                   (const uint64_t*)prio, (const float*)score, c, long_rows, cap, n_long));
  if (nnz > (few ? 256 : 1024))
    HNV_CHECK(launch("assign_long", assign_long_kernel<1>, (unsigned)(4 * num_sms()), kLongThreads,
                     0, s, (const int32_t*)long_rows, (const int32_t*)n_long,
                     (const int32_t*)fine->v_ptr, (const int32_t*)fine->v_edges,
                     (const uint64_t*)prio, (const float*)score, c, (Best*)nullptr));
  if (nnz > kHubRow) {
    Best* parts = nullptr;
    HNV_CHECK(pool.get(&parts, (size_t)(nnz / kHubRow + 1) * kHubParts));
    HNV_CHECK(launch("assign_hub_parts", assign_long_kernel<kHubParts>, (unsigned)(4 * num_sms()),
                     kLongThreads, 0, s, (const int32_t*)(long_rows + cap),
                     (const int32_t*)(n_long + 1), (const int32_t*)fine->v_ptr,
                     (const int32_t*)fine->v_edges, (const uint64_t*)prio, (const float*)score, c,
                     parts));
    HNV_CHECK(launch("assign_hub", assign_hub_kernel, 8, 256, 0, s,
                     (const int32_t*)(long_rows + cap), (const int32_t*)(n_long + 1),
                     (const Best*)parts, c));
  }

  // 2. Merge: coarse IDs are the ranks of the keys c(v) / m + v
  int32_t* rank = nullptr;
  const int64_t nkeys = (int64_t)m + n;
  HNV_CHECK(pool.get(&rank, (size_t)nkeys));
  HNV_CUDA(cudaMemsetAsync(rank, 0, sizeof(int32_t) * nkeys, s));
  HNV_CHECK(launch("mark_keys", mark_keys_kernel, grid_for(n, 256), 256, 0, s, n, m,
                   (const int32_t*)c, rank));
  HNV_CHECK(exclusive_scan_i32(rank, rank, nkeys, g->d_buf, s));
  HNV_CUDA(cudaMemsetAsync(g->d_buf + 1, 0, sizeof(int32_t), s));
  HNV_CHECK(launch("max_row_len", max_row_len, grid_for(m, 256), 256, 0, s, m,
                   (const int32_t*)fine->e_ptr, g->d_buf + 1));
  int32_t nm[2];
  HNV_CHECK(read_ints(g, g->d_buf, 2, nm, s));
  const int32_t n2 = nm[0], max_e_len = nm[1];
  HNV_CHECK(level_alloc(fine, (void**)&fine->rep_v, sizeof(int32_t) * (size_t)n, s));
  HNV_CHECK(level_alloc(fine, (void**)&fine->rep_e, sizeof(int32_t) * (size_t)m, s));
  HNV_CHECK(launch("rep_v", rep_v_kernel, grid_for(n, 256), 256, 0, s, n, m, (const int32_t*)c,
                   (const int32_t*)rank, fine->rep_v));

  // 3. Images of the hyperedges: sorted distinct rep_v of the members
  uint64_t *k0 = nullptr, *k1 = nullptr, *sorted = nullptr;
  int32_t *tiles = nullptr, *img_ptr = nullptr, *img_nodes = nullptr, *new_id = nullptr;
  HNV_CHECK(pool.get(&k0, (size_t)nnz));
  HNV_CHECK(launch("pack_image_keys", pack_image_keys, entry_grid(nnz), kEntryThreads, 0, s, m,
                   nnz, (const int32_t*)fine->e_ptr, (const int32_t*)fine->e_nodes,
                   (const int32_t*)fine->rep_v, k0));
  // the keys were packed hyperedge by hyperedge: sorting every hyperedge's
  // run by its low word gives what a full sort by (e, rep) would
  if (max_e_len <= kSegSortMax) {
    HNV_CHECK(segmented_sort_low32(m, fine->e_ptr, (const int64_t*)nullptr, max_e_len, nnz, k0, s,
                                   (uint32_t)n2));
    sorted = k0;
  } else {
    int shifts[16];
    const int np = radix_shifts(bits_for_count(n2), bits_for_count(m), shifts);
    HNV_CHECK(pool.get(&k1, (size_t)nnz));
    HNV_CHECK(radix_sort_u64(k0, k1, nnz, shifts, np, s, &sorted));
  }
  HNV_CHECK(pool.get(&tiles, (size_t)compact_tiles(nnz)));
  HNV_CHECK(pool.get(&img_ptr, (size_t)m + 1));
  HNV_CHECK(pool.get(&img_nodes, (size_t)nnz));
  HNV_CHECK(pool.get(&new_id, (size_t)m + 1));
  HNV_CHECK(unique_count(sorted, nnz, tiles, g->d_buf, s));
  HNV_CHECK(unique_csr(sorted, nnz, tiles, img_nodes, img_ptr, s));
  HNV_CUDA(cudaMemcpyAsync(img_ptr + m, g->d_buf, sizeof(int32_t), cudaMemcpyDeviceToDevice, s));

  // 4. addHedge: survivors have >= 2 distinct coarse members
  HNV_CHECK(launch("keep", keep_kernel, grid_for(m, 256), 256, 0, s, m, (const int32_t*)img_ptr,
                   new_id));
  HNV_CHECK(exclusive_scan_i32(new_id, new_id, m, g->d_buf + 1, s));
  int32_t h[2];
  HNV_CHECK(read_ints(g, g->d_buf, 2, h, s));
  const int32_t nnz_img = h[0];
  const int32_t m2 = h[1];
  const int32_t nnz2 = nnz_img - (m - m2);

  // 5. addNode/addEdge: the coarse level's CSR, weights and level-0 IDs
  *coarse = Level();
  coarse->n = n2;
  coarse->m = m2;
  coarse->nnz = nnz2;
  HNV_CHECK(level_alloc(coarse, (void**)&coarse->e_ptr, sizeof(int32_t) * ((size_t)m2 + 1), s));
  HNV_CHECK(level_alloc(coarse, (void**)&coarse->e_nodes, sizeof(int32_t) * (size_t)nnz2, s));
  HNV_CHECK(level_alloc(coarse, (void**)&coarse->w, sizeof(float) * (size_t)m2, s));
  HNV_CHECK(level_alloc(coarse, (void**)&coarse->orig_e, sizeof(int32_t) * (size_t)m2, s));
  HNV_CHECK(launch("survivor_rows", survivor_rows, grid_for(m, 256), 256, 0, s, m, m2, nnz2,
                   (const int32_t*)img_ptr, (const int32_t*)img_nodes, (const int32_t*)new_id,
                   (const float*)fine->w, (const int32_t*)fine->orig_e, fine->rep_e,
                   coarse->e_ptr, coarse->w, coarse->orig_e));
  HNV_CHECK(launch("survivor_nodes", survivor_nodes, entry_grid(nnz_img), kEntryThreads, 0, s, m,
                   (int64_t)nnz_img, (const int32_t*)img_ptr, (const int32_t*)img_nodes,
                   (const int32_t*)fine->rep_e, coarse->e_nodes));

  // 6. The coarse node features (feature rule): the mean of the merged
  // nodes' features, in ascending fine-node order (the CSC of rep_v).
  if (p->policy == HNV_ASSIGN_COSINE) {
    int32_t *iota = nullptr, *ch_ptr = nullptr, *ch_idx = nullptr;
    HNV_CHECK(pool.get(&iota, (size_t)n + 1));
    HNV_CHECK(pool.get(&ch_ptr, (size_t)n2 + 1));
    HNV_CHECK(pool.get(&ch_idx, (size_t)n));
    HNV_CHECK(launch("iota", iota_kernel, grid_for((int64_t)n + 1, 256), 256, 0, s, n + 1, iota));
    HNV_CHECK(transpose_csr(n, n2, n, iota, fine->rep_v, ch_ptr, ch_idx, s));
    HNV_CHECK(level_alloc(coarse, (void**)&coarse->feat, sizeof(float) * (size_t)n2 * k, s));
    coarse->feat_k = k;
    HNV_CHECK(segment_means(n2, n, k, ch_ptr, ch_idx, fine->feat, coarse->feat, pool, s));
  }
  return HNV_OK;
}

}  // namespace hnv
