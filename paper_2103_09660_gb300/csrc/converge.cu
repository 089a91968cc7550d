// The stopping rule of Section 4's experiments (stop once two consecutive
// iterates differ by at most eps): refinement one sweep at a time, with the
// largest change of any coordinate read back after each sweep.
#include <cuda_bf16.h>

#include <cstring>
#include <utility>

#include "refine_device.cuh"

namespace hnv {

using dev::VecT;

namespace {

// out = max(out, max_i |a_i - b_i|) over `count` 16-byte vectors of T rows.
// The bit patterns of non-negative floats order like the floats, so the
// running maximum is an unsigned atomicMax (exact and order-independent).
template <typename T>
__global__ void max_abs_diff_kernel(int64_t count, const uint4* __restrict__ a,
                                    const uint4* __restrict__ b, unsigned* __restrict__ out) {
  using V = VecT<T>;
  constexpr int U = 4;   // pairs of vectors in flight per thread
  float mx = 0.f;
  const int64_t step = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += U * step) {
    uint4 x[U], y[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int64_t k = i + u * step < count ? i + u * step : i;
      x[u] = a[k];
      y[u] = b[k];
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      float fa[V::N], fb[V::N];
      V::unpack(x[u], fa);
      V::unpack(y[u], fb);
#pragma unroll
      for (int e = 0; e < V::N; ++e) mx = fmaxf(mx, fabsf(fa[e] - fb[e]));
    }
  }
  for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  if ((threadIdx.x & 31) == 0 && mx > 0.f) atomicMax(out, __float_as_uint(mx));
}

}  // namespace

int refine_level_until(hnv_graph* g, int level, void* z_v, void* z_e, int dtype, int d,
                       float omega, int max_sweeps, float eps, int mode, int32_t* sweeps_done,
                       float* last_delta, cudaStream_t s) {
  const Level& lv = g->levels[level];
  int32_t done = 0;
  float delta = 0.f;
  if (max_sweeps > 0 && team_enabled(d) && team_fits(lv, dtype, d) && team_ready(g)) {
    // sweeps, changes and the test in one launch (at most kTeamMaxSweeps each)
    const int32_t* result = nullptr;
    int32_t res[3] = {0, 0, 0};
    int rc = HNV_OK;
    do {
      TeamGraph t;
      t.top = t.bottom = level;
      t.zv0 = static_cast<uint4*>(z_v);
      t.ze0 = static_cast<uint4*>(z_e);
      const int k = max_sweeps - done < kTeamMaxSweeps ? max_sweeps - done : kTeamMaxSweeps;
      rc = team_run(g, t, dtype, d, omega, k, mode, s, &eps, &result);
      if (rc == kTeamRefused) break;
      HNV_CHECK(rc);
      HNV_CHECK(read_ints(g, result, 3, res, s));
      // in whichever sweep: the rows are then half-written
      if (res[2]) HNV_FAIL(HNV_ERR_TIMEOUT, "a bounded wait of a refinement kernel gave up");
      done += res[0];
      std::memcpy(&delta, &res[1], sizeof(float));
    } while (done < max_sweeps && !(delta <= eps));
    if (rc != kTeamRefused) {
      *sweeps_done = done;
      *last_delta = delta;
      return HNV_OK;
    }
  }
  const size_t rb = (dtype == HNV_BF16 ? 2 : 4) * (size_t)d;
  const int64_t vec_v = (int64_t)lv.n * (int64_t)(rb / 16), vec_e = (int64_t)lv.m * (int64_t)(rb / 16);
  TempPool pool(s);
  uint8_t *pv = nullptr, *pe = nullptr;
  HNV_CHECK(pool.get(&pv, (size_t)lv.n * rb));
  HNV_CHECK(pool.get(&pe, (size_t)lv.m * rb));
  unsigned* dmax = reinterpret_cast<unsigned*>(g->d_buf + 32);
  // Iterates alternate between the caller's buffers and these: a sweep writes
  // the other pair, so the previous iterate needs no copy (copying it took 30
  // of 330 us a sweep at 200K nodes, d = 64).
  void *cv = z_v, *ce = z_e, *ov = pv, *oe = pe;
  for (int it = done; it < max_sweeps; ++it) {
    HNV_CHECK(refine_sweep_into(g, level, cv, ce, ov, oe, dtype, d, omega, mode, s));
    std::swap(cv, ov);
    std::swap(ce, oe);
    HNV_CUDA(cudaMemsetAsync(dmax, 0, sizeof(unsigned), s));
    auto kern = dtype == HNV_BF16 ? max_abs_diff_kernel<__nv_bfloat16> : max_abs_diff_kernel<float>;
    HNV_CHECK(launch("max_abs_diff", kern, grid_for(vec_v, 1024), 256, 0, s, vec_v,
                     (const uint4*)cv, (const uint4*)ov, dmax));
    HNV_CHECK(launch("max_abs_diff", kern, grid_for(vec_e, 1024), 256, 0, s, vec_e,
                     (const uint4*)ce, (const uint4*)oe, dmax));
    int32_t bits = 0;
    HNV_CHECK(read_ints(g, reinterpret_cast<const int32_t*>(dmax), 1, &bits, s));
    std::memcpy(&delta, &bits, sizeof(float));
    done = it + 1;
    if (delta <= eps) break;
  }
  if (cv != z_v) {
    if (lv.n) HNV_CUDA(cudaMemcpyAsync(z_v, cv, (size_t)lv.n * rb, cudaMemcpyDeviceToDevice, s));
    if (lv.m) HNV_CUDA(cudaMemcpyAsync(z_e, ce, (size_t)lv.m * rb, cudaMemcpyDeviceToDevice, s));
  }
  *sweeps_done = done;
  *last_delta = delta;
  return HNV_OK;
}

}  // namespace hnv
