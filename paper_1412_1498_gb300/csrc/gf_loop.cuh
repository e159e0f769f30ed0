// gf_loop.cuh -- the sweep loop of a small handle in one kernel.
//
// A sweep of a handle with many units is five launches (the time slices of a Coulomb lattice, a
// batch), and on up to kLoopSites sites each of them takes little longer than it costs to end
// one kernel and start the next.  Here every block stays for the whole loop, barriers over the
// grid take the place of the launches, the blocks take the decisions of the loop themselves,
// and the even-site pass is left out where no unit needs it.  One launch serves up to
// kLoopSweeps sweeps.
//
// The kernel is launched cooperatively, so all blocks are resident and the barrier ends.  Its
// wait is bounded all the same (LoopArgs.polls): a block that gives up sets DevState.fault and
// leaves, the others follow, and the host reports an error.
//
// A sweep: even half-sweep | odd half-sweep, with F and the odd-site theta per tile | the
// totals of each unit by one block and the decisions of FINISH_ODD | where some unit is
// undecided, and on the last sweep of the budget: the even-site theta pass over those units'
// tiles | their totals and FINISH_LOOP's decisions |.  "|" is a barrier (about 2.5 us on this
// GPU: the fence, the arrival and a poll are round trips to L2 each).  Per-site arithmetic, tile
// sums and the order of the totals are those of the kernels for other handles: the same bits.
// Links are read past L1, which other SMs' stores do not reach.  Only the first-order form of the
// overrelaxation runs here: nvcc contracts the exact form's products otherwise than in the
// sweep kernels, and the links would not be the same bits.
//
// Coulomb gauge, us a sweep, launches (blocks of 64 sites) -> this kernel: FP32-12 8^3x16 22.7 -> 14.8,
// 12^3x16 22.9 -> 15.5, 16^4 24.4 -> 17.9, 16^3x32 33.5 -> 26.0 (above that the pipelined kernels'
// bandwidth counts for more); FP32-18 23.5 -> 16.8, 23.6 -> 18.1, 26.7 -> 20.0, 38.9 -> 30.4.  A
// one-unit handle has three launches a sweep and gained nothing (8^4 12.2 against 12.7,
// 16^4 16.9 against 16.9), nor did a warp per direction here (8^4 11.5, 16^4 23.1): it keeps its
// launches.  Loops of several handles on streams of their own run side by side as far as their
// blocks fit the GPU together, and one after another beyond that, where launched loops share it: us a
// sweep over 1, 2, 4, 8 handles together, launches -> this kernel, 8^3x16 23.6 14.0 7.1 4.5 -> 15.6
// 8.5 4.6 3.6; 12^3x16 24.5 13.3 7.3 5.1 -> 15.6 8.5 8.5 8.6; 16^3x32 36.1 23.1 19.7 21.0 -> 26.2 25.7
// 26.0 26.0.  Such callers batch the lattices in one handle or take a block size of 64.
#pragma once

#include "gf_kernels.cuh"

namespace gf {

constexpr int kLoopThreads = 128;            // sites per tile
constexpr int kLoopUnits = 128;              // most convergence units of such a handle
constexpr long long kLoopSites = 1LL << 17;  // most sites
constexpr int kLoopSweeps = 4096;            // most sweeps of one launch

struct LoopArgs {
  char* links;
  const LatDev* lats;
  const int4* tiles;
  const int* unit_tiles;   // n_units + 1
  const double* unit_norm;
  int* active;
  int* iters;
  float2* part_F;
  float2* part_th_even;
  float2* part_th_odd;
  int* verdict;            // per unit, between blocks: 1 undecided by the odd part, 2 done, else 0
  double* unit_sumF;
  double* unit_sumTh;
  double* unit_sumTh_odd;
  double* unit_F;
  double* unit_theta;
  double* lat_F;
  double* lat_theta;
  DevState* st;
  int n_tiles, n_units, n_lat, nd;
  unsigned polls;          // most polls of one barrier wait
  Relax omega;
};

// Barrier over the grid: `target` arrivals since the launch (a multiple of the grid size).
// false: some block gave up.
__device__ __forceinline__ bool loop_barrier(DevState* st, unsigned target, unsigned polls, int* s_ok) {
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(&st->arrived, 1u);
    int ok = 1;
    for (unsigned spins = 0;; ++spins) {
      if (spins >= polls) {
        atomicExch(&st->fault, 1);
        ok = 0;
        break;
      }
      unsigned n;
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];\n" : "=r"(n) : "l"(&st->arrived) : "memory");
      if (n >= target) break;
    }
    __threadfence();
    *s_ok = ok && *(volatile int*)&st->fault == 0;
  }
  __syncthreads();
  return *s_ok != 0;
}

template <int S>
struct LoopStore;
template <>
struct LoopStore<GF_FP32_12> {
  __device__ static __forceinline__ void load(const char* base, long long V, int mu, int idx, cx<float> (&e)[6]) {
    const float4* p = reinterpret_cast<const float4*>(base);
#pragma unroll
    for (int w = 0; w < 3; ++w) {
      const float4 v = __ldcg(p + (long long)(w * 4 + mu) * V + idx);
      e[2 * w] = {v.x, v.y};
      e[2 * w + 1] = {v.z, v.w};
    }
  }
};
template <>
struct LoopStore<GF_FP32_18> {
  __device__ static __forceinline__ void load(const char* base, long long V, int mu, int idx, cx<float> (&e)[9]) {
    const float4* p = reinterpret_cast<const float4*>(base);
#pragma unroll
    for (int w = 0; w < 4; ++w) {
      const float4 v = __ldcg(p + (long long)(w * 4 + mu) * V + idx);
      e[2 * w] = {v.x, v.y};
      e[2 * w + 1] = {v.z, v.w};
    }
    const float2 v = __ldcg(reinterpret_cast<const float2*>(base + 256LL * V) + (long long)mu * V + idx);
    e[8] = {v.x, v.y};
  }
};

struct LoopSite {
  int idx_f, idx_b[4];
};
__device__ __forceinline__ LoopSite loop_site(const LatDev& lat, int parity, int t, int h3) {
  LoopSite r;
  const Site s = site_of_slice(lat, parity, t, h3);
  r.idx_f = parity * lat.Vh + t * lat.V3h + h3;
#pragma unroll
  for (int mu = 0; mu < 4; ++mu) r.idx_b[mu] = (1 - parity) * lat.Vh + (int)(back_lexi(lat, s, mu) >> 1);
  return r;
}

// The sum of a unit's tile partials by one block, in k_finish's order: virtual thread v of 256
// adds tiles tb + v + 256 j (j < 16) as a binary tree, then a binary tree over the threads.
// Valid in thread 0.
template <int NV>
__device__ __forceinline__ void loop_unit_sum(const float2* const (&p)[NV], int tb, int te, double (&out)[NV],
                                              float2 (*red)[kFinishThreads]) {
  const int tid = (int)threadIdx.x;
#pragma unroll
  for (int k = 0; k < NV; ++k)
    for (int v = tid; v < kFinishThreads; v += kLoopThreads) {
      float2 acc = make_float2(0.f, 0.f);
      for (int i0 = tb + v; i0 < te; i0 += kFinishUnroll * kFinishThreads) {
        float2 x[kFinishUnroll];
#pragma unroll
        for (int j = 0; j < kFinishUnroll; ++j) {
          const int i = i0 + j * kFinishThreads;
          x[j] = i < te ? __ldcg(p[k] + i) : make_float2(0.f, 0.f);
        }
#pragma unroll
        for (int w = kFinishUnroll / 2; w > 0; w >>= 1)
#pragma unroll
          for (int j = 0; j < w; ++j) x[j] = pair_add(x[j], x[j + w]);
        acc = pair_add(acc, x[0]);
      }
      red[k][v] = acc;
    }
  __syncthreads();
#pragma unroll
  for (int w = kFinishThreads / 2; w >= 32; w >>= 1) {
#pragma unroll
    for (int k = 0; k < NV; ++k)
      if (tid < w) red[k][tid] = pair_add(red[k][tid], red[k][tid + w]);
    __syncthreads();
  }
  if (tid < 32) {
#pragma unroll
    for (int k = 0; k < NV; ++k) {
      float2 x = red[k][tid];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1)
        x = pair_add(x, make_float2(__shfl_down_sync(0xffffffffu, x.x, o), __shfl_down_sync(0xffffffffu, x.y, o)));
      out[k] = pair_value(x);
    }
  }
  __syncthreads();
}

template <int S, int ND>
__global__ void __launch_bounds__(kLoopThreads, 2) k_loop(LoopArgs a) {
  using St = Store<S>;
  using Ld = LoopStore<S>;
  constexpr int NE = St::NE;
  __shared__ double red64[2][64];
  __shared__ float2 red[2][kFinishThreads];
  __shared__ int act[kLoopUnits], und[kLoopUnits];  // unit sweeps; unit undecided by its odd part
  __shared__ int done_sweeps[kLoopUnits];           // sweeps of each unit in this launch
  __shared__ int s_ok, s_count;
  const int tid = (int)threadIdx.x, G = (int)gridDim.x, blk = (int)blockIdx.x;
  const int sweep0 = a.st->sweep, limit = a.st->limit, ci = a.st->check_interval, ri = a.st->reunit_interval;
  const double eps = a.st->eps;
  int n_active = a.st->n_active;
  for (int u = tid; u < a.n_units; u += kLoopThreads) {
    act[u] = a.active[u] > 0;
    done_sweeps[u] = 0;
  }
  __syncthreads();
  unsigned target = 0;
  int rb = 0, sweep = sweep0;
#define BARRIER()                                             \
  do {                                                        \
    target += (unsigned)G;                                    \
    if (!loop_barrier(a.st, target, a.polls, &s_ok)) return;           \
  } while (0)
  while (n_active > 0 && sweep < limit && sweep - sweep0 < kLoopSweeps) {
    const bool check = ((sweep + 1) % ci) == 0 || sweep + 1 == limit;
    const bool forced = sweep + 1 == limit;
    const bool reunit_sweep = ri > 0 && ((sweep + 1) % ri) == 0;
#pragma unroll 1
    for (int parity = 0; parity < 2; ++parity) {
      const bool measure_now = parity == 1 && check, reunit_now = parity == 1 && reunit_sweep;
      for (int ti = blk; ti < a.n_tiles; ti += G) {
        const int4 tile = a.tiles[ti];
        if (!act[tile.w]) continue;
        const LatDev& lat = a.lats[tile.x];
        const int h3 = tile.z + tid;
        float v[2] = {0.f, 0.f};
        if (h3 < lat.V3h) {
          const LoopSite s = loop_site(lat, parity, tile.y, h3);
          char* base = a.links + lat.off_bytes;
          const long long V = lat.V;
          cx<float> K[9], Gx[9];
          cx<float> f[4][NE], b[4][NE];
#pragma unroll
          for (int mu = 0; mu < 4; ++mu) {
            Ld::load(base, V, mu, s.idx_f, f[mu]);
            Ld::load(base, V, mu, s.idx_b[mu], b[mu]);
          }
#pragma unroll
          for (int mu = 0; mu < ND; ++mu) add_to_K(K, f[mu], b[mu], mu == 0);
          su3_update<float, false, GF_OR_FIRST_ORDER>(K, Gx, a.omega, measure_now);
          if (measure_now) site_check_from_GK(K, v[0], v[1]);
#pragma unroll
          for (int mu = 0; mu < 4; ++mu) {
            left_mul<true>(Gx, f[mu]);
            right_mul_dag<true>(b[mu], Gx);
            if (reunit_now) {
              reunit<true>(f[mu]);
              reunit<true>(b[mu]);
            }
            St::store(base, V, mu, s.idx_f, f[mu]);
            St::store(base, V, mu, s.idx_b[mu], b[mu]);
          }
        }
        if (measure_now) {
          float2 o[2];
          block_sum_f32<2>(v, o, reinterpret_cast<float*>(red64[rb]));
          if (tid == 0) {
            a.part_F[ti] = o[0];
            a.part_th_odd[ti] = o[1];
          }
          rb ^= 1;  // (see k_or_sweep_pipe)
        }
      }
      BARRIER();
    }
    bool any = false;
    if (check) {
      for (int u = blk; u < a.n_units; u += G) {
        if (!act[u]) continue;
        const float2* const p[2] = {a.part_F, a.part_th_odd};
        double s[2];
        loop_unit_sum<2>(p, a.unit_tiles[u], a.unit_tiles[u + 1], s, red);
        if (tid == 0) {
          a.unit_sumF[u] = s[0];
          a.unit_F[u] = s[0] * a.unit_norm[2 * u];
          a.unit_sumTh_odd[u] = s[1];
          a.verdict[u] = forced || !(s[1] * a.unit_norm[2 * u + 1] >= eps);
        }
      }
      BARRIER();
      if (tid == 0) s_count = 0;
      __syncthreads();
      for (int u = tid; u < a.n_units; u += kLoopThreads) {
        und[u] = act[u] ? __ldcg(a.verdict + u) : 0;
        if (und[u]) s_count = 1;
      }
      __syncthreads();
      any = s_count != 0;
    }
    if (any) {
      // the even-site theta of the undecided units
      for (int ti = blk; ti < a.n_tiles; ti += G) {
        const int4 tile = a.tiles[ti];
        if (!act[tile.w] || !und[tile.w]) continue;
        const LatDev& lat = a.lats[tile.x];
        const int h3 = tile.z + tid;
        float v[1] = {0.f};
        if (h3 < lat.V3h) {
          const LoopSite s = loop_site(lat, 0, tile.y, h3);
          const char* base = a.links + lat.off_bytes;
          cx<float> A[9];
          cx<float> f[ND][NE], b[ND][NE];
          float fs = 0.f;
#pragma unroll
          for (int e = 0; e < 9; ++e) A[e] = {0.f, 0.f};
#pragma unroll
          for (int nu = 0; nu < ND; ++nu) {
            Ld::load(base, lat.V, nu, s.idx_f, f[nu]);
            Ld::load(base, lat.V, nu, s.idx_b[nu], b[nu]);
          }
#pragma unroll
          for (int nu = 0; nu < ND; ++nu) add_to_A_F(A, fs, f[nu], b[nu]);
          v[0] = theta_site(A);
        }
        float2 o[1];
        block_sum_f32<1>(v, o, reinterpret_cast<float*>(red64[rb]));
        if (tid == 0) a.part_th_even[ti] = o[0];
        rb ^= 1;
      }
      BARRIER();
      for (int u = blk; u < a.n_units; u += G) {
        if (!act[u] || !und[u]) continue;
        const float2* const p[1] = {a.part_th_even};
        double s[1];
        loop_unit_sum<1>(p, a.unit_tiles[u], a.unit_tiles[u + 1], s, red);
        if (tid == 0) {
          const double t = s[0] + __ldcg(a.unit_sumTh_odd + u), theta = t * a.unit_norm[2 * u + 1];
          a.verdict[u] = theta >= eps ? 0 : 2;
          a.unit_sumTh[u] = t;
          a.unit_theta[u] = theta;
        }
      }
      BARRIER();
      for (int u = tid; u < a.n_units; u += kLoopThreads)
        if (act[u] && und[u]) und[u] = __ldcg(a.verdict + u);
      __syncthreads();
    }
    // this sweep counts for every unit that was active; the done ones stop
    if (tid == 0) s_count = 0;
    __syncthreads();
    int n = 0;
    for (int u = tid; u < a.n_units; u += kLoopThreads) {
      if (!act[u]) continue;
      done_sweeps[u] += 1;
      if (any && und[u] == 2) act[u] = 0;
      n += act[u];
    }
    if (n) atomicAdd(&s_count, n);
    __syncthreads();
    n_active = s_count;
    ++sweep;
    __syncthreads();
  }
#undef BARRIER
  if (blk != 0) return;
  for (int u = tid; u < a.n_units; u += kLoopThreads) {
    a.active[u] = act[u];
    a.iters[u] += done_sweeps[u];
  }
  for (int l = tid; l < a.n_lat; l += kLoopThreads) {
    const LatDev& lat = a.lats[l];
    double sF = 0.0, sTh = 0.0;
    for (int k = 0; k < lat.n_units; ++k) {
      sF += __ldcg(a.unit_sumF + lat.unit0 + k);
      sTh += __ldcg(a.unit_sumTh + lat.unit0 + k);
    }
    a.lat_F[l] = sF * (1.0 / ((double)a.nd * 3.0 * (double)lat.V));
    a.lat_theta[l] = sTh * (1.0 / (3.0 * (double)lat.V));
  }
  if (tid == 0) {
    a.st->sweep = sweep;
    a.st->n_active = n_active;
  }
}

}  // namespace gf
