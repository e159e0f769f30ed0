// gf_sweep_dir.cuh -- half-sweep of a small lattice with one warp per direction.
//
// A lattice of a few thousand sites gives every SM a warp or two at most, and a half-sweep lasts
// as long as one thread takes to load a site's eight links, update them and store them.  Here
// a block of four warps updates 32 sites: warp mu holds U_mu(x) and U_mu(x - mu) of the 32 sites
// x, one site per lane.  Each warp forms its direction's share of K(x) and leaves it in shared
// memory; one warp adds the shares, runs the three subgroup steps and leaves g(x) there; each
// warp then applies g to the two links it still holds.  The warp that does the subgroup
// steps changes from block to block: warps of one number share a scheduler.
// The sums run in the order of the one-thread kernels: the same bits, in the links and in the
// check's F and theta of a site.
//
// us a sweep, one thread a site -> one warp a direction: Landau FP32-12 8^4 12.9 -> 9.9, 8x16x16x8
// (2^14 sites) 13.8 -> 11.2, 16^3x8 15.4 -> 14.0, 16^4 16.9 -> 21.9; FP32-18 8^4 14.0 -> 10.6,
// 2^14 sites 16.6 -> 11.8, 16^3x8 17.4 -> 15.4, 16^4 19.0 -> 23.8; FP64-18 8^4 94.8 -> 46.6, 2^14 sites
// 95.5 -> 73.4, 16^3x8 101 -> 115.  So the line is 2^14 sites.  Above it the SMs are full enough, and
// the barriers between the phases cost more than they give (24^4 FP32-18 66.7 -> 78.7).
#pragma once

#include "gf_kernels.cuh"

namespace gf {

constexpr int kDirThreads = 128;  // four directions x 32 sites

// where the links of a chunk's site live: forward at idx_f, backward at idx_b of the warp's
// direction
struct DirSite {
  int idx_f, idx_b;
};
__device__ __forceinline__ DirSite dir_site(const LatDev& lat, int parity, int t, int h3, int mu) {
  const Site s = site_of_slice(lat, parity, t, h3);
  return {parity * lat.Vh + t * lat.V3h + h3, (1 - parity) * lat.Vh + (int)(back_lexi(lat, s, mu) >> 1)};
}

template <int S>
constexpr int dir_min_blocks() {
  return sizeof(typename Store<S>::T) == 8 ? 2 : 4;
}

template <int S, int ND, int FORM>
__global__ void __launch_bounds__(kDirThreads, dir_min_blocks<S>()) k_or_sweep_dir(SweepArgs a) {
  using St = Store<S>;
  using T = typename St::T;
  constexpr int NE = St::NE;
  constexpr bool kCheckGK = sizeof(T) == 4;  // FP64 sums the stored links' A - A^dagger (Eq. (3))
  __shared__ T ks[4][18][32];                // K shares, later Delta shares of a check
  __shared__ T gs[18][32];
  __shared__ T fs4[4][32];
  grid_dep_wait();
  grid_dep_launch();
  bool reunit_now = a.reunit != 0, measure_now = a.measure != 0;
  if (a.st) {
    if (!state_sweeping(a.st)) return;
    reunit_now = a.parity == 1 && state_reunit_sweep(a.st);
    measure_now = a.parity == 1 && state_check_sweep(a.st);
  }
  const int ti = a.reverse ? a.n_tiles - 1 - (int)blockIdx.x : (int)blockIdx.x;
  const int4 tile = a.tiles[ti];
  if (a.active && a.active[tile.w] != a.level) return;
  const LatDev lat = a.lats[tile.x];
  const int mu = (int)threadIdx.x >> 5, lane = (int)threadIdx.x & 31;
  char* base = a.links + lat.off_bytes;
  const long long V = lat.V;
  const int turn = ti & 3;  // the warp of the subgroup steps
  const int h3 = tile.z + lane;
  const bool valid = h3 < lat.V3h;
  cx<T> f[NE], b[NE];
  DirSite ds{0, 0};
  if (valid) {
    ds = dir_site(lat, a.parity, tile.y, h3, mu);
    St::load(base, V, mu, ds.idx_f, f);
    St::load(base, V, mu, ds.idx_b, b);
    if (mu < ND) {
      cx<T> s[9];
      add_to_K(s, f, b, true);
#pragma unroll
      for (int e = 0; e < 9; ++e) {
        ks[mu][2 * e][lane] = s[e].re;
        ks[mu][2 * e + 1][lane] = s[e].im;
      }
    }
  }
  __syncthreads();
  T q = T(0), fs = T(0);
  if (mu == turn && valid) {
    cx<T> K[9], G[9];
#pragma unroll
    for (int e = 0; e < 9; ++e) K[e] = {ks[0][2 * e][lane], ks[0][2 * e + 1][lane]};
#pragma unroll
    for (int d = 1; d < ND; ++d)
#pragma unroll
      for (int e = 0; e < 9; ++e) K[e] = cadd(K[e], cx<T>{ks[d][2 * e][lane], ks[d][2 * e + 1][lane]});
    su3_update<T, false, FORM>(K, G, a.omega, kCheckGK && measure_now);
    if (kCheckGK && measure_now) site_check_from_GK(K, fs, q);
#pragma unroll
    for (int e = 0; e < 9; ++e) {
      gs[2 * e][lane] = G[e].re;
      gs[2 * e + 1][lane] = G[e].im;
    }
  }
  __syncthreads();
  if (valid) {
    cx<T> G[9];
#pragma unroll
    for (int e = 0; e < 9; ++e) G[e] = {gs[2 * e][lane], gs[2 * e + 1][lane]};
    left_mul<kPlain<T>>(G, f);
    right_mul_dag<kPlain<T>>(b, G);
    if (reunit_now) {
      reunit<kPlain<T>>(f);
      reunit<kPlain<T>>(b);
    }
    if (!kCheckGK && mu < ND && measure_now) {
      cx<T> fu[9], bu[9];
      to_full(f, fu);
      to_full(b, bu);
      AntiHermSum<T> D;
      D.add(fu, bu, true);
      const T d[9] = {D.d01.re, D.d01.im, D.d02.re, D.d02.im, D.d12.re, D.d12.im, D.e0, D.e1, D.e2};
#pragma unroll
      for (int e = 0; e < 9; ++e) ks[mu][e][lane] = d[e];
      fs4[mu][lane] = (fu[0].re + fu[4].re + fu[8].re) + (bu[0].re + bu[4].re + bu[8].re);
    }
    St::store(base, V, mu, ds.idx_f, f);
    St::store(base, V, mu, ds.idx_b, b);
  }
  if (!kCheckGK && measure_now) {
    __syncthreads();
    if (mu == turn && valid) {
      T s[9];
#pragma unroll
      for (int e = 0; e < 9; ++e) s[e] = ks[0][e][lane];
      fs = fs4[0][lane];
#pragma unroll
      for (int d = 1; d < ND; ++d) {
#pragma unroll
        for (int e = 0; e < 9; ++e) s[e] = s[e] + ks[d][e][lane];
        fs = fs + fs4[d][lane];
      }
      AntiHermSum<T> D = {{s[0], s[1]}, {s[2], s[3]}, {s[4], s[5]}, s[6], s[7], s[8]};
      q = D.finish();
    }
  }
  if (measure_now && mu == turn) {
    const T v[2] = {fs, q};
    float2 o[2];
    if constexpr (sizeof(T) == 4) {
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        float hi = v[j], lo = 0.f;
#pragma unroll
        for (int o2 = 16; o2 > 0; o2 >>= 1) {
          const float oh = __shfl_down_sync(0xffffffffu, hi, o2), ol = __shfl_down_sync(0xffffffffu, lo, o2);
          float s, e;
          two_sum(hi, oh, s, e);
          hi = s;
          lo = (lo + ol) + e;
        }
        o[j] = make_float2(hi, lo);
      }
    } else {
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        double d = v[j];
#pragma unroll
        for (int o2 = 16; o2 > 0; o2 >>= 1) d += __shfl_down_sync(0xffffffffu, d, o2);
        o[j] = pair_of(d);
      }
    }
    if (lane == 0) {
      if (a.part_F) a.part_F[ti] = o[0];
      a.part_theta[ti] = o[1];
    }
  }
}

}  // namespace gf
