// The CG solve of one Newton step in one launch, for small frames: a thread-block cluster with one block per coil runs
// every iteration of q_cg_iter (nlinv.cu) on chip.
//
// What bounds it: at 64 x 64 with 4 coils an iteration as four launches takes 13.6 us although each pass has about a
// microsecond of work, and the launches of a solve that has stopped at its rounding floor still cost 4.6 us an
// iteration.  Here the four passes are phases of one block: its coil's T, W^-1 p and coil map stay in its shared memory,
// its elements of r, p, dx and w in registers, so the transposes between column and row phases need __syncthreads only.
// Only the channel sum, the rho plane and the scalars cross blocks, through the cluster's shared memory, with two
// cluster barriers an iteration; the loop touches no global memory (a barrier would wait for its stores).  One block per
// coil leaves most SMs idle, so it pays only while a coil's plane is small: with the vectors of 80 x 80 and 96 x 96 planes
// in global memory, one SM's share of the L2 bandwidth made an iteration 30 us.  A stopped solve ends the loop.
// 64 x 64 with 4 coils: 13.6 -> 7.8 us an iteration, 2.00 -> 0.94 ms a frame.
#pragma once
#include "kernels.cuh"

namespace nlv {

constexpr int kClusterMaxSide = 64;      // largest grid side of the cluster solve
constexpr int kClusterMaxCoils = 16;     // largest cluster (non-portable size)

// Shared-memory layout in float2 elements, then the mask; the block's share of the rho plane (r, p, dx) follows.  T rows
// are padded so that the rows that a half-warp reads together fall on different banks.
template <int N1, int N2> struct ClusterSmem {
  using S = Split<N1, N2>;
  static constexpr int N = S::N, Wc = N / 2, P = Wc + 8, T = N * N2;
  static constexpr int XR = N * S::SM_LANE, XC = Wc * S::SM_LANE_COL;
  static constexpr int tw = 0, t = tw + 2 * N, xch = t + N * P, coil = xch + (XR > XC ? XR : XC), u = coil + Wc * Wc,
                       rho = u + Wc * Wc, z = rho + Wc * Wc, mask = z + Wc * Wc, share = mask + N * N / 8;
  static_assert(T % 32 == 0 && T <= 1024, "cluster solve thread maps");
};
// Pixels of the rho plane per block, and the kernel's dynamic shared memory.
__host__ __device__ constexpr int cluster_share(int N, int J) { return (N * N + J - 1) / J; }
template <int N1, int N2> size_t cluster_smem_bytes(int J) {
  using M = ClusterSmem<N1, N2>;
  return ((size_t)M::share + 3 * (size_t)cluster_share(M::N, J)) * 8;
}

__device__ __forceinline__ unsigned cluster_rank() {
  unsigned r;
  asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// Barrier of the whole cluster: what its threads wrote before is visible after.
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// The address of this block's shared `p` in block `rank` of the cluster, and 8 bytes read there.
__device__ __forceinline__ unsigned cluster_addr(const void* p, unsigned rank) {
  unsigned ra;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"((unsigned)__cvta_generic_to_shared(p)), "r"(rank));
  return ra;
}
__device__ __forceinline__ float2 cluster_ld(unsigned addr) {
  float2 v;
  asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(addr) : "memory");
  return v;
}

// Block sums of K pairs per thread into slot[0 .. K); every thread calls it (one barrier).  wsum: K * 32 pairs.
template <int K> __device__ __forceinline__ void cluster_block_sums(const Pair (&v)[K], Pair* wsum, Pair* slot) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
  for (int k = 0; k < K; ++k) {
    const Pair s = warp_sum(v[k], 32);
    if (lane == 0) wsum[k * 32 + warp] = s;
  }
  __syncthreads();
  for (int k = warp; k < K; k += nw) {
    Pair s = {0.f, 0.f};
    if (lane < nw) s = wsum[k * 32 + lane];
    s = warp_sum(s, 32);
    if (lane == 0) slot[k] = s;
  }
}
// Sum over the cluster's blocks of a slot, by the calling warp, the same in every block; valid in lane 0.
__device__ __forceinline__ Pair cluster_sum(const Pair* slot, int J) {
  const int lane = threadIdx.x & 31;
  Pair s = {0.f, 0.f};
  if (lane < J) {
    const float2 v = cluster_ld(cluster_addr(slot, lane));
    s = {v.x, v.y};
  }
  return warp_sum(s, 32);
}

// A.iter: the scheduled iterations; src: T (row transform of w r from the right-hand side); r, coil, rho, mask, alpha, slot
// as in the four passes.  Writes dst = x + dx (x NULL: dx alone) and the iteration that stopped.
template <int N1, int N2>
__global__ void __launch_bounds__(ClusterSmem<N1, N2>::T, 1) cg_solve_cluster(const KArgs A) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  pdl_enter();
  using M = ClusterSmem<N1, N2>;
  using S = Split<N1, N2>;
  constexpr int N = M::N, Wc = M::Wc, P = M::P, T = M::T, E = S::E, f = N / 4, H = N1 / 2;
  constexpr int plane = N * N;
  const int J = A.J, tid = threadIdx.x;
  const int j = (int)cluster_rank();
  float2* sm2 = (float2*)smem_raw;
  float2* sT = sm2 + M::t;
  const float2 *twA = sm2 + M::tw, *twB = twA + N;
  float2 *sc = sm2 + M::coil, *su = sm2 + M::u, *srho = sm2 + M::rho, *sz = sm2 + M::z;
  const uint8_t* smask = (const uint8_t*)(sm2 + M::mask);
  __shared__ Pair wsum[3 * 32];
  __shared__ Pair slots[4];            // |DF p|^2; |r|^2, Re<r, p>, |p|^2 of this block
  __shared__ CgStep s_cg;
  __shared__ int s_stop;

  // thread maps: columns (adjacent threads on adjacent columns), rows in layouts A and B
  const int cl = tid % Wc, ci = tid / Wc;
  const bool colA = ci < N1, colB = ci < N2;
  float2* xc = sm2 + M::xch + cl * S::SM_LANE_COL;
  const int laneA = tid / N1, idxA = tid % N1, laneB = tid / N2, idxB = tid % N2;
  const bool mapA = laneA < N;
  float2* xA = sm2 + M::xch + laneA * S::SM_LANE;
  float2* xB = sm2 + M::xch + laneB * S::SM_LANE;
  const float rs = rsqrtf((float)N);
  const int ob = laneB * N + idxB;                               // element m of layout B: ob + N2 m
  const size_t coil0 = (size_t)(1 + j) * plane;
  // this block's share of the rho plane: pixels o_begin + tid + k T
  const int share = cluster_share(N, J), o_begin = j * share, o_cnt = max(0, min(share, plane - o_begin));
  float2 *qr = sm2 + M::share, *qp = qr + share, *qd = qp + share;

  // ---- everything the iterations read
  stage_bytes((void*)twA, A.twA, N * 8);
  stage_bytes((void*)twB, A.twB, N * 8);
  stage_bytes((void*)smask, A.mask, plane);
  stage_bytes(sc, A.coil + (size_t)j * Wc * Wc, Wc * Wc * 8);
  for (int i = tid; i < N * Wc / 2; i += T) {
    const int e = i / (Wc / 2), k = i % (Wc / 2);
    cp_async16(sT + e * P + 2 * k, A.src + ((size_t)j * N + e) * Wc + 2 * k);
  }
  for (int i = tid; i < Wc * Wc / 2; i += T) {
    const int cr = i / (Wc / 2), k = i % (Wc / 2);
    cp_async16(srho + cr * Wc + 2 * k, A.rho + (size_t)to_natural(cr, N, f) * N + to_natural(2 * k, N, f));
  }
  const float unit = A.sc->unit;
  for (int o = tid; o < o_cnt; o += T) {
    qr[o] = cscale(A.r[o_begin + o], unit);
    qp[o] = qd[o] = make_float2(0.f, 0.f);
  }
  float2 r[N1], p[N1], dx[N1];
  float w[N1];
#pragma unroll
  for (int m = 0; m < N1; ++m) {
    r[m] = cscale(A.r[coil0 + ob + N2 * m], unit);
    w[m] = A.wtab[ob + N2 * m] * rs;
    p[m] = dx[m] = make_float2(0.f, 0.f);
  }
  // where this thread's Omega elements of the rho plane live (r there; p `share` elements on)
  unsigned ro_at[H];
#pragma unroll
  for (int h = 0; h < H; ++h) {
    const int m = h < H / 2 ? h : h + N1 - H;                    // the Omega elements of layout B
    const int o = min((ci + N2 * m) * N + to_natural(cl, N, f), plane - 1), own = o / share;
    ro_at[h] = cluster_addr(qr + (o - own * share), own);
  }
  // The scalars live in thread 0 of every block, formed there from the same sums in the same order: pairs, all in the
  // unit of the solve (cg_unit), as r, p and dx.  s_cg and s_stop pass the decisions on (s_stop: 1 the solve stops before
  // iteration `it` takes its step, 2 on a non-finite value).  In FP64 they took 15000 of 34600 cycles an iteration.
  Pair rr = {0.f, 0.f}, floor = rr, pp = rr, beta = rr, inv_rs2 = rr;
  if (tid == 0) {
    rr = pp = A.sc->rr_pair;
    floor = pair_scale(rr, (float)kCgFloor2);
    inv_rs2 = pair_div({1.f, 0.f}, pair_mul({rs, 0.f}, {rs, 0.f}));
    s_cg.a = s_cg.a_prev = s_cg.beta = 0.f;
    s_cg.alpha = A.alpha;
    s_stop = !isfinite(rr.h) ? 2 : pair_gt(rr, floor) ? 0 : 1;
  }
  cp_async_wait_all();
  float2 v[E];
  __syncthreads();
  cluster_sync_all();           // every block's share of the rho plane is in place

  int it = 0;
  for (; it < A.iter && !s_stop; ++it) {
    const bool first = it == 0;
    const float bf = s_cg.beta;
    // ---- columns: u = W^-1 p, T = FFT_col(M (p_rho c + rho u))
    {
      float2 ro[H], po[H];
      if (colB) {
#pragma unroll
        for (int h = 0; h < H; ++h) {
          ro[h] = cluster_ld(ro_at[h]);
          po[h] = cluster_ld(ro_at[h] + 8 * share);
        }
      }
      if (colA) {
#pragma unroll
        for (int m = 0; m < N2; ++m) v[m] = sT[(ci + N1 * m) * P + cl];
      }
      fft_AtoB2<N1, N2, +1, E>(v, xc, ci, colA, xc, ci, colB, twA);
      if (colB) {
#pragma unroll
        for (int m = 0; m < N1; ++m) {
          const int e1 = ci + N2 * m;
          float2 out = make_float2(0.f, 0.f);
          if (m < H / 2 || m >= N1 - H / 2) {                    // Omega
            const int h = m < H / 2 ? m : m - (N1 - H);
            const int o = to_compact(e1, N, f) * Wc + cl;
            float2 u = cscale(v[m], first ? rs * unit : rs), dr = ro[h];      // (T as staged holds b)
            if (!first) {
              const float2 uo = su[o];
              dr = make_float2(fmaf(bf, po[h].x, dr.x), fmaf(bf, po[h].y, dr.y));
              u = make_float2(fmaf(bf, uo.x, u.x), fmaf(bf, uo.y, u.y));
            }
            su[o] = u;
            out = cadd(cmul(dr, sc[o]), cmul(srho[o], u));
          }
          v[m] = out;
        }
      }
      fft_AtoB2<N2, N1, -1, E, NoTc, false>(v, xc, ci, colB, xc, ci, colA, twB);
      if (colA) {
#pragma unroll
        for (int m = 0; m < N2; ++m) sT[(ci + N1 * m) * P + cl] = cscale(v[m], rs);
      }
    }
    __syncthreads();
    // ---- rows: PSF, |DF p|^2
    Pair dd[1] = {{0.f, 0.f}};
    {
      float2 acc = make_float2(0.f, 0.f);
      if (mapA) {
#pragma unroll
        for (int m = 0; m < N2; ++m) {
          const int e2 = idxA + N1 * m;
          v[m] = in_omega(e2, N, f) ? sT[laneA * P + to_compact(e2, N, f)] : make_float2(0.f, 0.f);
        }
      }
      fft_AtoB2<N1, N2, -1, E>(v, xA, idxA, mapA, xB, idxB, true, twA);
#pragma unroll
      for (int m = 0; m < N1; ++m) {
        v[m] = smask[ob + N2 * m] ? cscale(v[m], rs * rs) : make_float2(0.f, 0.f);
        dot_acc(acc, v[m], v[m]);
      }
      dot_flush(acc, dd[0]);
      fft_AtoB2<N2, N1, +1, E, NoTc, false>(v, xB, idxB, true, xA, idxA, mapA, twB);
      if (mapA) {
#pragma unroll
        for (int m = 0; m < N2; ++m) {
          const int e2 = idxA + N1 * m;
          if (in_omega(e2, N, f)) sT[laneA * P + to_compact(e2, N, f)] = v[m];
        }
      }
    }
    cluster_block_sums<1>(dd, wsum, slots);        // its barrier also ends the row phase
    // ---- columns: channel products, T = FFT_col(conj(rho) z)
    if (colA) {
#pragma unroll
      for (int m = 0; m < N2; ++m) v[m] = sT[(ci + N1 * m) * P + cl];
    }
    fft_AtoB2<N1, N2, +1, E>(v, xc, ci, colA, xc, ci, colB, twA);
    if (colB) {
#pragma unroll
      for (int m = 0; m < N1; ++m) {
        const int e1 = ci + N2 * m;
        float2 out = make_float2(0.f, 0.f);
        if (m < H / 2 || m >= N1 - H / 2) {
          const int o = to_compact(e1, N, f) * Wc + cl;
          const float2 u = cscale(v[m], rs);
          sz[o] = cmulc(sc[o], u);
          out = cmulc(srho[o], u);
        }
        v[m] = out;
      }
    }
    fft_AtoB2<N2, N1, -1, E, NoTc, false>(v, xc, ci, colB, xc, ci, colA, twB);
    if (colA) {
#pragma unroll
      for (int m = 0; m < N2; ++m) sT[(ci + N1 * m) * P + cl] = cscale(v[m], rs);
    }
    cluster_sync_all();
    // ---- step length, the same in every block, while the other warps start on the rows' transform
    if (tid < 32) {
      const Pair d = cluster_sum(slots, J);
      if (tid == 0) {
        const Pair t = pair_sum(pair_mul(d, inv_rs2), pair_mul(pp, {A.alpha, 0.f}));
        s_stop = !isfinite(t.h) ? 2 : t.h > 0.f ? 0 : 1;
        s_cg.a = pair_div(rr, t).h;
      }
    }
    // ---- rows: q, p, r, dx; T = row transform of w r
    if (mapA) {
#pragma unroll
      for (int m = 0; m < N2; ++m) {
        const int e2 = idxA + N1 * m;
        v[m] = in_omega(e2, N, f) ? sT[laneA * P + to_compact(e2, N, f)] : make_float2(0.f, 0.f);
      }
    }
    fft_AtoB2<N1, N2, -1, E>(v, xA, idxA, mapA, xB, idxB, true, twA);      // (its barriers publish s_cg and s_stop)
    if (s_stop) break;
    const float a = s_cg.a;
    CgStep cg;
    cg.a = a;
    cg.a_prev = 0.f;
    cg.beta = bf;
    cg.alpha = A.alpha;
    cg.unit = 1.f;
    cg.first = first;
    CgDots dots;
    dots.rr = dots.rp = dots.pp = make_float2(0.f, 0.f);
#pragma unroll
    for (int m = 0; m < N1; ++m) {
      float2 g;
      r[m] = cg_point(cg, cscale(v[m], w[m]), r[m], p[m], g, dots);
      dx[m] = make_float2(fmaf(a, p[m].x, dx[m].x), fmaf(a, p[m].y, dx[m].y));
      v[m] = cscale(r[m], w[m]);
    }
    Pair sums[3] = {{0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}};
    cg_flush(dots, sums);
    fft_AtoB2<N2, N1, +1, E, NoTc, false>(v, xB, idxB, true, xA, idxA, mapA, twB);
    if (mapA) {
#pragma unroll
      for (int m = 0; m < N2; ++m) {
        const int e2 = idxA + N1 * m;
        if (in_omega(e2, N, f)) sT[laneA * P + to_compact(e2, N, f)] = v[m];
      }
    }
    // ---- this block's share of the rho plane: the channel sum over the blocks' shared memory, eight coils in flight
    for (int o = tid; o < o_cnt; o += T) {
      const int e1 = (o_begin + o) / N, e2 = (o_begin + o) - e1 * N;
      float2 z0 = make_float2(0.f, 0.f), z1 = z0, pv = qp[o], g;
      if (in_omega(e1, N, f) && in_omega(e2, N, f)) {
        const float2* za = sz + to_compact(e1, N, f) * Wc + to_compact(e2, N, f);
        for (int k0 = 0; k0 < J; k0 += 8) {
          float2 zk[8];
#pragma unroll
          for (int k = 0; k < 8; ++k) zk[k] = k0 + k < J ? cluster_ld(cluster_addr(za, k0 + k)) : make_float2(0.f, 0.f);
#pragma unroll
          for (int k = 0; k < 8; k += 2) {
            z0 = cadd(z0, zk[k]);
            z1 = cadd(z1, zk[k + 1]);
          }
        }
      }
      qr[o] = cg_point(cg, cadd(z0, z1), qr[o], pv, g, dots);
      qp[o] = pv;
      qd[o] = make_float2(fmaf(a, pv.x, qd[o].x), fmaf(a, pv.y, qd[o].y));
      cg_flush(dots, sums);
    }
    cluster_block_sums<3>(sums, wsum, slots + 1);
    cluster_sync_all();
    // ---- |r|^2, beta and |p|^2 of the next direction, the same in every block
    if (tid < 32) {
      const Pair sr = cluster_sum(slots + 1, J), srp = cluster_sum(slots + 2, J), spp = cluster_sum(slots + 3, J);
      if (tid == 0) {
        beta = pair_gt(rr, {0.f, 0.f}) ? pair_div(sr, rr) : Pair{0.f, 0.f};
        rr = sr;
        pp = cg_direction_norm(rr, beta, srp, spp);
        s_cg.beta = beta.h;
        s_stop = !isfinite(rr.h) ? 2 : pair_gt(rr, floor) ? 0 : 1;
      }
    }
    __syncthreads();
  }
  // ---- x + dx
  const float inv = 1.f / unit;
#pragma unroll
  for (int m = 0; m < N1; ++m) {
    const size_t o = coil0 + ob + N2 * m;
    const float2 d = cscale(dx[m], inv);
    A.dst[o] = A.x ? cadd(A.x[o], d) : d;
  }
  for (int o = tid; o < o_cnt; o += T) {
    const float2 d = cscale(qd[o], inv);
    A.dst[o_begin + o] = A.x ? cadd(A.x[o_begin + o], d) : d;
  }
  if (j == 0 && tid == 0) {
    // (`it` iterations took a step; a floor reached by the last scheduled one is not a stop)
    A.sc->cg_stop[A.slot] = it < A.iter ? it : -1;
    if (s_stop == 2 && it < A.iter) atomicOr(&A.sc->flags, kFlagBreakdown);
  }
  cluster_sync_all();          // no block leaves while another may read its shared memory
}

}  // namespace nlv
