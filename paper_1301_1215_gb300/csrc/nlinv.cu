// C interface, context and solver driver of the GB300 NLINV library (declared in include/nlinv.h).
//
// The driver queues the pass kernels of kernels.cuh on the context's stream:
//   coil maps      c_j = W^-1 chat_j on Omega                  row ROW_W_IFFT, col COL_IFFT_C
//   F x            P FFT(M rho c_j)                            col COL_PROD_FFT, row ROW_FFT_P_OUT / ROW_FFT_RESID
//   DF dx          P FFT(M (drho c_j + rho W^-1 dchat_j))       row ROW_W_IFFT, col COL_IFFT_PROD_FFT, row ROW_FFT_P_OUT
//   DF^H r         (sum_j conj(c_j) z_j, w FFT(conj(rho) z_j)) row ROW_P_IFFT, col COL_IFFT_ADJ_FFT, row ROW_FFT_W_ADJ
//   (DF^H DF + alpha) p   the PSF form of Sec. 3.1: row ROW_W_IFFT, col COL_IFFT_PROD_FFT, row ROW_PSF,
//                         col COL_IFFT_ADJ_FFT, row ROW_FFT_W_NORMAL
//   CG iteration   col COL_CG_DIR, row ROW_PSF, col COL_IFFT_ADJ_FFT, row ROW_CG_UPDATE (q_cg_iter)
// Each operator application performs the two 2D transforms per operator of Table 1, batched over all coils.
// Beyond the paper's method: the gradient through the reconstruction (nlinv_reconstruct_checkpoints and
// nlinv_reconstruct_vjp: the same operators at other linearisation points, plus a CG solve per Newton step),
// batches of independent frames (nlinv_batch_*: the same passes, one launch per grid side), and the launch-shape
// autotuner (nlinv_autotune: whole graph-replayed frames per candidate).
#include <algorithm>
#include <chrono>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <functional>
#include <mutex>
#include <new>
#include <string>
#include <thread>
#include <vector>

#include "nlinv.h"
#include "call_order.h"
#include "sizes.cuh"

using nlv::KArgs;
using nlv::Scalars;
using nlv::SizeKernels;

namespace {

thread_local std::string g_create_error;

// ------------------------------------------------------------------------------------------ vector kernels ----
constexpr int kVecThreads = 256;     // threads per block of the vector kernels

// The CG step of batches.  float4 groups of its operands in flight per thread.  Two keep the kernel at 64 registers, four blocks of 256
// threads per SM; four groups need 96 registers (two blocks per SM, measured 13.2 against 11.5 us per step at
// 384 x 384 with 10 coils) or spill at 64.
constexpr int kCgGroups = 2;
// dx += alpha p; r -= alpha q; partial of |r|^2 -> brr_part[bid], over this block's share of the A.n2 float4.
// A thread sums the squares of at most two float4 (8 products) in FP32 before adding them to its pair.
__device__ __forceinline__ void cg_step_update(float4& d, float4& r, const float4& p, const float4& q, float a,
                                               float& acc) {
  d.x = fmaf(a, p.x, d.x); d.y = fmaf(a, p.y, d.y); d.z = fmaf(a, p.z, d.z); d.w = fmaf(a, p.w, d.w);
  r.x = fmaf(-a, q.x, r.x); r.y = fmaf(-a, q.y, r.y); r.z = fmaf(-a, q.z, r.z); r.w = fmaf(-a, q.w, r.w);
  acc += r.x * r.x + r.y * r.y + r.z * r.z + r.w * r.w;
}

// The CG step's scalars, the same in every block: t = Re<p, A p> from the n_pq partials, alpha = |r|^2 / t, and the
// rounding-floor test (see cg_step_body), formed as pairs by the block's first warp (in FP64, a tree over the block and a
// quotient, each some thousand cycles a block).  Block 0 publishes them; s_alpha is valid for every thread of the block
// on return, as is s_unit, the solve's unit.
__device__ __forceinline__ void cg_step_decide(const KArgs& A, int bid, float& s_alpha, float& s_unit) {
  if (threadIdx.x < 32) {
    const nlv::Pair t = nlv::warp_sum_of(A.pq_part, A.n_pq);
    if (threadIdx.x == 0) {
      s_unit = A.sc->unit;
      const nlv::Pair rr = A.sc->rr_i[0], floor = nlv::pair_scale(A.sc->rr_pair, (float)nlv::kCgFloor2);
      const bool finite = isfinite(t.h) && isfinite(rr.h);
      const bool go = finite && nlv::pair_gt(rr, floor) && t.h > 0.f;
      if (bid == 0) {
        A.sc->rr_i[1] = rr;
        if (!go) A.sc->cg_stop[A.slot] = A.iter;
        if (!finite) atomicOr(&A.sc->flags, nlv::kFlagBreakdown);
      }
      s_alpha = go ? nlv::pair_div(rr, t).h : 0.f;
    }
  }
  __syncthreads();
}

template <int G>
__device__ __forceinline__ void cg_step_body(const KArgs& A, int bid, int nblk) {
  const float4* __restrict__ p4 = (const float4*)A.p;
  const float4* __restrict__ q4 = (const float4*)A.q;
  float4* __restrict__ r4 = (float4*)A.r;
  float4* __restrict__ dx4 = (float4*)A.dx;
  // Two groups of operands per thread in flight: the first two are loaded while the block forms
  // alpha = |r|^2 / Re<p, A p> from the partials of the normal-operator pass (every block sums them in the same
  // fixed order).  The solve stops at the rounding floor: |r|^2 <= kCgFloor2 |b|^2 (|r| at the FP32 unit roundoff
  // relative to |b|, including b = 0), Re<p, A p> <= 0 (impossible in exact arithmetic for the positive definite
  // system of Eq. 3) or a non-finite value.  This step and every later step of the same solve are then empty
  // (alpha = 0): block 0 records the iteration, and the passes of later iterations skip (cg_stopped).  Non-finite values
  // also set the breakdown flag.  Every block takes the same decision from the same partials.
  const long stride = (long)nblk * blockDim.x;
  long i = bid * (long)blockDim.x + threadIdx.x;
  float4 pg[G], qg[G], rg[G], dg[G];
#pragma unroll
  for (int g = 0; g < G; ++g)
    if (i + g * stride < A.n2) {
      const long k = i + g * stride;
      pg[g] = p4[k]; qg[g] = q4[k]; rg[g] = r4[k]; dg[g] = dx4[k];
    }
  __shared__ float s_alpha, s_unit;
  __shared__ nlv::Pair s_pairs[kVecThreads];
  cg_step_decide(A, bid, s_alpha, s_unit);
  const float a = s_alpha;
  const bool first = A.iter == 0;        // r holds b
  nlv::Pair sum = {0.f, 0.f};
  // G groups in flight per thread; each group's operands for the next round are loaded right after it is stored,
  // while the other groups of this round are processed
  while (i < A.n2) {
    float acc = 0.f;
#pragma unroll
    for (int g = 0; g < G; ++g) {
      const long k = i + g * stride;
      if (k < A.n2) {
        if (first) rg[g] = make_float4(rg[g].x * s_unit, rg[g].y * s_unit, rg[g].z * s_unit, rg[g].w * s_unit);
        cg_step_update(dg[g], rg[g], pg[g], qg[g], a, acc);
        dx4[k] = dg[g];
        r4[k] = rg[g];
        const long kn = k + G * stride;
        if (kn < A.n2) { pg[g] = p4[kn]; qg[g] = q4[kn]; rg[g] = r4[kn]; dg[g] = dx4[kn]; }
      }
    }
    nlv::acc_add(sum, acc);
    i += G * stride;
  }
  s_pairs[threadIdx.x] = sum;
  __syncthreads();
  nlv::block_pairs<1>(s_pairs, {A.brr_part + bid});
}

// x += dx (x = A.dst; dx in the unit of the solve)
__device__ __forceinline__ void add_body(const KArgs& A, int bid, int nblk) {
  const float4* __restrict__ d4 = (const float4*)A.dx;
  float4* __restrict__ x4 = (float4*)A.dst;
  const float inv = 1.f / A.sc->unit;
  for (long i = bid * (long)blockDim.x + threadIdx.x; i < A.n2; i += (long)nblk * blockDim.x) {
    float4 d = d4[i], x = x4[i];
    x.x = fmaf(inv, d.x, x.x); x.y = fmaf(inv, d.y, x.y); x.z = fmaf(inv, d.z, x.z); x.w = fmaf(inv, d.w, x.w);
    x4[i] = x;
  }
}

// out = base + dx_total (out = A.dst, base = A.src or zero): the end of a CG solve, which leaves its unit.  The CG update pass adds the steps of
// an even iteration and of the odd one after it to A.dx together, in the odd one (the first pair without reading it),
// so that after an odd number of executed iterations the last step a p is still to be added, and A.dx holds nothing
// before iteration 1.  A.iter: the scheduled iterations; A.slot: the Newton step.
__global__ void cg_finish_kernel(const KArgs A) {
  nlv::pdl_enter();
  const int stop = A.sc->cg_stop[A.slot];
  const int done = stop < 0 ? A.iter : stop;
  const bool has_dx = done >= 2, has_p = (done & 1) != 0;
  const float a = has_p ? A.sc->step[0] : 0.f;        // the last executed iteration is an even one
  const float inv = 1.f / A.sc->unit;
  const float4* d4 = (const float4*)A.dx;        // A.dst itself in the gradient
  const float4* __restrict__ p4 = (const float4*)A.p;
  const float4* x4 = (const float4*)A.src;
  float4* o4 = (float4*)A.dst;
  const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < A.n2; i += (long)gridDim.x * blockDim.x) {
    const float4 x = x4 ? x4[i] : zero, p = has_p ? p4[i] : zero;
    float4 d = has_dx ? d4[i] : zero;
    if (has_p) {
      d.x = fmaf(a, p.x, d.x); d.y = fmaf(a, p.y, d.y); d.z = fmaf(a, p.z, d.z); d.w = fmaf(a, p.w, d.w);
    }
    o4[i] = make_float4(fmaf(inv, d.x, x.x), fmaf(inv, d.y, x.y), fmaf(inv, d.z, x.z), fmaf(inv, d.w, x.w));
  }
}

// Display image rho * sqrt(sum_j |c_j|^2) on Omega, centred: out[i][k] for the signed coordinates (i - f, k - f).
__global__ void image_kernel(const KArgs A) {
  nlv::pdl_enter();
  const int N = A.N, f = A.f, Wc = A.Wc, J = A.J;
  const long total = (long)Wc * Wc;
  for (long o = blockIdx.x * (long)blockDim.x + threadIdx.x; o < total; o += (long)gridDim.x * blockDim.x) {
    const int i = (int)(o / Wc), k = (int)(o % Wc);
    const int cr = (i + f) % Wc, cc = (k + f) % Wc;           // compact indices of the signed coordinates
    float s = 0.f;
    for (int j = 0; j < J; ++j) {
      const float2 c = A.coil[((size_t)j * Wc + cr) * Wc + cc];
      s = fmaf(c.x, c.x, fmaf(c.y, c.y, s));
    }
    const float2 r = A.rho[(size_t)nlv::to_natural(cr, N, f) * N + nlv::to_natural(cc, N, f)];
    A.dst[o] = nlv::cscale(r, sqrtf(s));
  }
}

// out = alpha X + coef Y (X = A.src, Y = A.q, out = A.dst, which may be X or Y) over A.n2 float4, or, for a caller's array
// off the 16-byte boundary, 2 A.n2 float2
__device__ __forceinline__ float4 axpby(float a, float4 x, float b, float4 y) {
  return make_float4(fmaf(a, x.x, b * y.x), fmaf(a, x.y, b * y.y), fmaf(a, x.z, b * y.z), fmaf(a, x.w, b * y.w));
}
__device__ __forceinline__ float2 axpby(float a, float2 x, float b, float2 y) {
  return make_float2(fmaf(a, x.x, b * y.x), fmaf(a, x.y, b * y.y));
}
template <class V> __global__ void axpby_kernel(const KArgs A) {
  nlv::pdl_enter();
  const V *x = (const V*)A.src, *y = (const V*)A.q;
  V* o = (V*)A.dst;
  const long n = A.n2 * (long)(sizeof(float4) / sizeof(V));
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x)
    o[i] = axpby(A.alpha, x[i], A.coef, y[i]);
}

// CG from dx = 0 for the right-hand side b = A.src: r = b, |b|^2 -> RED_RR_INIT
__global__ void cg_init_kernel(const KArgs A) {
  nlv::pdl_enter();
  const float4* __restrict__ b4 = (const float4*)A.src;
  float4* __restrict__ r4 = (float4*)A.r;
  double acc = 0.0;
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < A.n2; i += (long)gridDim.x * blockDim.x) {
    const float4 b = b4[i];
    r4[i] = b;
    acc += (double)(b.x * b.x + b.y * b.y + b.z * b.z + b.w * b.w);
  }
  nlv::grid_reduce(acc, A, blockIdx.x, gridDim.x);
}

__global__ void __launch_bounds__(256, 4) cg_step_batch(const nlv::BatchArgs B) {
  __shared__ nlv::BatchQueue q;
  nlv::pdl_enter();
  nlv::batch_items(B, q, [&](const KArgs& A, int bid, int nblk, bool stopped) {
    if (!stopped) cg_step_body<kCgGroups>(A, bid, nblk);
  });
}
__global__ void add_batch(const nlv::BatchArgs B) {
  __shared__ nlv::BatchQueue q;
  nlv::pdl_enter();
  nlv::batch_items(B, q, [&](const KArgs& A, int bid, int nblk, bool stopped) {
    if (!stopped) add_body(A, bid, nblk);
  });
}

constexpr int kTuneVecMax = 8;       // largest vector-kernel blocks per SM that nlinv_autotune tries
constexpr int kTuneMaxCandidates = 16;   // most candidates it times (2 splits + 3 strips + 3 row + 6 vector shapes)
constexpr double kTuneMargin = 0.03; // a candidate replaces the compiled default only when this much faster
#ifndef NLV_VEC_BLOCKS_PER_SM
#define NLV_VEC_BLOCKS_PER_SM 4   // blocks per SM of the vector passes
#endif
// One shared-memory carve-out for every pass of a batch (percent of an SM's; 72 to 84 select the same one): a launch that
// asks for another split of the L1 than its predecessor's waits until the SM is empty, and streams of different sides then
// hold each other up.  Left to the driver, per pass, or at the maximum, whose 28 KB of L1 limit the loads in flight, 64
// frames (5 Newton steps of 12 iterations) take 107.3 ms, at 50 percent 107.8, at 60 102.8, here 100.0; three 384^2
// frames 12.7, 13.3, 12.5 and 11.9.
constexpr int kBatchCarveout = 76;
constexpr int kProfileSteps = 6;   // steps of one CG iteration, in the order nlinv_profile_cg reports them

size_t align_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

}  // namespace

// ----------------------------------------------------------------------------------------------- context ----
struct nlinv_ctx {
  nlinv_params prm{};
  int N = 0, J = 0, f = 0, Wc = 0;
  long plane = 0;             // N*N
  long vec = 0;               // (1+J)*N*N complex values of an unknown-space vector
  const SizeKernels* k = nullptr;
  cudaStream_t stream = nullptr;
  bool own_stream = false;
  nlv::StreamOrder order;     // operator calls on a caller's stream (nlinv_use_stream): all share the workspace
  int device = 0;
  int vec_blocks = 0;         // grid of the vector kernels
  int sms = 0;                // streaming multiprocessors of the device
  int row_ctas_per_sm = nlv::kRowCtasPerSM;   // blocks per SM of the row passes
  int carveout = 100;         // shared-memory carve-out of the launches, percent (choose_carveout)
  // workspace (one allocation)
  void* base = nullptr;
  float2 *x = nullptr, *xref = nullptr, *y = nullptr, *r0 = nullptr;
  float2 *r = nullptr, *p = nullptr, *dx = nullptr;
  float2* q = nullptr;        // A p (frames of a batch)
  float2 *T = nullptr, *coil = nullptr, *zsum = nullptr;
  float2* U = nullptr;        // W^-1 p on Omega of the CG direction (single frames)
  float2 *twA = nullptr, *twB = nullptr;
  float* wtab = nullptr;      // Sobolev weight, N x N
  uint8_t* mask = nullptr;
  double* partials = nullptr;
  nlv::Pair* pq_part = nullptr;  // frames of a batch: per-block partials of Re<p, A p> and of |r|^2
  nlv::Pair* brr_part = nullptr;
  nlv::Pair* dd_part = nullptr;  // single frames: per-block partials of |DF p|^2 of the PSF pass
  nlv::Pair* rr_part = nullptr;  // per-block partials of |r|^2, Re<r, p> and |p|^2 of the CG update pass
  Scalars* sc = nullptr;
  // graph of one reconstruction
  cudaGraphExec_t graph = nullptr;
  long graph_launches = 0;
  long launches = 0;
  bool have_state = false;    // a reconstruction has filled the workspace
  int batch_lanes = 0;        // > 0: frame of a batch; row passes use this many lanes and one round per block
  bool batch_split = true;    // those blocks may be divided (batch_row_split); not under the multi-side kernels, which
                              // run kRowMaxThreads threads whatever the side
  struct Rec {
    const void* fn;
    int grid, block;
    size_t smem;
    KArgs args;
    int step;                 // 1..6: pass of the CG iteration that nlinv_batch_profile_cg times, 0 otherwise
  };
  int rec_step = 0;           // the `step` of the launches being recorded
  std::vector<Rec>* rec = nullptr;   // non-null: launches are recorded instead of issued
  bool pdl = true;            // programmatic dependent launches (NLINV_PDL=0 turns them off)
  bool std_fov = false;       // fov = N/4: the passes specialised for it (SizeKernels::row_std, col_std) apply
  bool cluster = false;       // the CG solves run as one cluster launch each (cluster_fits)
  bool tc = false;            // radix-16 DFT stages on the tensor cores (params.tensor_dft)
  void* tcB = nullptr;        // their B tiles (workspace)
  double last_alpha = 0.0;    // alpha_n of the last Newton step
  float2* ckpt = nullptr;     // non-null: q_reconstruct writes x_0 .. x_N here (nlinv_reconstruct_checkpoints)
  void* vjp_base = nullptr;   // scratch of nlinv_reconstruct_vjp (allocated on first use)
  std::string err;
};

namespace {

}  // namespace

// Records the message returned by nlinv_last_error(NULL) (used by the calls that take no context).
void nlv_set_global_error(const std::string& msg) { g_create_error = msg; }

namespace {

nlinv_status fail(nlinv_ctx* c, nlinv_status s, const std::string& msg) {
  if (c) c->err = msg; else g_create_error = msg;
  return s;
}

nlinv_status cuda_fail(nlinv_ctx* c, cudaError_t e, const char* where) {
  return fail(c, NLINV_ECUDA, std::string(where) + ": " + cudaGetErrorString(e));
}

#define NLV_TRY(call, where)                           \
  do {                                                 \
    cudaError_t e_ = (call);                           \
    if (e_ != cudaSuccess) return cuda_fail(c, e_, where); \
  } while (0)

KArgs base_args(const nlinv_ctx* c) {
  KArgs a{};
  a.N = c->N;
  a.J = c->J;
  a.f = c->f;
  a.Wc = c->Wc;
  a.wtab = c->wtab;
  a.twA = c->twA;
  a.twB = c->twB;
  a.partials = c->partials;
  a.sc = c->sc;
  a.reduce = nlv::RED_NONE;
  a.tcB = c->tcB;
  return a;
}

nlv::RowGrid row_geom(const nlinv_ctx* c, bool with_rho, int arrays = 1) {
  if (c->batch_lanes > 0) {           // batch frames: equal block shapes for every frame of a grid side
    nlv::RowGrid g{};
    const int rows = c->J * c->N;
    g.rows_per_cta = std::min(c->batch_lanes, rows);
    const int groups = (rows + g.rows_per_cta - 1) / g.rows_per_cta;
    g.sub = c->batch_split ? nlv::batch_row_split(c->k, g.rows_per_cta) : 1;
    g.lanes = g.rows_per_cta / g.sub;
    g.blocks = groups * g.sub;
    g.rho_per_cta = with_rho ? (int)((c->plane + groups - 1) / groups) : 0;
    return g;
  }
  nlv::RowGrid g = nlv::row_grid(c->k, arrays * c->J * c->N, with_rho ? c->plane : 0, c->sms, c->row_ctas_per_sm);
  // tensor-core passes: whole warps (every lane of a warp takes part in tcgen05.ld), the extra lanes idle
  if (c->tc)
    while ((g.lanes * c->k->tl) % 32 != 0) ++g.lanes;
  return g;
}

int col_blocks(const nlinv_ctx* c) {
  const int C = c->k->col_lanes;
  return c->J * ((c->Wc + C - 1) / C);
}

// Launches with programmatic stream serialisation (see pdl_enter in kernels.cuh): the next pass is scheduled while
// the current one drains (about 1% per frame on the 384 x 384, 10-coil series).  Every kernel launched here must
// call nlv::pdl_enter() before its first global memory access.
// cluster > 1: the grid in clusters of that many blocks.
cudaError_t launch(nlinv_ctx* c, const void* fn, int grid, int block, size_t smem, void** args, int cluster = 1) {
  c->launches++;
  if (c->rec) {                       // every pass takes one KArgs
    c->rec->push_back({fn, grid, block, smem, *(const KArgs*)args[0], c->rec_step});
    return cudaSuccess;
  }
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = c->order.run;
  cudaLaunchAttribute attr[3];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = c->pdl ? 1 : 0;
  attr[1].id = cudaLaunchAttributePreferredSharedMemoryCarveout;
  attr[1].val.sharedMemCarveout = c->carveout;
  attr[2].id = cudaLaunchAttributeClusterDimension;
  attr[2].val.clusterDim.x = cluster;
  attr[2].val.clusterDim.y = attr[2].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = cluster > 1 ? 3 : 2;
  return cudaLaunchKernelExC(&cfg, fn, args);
}

// Scope of a call on the context's own stream.
struct OwnStream {
  nlinv_ctx* c;
  cudaError_t err;
  explicit OwnStream(nlinv_ctx* ctx) : c(ctx), err(ctx->order.enter_own()) {}
  ~OwnStream() { c->order.leave(); }
};

// Passes copy the planes of rho, drho and the sampling pattern into shared memory in 16-byte pieces.  A caller's array may
// lie off that boundary (a slice of a larger one): its plane then goes to `room` first, part of a vector that holds
// nothing outside a CG solve, whose own arrays all lie on it.
bool on_boundary(const void* p) { return (uintptr_t)p % 16 == 0; }
template <class T> cudaError_t stageable(const nlinv_ctx* c, const T*& p, void* room) {
  if (on_boundary(p)) return cudaSuccess;
  const T* from = p;
  p = (const T*)room;
  return cudaMemcpyAsync(room, from, (size_t)c->plane * sizeof(T), cudaMemcpyDeviceToDevice, c->order.run);
}
bool row_stages_mask(int mode) {
  return mode == nlv::ROW_PSF || mode == nlv::ROW_CG_PSF || mode == nlv::ROW_FFT_P_OUT || mode == nlv::ROW_FFT_RESID;
}
bool col_stages_rho(int mode) {
  return mode != nlv::COL_IFFT_C && mode != nlv::COL_PROD_FFT && mode != nlv::COL_SIM_FFT;
}
bool col_stages_drho(int mode) { return mode == nlv::COL_IFFT_PROD_FFT || mode == nlv::COL_COIL_DIR; }

bool row_two_arrays(int mode) { return mode == nlv::ROW_W_W_IFFT || mode == nlv::ROW_W_P_IFFT; }
bool row_has_rho(int mode) {
  return mode >= nlv::ROW_FFT_W_ADJ && mode != nlv::ROW_CG_PSF && mode != nlv::ROW_BCG_DIR && !row_two_arrays(mode);
}

// One shared-memory carve-out for all launches of a single frame (with the driver's own choice consecutive passes differ,
// and an SM changes its carve-out only when it is empty): the smallest of 164, 196 and 228 KB per SM that holds the row
// passes' resident blocks, and the column passes' where 228 KB holds them all at once.  What is left is L1, which holds the
// loads in flight.  Four Newton steps of 20 iterations with 164 / 196 / 228 KB: 192^2/13 coils 1450 / 1516 / 1625 us,
// 320^2/7 2007 / 2016 / 2119, 384^2/22 6227 / 5334 / 5629, 512^2/3 2442 / 2432 / 2673, 320^2/22 4201 / 3718 / 3611; 7 x 30
// iterations, 384^2/10 7240 / 7302 / 6526, 512^2/16 22.2 / 22.7 / 18.6 ms.  Two lines rest on measurements without a mechanism behind them, both
// within a few percent either way (3 Newton steps of 20): side 256 does not go below 196 -- 164 / 196 KB: 4 coils 1110 / 1082,
// gradient with 9 1444 / 1391, normal operator with 16 and half-width 100 37.2 / 34.3, but 12 coils 1313 / 1379, 24 1927 /
// 2080 --, and sides up to 128 keep the largest -- 164 / 228 KB: 128^2/3 726 / 710, /6 714 / 712, /12 737 / 747, /22 821 /
// 832, 96^2/8 646 / 647 --, as do the tensor-core passes.
void choose_carveout(nlinv_ctx* c) {
  c->carveout = 100;
  if (c->tc || c->N <= 128) return;
  size_t need = 0;
  for (int m = 0; m < nlv::NUM_ROW_MODES; ++m) {
    if (!c->k->row[m]) continue;
    const nlv::RowGrid g = row_geom(c, row_has_rho(m), row_two_arrays(m) ? 2 : 1);
    const size_t resident = (size_t)std::min(c->row_ctas_per_sm, (g.blocks + c->sms - 1) / c->sms);
    need = std::max(need, resident * (c->k->row_smem(m, g.lanes) + 2048));     // static and system use: under 2 KB a block
  }
  // column blocks that the full 228 KB would hold all at once stay resident together (320^2/22: 440 blocks, three per SM)
  const size_t blocks = col_blocks(c) + 1;
  for (int m = 0; m < nlv::NUM_COL_MODES; ++m) {
    if (!c->k->col[m]) continue;
    const size_t per = c->k->col_smem(m, c->Wc) + 2048, resident = (blocks + c->sms - 1) / c->sms;
    if (resident * per <= (size_t)228 << 10) need = std::max(need, resident * per);
  }
  c->carveout = need <= (size_t)164 << 10 && c->N != 256 ? 66 : need <= (size_t)196 << 10 ? 84 : 100;
}

cudaError_t row(nlinv_ctx* c, int mode, KArgs a) {
  if (row_stages_mask(mode)) {
    const cudaError_t e = stageable(c, a.mask, c->dx);
    if (e != cudaSuccess) return e;
  }
  const bool both = row_two_arrays(mode), rho = row_has_rho(mode);
  const nlv::RowGrid g = row_geom(c, rho, both ? 2 : 1);
  a.nrows1 = c->J * c->N;
  a.nrows = (both ? 2 : 1) * a.nrows1;
  a.rows_per_cta = g.rows_per_cta;
  a.rho_per_cta = g.rho_per_cta;
  a.sub = g.sub;
  a.sub_lanes = g.lanes;
  a.group_threads = g.rows_per_cta * c->k->tl;
  void* args[] = {&a};
  if (c->tc) {
    const void* fn = (c->std_fov && c->k->row_tc_std[mode]) ? c->k->row_tc_std[mode] : c->k->row_tc[mode];
    return launch(c, fn, g.blocks, g.lanes * c->k->tl, c->k->row_smem_tc(mode, g.lanes), args);
  }
  const void* fn = (c->std_fov && c->k->row_std[mode]) ? c->k->row_std[mode] : c->k->row[mode];
  if (c->batch_lanes > 0)           // recorded for the batch's launch
    fn = c->k->row_std_batch[mode] ? c->k->row_std_batch[mode] : c->k->row_batch[mode];
  return launch(c, fn, g.blocks, g.lanes * c->k->tl, c->k->row_smem(mode, g.lanes), args);
}

cudaError_t col(nlinv_ctx* c, int mode, KArgs a) {
  cudaError_t e = cudaSuccess;
  if (col_stages_rho(mode)) e = stageable(c, a.rho, c->p);
  if (e == cudaSuccess && col_stages_drho(mode)) e = stageable(c, a.drho, c->r);
  if (e != cudaSuccess) return e;
  a.nrows = c->J;
  const int blocks = col_blocks(c) + (a.scalars ? 1 : 0);
  void* args[] = {&a};
  if (c->tc) {
    const void* fn = (c->std_fov && c->k->col_tc_std[mode]) ? c->k->col_tc_std[mode] : c->k->col_tc[mode];
    return launch(c, fn, blocks, c->k->col_threads, c->k->col_smem_tc(mode, c->Wc), args);
  }
  const void* fn = (c->std_fov && c->k->col_std[mode]) ? c->k->col_std[mode] : c->k->col[mode];
  if (c->batch_lanes > 0)
    fn = c->k->col_std_batch[mode] ? c->k->col_std_batch[mode] : c->k->col_batch[mode];
  return launch(c, fn, blocks, c->k->col_threads, c->k->col_smem(mode, c->Wc), args);
}

// c_j = W^-1 chat_j on Omega, for the coil planes of x (1+J planes).
cudaError_t q_coils(nlinv_ctx* c, const float2* x) {
  KArgs a = base_args(c);
  a.src = x + c->plane;
  a.dst = c->T;
  cudaError_t e = row(c, nlv::ROW_W_IFFT, a);
  if (e != cudaSuccess) return e;
  a = base_args(c);
  a.src = c->T;
  a.dst = c->coil;
  return col(c, nlv::COL_IFFT_C, a);
}

// T <- FFT_col(M rho c_j) for rho = plane 0 of x (coil maps already in c->coil)
cudaError_t q_prod(nlinv_ctx* c, const float2* rho) {
  KArgs a = base_args(c);
  a.rho = rho;
  a.coil = c->coil;
  a.dst = c->T;
  return col(c, nlv::COL_PROD_FFT, a);
}

// The operators' passes that form the coil maps on the way (the FP32 transforms of single frames): W^-1 of the coil
// planes and the other operator's input go through one row launch, and the column pass transforms both, where coil maps,
// then the operator, took two launches each and a pass over the maps.  The calls are bound by launches and by each
// pass's latency (1.5 to 6 us a launch, against 1 to 4 us of arithmetic).  Before and after: normal operator 384^2/10
// coils 47.4 -> 40.0 us, 512^2/16 113.6 -> 109.8; DF^H 192^2/13 23.4 -> 18.1, DF 26.6 -> 21.5; F 64^2/4 19.3 -> 16.6.
// The results are the same bits on most shapes and within 1.2e-7 on the others.  The tensor-core passes have one input, and the batch's item
// tables one launch per pass for all frames: both keep the separate passes.
bool fused_ops(const nlinv_ctx* c) { return !c->tc && c->batch_lanes == 0; }

// T <- FFT_col(M rho c_j), c_j = W^-1 chat_j of x (1+J planes); the maps to c->coil if keep.
cudaError_t q_op_prod(nlinv_ctx* c, const float2* x, bool keep) {
  KArgs a = base_args(c);
  a.src = x + c->plane;
  a.dst = c->T;
  cudaError_t e = row(c, nlv::ROW_W_IFFT, a);
  if (e != cudaSuccess) return e;
  a = base_args(c);
  a.src = c->T;
  a.dst = c->T;
  a.rho = x;
  a.coil_out = keep ? c->coil : nullptr;
  return col(c, nlv::COL_COIL_PROD, a);
}

// T <- FFT_col(M (drho c_j + rho W^-1 dchat_j)), c_j of x, for direction d; the maps to c->coil if keep.
cudaError_t q_op_dir(nlinv_ctx* c, const float2* x, const float2* d, bool keep) {
  KArgs a = base_args(c);
  a.src = x + c->plane;
  a.src2 = d + c->plane;
  a.dst = c->T;
  a.dst2 = c->r0;                 // the data residual's buffer, free outside a Newton step
  cudaError_t e = row(c, nlv::ROW_W_W_IFFT, a);
  if (e != cudaSuccess) return e;
  a = base_args(c);
  a.src = c->T;
  a.src2 = c->r0;
  a.dst = c->T;
  a.rho = x;
  a.drho = d;
  a.coil_out = keep ? c->coil : nullptr;
  return col(c, nlv::COL_COIL_DIR, a);
}

// T <- FFT_col(conj(rho) z_j), zsum_j <- conj(c_j) z_j with z_j = M FFT^-1(P r_j), c_j of x.
cudaError_t q_op_adj(nlinv_ctx* c, const float2* x, const float2* r, const uint8_t* mask) {
  KArgs a = base_args(c);
  a.src = x + c->plane;
  a.src2 = r;
  a.mask = mask;
  a.dst = c->T;
  a.dst2 = c->r0;
  cudaError_t e = row(c, nlv::ROW_W_P_IFFT, a);
  if (e != cudaSuccess) return e;
  a = base_args(c);
  a.src = c->T;
  a.src2 = c->r0;
  a.dst = c->T;
  a.rho = x;
  a.zsum = c->zsum;
  return col(c, nlv::COL_COIL_ADJ, a);
}

// T <- FFT_col(M (drho c_j + rho W^-1 dchat_j)) for direction d and linearisation point x
cudaError_t q_dir(nlinv_ctx* c, const float2* x, const float2* d) {
  KArgs a = base_args(c);
  a.src = d + c->plane;
  a.dst = c->T;
  cudaError_t e = row(c, nlv::ROW_W_IFFT, a);
  if (e != cudaSuccess) return e;
  a = base_args(c);
  a.src = c->T;
  a.dst = c->T;
  a.rho = x;
  a.drho = d;
  a.coil = c->coil;
  return col(c, nlv::COL_IFFT_PROD_FFT, a);
}

// T <- FFT_col(conj(rho) z_j), zsum_j <- conj(c_j) z_j, with z_j = M FFT^-1_col(T).
cudaError_t q_adj_col(nlinv_ctx* c, const float2* x) {
  KArgs a = base_args(c);
  a.src = c->T;
  a.dst = c->T;
  a.rho = x;
  a.coil = c->coil;
  a.zsum = c->zsum;
  return col(c, nlv::COL_IFFT_ADJ_FFT, a);
}

// End of a CG solve: out = base + dx_total (base NULL: dx_total alone).
cudaError_t q_cg_finish(nlinv_ctx* c, const float2* base, float2* out, int newton) {
  KArgs a = base_args(c);
  a.src = base;
  a.dst = out;
  a.dx = c->dx;
  a.p = c->p;
  a.iter = c->prm.cg_iters;
  a.slot = newton;
  a.n2 = c->vec / 2;
  void* args[] = {&a};
  return launch(c, (const void*)cg_finish_kernel, c->vec_blocks, kVecThreads, 0, args);
}

// One CG iteration i on (DF^H DF + alpha) for linearisation point x, in four passes.  W^-1 and its row transform are
// linear, so the row pass that finishes q = (DF^H DF + alpha) p goes straight on to r_{i+1} = r_i - a_i q and to the row
// transform of w r_{i+1} (into T), without beta_{i+1}: W^-1 p_{i+1} = W^-1 r_{i+1} + beta_{i+1} W^-1 p_i is formed by the
// next column pass, which carries W^-1 p on Omega (U).  a_i is known before that row pass because
// Re<p, A p> = |DF p|^2 + alpha |p|^2 with |DF p|^2 summed by the PSF pass.  q is never stored, and p, r, dx cross memory
// 5 times per iteration on average (p, r in and out; dx in and out every other iteration, with two steps at once)
// where q, p, r and dx crossed it 11 times in separate p-update, q and CG-step passes: 277 -> 145 MB of algorithmic
// traffic an iteration at 384^2 with 10 coils.  An iteration inside a graph, before (six passes) and after: 64^2/4 coils
// 25.6 -> 13.7 us, 256^2/8 29.9 -> 24.6, 384^2/10 44.2 -> 31.8, 512^2/16 126 -> 104.
//   col  beta_i from the |r|^2 partials; u = W^-1 p; T = FFT_col(M (p_rho c_j + rho u))
//   row  PSF, |DF p|^2 partials
//   col  adjoint products; one more block: a_i, the stop test
//   row  p = r + beta p, q, r -= a q, dx += a_{i-1} p_{i-1} + a_i p (odd i); T = row transform of w r; partials
// The passes are separate functions so that nlinv_profile_cg times exactly what a reconstruction launches.
cudaError_t q_cg_col_dir(nlinv_ctx* c, const float2* x, int newton, int iter) {
  KArgs a = base_args(c);
  a.skip = iter;
  a.src = c->T;
  a.dst = c->T;
  a.rho = x;
  a.drho = c->p;
  a.r = c->r;
  a.U = c->U;
  a.coil = c->coil;
  a.rr_part = c->rr_part;
  a.n_rr = row_geom(c, true).blocks;
  a.slot = newton;
  a.iter = iter;
  return col(c, nlv::COL_CG_DIR, a);
}

cudaError_t q_cg_row_psf(nlinv_ctx* c, int newton, int iter) {
  KArgs a = base_args(c);
  a.skip = iter;
  a.slot = newton;
  a.src = c->T;
  a.dst = c->T;
  a.mask = c->mask;
  a.dd_part = c->dd_part;
  return row(c, nlv::ROW_CG_PSF, a);
}

cudaError_t q_cg_col_adj(nlinv_ctx* c, const float2* x, float alpha, int newton, int iter) {
  KArgs a = base_args(c);
  a.skip = iter;
  a.src = c->T;
  a.dst = c->T;
  a.rho = x;
  a.coil = c->coil;
  a.zsum = c->zsum;
  a.scalars = 1;
  a.alpha = alpha;
  a.dd_part = c->dd_part;
  a.n_dd = row_geom(c, false).blocks;
  a.rr_part = c->rr_part;
  a.n_rr = row_geom(c, true).blocks;
  a.slot = newton;
  a.iter = iter;
  return col(c, nlv::COL_IFFT_ADJ_FFT, a);
}

// early: p and r may be loaded before the dependent-launch wait (false for back-to-back launches of this pass alone,
// where each launch would read what the one before writes)
cudaError_t q_cg_row_update(nlinv_ctx* c, float alpha, int newton, int iter, bool last, bool early = true) {
  KArgs a = base_args(c);
  a.skip = iter + 1;
  a.skip_after = 1;
  a.slot = newton;
  a.src_early = early ? 1 : 0;
  a.src = c->T;
  a.dst = c->T;
  a.p = c->p;
  a.r = c->r;
  a.dx = c->dx;
  a.zsum = c->zsum;
  a.alpha = alpha;
  a.rr_part = c->rr_part;
  a.n_rr = row_geom(c, true).blocks;
  a.iter = iter;
  a.last = last ? 1 : 0;
  return row(c, nlv::ROW_CG_UPDATE, a);
}

cudaError_t q_cg_iter(nlinv_ctx* c, const float2* x, float alpha, int newton, int iter) {
  cudaError_t e;
  if ((e = q_cg_col_dir(c, x, newton, iter)) != cudaSuccess) return e;
  if ((e = q_cg_row_psf(c, newton, iter)) != cudaSuccess) return e;
  if ((e = q_cg_col_adj(c, x, alpha, newton, iter)) != cudaSuccess) return e;
  return q_cg_row_update(c, alpha, newton, iter, iter == c->prm.cg_iters - 1);
}

// The CG solve of a Newton step and out = base + dx (base NULL: dx alone): one cluster launch, or one launch per pass.
cudaError_t q_cg_solve(nlinv_ctx* c, const float2* x, float alpha, int newton, const float2* base, float2* out) {
  if (!c->cluster || c->prm.cg_iters == 0) {
    cudaError_t e = cudaSuccess;
    for (int i = 0; i < c->prm.cg_iters && e == cudaSuccess; ++i) e = q_cg_iter(c, x, alpha, newton, i);
    return e == cudaSuccess ? q_cg_finish(c, base, out, newton) : e;
  }
  KArgs a = base_args(c);
  a.src = c->T;
  a.rho = x;
  a.coil = c->coil;
  a.mask = c->mask;
  a.r = c->r;
  a.x = base;
  a.dst = out;
  a.alpha = alpha;
  a.slot = newton;
  a.iter = c->prm.cg_iters;
  void* args[] = {&a};
  return launch(c, c->k->cluster, c->J, c->k->cluster_threads, c->k->cluster_smem(c->J), args, c->J);
}

// Whether the CG solves of a single frame run as one cluster launch each: the side has that kernel, the field of view is
// n/4, one block per coil makes a cluster the device can hold, and the transforms run in FP32.  Sets the kernel's limits.
bool cluster_fits(nlinv_ctx* c) {
  if (!c->k->cluster || !c->std_fov || c->tc || c->batch_lanes > 0 || c->J > nlv::kClusterMaxCoils) return false;
  const void* fn = c->k->cluster;
  int n = 0, smem_optin = 0;
  cudaFuncAttributes fa{};
  if (cudaDeviceGetAttribute(&smem_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, c->device) != cudaSuccess ||
      cudaFuncGetAttributes(&fa, fn) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  const int dyn_max = smem_optin - (int)fa.sharedSizeBytes;
  if ((size_t)dyn_max < c->k->cluster_smem(c->J)) return false;
  cudaLaunchConfig_t cfg{};
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = c->J;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  cfg.gridDim = dim3(c->J);
  cfg.blockDim = dim3(c->k->cluster_threads);
  cfg.dynamicSmemBytes = c->k->cluster_smem(c->J);
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  const bool ok =
      cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, dyn_max) == cudaSuccess &&
      cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
      cudaFuncSetAttribute(fn, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared) ==
          cudaSuccess &&
      cudaOccupancyMaxActiveClusters(&n, fn, &cfg) == cudaSuccess && n >= 1;
  if (!ok) cudaGetLastError();
  return ok;
}

// One CG iteration of a batch's frame, in six passes with q stored and Re<p, q> taken from it.  A batch keeps this
// form although the four passes above move fewer bytes: FP32 CG that ends unconverged (30 iterations at small alpha_n)
// lies between two iterates of exact CG, and any other rounding moves it there -- of the 64 frames of the uneven
// batch, two or so change their distance to the FP64 solution by more than 1.5x either way.  The batch's results stay
// what they were, bit for bit.
//   row  beta from the |r|^2 partials of the CG step before; p_c = r_c + beta p_c; T = W^-1 p_c (first axis)
//   col  drho = r_rho + beta p_rho; T = FFT_col(M (drho c_j + rho W^-1 p_c))
//   row  PSF;  col  adjoint products;  row  q = DF^H DF p + alpha p, p_rho written, Re<p, q> partials
//   vec  alpha from those; dx += alpha p, r -= alpha q, per-block partials of |r|^2
// The direction update p = r + beta p of the previous iteration is folded into the passes that first read p (beta = 0
// right after the right-hand side).
cudaError_t q_bcg_iter(nlinv_ctx* c, const float2* x, float alpha, int newton, int iter) {
  cudaError_t e;
  const bool timed = iter == 1 && newton == 0;      // the iteration that nlinv_batch_profile_cg times
  auto cg_args = [&](int step) {
    KArgs a = base_args(c);
    a.skip = iter;
    a.skip_after = 1;
    a.slot = newton;
    a.iter = iter;
    c->rec_step = timed ? step : 0;
    return a;
  };
  KArgs a = cg_args(1);
  a.src = c->p + c->plane;
  a.r = c->r + c->plane;
  if (iter > 0) {
    a.brr_part = c->brr_part;
    a.n_rr = c->vec_blocks;
  }
  a.dst = c->T;
  if ((e = row(c, nlv::ROW_BCG_DIR, a)) != cudaSuccess) return e;
  a = cg_args(2);
  a.src = c->T;
  a.dst = c->T;
  a.rho = x;
  a.drho = c->p;
  a.r = c->r;
  a.coil = c->coil;
  if ((e = col(c, nlv::COL_BCG_DIR, a)) != cudaSuccess) return e;
  a = cg_args(3);
  a.src = c->T;
  a.dst = c->T;
  a.mask = c->mask;
  if ((e = row(c, nlv::ROW_PSF, a)) != cudaSuccess) return e;
  a = cg_args(4);
  a.src = c->T;
  a.dst = c->T;
  a.rho = x;
  a.coil = c->coil;
  a.zsum = c->zsum;
  if ((e = col(c, nlv::COL_IFFT_ADJ_FFT, a)) != cudaSuccess) return e;
  a = cg_args(5);
  a.src = c->T;
  a.dst = c->q;
  a.p = c->p;
  a.r = c->r;
  a.zsum = c->zsum;
  a.alpha = alpha;
  a.pq_part = c->pq_part;
  if ((e = row(c, nlv::ROW_BCG_NORMAL, a)) != cudaSuccess) return e;
  a = cg_args(6);
  a.pq_part = c->pq_part;
  a.n_pq = row_geom(c, true).blocks;
  a.brr_part = c->brr_part;
  a.p = c->p;
  a.q = c->q;
  a.r = c->r;
  a.dx = c->dx;
  a.n2 = c->vec / 2;
  void* args[] = {&a};
  e = launch(c, (const void*)cg_step_batch, c->vec_blocks, kVecThreads, 0, args);
  c->rec_step = 0;
  return e;
}

// x += dx, after the CG solve of a batch's frame
cudaError_t q_bcg_add(nlinv_ctx* c) {
  KArgs a = base_args(c);
  a.dx = c->dx;
  a.dst = c->x;
  a.n2 = c->vec / 2;
  void* args[] = {&a};
  return launch(c, (const void*)add_batch, c->vec_blocks, kVecThreads, 0, args);
}

// Coil maps of c->x and the Newton residual r0 = y - F x with |r0| into resid[slot].
cudaError_t q_residual(nlinv_ctx* c, int slot) {
  cudaError_t e = fused_ops(c) ? q_op_prod(c, c->x, true) : q_coils(c, c->x);
  if (e == cudaSuccess && !fused_ops(c)) e = q_prod(c, c->x);
  if (e != cudaSuccess) return e;
  KArgs a = base_args(c);
  a.src = c->T;
  a.dst = c->r0;
  a.y = c->y;
  a.mask = c->mask;
  a.reduce = nlv::RED_RESID;
  a.slot = slot;
  return row(c, nlv::ROW_FFT_RESID, a);
}

// out = a X + b Y over one unknown-space vector ((1+J) planes) or, with planes = J, one data array.
cudaError_t q_axpby(nlinv_ctx* c, float2* out, float a, const float2* X, float b, const float2* Y, long planes) {
  KArgs k = base_args(c);
  k.src = X;
  k.q = Y;
  k.dst = out;
  k.alpha = a;
  k.coef = b;
  k.n2 = planes * c->plane / 2;
  void* args[] = {&k};
  const bool wide = on_boundary(out) && on_boundary(X) && on_boundary(Y);
  return launch(c, wide ? (const void*)axpby_kernel<float4> : (const void*)axpby_kernel<float2>, c->vec_blocks,
                kVecThreads, 0, args);
}

// out = DF_z d (J data planes) at the linearisation point z.
cudaError_t q_derivative_to(nlinv_ctx* c, const float2* z, const float2* d, const uint8_t* mask, float2* out) {
  cudaError_t e = fused_ops(c) ? q_op_dir(c, z, d, false) : q_coils(c, z);
  if (e == cudaSuccess && !fused_ops(c)) e = q_dir(c, z, d);
  if (e != cudaSuccess) return e;
  KArgs a = base_args(c);
  a.src = c->T;
  a.dst = out;
  a.mask = mask;
  return row(c, nlv::ROW_FFT_P_OUT, a);
}

// out = DF_z^H r (one unknown-space vector) at the linearisation point z.
cudaError_t q_adjoint_to(nlinv_ctx* c, const float2* z, const float2* r, const uint8_t* mask, float2* out) {
  cudaError_t e;
  KArgs a = base_args(c);
  if (fused_ops(c)) {
    if ((e = q_op_adj(c, z, r, mask)) != cudaSuccess) return e;
  } else {
    if ((e = q_coils(c, z)) != cudaSuccess) return e;
    a.src = r;
    a.dst = c->T;
    a.mask = mask;
    if ((e = row(c, nlv::ROW_P_IFFT, a)) != cudaSuccess) return e;
    if ((e = q_adj_col(c, z)) != cudaSuccess) return e;
  }
  a = base_args(c);
  a.src = c->T;
  a.dst = out;
  a.zsum = c->zsum;
  return row(c, nlv::ROW_FFT_W_ADJ, a);
}

// The whole reconstruction on the workspace buffers (x, xref, y, mask already in place).
cudaError_t q_reconstruct(nlinv_ctx* c) {
  const nlinv_params& P = c->prm;
  double alpha = P.alpha0;
  cudaError_t e;
  const size_t vb = c->vec * sizeof(float2);
  if (c->ckpt && (e = cudaMemcpyAsync(c->ckpt, c->x, vb, cudaMemcpyDeviceToDevice, c->stream)) != cudaSuccess) return e;
  for (int n = 0; n < P.newton_steps; ++n) {
    const float al = (float)alpha;
    if ((e = q_residual(c, n)) != cudaSuccess) return e;
    // b = DF^H r0 - alpha (x - xref) -> r = b, rr = |b|^2 and, for the first iteration, T = row transform of w b (a
    // single frame) or p = b, dx = 0 (a frame of a batch)
    const bool batch = c->batch_lanes > 0;
    KArgs a = base_args(c);
    a.src = c->r0;
    a.dst = c->T;
    a.mask = c->mask;
    if ((e = row(c, nlv::ROW_P_IFFT, a)) != cudaSuccess) return e;
    if ((e = q_adj_col(c, c->x)) != cudaSuccess) return e;
    a = base_args(c);
    a.src = c->T;
    a.zsum = c->zsum;
    a.x = c->x;
    a.xref = c->xref;
    a.r = c->r;
    a.dst = c->T;
    a.pout = c->p;
    a.dx = c->dx;
    a.alpha = al;
    a.reduce = nlv::RED_RR_INIT;
    a.slot = n;
    if ((e = row(c, batch ? nlv::ROW_BCG_RHS : nlv::ROW_CG_RHS, a)) != cudaSuccess) return e;
    for (int i = 0; i < P.cg_iters && batch; ++i)
      if ((e = q_bcg_iter(c, c->x, al, n, i)) != cudaSuccess) return e;
    if ((e = batch ? q_bcg_add(c) : q_cg_solve(c, c->x, al, n, c->x, c->x)) != cudaSuccess) return e;
    if (c->ckpt &&
        (e = cudaMemcpyAsync(c->ckpt + (size_t)(n + 1) * c->vec, c->x, vb, cudaMemcpyDeviceToDevice, c->stream)) !=
            cudaSuccess)
      return e;
    c->last_alpha = alpha;
    alpha = std::max(alpha * P.alpha_q, P.alpha_min);
  }
  return q_residual(c, P.newton_steps);
}

bool is_device_ptr(const void* p) {
  cudaPointerAttributes at{};
  if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return at.type == cudaMemoryTypeDevice || at.type == cudaMemoryTypeManaged;
}

nlinv_status check_dev(nlinv_ctx* c, const void* p, const char* name) {
  if (!p) return fail(c, NLINV_EINVAL, std::string(name) + " is NULL");
  if (!is_device_ptr(p)) return fail(c, NLINV_EINVAL, std::string(name) + " must be a device pointer");
  return NLINV_OK;
}

nlinv_status validate(const nlinv_params* p, std::string* why) {
  if (!p) { *why = "params is NULL"; return NLINV_EINVAL; }
  if (!nlinv_supported_size(p->n)) { *why = "grid side n=" + std::to_string(p->n) + " has no compiled transform"; return NLINV_EINVAL; }
  if (p->ncoils < 1 || p->ncoils > 64) { *why = "ncoils must be in 1..64"; return NLINV_EINVAL; }
  if (p->newton_steps < 1 || p->newton_steps > nlv::kMaxNewton) { *why = "newton_steps must be in 1..64"; return NLINV_EINVAL; }
  if (p->cg_iters < 0 || p->cg_iters > 100000) { *why = "cg_iters must be in 0..100000"; return NLINV_EINVAL; }
  if (!(p->alpha0 > 0) || !std::isfinite(p->alpha0)) { *why = "alpha0 must be positive"; return NLINV_EINVAL; }
  if (!(p->alpha_q > 0 && p->alpha_q <= 1)) { *why = "alpha_q must be in (0, 1]"; return NLINV_EINVAL; }
  if (!(p->alpha_min >= 0) || !std::isfinite(p->alpha_min)) { *why = "alpha_min must be >= 0"; return NLINV_EINVAL; }
  if (!(p->sobolev_a >= 0) || !std::isfinite(p->sobolev_a)) { *why = "sobolev_a must be >= 0"; return NLINV_EINVAL; }
  if (!(p->sobolev_l >= 0) || !std::isfinite(p->sobolev_l)) { *why = "sobolev_l must be >= 0"; return NLINV_EINVAL; }
  if (p->fov < 1 || p->fov > p->n / 2) { *why = "fov must be in 1..n/2"; return NLINV_EINVAL; }
  if (p->tensor_dft != 0 && p->tensor_dft != 1) { *why = "tensor_dft must be 0 or 1"; return NLINV_EINVAL; }
  if (p->tensor_dft && !nlv::find_size(p->n)->row_tc[0]) {
    *why = "tensor-core DFT stages are compiled for n = 256 and 512 only";
    return NLINV_EINVAL;
  }
  return NLINV_OK;
}

// For the timing calls: marks the CG solve of a Newton step as running and takes the rounding floor away (until the
// next right-hand side), so that every kernel does its full work.  Synchronous.
cudaError_t mark_running(nlinv_ctx* c, int newton) {
  const int running = -1;
  const nlv::Pair none = {0.f, 0.f};
  cudaError_t e = cudaMemcpy(&c->sc->cg_stop[newton], &running, sizeof(int), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemcpy(&c->sc->rr_pair, &none, sizeof(none), cudaMemcpyHostToDevice);
  return e;
}

// The same for a single frame's passes, with a CG state that none of them takes for a stopped or broken solve: what the
// passes find otherwise depends on the solve before (the cluster solve writes no partial sums at all; a diverged or
// finished one leaves NaN or zeros).  Synchronous; the context's stream is idle.
cudaError_t seed_running(nlinv_ctx* c, int newton) {
  const nlv::Pair one = {1.f, 0.f};
  const int n_dd = row_geom(c, false).blocks, n_rr = row_geom(c, true).blocks;
  const std::vector<nlv::Pair> part(std::max(n_dd, 3 * n_rr), one);
  Scalars hs{};
  cudaError_t e = mark_running(c, newton);
  if (e == cudaSuccess) e = cudaMemcpy(&hs, c->sc, sizeof(hs), cudaMemcpyDeviceToHost);
  hs.rr_i[0] = hs.rr_i[1] = hs.beta_p = one;
  if (e == cudaSuccess) e = cudaMemcpy(c->sc, &hs, sizeof(hs), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemcpy(c->dd_part, part.data(), n_dd * sizeof(one), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemcpy(c->rr_part, part.data(), 3 * n_rr * sizeof(one), cudaMemcpyHostToDevice);
  return e;
}

nlinv_status finish_call(nlinv_ctx* c, cudaError_t e, const char* where) {
  if (e != cudaSuccess) return cuda_fail(c, e, where);
  return NLINV_OK;
}

// Begin and end of an operator call: on the stream that nlinv_use_stream chose for it (taken first thing, so that a
// refused call uses the choice up too), else on the context's own.
cudaStream_t op_stream(nlinv_ctx* c) { return c->order.take(); }
cudaError_t op_begin(nlinv_ctx* c, cudaStream_t s) {
  c->launches = 0;
  return c->order.enter(s);
}
nlinv_status op_end(nlinv_ctx* c, cudaError_t e, const char* where) {
  const cudaError_t e2 = c->order.leave();
  return finish_call(c, e != cudaSuccess ? e : e2, where);
}

}  // namespace

// ---------------------------------------------------------------------------------------------- C-ABI ----
extern "C" {

int nlinv_supported_size(int n) { return nlv::find_size(n) != nullptr ? 1 : 0; }

nlinv_status nlinv_default_params(nlinv_params* p, int n, int ncoils) {
  if (!p) return NLINV_EINVAL;
  std::memset(p, 0, sizeof(*p));
  p->n = n;
  p->ncoils = ncoils;
  p->newton_steps = 7;
  p->cg_iters = 30;
  p->alpha0 = 1.0;
  p->alpha_q = 0.5;
  p->alpha_min = 0.0;
  p->sobolev_a = 220.0;
  p->sobolev_l = 32.0;
  p->fov = n / 4;
  p->use_graph = 1;
  p->tensor_dft = 0;
  return NLINV_OK;
}

}  // extern "C"

namespace {

// Twiddle tables of the context's split: twA[k2*N1 + a] = exp(-2 pi i a k2 / N) (a < N1, k2 < N2), twB likewise
// for (N2, N1).  Synchronous.
cudaError_t upload_twiddles(nlinv_ctx* c) {
  const int N = c->N, N1 = c->k->N1, N2 = c->k->N2;
  std::vector<float2> ta(N), tb(N);
  auto tw = [N](long m) {
    m %= N;
    const double t = 2.0 * 3.14159265358979323846 * (double)m / (double)N;
    return make_float2((float)std::cos(t), (float)-std::sin(t));
  };
  for (int k2 = 0; k2 < N2; ++k2)
    for (int a = 0; a < N1; ++a) ta[k2 * N1 + a] = tw((long)a * k2);
  for (int k2 = 0; k2 < N1; ++k2)
    for (int a = 0; a < N2; ++a) tb[k2 * N2 + a] = tw((long)a * k2);
  cudaError_t e = cudaMemcpy(c->twA, ta.data(), N * sizeof(float2), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemcpy(c->twB, tb.data(), N * sizeof(float2), cudaMemcpyHostToDevice);
  return e;
}

// Raises the dynamic shared-memory limit of every single-frame pass of table k for the context's shapes; false
// when one of them needs more than the device allows.
bool allow_passes(nlinv_ctx* c, const SizeKernels* k) {
  int smem_optin = 0;
  cudaDeviceGetAttribute(&smem_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, c->device);
  const SizeKernels* saved = c->k;
  c->k = k;
  const int lanes = std::max({row_geom(c, false).lanes, row_geom(c, true).lanes, row_geom(c, false, 2).lanes});
  c->k = saved;
  auto allow = [&](const void* fn, size_t need) {
    if (!fn) return true;
    cudaFuncAttributes fa{};
    if (cudaFuncGetAttributes(&fa, fn) != cudaSuccess) { cudaGetLastError(); return false; }
    const int dyn_max = smem_optin - (int)fa.sharedSizeBytes;
    if ((size_t)dyn_max < need) return false;
    if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, dyn_max) != cudaSuccess) {
      cudaGetLastError();
      return false;
    }
    return true;
  };
  bool ok = true;
  for (int m = 0; m < nlv::NUM_ROW_MODES && ok; ++m)
    ok = allow(k->row[m], k->row_smem(m, lanes)) && allow(k->row_std[m], k->row_smem(m, lanes));
  for (int m = 0; m < nlv::NUM_COL_MODES && ok; ++m)
    ok = allow(k->col[m], k->col_smem(m, c->Wc)) && allow(k->col_std[m], k->col_smem(m, c->Wc));
  return ok;
}

// Switches the context to the kernel table k (a tuning variant of its side): false, and no change, when its passes
// do not fit; rewrites the twiddle tables when the split differs.  Drops the captured graph.
bool use_variant(nlinv_ctx* c, const SizeKernels* k) {
  if (k == c->k) return true;
  if (!allow_passes(c, k)) return false;
  const bool resplit = k->N1 != c->k->N1;
  c->k = k;
  choose_carveout(c);
  if (resplit && upload_twiddles(c) != cudaSuccess) return false;
  if (c->graph) { cudaGraphExecDestroy(c->graph); c->graph = nullptr; }
  return true;
}

// Context set-up shared by nlinv_create and the frames of a batch (batch_lanes > 0: fixed row-pass block shape).
nlinv_status create_ctx(const nlinv_params* params, void* stream, int batch_lanes, nlinv_ctx** out) {
  nlinv_ctx* c = nullptr;
  if (!out) return fail(nullptr, NLINV_EINVAL, "out is NULL");
  *out = nullptr;
  std::string why;
  if (validate(params, &why) != NLINV_OK) return fail(nullptr, NLINV_EINVAL, why);
  c = new (std::nothrow) nlinv_ctx();
  if (!c) return fail(nullptr, NLINV_ENOMEM, "host allocation failed");
  c->prm = *params;
  c->N = params->n;
  c->J = params->ncoils;
  c->f = params->fov;
  c->Wc = 2 * params->fov;
  c->std_fov = 4 * params->fov == params->n;
  c->tc = params->tensor_dft != 0;
  c->plane = (long)c->N * c->N;
  c->vec = (long)(1 + c->J) * c->plane;
  c->k = nlv::find_size(c->N);
  c->batch_lanes = batch_lanes;
  cudaError_t e = cudaGetDevice(&c->device);
  if (e != cudaSuccess) { g_create_error = std::string("cudaGetDevice: ") + cudaGetErrorString(e); delete c; return NLINV_ECUDA; }
  if (stream) {
    c->stream = (cudaStream_t)stream;
  } else {
    e = cudaStreamCreateWithFlags(&c->stream, cudaStreamNonBlocking);
    if (e != cudaSuccess) { g_create_error = std::string("cudaStreamCreate: ") + cudaGetErrorString(e); delete c; return NLINV_ECUDA; }
    c->own_stream = true;
  }
  c->order.init(c->stream, c->device);
  int sms = 0;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, c->device);
  if (const char* v = std::getenv("NLINV_PDL")) c->pdl = std::strcmp(v, "0") != 0;
  c->sms = std::max(1, sms);
  c->vec_blocks = c->sms * NLV_VEC_BLOCKS_PER_SM;
  if (batch_lanes > 0)   // a frame of a batch: vector passes get blocks in proportion to its size
    c->vec_blocks = (int)std::min<long>(c->vec_blocks, std::max<long>(1, c->vec / 2 / (kVecThreads * 8)));

  // dynamic shared memory above the 48 KB default, within the device's opt-in limit
  int smem_optin = 0;
  cudaDeviceGetAttribute(&smem_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, c->device);
  // (the limit is raised to the device maximum so that contexts with different fov can share the kernels)
  std::string smem_err;
  auto allow = [&](const void* fn, size_t need) {
    cudaFuncAttributes fa{};
    if (cudaFuncGetAttributes(&fa, fn) != cudaSuccess) { smem_err = "cudaFuncGetAttributes failed"; return; }
    const int dyn_max = smem_optin - (int)fa.sharedSizeBytes;
    if ((size_t)dyn_max < need) {
      smem_err = "a pass needs " + std::to_string(need) + " bytes of dynamic shared memory, the device allows " +
                 std::to_string(dyn_max);
      return;
    }
    if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, dyn_max) != cudaSuccess)
      smem_err = "cudaFuncSetAttribute failed";
  };
  const int lanes_max = std::max({row_geom(c, false).lanes, row_geom(c, true).lanes, row_geom(c, false, 2).lanes});
  for (int m = 0; m < nlv::NUM_ROW_MODES && smem_err.empty(); ++m) {
    if (c->k->row[m]) allow(c->k->row[m], c->k->row_smem(m, lanes_max));
    if (smem_err.empty() && c->k->row_batch[m]) allow(c->k->row_batch[m], c->k->row_smem(m, lanes_max));
    if (smem_err.empty() && c->k->row_std[m]) allow(c->k->row_std[m], c->k->row_smem(m, lanes_max));
    if (smem_err.empty() && c->k->row_std_batch[m]) allow(c->k->row_std_batch[m], c->k->row_smem(m, lanes_max));
  }
  for (int m = 0; m < nlv::NUM_COL_MODES && smem_err.empty(); ++m) {
    if (c->k->col[m]) allow(c->k->col[m], c->k->col_smem(m, c->Wc));
    if (smem_err.empty() && c->k->col_batch[m]) allow(c->k->col_batch[m], c->k->col_smem(m, c->Wc));
    if (smem_err.empty() && c->k->col_std[m]) allow(c->k->col_std[m], c->k->col_smem(m, c->Wc));
    if (smem_err.empty() && c->k->col_std_batch[m]) allow(c->k->col_std_batch[m], c->k->col_smem(m, c->Wc));
  }
  if (c->tc) {
    for (int m = 0; m < nlv::NUM_ROW_MODES && smem_err.empty(); ++m) {
      if (c->k->row_tc[m]) allow(c->k->row_tc[m], c->k->row_smem_tc(m, lanes_max));
      if (smem_err.empty() && c->k->row_tc_std[m]) allow(c->k->row_tc_std[m], c->k->row_smem_tc(m, lanes_max));
    }
    for (int m = 0; m < nlv::NUM_COL_MODES && smem_err.empty(); ++m) {
      if (c->k->col_tc[m]) allow(c->k->col_tc[m], c->k->col_smem_tc(m, c->Wc));
      if (smem_err.empty() && c->k->col_tc_std[m]) allow(c->k->col_tc_std[m], c->k->col_smem_tc(m, c->Wc));
    }
  }
  if (!smem_err.empty()) {
    cudaGetLastError();
    g_create_error = smem_err;
    if (c->own_stream) cudaStreamDestroy(c->stream);
    delete c;
    return NLINV_EINVAL;
  }

  c->cluster = cluster_fits(c);
  choose_carveout(c);

  // workspace layout
  const size_t cplx = sizeof(float2);
  const size_t vecb = align_up(c->vec * cplx, 256), datab = align_up((size_t)c->J * c->plane * cplx, 256);
  const size_t Tb = align_up((size_t)c->J * c->N * c->Wc * cplx, 256);
  const size_t cb = align_up((size_t)c->J * c->Wc * c->Wc * cplx, 256);
  const size_t twb = align_up((size_t)c->N * cplx, 256);
  const size_t wb = align_up((size_t)c->plane * sizeof(float), 256);
  const size_t maskb = align_up((size_t)c->plane, 256);
  // partials sized for the largest vector grid that nlinv_autotune tries
  const int max_blocks = std::max(row_geom(c, true).blocks, std::max(c->vec_blocks, c->sms * kTuneVecMax));
  const size_t partb = align_up((size_t)max_blocks * sizeof(double), 256);
  const size_t scb = align_up(sizeof(Scalars), 256);
  const size_t tcb = c->tc ? align_up(nlv::kTcBBytes, 256) : 0;
  const bool batch = batch_lanes > 0;
  const size_t total = (batch ? 6 : 5) * vecb + 2 * datab + Tb + (batch ? 2 : 3) * cb + 2 * twb + wb + maskb +
                       (batch ? 3 : 5) * partb + scb + tcb;
  // NLINV_TEST_FAIL_ALLOC=1 (tests only): the workspace allocation reports out-of-memory without trying, so that
  // the ENOMEM path can be exercised without exhausting a GPU.
  const char* fail_alloc = std::getenv("NLINV_TEST_FAIL_ALLOC");
  e = (fail_alloc && std::strcmp(fail_alloc, "1") == 0) ? cudaErrorMemoryAllocation : cudaMalloc(&c->base, total);
  if (e != cudaSuccess) {
    cudaGetLastError();
    c->base = nullptr;
    g_create_error = "cudaMalloc of " + std::to_string(total) + " bytes failed: " + cudaGetErrorString(e);
    if (c->own_stream) cudaStreamDestroy(c->stream);
    delete c;
    return NLINV_ENOMEM;
  }
  char* b = (char*)c->base;
  auto take = [&](size_t n) { char* r = b; b += n; return r; };
  c->x = (float2*)take(vecb);
  c->xref = (float2*)take(vecb);
  c->r = (float2*)take(vecb);
  c->p = (float2*)take(vecb);
  c->dx = (float2*)take(vecb);
  if (batch) c->q = (float2*)take(vecb);
  c->y = (float2*)take(datab);
  c->r0 = (float2*)take(datab);
  c->T = (float2*)take(Tb);
  c->coil = (float2*)take(cb);
  c->zsum = (float2*)take(cb);
  if (!batch) c->U = (float2*)take(cb);
  c->twA = (float2*)take(twb);
  c->twB = (float2*)take(twb);
  c->wtab = (float*)take(wb);
  c->mask = (uint8_t*)take(maskb);
  c->partials = (double*)take(partb);
  if (batch) {
    c->pq_part = (nlv::Pair*)take(partb);
    c->brr_part = (nlv::Pair*)take(partb);
  } else {
    c->dd_part = (nlv::Pair*)take(partb);
    c->rr_part = (nlv::Pair*)take(3 * partb);
  }
  c->sc = (Scalars*)take(scb);
  if (c->tc) c->tcB = take(tcb);

  const int N = c->N;
  // Sobolev weight w(k) = (1 + a |k|^2)^(-l/2), |k|^2 = (g1^2 + g2^2) / N^2 with signed natural-order indices
  std::vector<float> wt((size_t)c->plane);
  for (int k1 = 0; k1 < N; ++k1)
    for (int k2 = 0; k2 < N; ++k2) {
      const double g1 = k1 < N / 2 ? k1 : k1 - N, g2 = k2 < N / 2 ? k2 : k2 - N;
      const double kk = (g1 * g1 + g2 * g2) / ((double)N * N);
      wt[(size_t)k1 * N + k2] = (float)std::pow(1.0 + params->sobolev_a * kk, -0.5 * params->sobolev_l);
    }
  e = cudaMemset(c->base, 0, total);
  if (e == cudaSuccess) e = upload_twiddles(c);
  if (e == cudaSuccess) e = cudaMemcpy(c->wtab, wt.data(), wt.size() * sizeof(float), cudaMemcpyHostToDevice);
  if (e == cudaSuccess && c->tc) {
    std::vector<uint16_t> bt(nlv::kTcBBytes / 2);
    nlv::host_tc_btables(bt.data());
    e = cudaMemcpy(c->tcB, bt.data(), nlv::kTcBBytes, cudaMemcpyHostToDevice);
  }
  if (e == cudaSuccess) e = cudaDeviceSynchronize();
  if (e != cudaSuccess) {
    g_create_error = std::string("context set-up: ") + cudaGetErrorString(e);
    cudaFree(c->base);
    if (c->own_stream) cudaStreamDestroy(c->stream);
    delete c;
    return NLINV_ECUDA;
  }
  *out = c;
  return NLINV_OK;
}

}  // namespace

extern "C" {

nlinv_status nlinv_create(const nlinv_params* params, void* stream, nlinv_ctx** out) {
  return create_ctx(params, stream, 0, out);
}

int nlinv_use_stream(nlinv_ctx* c, void* stream) { return c && c->order.choose((cudaStream_t)stream) ? 1 : 0; }

nlinv_status nlinv_join(nlinv_ctx* c) {
  if (!c) return NLINV_EINVAL;
  OwnStream on(c);
  NLV_TRY(on.err, "order after the last call");
  return NLINV_OK;
}

nlinv_status nlinv_destroy(nlinv_ctx* c) {
  if (!c) return NLINV_OK;
  cudaStreamSynchronize(c->stream);
  c->order.finish();
  if (c->graph) cudaGraphExecDestroy(c->graph);
  cudaFree(c->base);
  if (c->vjp_base) cudaFree(c->vjp_base);
  if (c->own_stream) cudaStreamDestroy(c->stream);
  delete c;
  return NLINV_OK;
}

nlinv_status nlinv_forward(nlinv_ctx* c, const nlinv_c32* x, const uint8_t* mask, nlinv_c32* y_out) {
  if (!c) return NLINV_EINVAL;
  const cudaStream_t on = op_stream(c);
  nlinv_status s;
  if ((s = check_dev(c, x, "x")) || (s = check_dev(c, mask, "mask")) || (s = check_dev(c, y_out, "y_out"))) return s;
  const float2* xv = (const float2*)x;
  cudaError_t e = op_begin(c, on);
  if (e == cudaSuccess) e = fused_ops(c) ? q_op_prod(c, xv, false) : q_coils(c, xv);
  if (e == cudaSuccess && !fused_ops(c)) e = q_prod(c, xv);
  if (e == cudaSuccess) {
    KArgs a = base_args(c);
    a.src = c->T;
    a.dst = (float2*)y_out;
    a.mask = mask;
    e = row(c, nlv::ROW_FFT_P_OUT, a);
  }
  return op_end(c, e, "nlinv_forward");
}

nlinv_status nlinv_derivative(nlinv_ctx* c, const nlinv_c32* x, const uint8_t* mask, const nlinv_c32* dx,
                              nlinv_c32* out) {
  if (!c) return NLINV_EINVAL;
  const cudaStream_t on = op_stream(c);
  nlinv_status s;
  if ((s = check_dev(c, x, "x")) || (s = check_dev(c, mask, "mask")) || (s = check_dev(c, dx, "dx")) ||
      (s = check_dev(c, out, "out")))
    return s;
  cudaError_t e = op_begin(c, on);
  if (e == cudaSuccess) e = q_derivative_to(c, (const float2*)x, (const float2*)dx, mask, (float2*)out);
  return op_end(c, e, "nlinv_derivative");
}

nlinv_status nlinv_adjoint(nlinv_ctx* c, const nlinv_c32* x, const uint8_t* mask, const nlinv_c32* r,
                           nlinv_c32* out) {
  if (!c) return NLINV_EINVAL;
  const cudaStream_t on = op_stream(c);
  nlinv_status s;
  if ((s = check_dev(c, x, "x")) || (s = check_dev(c, mask, "mask")) || (s = check_dev(c, r, "r")) ||
      (s = check_dev(c, out, "out")))
    return s;
  cudaError_t e = op_begin(c, on);
  if (e == cudaSuccess) e = q_adjoint_to(c, (const float2*)x, (const float2*)r, mask, (float2*)out);
  return op_end(c, e, "nlinv_adjoint");
}

nlinv_status nlinv_normal(nlinv_ctx* c, const nlinv_c32* x, const uint8_t* mask, const nlinv_c32* d, double alpha,
                          nlinv_c32* out) {
  if (!c) return NLINV_EINVAL;
  const cudaStream_t on = op_stream(c);
  nlinv_status s;
  if ((s = check_dev(c, x, "x")) || (s = check_dev(c, mask, "mask")) || (s = check_dev(c, d, "d")) ||
      (s = check_dev(c, out, "out")))
    return s;
  if (!std::isfinite(alpha)) return fail(c, NLINV_EINVAL, "alpha must be finite");
  const float2* xv = (const float2*)x;
  cudaError_t e = op_begin(c, on);
  if (e == cudaSuccess) e = fused_ops(c) ? q_op_dir(c, xv, (const float2*)d, true) : q_coils(c, xv);
  if (e == cudaSuccess && !fused_ops(c)) e = q_dir(c, xv, (const float2*)d);
  if (e == cudaSuccess) {
    KArgs a = base_args(c);
    a.src = c->T;
    a.dst = c->T;
    a.mask = mask;
    e = row(c, nlv::ROW_PSF, a);
  }
  if (e == cudaSuccess) e = q_adj_col(c, xv);
  if (e == cudaSuccess) {
    KArgs a = base_args(c);
    a.src = c->T;
    a.dst = (float2*)out;
    a.p = (const float2*)d;
    a.zsum = c->zsum;
    a.alpha = (float)alpha;
    e = row(c, nlv::ROW_FFT_W_NORMAL, a);
  }
  return op_end(c, e, "nlinv_normal");
}

nlinv_status nlinv_image(nlinv_ctx* c, const nlinv_c32* x, nlinv_c32* image_out) {
  if (!c) return NLINV_EINVAL;
  const cudaStream_t on = op_stream(c);
  nlinv_status s;
  if ((s = check_dev(c, x, "x")) || (s = check_dev(c, image_out, "image_out"))) return s;
  cudaError_t e = op_begin(c, on);
  if (e == cudaSuccess) e = q_coils(c, (const float2*)x);
  if (e == cudaSuccess) {
    KArgs a = base_args(c);
    a.rho = (const float2*)x;
    a.coil = c->coil;
    a.dst = (float2*)image_out;
    void* args[] = {&a};
    e = launch(c, (const void*)image_kernel, c->vec_blocks, kVecThreads, 0, args);
  }
  return op_end(c, e, "nlinv_image");
}

nlinv_status nlinv_simulate(nlinv_ctx* c, const nlinv_c32* rho, const nlinv_c32* coil_img, const uint8_t* mask,
                            nlinv_c32* y_out) {
  if (!c) return NLINV_EINVAL;
  const cudaStream_t on = op_stream(c);
  nlinv_status s;
  if ((s = check_dev(c, rho, "rho")) || (s = check_dev(c, coil_img, "coil_img")) ||
      (s = check_dev(c, mask, "mask")) || (s = check_dev(c, y_out, "y_out")))
    return s;
  KArgs a = base_args(c);
  a.rho = (const float2*)rho;
  a.cimg = (const float2*)coil_img;
  a.dst = c->T;
  cudaError_t e = op_begin(c, on);
  if (e == cudaSuccess) e = col(c, nlv::COL_SIM_FFT, a);
  if (e == cudaSuccess) {
    a = base_args(c);
    a.src = c->T;
    a.dst = (float2*)y_out;
    a.mask = mask;
    e = row(c, nlv::ROW_FFT_P_OUT, a);
  }
  return op_end(c, e, "nlinv_simulate");
}

nlinv_status nlinv_reconstruct(nlinv_ctx* c, const nlinv_c32* y, const uint8_t* mask, const nlinv_c32* x_ref,
                               nlinv_c32* x_inout, double* resid) {
  if (!c) return NLINV_EINVAL;
  if (!y || !mask || !x_inout) return fail(c, NLINV_EINVAL, "y, mask and x_inout must not be NULL");
  const size_t vb = c->vec * sizeof(float2), db = (size_t)c->J * c->plane * sizeof(float2);
  const bool host_x = !is_device_ptr(x_inout);
  OwnStream on(c);
  NLV_TRY(on.err, "order after the last call");
  NLV_TRY(cudaMemcpyAsync(c->y, y, db, cudaMemcpyDefault, c->stream), "copy y");
  NLV_TRY(cudaMemcpyAsync(c->mask, mask, (size_t)c->plane, cudaMemcpyDefault, c->stream), "copy mask");
  NLV_TRY(cudaMemcpyAsync(c->x, x_inout, vb, cudaMemcpyDefault, c->stream), "copy x");
  NLV_TRY(cudaMemcpyAsync(c->xref, x_ref ? (const void*)x_ref : (const void*)c->x, vb, cudaMemcpyDefault, c->stream),
          "copy x_ref");
  if (c->prm.use_graph) {
    if (!c->graph) {
      cudaGraph_t g = nullptr;
      c->launches = 0;
      NLV_TRY(cudaStreamBeginCapture(c->stream, cudaStreamCaptureModeThreadLocal), "begin capture");
      cudaError_t e = q_reconstruct(c);
      cudaError_t e2 = cudaStreamEndCapture(c->stream, &g);
      if (e != cudaSuccess || e2 != cudaSuccess) {
        if (g) cudaGraphDestroy(g);
        return cuda_fail(c, e != cudaSuccess ? e : e2, "capture reconstruction");
      }
      e = cudaGraphInstantiate(&c->graph, g, 0);
      cudaGraphDestroy(g);
      if (e != cudaSuccess) { c->graph = nullptr; return cuda_fail(c, e, "instantiate graph"); }
      c->graph_launches = c->launches;
    }
    NLV_TRY(cudaGraphLaunch(c->graph, c->stream), "graph launch");
    c->launches = c->graph_launches;
  } else {
    c->launches = 0;
    NLV_TRY(q_reconstruct(c), "reconstruction");
  }
  c->have_state = true;
  NLV_TRY(cudaMemcpyAsync(x_inout, c->x, vb, cudaMemcpyDefault, c->stream), "copy x out");
  if (resid || host_x) {
    Scalars hs{};
    NLV_TRY(cudaMemcpyAsync(&hs, c->sc, sizeof(Scalars), cudaMemcpyDeviceToHost, c->stream), "read scalars");
    NLV_TRY(cudaStreamSynchronize(c->stream), "synchronize");
    if (resid)
      for (int n = 0; n <= c->prm.newton_steps; ++n) resid[n] = hs.resid[n];
    if (hs.flags & nlv::kFlagTcTimeout) {
      int zero = 0;
      cudaMemcpy(&c->sc->flags, &zero, sizeof(int), cudaMemcpyHostToDevice);
      return fail(c, NLINV_ECUDA, "a tensor-core stage did not complete within its time limit");
    }
    if (hs.flags & 1) {
      int zero = 0;
      cudaMemcpy(&c->sc->flags, &zero, sizeof(int), cudaMemcpyHostToDevice);
      return fail(c, NLINV_EBREAKDOWN, "CG breakdown: a non-finite |r|^2 or Re<p, A p>");
    }
  }
  return NLINV_OK;
}

nlinv_status nlinv_wait(nlinv_ctx* c, double timeout_s) {
  if (!c) return NLINV_EINVAL;
  OwnStream on(c);
  NLV_TRY(on.err, "order after the last call");
  cudaEvent_t ev;
  NLV_TRY(cudaEventCreateWithFlags(&ev, cudaEventDisableTiming), "event create");
  cudaError_t e = cudaEventRecord(ev, c->stream);
  if (e != cudaSuccess) { cudaEventDestroy(ev); return cuda_fail(c, e, "event record"); }
  const auto t0 = std::chrono::steady_clock::now();
  for (;;) {
    e = cudaEventQuery(ev);
    if (e == cudaSuccess) break;
    if (e != cudaErrorNotReady) { cudaEventDestroy(ev); return cuda_fail(c, e, "wait"); }
    const double el = std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
    if (timeout_s >= 0 && el > timeout_s) {
      cudaEventDestroy(ev);
      return fail(c, NLINV_ETIMEOUT, "queued work did not finish within the time limit");
    }
    std::this_thread::sleep_for(std::chrono::microseconds(50));
  }
  cudaEventDestroy(ev);
  int flags = 0;
  NLV_TRY(cudaMemcpy(&flags, &c->sc->flags, sizeof(int), cudaMemcpyDeviceToHost), "read flags");
  if (flags & nlv::kFlagTcTimeout) {
    int zero = 0;
    NLV_TRY(cudaMemcpy(&c->sc->flags, &zero, sizeof(int), cudaMemcpyHostToDevice), "clear flags");
    return fail(c, NLINV_ECUDA, "a tensor-core stage did not complete within its time limit");
  }
  if (flags & 1) {
    int zero = 0;
    NLV_TRY(cudaMemcpy(&c->sc->flags, &zero, sizeof(int), cudaMemcpyHostToDevice), "clear flags");
    return fail(c, NLINV_EBREAKDOWN, "CG breakdown: a non-finite |r|^2 or Re<p, A p>");
  }
  return NLINV_OK;
}

nlinv_status nlinv_reconstruct_checkpoints(nlinv_ctx* c, const nlinv_c32* y, const uint8_t* mask,
                                           const nlinv_c32* x_ref, nlinv_c32* x_inout, nlinv_c32* ckpt,
                                           double* resid) {
  if (!c) return NLINV_EINVAL;
  nlinv_status s;
  if ((s = check_dev(c, y, "y")) || (s = check_dev(c, mask, "mask")) || (s = check_dev(c, x_inout, "x_inout")) ||
      (s = check_dev(c, ckpt, "ckpt")))
    return s;
  if (x_ref && (s = check_dev(c, x_ref, "x_ref"))) return s;
  const size_t vb = c->vec * sizeof(float2), db = (size_t)c->J * c->plane * sizeof(float2);
  OwnStream on(c);
  NLV_TRY(on.err, "order after the last call");
  NLV_TRY(cudaMemcpyAsync(c->y, y, db, cudaMemcpyDeviceToDevice, c->stream), "copy y");
  NLV_TRY(cudaMemcpyAsync(c->mask, mask, (size_t)c->plane, cudaMemcpyDeviceToDevice, c->stream), "copy mask");
  NLV_TRY(cudaMemcpyAsync(c->x, x_inout, vb, cudaMemcpyDeviceToDevice, c->stream), "copy x");
  NLV_TRY(cudaMemcpyAsync(c->xref, x_ref ? (const void*)x_ref : (const void*)c->x, vb, cudaMemcpyDeviceToDevice,
                          c->stream), "copy x_ref");
  c->launches = 0;
  c->ckpt = (float2*)ckpt;
  const cudaError_t e = q_reconstruct(c);
  c->ckpt = nullptr;
  NLV_TRY(e, "reconstruction");
  c->have_state = true;
  NLV_TRY(cudaMemcpyAsync(x_inout, c->x, vb, cudaMemcpyDeviceToDevice, c->stream), "copy x out");
  if (resid) {
    Scalars hs{};
    NLV_TRY(cudaMemcpyAsync(&hs, c->sc, sizeof(Scalars), cudaMemcpyDeviceToHost, c->stream), "read scalars");
    NLV_TRY(cudaStreamSynchronize(c->stream), "synchronize");
    for (int n = 0; n <= c->prm.newton_steps; ++n) resid[n] = hs.resid[n];
    if (hs.flags & 1) {
      int zero = 0;
      cudaMemcpy(&c->sc->flags, &zero, sizeof(int), cudaMemcpyHostToDevice);
      return fail(c, NLINV_EBREAKDOWN, "CG breakdown: a non-finite |r|^2 or Re<p, A p>");
    }
  }
  return NLINV_OK;
}

nlinv_status nlinv_reconstruct_vjp(nlinv_ctx* c, const nlinv_c32* y, const uint8_t* mask, const nlinv_c32* ckpt,
                                   const nlinv_c32* grad_x, int tied, nlinv_c32* grad_y, nlinv_c32* grad_x0,
                                   nlinv_c32* grad_xref) {
  if (!c) return NLINV_EINVAL;
  nlinv_status s;
  if ((s = check_dev(c, y, "y")) || (s = check_dev(c, mask, "mask")) || (s = check_dev(c, ckpt, "ckpt")) ||
      (s = check_dev(c, grad_x, "grad_x")) || (s = check_dev(c, grad_y, "grad_y")) ||
      (s = check_dev(c, grad_x0, "grad_x0")))
    return s;
  if (grad_xref && (s = check_dev(c, grad_xref, "grad_xref"))) return s;
  const nlinv_params& P = c->prm;
  const long J = c->J, V = 1 + J;
  const size_t vb = c->vec * sizeof(float2), db = (size_t)J * c->plane * sizeof(float2);
  if (!c->vjp_base) {   // g, dx_n, one adjoint result, dL/dx_ref; s and DF_x u (data arrays)
    cudaError_t e = cudaMalloc(&c->vjp_base, 4 * vb + 2 * db);
    if (e != cudaSuccess) {
      cudaGetLastError();
      c->vjp_base = nullptr;
      return fail(c, NLINV_ENOMEM, "nlinv_reconstruct_vjp: scratch allocation failed");
    }
  }
  float2* g = (float2*)c->vjp_base;
  float2* dxn = g + c->vec;
  float2* tmp = dxn + c->vec;
  float2* gref = tmp + c->vec;
  float2* sres = gref + c->vec;
  float2* v = sres + J * c->plane;
  const float2* X = (const float2*)ckpt;
  c->launches = 0;
  OwnStream on(c);
  NLV_TRY(on.err, "order after the last call");
  NLV_TRY(cudaMemcpyAsync(c->y, y, db, cudaMemcpyDeviceToDevice, c->stream), "copy y");
  NLV_TRY(cudaMemcpyAsync(c->mask, mask, (size_t)c->plane, cudaMemcpyDeviceToDevice, c->stream), "copy mask");
  NLV_TRY(cudaMemcpyAsync(g, grad_x, vb, cudaMemcpyDeviceToDevice, c->stream), "copy grad_x");
  NLV_TRY(cudaMemsetAsync(grad_y, 0, db, c->stream), "clear grad_y");
  NLV_TRY(cudaMemsetAsync(gref, 0, vb, c->stream), "clear dL/dx_ref");
  std::vector<double> alphas(P.newton_steps);
  double al = P.alpha0;
  for (int n = 0; n < P.newton_steps; ++n) {
    alphas[n] = al;
    al = std::max(al * P.alpha_q, P.alpha_min);
  }
  cudaError_t e = cudaSuccess;
  for (int k = P.newton_steps - 1; k >= 0 && e == cudaSuccess; --k) {
    const float alpha = (float)alphas[k];
    const float2* xk = X + (size_t)k * c->vec;
    e = cudaMemcpyAsync(c->x, xk, vb, cudaMemcpyDeviceToDevice, c->stream);
    if (e == cudaSuccess) e = q_axpby(c, dxn, 1.f, xk + c->vec, -1.f, xk, V);
    // r0 = y - F x_k, then s = r0 - DF_x dx_k (both as "data minus masked transform" row passes)
    if (e == cudaSuccess) e = q_coils(c, c->x);
    if (e == cudaSuccess) e = q_prod(c, c->x);
    if (e == cudaSuccess) {
      KArgs a = base_args(c);
      a.src = c->T; a.dst = c->r0; a.y = c->y; a.mask = c->mask;
      e = row(c, nlv::ROW_FFT_RESID, a);
    }
    if (e == cudaSuccess) e = q_dir(c, c->x, dxn);
    if (e == cudaSuccess) {
      KArgs a = base_args(c);
      a.src = c->T; a.dst = sres; a.y = c->r0; a.mask = c->mask;
      e = row(c, nlv::ROW_FFT_RESID, a);
    }
    // u = (DF^H DF + alpha)^-1 g by the reconstruction's CG (u in c->dx)
    if (e == cudaSuccess) {
      KArgs a = base_args(c);
      a.src = g; a.r = c->r; a.n2 = c->vec / 2; a.reduce = nlv::RED_RR_INIT;
      a.slot = k;
      void* args[] = {&a};
      e = launch(c, (const void*)cg_init_kernel, c->vec_blocks, kVecThreads, 0, args);
    }
    if (e == cudaSuccess) {      // T = row transform of w r, which the first iteration starts from
      KArgs a = base_args(c);
      a.src = c->r + c->plane; a.dst = c->T;
      e = row(c, nlv::ROW_W_IFFT, a);
    }
    if (e == cudaSuccess) e = q_cg_solve(c, c->x, alpha, k, nullptr, c->dx);
    // v = DF_x u; dL/dy += v; dL/dx_ref += alpha u
    if (e == cudaSuccess) e = q_dir(c, c->x, c->dx);
    if (e == cudaSuccess) {
      KArgs a = base_args(c);
      a.src = c->T; a.dst = v; a.mask = c->mask;
      e = row(c, nlv::ROW_FFT_P_OUT, a);
    }
    if (e == cudaSuccess) e = q_axpby(c, (float2*)grad_y, 1.f, (const float2*)grad_y, 1.f, v, J);
    if (e == cudaSuccess) e = q_axpby(c, gref, 1.f, gref, alpha, c->dx, V);
    // g <- DF_u^H s - DF_dx^H v
    if (e == cudaSuccess) e = q_adjoint_to(c, c->dx, sres, c->mask, tmp);
    if (e == cudaSuccess) e = q_adjoint_to(c, dxn, v, c->mask, g);
    if (e == cudaSuccess) e = q_axpby(c, g, 1.f, tmp, -1.f, g, V);
  }
  // dL/dx_0 (plus dL/dx_ref when the reference is the start value)
  if (e == cudaSuccess) e = q_axpby(c, (float2*)grad_x0, 1.f, g, tied ? 1.f : 0.f, gref, V);
  if (e == cudaSuccess && grad_xref) e = cudaMemcpyAsync(grad_xref, gref, vb, cudaMemcpyDeviceToDevice, c->stream);
  return finish_call(c, e, "nlinv_reconstruct_vjp");
}

nlinv_status nlinv_profile_cg(nlinv_ctx* c, int reps, double* ms_out) {
  if (!c) return NLINV_EINVAL;
  if (reps < 1 || !ms_out) return fail(c, NLINV_EINVAL, "reps must be >= 1 and ms_out non-NULL");
  if (!c->have_state) return fail(c, NLINV_EINVAL, "run nlinv_reconstruct before nlinv_profile_cg");
  OwnStream on(c);
  NLV_TRY(on.err, "order after the last call");
  NLV_TRY(cudaStreamSynchronize(c->stream), "synchronize");      // a reconstruction may still be running
  NLV_TRY(seed_running(c, nlv::kMaxNewton), "mark the solve running");
  cudaEvent_t ev[2];
  for (int i = 0; i < 2; ++i) NLV_TRY(cudaEventCreate(&ev[i]), "event create");
  const float al = (float)c->last_alpha;
  // pass k of the CG iteration, reps launches back to back between two events: its steady-state launch duration
  // (consecutive launches overlap ramp and drain through the dependent launch, as in a graph replay).  The CG update
  // pass alternates between the iteration that updates dx and the one that does not.
  auto one = [&](int k, int it) -> cudaError_t {
    switch (k) {
      case 0: return q_cg_col_dir(c, c->x, nlv::kMaxNewton, 2);
      case 1: return q_cg_row_psf(c, nlv::kMaxNewton, 2);
      case 2: return q_cg_col_adj(c, c->x, al, nlv::kMaxNewton, 2);
      default: return q_cg_row_update(c, al, nlv::kMaxNewton, 2 + (it & 1), false, false);
    }
  };
  cudaError_t e = cudaSuccess;
  double ms4[4] = {};
  for (int k = 0; k < 4 && e == cudaSuccess; ++k) {
    e = cudaEventRecord(ev[0], c->stream);
    for (int it = 0; it < reps && e == cudaSuccess; ++it) e = one(k, it);
    if (e == cudaSuccess) e = cudaEventRecord(ev[1], c->stream);
    if (e == cudaSuccess) e = cudaEventSynchronize(ev[1]);
    float ms = 0.f;
    if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, ev[0], ev[1]);
    ms4[k] = ms / reps;
    if (e == cudaSuccess) e = seed_running(c, nlv::kMaxNewton);
  }
  for (int i = 0; i < 2; ++i) cudaEventDestroy(ev[i]);
  if (e != cudaSuccess) return cuda_fail(c, e, "nlinv_profile_cg");
  const double six[kProfileSteps] = {0.0, ms4[0], ms4[1], ms4[2], 0.0, ms4[3]};   // the update pass does [0] and [4] too
  std::copy(six, six + kProfileSteps, ms_out);
  return NLINV_OK;
}

long nlinv_last_launch_count(const nlinv_ctx* c) { return c ? c->launches : -1; }

nlinv_status nlinv_cg_stops(nlinv_ctx* c, int* out, int len) {
  if (!c) return NLINV_EINVAL;
  if (!out || len < c->prm.newton_steps) return fail(c, NLINV_EINVAL, "out must hold newton_steps entries");
  if (!c->have_state) return fail(c, NLINV_EINVAL, "no reconstruction has run on this context");
  OwnStream on(c);
  NLV_TRY(on.err, "order after the last call");
  Scalars hs{};
  NLV_TRY(cudaMemcpyAsync(&hs, c->sc, sizeof(Scalars), cudaMemcpyDeviceToHost, c->stream), "read scalars");
  NLV_TRY(cudaStreamSynchronize(c->stream), "synchronize");
  for (int n = 0; n < c->prm.newton_steps; ++n) out[n] = hs.cg_stop[n];
  return NLINV_OK;
}

nlinv_status nlinv_set_shapes(nlinv_ctx* c, const nlinv_tuning* t) {
  if (!c) return NLINV_EINVAL;
  if (!t) return fail(c, NLINV_EINVAL, "t is NULL");
  if (c->batch_lanes > 0) return fail(c, NLINV_EINVAL, "batch frames keep the batch's shapes");
  if (t->vec_blocks_per_sm < 1 || t->vec_blocks_per_sm > kTuneVecMax)
    return fail(c, NLINV_EINVAL, "vec_blocks_per_sm must be in 1..8");
  if (t->row_blocks_per_sm < 1 || t->row_blocks_per_sm > 3) return fail(c, NLINV_EINVAL, "row_blocks_per_sm must be in 1..3");
  const SizeKernels* variants[8];
  const int nvar = nlv::size_variants(c->N, variants, 8);
  const SizeKernels* pick = nullptr;
  for (int v = 0; v < nvar && !pick; ++v)
    if (variants[v]->N1 == t->split_n1 && variants[v]->col_lanes == t->col_strip) pick = variants[v];
  if (!pick) return fail(c, NLINV_EINVAL, "no compiled transform with that split and column strip for this n");
  if (c->tc && pick != variants[0]) return fail(c, NLINV_EINVAL, "the tensor-core passes keep the compiled split and strips");
  const int saved_rc = c->row_ctas_per_sm;
  c->row_ctas_per_sm = t->row_blocks_per_sm;
  if (!use_variant(c, pick) || !allow_passes(c, c->k)) {
    c->row_ctas_per_sm = saved_rc;
    choose_carveout(c);
    return fail(c, NLINV_EINVAL, "the passes of these shapes do not fit in shared memory");
  }
  c->vec_blocks = c->sms * t->vec_blocks_per_sm;
  c->pdl = t->pdl != 0;
  choose_carveout(c);
  if (c->graph) { cudaGraphExecDestroy(c->graph); c->graph = nullptr; }
  return NLINV_OK;
}

nlinv_status nlinv_autotune(nlinv_ctx* c, const nlinv_c32* y, const uint8_t* mask, const nlinv_c32* x0, int reps,
                            nlinv_tuning* out, nlinv_tuning* table, int table_len) {
  if (!c) return NLINV_EINVAL;
  nlinv_status st;
  if ((st = check_dev(c, y, "y")) || (st = check_dev(c, mask, "mask")) || (st = check_dev(c, x0, "x0"))) return st;
  if (reps < 1 || reps > 1000) return fail(c, NLINV_EINVAL, "reps must be in 1..1000");
  if (c->batch_lanes > 0) return fail(c, NLINV_EINVAL, "batch frames are not tuned one by one");
  if (table && table_len < kTuneMaxCandidates)
    return fail(c, NLINV_EINVAL, "table needs " + std::to_string(kTuneMaxCandidates) + " entries");
  struct Key { int dev, n, J, fov, newton, cg, tc; };
  struct Entry { Key k; const SizeKernels* kern; nlinv_tuning t; std::vector<nlinv_tuning> all; };
  static std::mutex mtx;
  static std::vector<Entry> cache;
  const Key key{c->device, c->N, c->J, c->f, c->prm.newton_steps, c->prm.cg_iters, c->tc ? 1 : 0};
  auto same = [&](const Key& a) {
    return a.dev == key.dev && a.n == key.n && a.J == key.J && a.fov == key.fov && a.newton == key.newton &&
           a.cg == key.cg && a.tc == key.tc;
  };
  // the context's launch shapes as one tuning record (ms_per_frame and stage filled by the caller)
  auto shape = [&]() {
    nlinv_tuning t{};
    t.vec_blocks_per_sm = c->vec_blocks / c->sms;
    t.pdl = c->pdl ? 1 : 0;
    t.split_n1 = c->k->N1;
    t.col_strip = c->k->col_lanes;
    t.row_blocks_per_sm = c->row_ctas_per_sm;
    return t;
  };
  auto set_shapes = [&](int vbk, bool pdl, int row_ctas) {
    c->vec_blocks = c->sms * vbk;
    c->pdl = pdl;
    c->row_ctas_per_sm = row_ctas;
    choose_carveout(c);
    if (c->graph) { cudaGraphExecDestroy(c->graph); c->graph = nullptr; }
  };
  {
    std::lock_guard<std::mutex> lk(mtx);
    for (const Entry& e : cache)
      if (same(e.k)) {
        if (!use_variant(c, e.kern)) return fail(c, NLINV_ECUDA, "nlinv_autotune: cached variant does not fit");
        set_shapes(e.t.vec_blocks_per_sm, e.t.pdl != 0, e.t.row_blocks_per_sm);
        if (out) *out = e.t;
        if (table) {
          for (int i = 0; i < table_len; ++i) table[i] = nlinv_tuning{};
          std::copy(e.all.begin(), e.all.end(), table);
        }
        return NLINV_OK;
      }
  }
  OwnStream on(c);
  NLV_TRY(on.err, "order after the last call");
  // Whole reconstructions of the caller's frame, replayed as graphs (each replay starts from the same start value):
  // only the whole graph shows how neighbouring passes overlap, and an all-zero workspace times differently from
  // data.  Every timed replay starts with a cold L2 (a write of twice its size outside the events), as a frame of a
  // series does after the rest of an application has run.
  const size_t vb = c->vec * sizeof(float2), db = (size_t)c->J * c->plane * sizeof(float2);
  NLV_TRY(cudaMemcpyAsync(c->y, y, db, cudaMemcpyDeviceToDevice, c->stream), "copy y");
  NLV_TRY(cudaMemcpyAsync(c->mask, mask, (size_t)c->plane, cudaMemcpyDeviceToDevice, c->stream), "copy mask");
  int l2 = 0;
  cudaDeviceGetAttribute(&l2, cudaDevAttrL2CacheSize, c->device);
  const size_t flush_bytes = std::max<size_t>(2 * (size_t)l2, 64u << 20);
  void* flush = nullptr;
  if (cudaMalloc(&flush, flush_bytes) != cudaSuccess) {
    cudaGetLastError();
    return fail(c, NLINV_ENOMEM, "nlinv_autotune: L2 flush buffer allocation failed");
  }
  cudaEvent_t ev[2];
  for (int i = 0; i < 2; ++i) {
    cudaError_t ee = cudaEventCreate(&ev[i]);
    if (ee != cudaSuccess) { cudaFree(flush); return cuda_fail(c, ee, "event create"); }
  }
  cudaError_t e = cudaSuccess;
  // ms per frame of the context's current shapes
  auto time_frame = [&]() -> double {
    if (e != cudaSuccess) return 1e30;
    e = cudaMemcpyAsync(c->x, x0, vb, cudaMemcpyDeviceToDevice, c->stream);
    if (e == cudaSuccess) e = cudaMemcpyAsync(c->xref, x0, vb, cudaMemcpyDeviceToDevice, c->stream);
    if (e != cudaSuccess) return 1e30;
    cudaGraph_t g = nullptr;
    cudaGraphExec_t ge = nullptr;
    e = cudaStreamBeginCapture(c->stream, cudaStreamCaptureModeThreadLocal);
    if (e != cudaSuccess) return 1e30;
    cudaError_t e1 = q_reconstruct(c);
    cudaError_t e2 = cudaStreamEndCapture(c->stream, &g);
    e = e1 != cudaSuccess ? e1 : e2;
    if (e == cudaSuccess) e = cudaGraphInstantiate(&ge, g, 0);
    if (g) cudaGraphDestroy(g);
    double tot = 0.0;
    for (int r = 0; r <= reps && e == cudaSuccess; ++r) {          // r = 0: warm-up
      e = cudaMemcpyAsync(c->x, x0, vb, cudaMemcpyDeviceToDevice, c->stream);
      if (e == cudaSuccess) e = cudaMemsetAsync(flush, r & 0xff, flush_bytes, c->stream);
      if (e == cudaSuccess) e = cudaEventRecord(ev[0], c->stream);
      if (e == cudaSuccess) e = cudaGraphLaunch(ge, c->stream);
      if (e == cudaSuccess) e = cudaEventRecord(ev[1], c->stream);
      if (e == cudaSuccess) e = cudaEventSynchronize(ev[1]);
      float ms = 0.f;
      if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, ev[0], ev[1]);
      if (r > 0) tot += ms;
    }
    if (ge) cudaGraphExecDestroy(ge);
    return e == cudaSuccess ? tot / reps : 1e30;
  };
  Entry ent{};
  // Coordinate descent, one launch-shape dimension per stage, each from the best shapes of the stages before:
  // stage 0 the four-step split of the transforms, 1 the column-strip width, 2 the row-pass blocks per SM, 3 the
  // vector-pass blocks per SM with dependent launch off and on.  Within a stage a candidate replaces the incumbent
  // only when it is kTuneMargin faster (closer shapes swap places with small changes of conditions).
  const SizeKernels* variants[8];
  const int nvar = nlv::size_variants(c->N, variants, 8);
  const SizeKernels* base = c->k;
  auto stage = [&](int id, const std::vector<std::function<bool()>>& cands) {
    // cands[0] restores the incumbent; each candidate applies its shapes and returns false if they do not fit
    double inc_ms = -1.0;
    int best = 0;
    double best_ms = 1e30;
    for (size_t i = 0; i < cands.size() && e == cudaSuccess; ++i) {
      if (!cands[i]()) continue;
      nlinv_tuning t = shape();
      t.ms_per_frame = time_frame();
      t.stage = id;
      if (e != cudaSuccess) break;
      ent.all.push_back(t);
      if (i == 0) inc_ms = t.ms_per_frame;
      if (t.ms_per_frame < best_ms) { best_ms = t.ms_per_frame; best = (int)i; }
    }
    if (inc_ms > 0.0 && best_ms > (1.0 - kTuneMargin) * inc_ms) best = 0;
    if (e == cudaSuccess) cands[best]();
  };
  // stage 0: splits (the default table, and the alternative split if the side has one; the tensor-core passes
  // exist for the default split only)
  {
    std::vector<std::function<bool()>> cands{[&] { return use_variant(c, base); }};
    for (int v = 1; v < nvar && !c->tc; ++v)
      if (variants[v]->N1 != base->N1) cands.push_back([&, v] { return use_variant(c, variants[v]); });
    stage(0, cands);
  }
  // stage 1: column strips of the chosen split (variants of the default split only)
  if (c->k->N1 == base->N1 && !c->tc) {
    std::vector<std::function<bool()>> cands{[&] { return use_variant(c, base); }};
    for (int v = 1; v < nvar; ++v)
      if (variants[v]->N1 == base->N1 && variants[v]->col_lanes != base->col_lanes)
        cands.push_back([&, v] { return use_variant(c, variants[v]); });
    stage(1, cands);
  }
  // stage 2: row-pass blocks per SM
  {
    const int inc = c->row_ctas_per_sm;
    std::vector<std::function<bool()>> cands{[&, inc] { set_shapes(c->vec_blocks / c->sms, c->pdl, inc); return true; }};
    for (int rc : {1, 2, 3})
      if (rc != inc)
        cands.push_back([&, rc] { set_shapes(c->vec_blocks / c->sms, c->pdl, rc); return allow_passes(c, c->k); });
    stage(2, cands);
  }
  // stage 3: vector-pass blocks per SM x dependent launch
  {
    const int ivb = c->vec_blocks / c->sms;
    const bool ipdl = c->pdl;
    std::vector<std::function<bool()>> cands{[&, ivb, ipdl] { set_shapes(ivb, ipdl, c->row_ctas_per_sm); return true; }};
    for (int pdl = 0; pdl < 2; ++pdl)
      for (int vbk : {2, 4, kTuneVecMax})
        if (vbk != ivb || (pdl != 0) != ipdl)
          cands.push_back([&, vbk, pdl] { set_shapes(vbk, pdl != 0, c->row_ctas_per_sm); return true; });
    stage(3, cands);
  }
  for (int i = 0; i < 2; ++i) cudaEventDestroy(ev[i]);
  cudaFree(flush);
  int zero = 0;   // the timing runs are not the caller's results: drop any flag they raised
  if (e == cudaSuccess) e = cudaMemcpy(&c->sc->flags, &zero, sizeof(int), cudaMemcpyHostToDevice);
  if (e != cudaSuccess) return cuda_fail(c, e, "nlinv_autotune");
  ent.k = key;
  ent.kern = c->k;
  ent.t = shape();
  // the chosen shapes' own measurement: the last stage's entry for them
  for (const nlinv_tuning& t : ent.all)
    if (t.vec_blocks_per_sm == ent.t.vec_blocks_per_sm && t.pdl == ent.t.pdl && t.split_n1 == ent.t.split_n1 &&
        t.col_strip == ent.t.col_strip && t.row_blocks_per_sm == ent.t.row_blocks_per_sm)
      ent.t.ms_per_frame = t.ms_per_frame, ent.t.stage = t.stage;
  {
    std::lock_guard<std::mutex> lk(mtx);
    cache.push_back(ent);
  }
  if (out) *out = ent.t;
  if (table) {
    for (int i = 0; i < table_len; ++i) table[i] = nlinv_tuning{};
    std::copy(ent.all.begin(), ent.all.end(), table);
  }
  return NLINV_OK;
}

}  // extern "C"

// ---------------------------------------------------------------------------------------------- batches ----
struct nlinv_batch {
  nlinv_params prm{};
  std::vector<nlinv_ctx*> frames;           // per-frame workspaces (they never launch by themselves)
  std::vector<std::vector<int>> groups;     // frame indices per grid side
  cudaStream_t stream = nullptr;
  bool own_stream = false;
  std::vector<cudaStream_t> gstream;        // branch stream per group (group 0 runs on `stream`)
  cudaEvent_t ev_fork = nullptr;
  std::vector<cudaEvent_t> ev_join;
  void* tables = nullptr;                   // device: per-launch frame arguments and block offsets
  struct Launch {
    int group;
    const void* fn;
    int grid, block;
    size_t smem;
    nlv::BatchArgs args;
    int step;                               // nlinv_ctx::Rec::step
  };
  std::vector<Launch> launches;
  cudaGraphExec_t graph = nullptr;
  bool have_state = false;                  // a reconstruction has filled the workspaces
  bool pdl = true;
  bool multi = false;                       // one launch per pass for all sides the multi-side kernels cover
                                            // (NLINV_BATCH_MULTI=1; measured slower, see nlinv_batch_create)
};

namespace {

void batch_free(nlinv_batch* b) {
  if (!b) return;
  if (b->stream) cudaStreamSynchronize(b->stream);
  if (b->graph) cudaGraphExecDestroy(b->graph);
  for (size_t g = 1; g < b->gstream.size(); ++g)
    if (b->gstream[g]) cudaStreamDestroy(b->gstream[g]);
  for (cudaEvent_t e : b->ev_join)
    if (e) cudaEventDestroy(e);
  if (b->ev_fork) cudaEventDestroy(b->ev_fork);
  if (b->tables) cudaFree(b->tables);
  for (nlinv_ctx* c : b->frames) nlinv_destroy(c);
  if (b->own_stream && b->stream) cudaStreamDestroy(b->stream);
  delete b;
}

// The multi-side kernel (kernels.cuh, "batches of several sides") that runs the batched pass fn of side k for frames of
// every side, and its dynamic shared memory (0 and fn itself when fn is a vector pass, which knows no side).
const void* multi_kernel(const SizeKernels* k, const void* fn, size_t* smem) {
  const nlv::MultiKernels* mk = nlv::multi_kernels();
  for (int m = 0; m < nlv::NUM_ROW_MODES; ++m) {
    if (fn == k->row_batch[m]) { *smem = mk->row_smem[m]; return mk->row[m]; }
    if (k->row_std_batch[m] && fn == k->row_std_batch[m]) { *smem = mk->row_smem[m]; return mk->row_std[m]; }
  }
  for (int m = 0; m < nlv::NUM_COL_MODES; ++m) {
    if (fn == k->col_batch[m]) { *smem = mk->col_smem[m]; return mk->col[m]; }
    if (k->col_std_batch[m] && fn == k->col_std_batch[m]) { *smem = mk->col_smem[m]; return mk->col_std[m]; }
  }
  *smem = 0;
  return fn;
}

// One batched launch on stream st (with the batch's dependent-launch setting).
cudaError_t launch_batched(nlinv_batch* b, nlinv_batch::Launch& bl, cudaStream_t st) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(bl.grid);
  cfg.blockDim = dim3(bl.block);
  cfg.dynamicSmemBytes = bl.smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = b->pdl ? 1 : 0;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  void* args[] = {&bl.args};
  return cudaLaunchKernelExC(&cfg, bl.fn, args);
}

nlinv_status batch_fail(nlinv_batch* b, nlinv_status st, const std::string& msg) {
  g_create_error = msg;
  batch_free(b);
  return st;
}

}  // namespace

extern "C" {

nlinv_status nlinv_batch_create(const nlinv_params* params, int nframes, const nlinv_frame_desc* frames,
                                void* stream, nlinv_batch** out) {
  if (!out) return fail(nullptr, NLINV_EINVAL, "out is NULL");
  *out = nullptr;
  if (!params || !frames || nframes < 1 || nframes > 4096)
    return fail(nullptr, NLINV_EINVAL, "params, frames and 1 <= nframes <= 4096 are required");
  nlinv_batch* b = new (std::nothrow) nlinv_batch();
  if (!b) return fail(nullptr, NLINV_ENOMEM, "host allocation failed");
  b->prm = *params;
  if (const char* v = std::getenv("NLINV_PDL")) b->pdl = std::strcmp(v, "0") != 0;
  if (const char* v = std::getenv("NLINV_BATCH_MULTI")) b->multi = std::strcmp(v, "0") != 0;
  cudaError_t e = cudaSuccess;
  if (stream) {
    b->stream = (cudaStream_t)stream;
  } else {
    e = cudaStreamCreateWithFlags(&b->stream, cudaStreamNonBlocking);
    if (e != cudaSuccess) return batch_fail(b, NLINV_ECUDA, std::string("cudaStreamCreate: ") + cudaGetErrorString(e));
    b->own_stream = true;
  }
  // one workspace per frame, grouped by grid side
  std::vector<int> sides;
  for (int i = 0; i < nframes; ++i) {
    nlinv_params fp = *params;
    fp.n = frames[i].n;
    fp.ncoils = frames[i].ncoils;
    fp.fov = frames[i].n / 4;
    fp.use_graph = 0;
    fp.tensor_dft = 0;        // batches run the FP32 transforms
    const SizeKernels* k = nlv::find_size(fp.n);
    if (!k) return batch_fail(b, NLINV_EINVAL, "frame " + std::to_string(i) + ": unsupported grid side");
    nlinv_ctx* c = nullptr;
    const nlinv_status st = create_ctx(&fp, b->stream, nlv::kRowMaxThreads / k->tl, &c);
    if (st != NLINV_OK) return batch_fail(b, st, "frame " + std::to_string(i) + ": " + g_create_error);
    b->frames.push_back(c);
    // frames of the sides the multi-side kernels cover form one group (side key 0); other sides one group each
    const int key = (b->multi && nlv::multi_side(fp.n)) ? 0 : fp.n;
    c->batch_split = key != 0;
    size_t g = 0;
    while (g < sides.size() && sides[g] != key) ++g;
    if (g == sides.size()) {
      sides.push_back(key);
      b->groups.emplace_back();
    }
    b->groups[g].push_back(i);
  }
  int sms = 1, dev = 0, smem_optin = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  cudaDeviceGetAttribute(&smem_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  // the launch sequence of every frame, merged launch by launch within each group
  std::vector<std::vector<nlinv_ctx::Rec>> recs(nframes);
  for (int i = 0; i < nframes; ++i) {
    nlinv_ctx* c = b->frames[i];
    c->rec = &recs[i];
    e = q_reconstruct(c);
    c->rec = nullptr;
    if (e != cudaSuccess) return batch_fail(b, NLINV_ECUDA, std::string("recording: ") + cudaGetErrorString(e));
  }
  std::vector<char> host;
  std::vector<size_t> arg_off, first_off, stop_off;
  for (size_t g = 0; g < b->groups.size(); ++g) {
    const std::vector<int>& fr = b->groups[g];
    const size_t L = recs[fr[0]].size();
    const SizeKernels* k = b->frames[fr[0]]->k;
    for (int i : fr)
      if (recs[i].size() != L) return batch_fail(b, NLINV_EINVAL, "frames of one grid side differ in schedule");
    const bool multi = sides[g] == 0;
    stop_off.push_back((host.size() + 15) / 16 * 16);
    host.resize(stop_off.back() + fr.size() * sizeof(const int*));
    for (size_t t = 0; t < fr.size(); ++t) {
      const int* at = b->frames[fr[t]]->sc->cg_stop;      // a device address
      std::memcpy(host.data() + stop_off.back() + t * sizeof(at), &at, sizeof(at));
    }
    for (size_t l = 0; l < L; ++l) {
      nlinv_batch::Launch bl{};
      bl.group = (int)g;
      bl.step = recs[fr[0]][l].step;
      size_t msmem = 0;
      bl.fn = multi ? multi_kernel(k, recs[fr[0]][l].fn, &msmem) : recs[fr[0]][l].fn;
      if (!bl.fn) return batch_fail(b, NLINV_EINVAL, "internal: no batched form of a pass");
      size_t off = (host.size() + 15) / 16 * 16;
      host.resize(off + fr.size() * sizeof(KArgs));
      arg_off.push_back(off);
      std::vector<int> first(fr.size() + 1, 0);
      bl.block = 0;
      for (size_t t = 0; t < fr.size(); ++t) {
        const nlinv_ctx::Rec& r = recs[fr[t]][l];
        size_t ms = 0;
        const void* same = multi ? multi_kernel(b->frames[fr[t]]->k, r.fn, &ms) : r.fn;
        if (same != bl.fn || (!multi && r.block != recs[fr[0]][l].block))
          return batch_fail(b, NLINV_EINVAL, "frames of one group differ in pass shapes");
        std::memcpy(host.data() + off + t * sizeof(KArgs), &r.args, sizeof(KArgs));
        first[t + 1] = first[t] + r.grid;
        bl.smem = multi ? msmem : std::max(bl.smem, r.smem);
        bl.block = std::max(bl.block, r.block);
      }
      if (multi) {   // the multi-side kernels run fixed block shapes
        const nlv::MultiKernels* mk = nlv::multi_kernels();
        bool is_col = false;
        for (int m = 0; m < nlv::NUM_COL_MODES; ++m)
          is_col = is_col || bl.fn == mk->col[m] || (mk->col_std[m] && bl.fn == mk->col_std[m]);
        bool is_row = false;
        for (int m = 0; m < nlv::NUM_ROW_MODES; ++m)
          is_row = is_row || bl.fn == mk->row[m] || (mk->row_std[m] && bl.fn == mk->row_std[m]);
        if (is_row) bl.block = nlv::kRowMaxThreads;
        if (is_col) bl.block = nlv::kMultiColThreads;
      }
      // persistent blocks: as many as are resident at once, each looping over the work items
      cudaFuncAttributes fa{};
      if (cudaFuncGetAttributes(&fa, bl.fn) == cudaSuccess && bl.smem > 0)
        cudaFuncSetAttribute(bl.fn, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_optin - (int)fa.sharedSizeBytes);
      cudaFuncSetAttribute(bl.fn, cudaFuncAttributePreferredSharedMemoryCarveout, kBatchCarveout);
      int occ = 0;
      if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, bl.fn, bl.block, bl.smem) != cudaSuccess || occ < 1) {
        cudaGetLastError();
        return batch_fail(b, NLINV_EINVAL, "a batched pass does not fit on a multiprocessor");
      }
      bl.grid = std::min(first.back(), occ * sms);
      off = (host.size() + 15) / 16 * 16;
      host.resize(off + first.size() * sizeof(int));
      std::memcpy(host.data() + off, first.data(), first.size() * sizeof(int));
      first_off.push_back(off);
      bl.args.nframes = (int)fr.size();
      bl.args.total = first.back();
      bl.args.slot = recs[fr[0]][l].args.slot;
      bl.args.skip = recs[fr[0]][l].args.skip;
      b->launches.push_back(bl);
    }
  }
  e = cudaMalloc(&b->tables, host.size());
  if (e != cudaSuccess) { cudaGetLastError(); return batch_fail(b, NLINV_ENOMEM, "batch tables: cudaMalloc failed"); }
  e = cudaMemcpy(b->tables, host.data(), host.size(), cudaMemcpyHostToDevice);
  if (e != cudaSuccess) return batch_fail(b, NLINV_ECUDA, std::string("batch tables: ") + cudaGetErrorString(e));
  for (size_t l = 0; l < b->launches.size(); ++l) {
    b->launches[l].args.args = (const KArgs*)((char*)b->tables + arg_off[l]);
    b->launches[l].args.first = (const int*)((char*)b->tables + first_off[l]);
    b->launches[l].args.stops = (const int* const*)((char*)b->tables + stop_off[b->launches[l].group]);
  }
  // one graph: the groups as parallel branches
  const size_t G = b->groups.size();
  b->gstream.assign(G, nullptr);
  b->ev_join.assign(G, nullptr);
  b->gstream[0] = b->stream;
  for (size_t g = 1; g < G && e == cudaSuccess; ++g) {
    e = cudaStreamCreateWithFlags(&b->gstream[g], cudaStreamNonBlocking);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&b->ev_join[g], cudaEventDisableTiming);
  }
  if (e == cudaSuccess) e = cudaEventCreateWithFlags(&b->ev_fork, cudaEventDisableTiming);
  if (e != cudaSuccess) return batch_fail(b, NLINV_ECUDA, std::string("batch streams: ") + cudaGetErrorString(e));
  cudaGraph_t graph = nullptr;
  e = cudaStreamBeginCapture(b->stream, cudaStreamCaptureModeThreadLocal);
  if (e == cudaSuccess) e = cudaEventRecord(b->ev_fork, b->stream);
  for (size_t g = 1; g < G && e == cudaSuccess; ++g) e = cudaStreamWaitEvent(b->gstream[g], b->ev_fork, 0);
  for (size_t l = 0; l < b->launches.size() && e == cudaSuccess; ++l)
    e = launch_batched(b, b->launches[l], b->gstream[b->launches[l].group]);
  for (size_t g = 1; g < G && e == cudaSuccess; ++g) {
    e = cudaEventRecord(b->ev_join[g], b->gstream[g]);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(b->stream, b->ev_join[g], 0);
  }
  cudaError_t e2 = cudaStreamEndCapture(b->stream, &graph);
  if (e == cudaSuccess) e = e2;
  if (e == cudaSuccess) e = cudaGraphInstantiate(&b->graph, graph, 0);
  if (graph) cudaGraphDestroy(graph);
  if (e != cudaSuccess) {
    b->graph = nullptr;
    return batch_fail(b, NLINV_ECUDA, std::string("batch graph: ") + cudaGetErrorString(e));
  }
  *out = b;
  return NLINV_OK;
}

nlinv_status nlinv_reconstruct_batch(nlinv_batch* b, int nframes, const nlinv_frame_desc* frames) {
  if (!b) return NLINV_EINVAL;
  if (!frames || nframes != (int)b->frames.size())
    return fail(nullptr, NLINV_EINVAL, "nframes and the frames must match the batch");
  bool wait = false;
  for (int i = 0; i < nframes; ++i) {
    nlinv_ctx* c = b->frames[i];
    const nlinv_frame_desc& d = frames[i];
    if (d.n != c->N || d.ncoils != c->J) return fail(nullptr, NLINV_EINVAL, "frame " + std::to_string(i) + ": shape differs");
    if (!d.y || !d.mask || !d.x_inout) return fail(nullptr, NLINV_EINVAL, "frame " + std::to_string(i) + ": NULL buffer");
    wait = wait || d.resid || !is_device_ptr(d.x_inout);
  }
  cudaError_t e = cudaSuccess;
  for (int i = 0; i < nframes && e == cudaSuccess; ++i) {
    nlinv_ctx* c = b->frames[i];
    const nlinv_frame_desc& d = frames[i];
    const size_t vb = c->vec * sizeof(float2), db = (size_t)c->J * c->plane * sizeof(float2);
    e = cudaMemcpyAsync(c->y, d.y, db, cudaMemcpyDefault, b->stream);
    if (e == cudaSuccess) e = cudaMemcpyAsync(c->mask, d.mask, (size_t)c->plane, cudaMemcpyDefault, b->stream);
    if (e == cudaSuccess) e = cudaMemcpyAsync(c->x, d.x_inout, vb, cudaMemcpyDefault, b->stream);
    if (e == cudaSuccess)
      e = cudaMemcpyAsync(c->xref, d.x_ref ? (const void*)d.x_ref : (const void*)c->x, vb, cudaMemcpyDefault, b->stream);
  }
  if (e == cudaSuccess) e = cudaGraphLaunch(b->graph, b->stream);
  if (e == cudaSuccess) b->have_state = true;
  for (int i = 0; i < nframes && e == cudaSuccess; ++i) {
    nlinv_ctx* c = b->frames[i];
    e = cudaMemcpyAsync(frames[i].x_inout, c->x, c->vec * sizeof(float2), cudaMemcpyDefault, b->stream);
  }
  if (e != cudaSuccess) return fail(nullptr, NLINV_ECUDA, std::string("nlinv_reconstruct_batch: ") + cudaGetErrorString(e));
  if (!wait) return NLINV_OK;
  std::vector<Scalars> hs(nframes);
  for (int i = 0; i < nframes && e == cudaSuccess; ++i)
    e = cudaMemcpyAsync(&hs[i], b->frames[i]->sc, sizeof(Scalars), cudaMemcpyDeviceToHost, b->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(b->stream);
  if (e != cudaSuccess) return fail(nullptr, NLINV_ECUDA, std::string("nlinv_reconstruct_batch: ") + cudaGetErrorString(e));
  bool broke = false;
  for (int i = 0; i < nframes; ++i) {
    if (frames[i].resid)
      for (int n = 0; n <= b->prm.newton_steps; ++n) frames[i].resid[n] = hs[i].resid[n];
    if (hs[i].flags & 1) {
      broke = true;
      int zero = 0;
      cudaMemcpy(&b->frames[i]->sc->flags, &zero, sizeof(int), cudaMemcpyHostToDevice);
    }
  }
  if (broke) return fail(nullptr, NLINV_EBREAKDOWN, "CG breakdown in at least one frame");
  return NLINV_OK;
}

long nlinv_batch_launch_count(const nlinv_batch* b) { return b ? (long)b->launches.size() : -1; }

nlinv_status nlinv_batch_profile_cg(nlinv_batch* b, int reps, double* ms_out) {
  if (!b) return NLINV_EINVAL;
  if (reps < 1 || !ms_out) return fail(nullptr, NLINV_EINVAL, "reps must be >= 1 and ms_out non-NULL");
  if (!b->have_state) return fail(nullptr, NLINV_EINVAL, "run nlinv_reconstruct_batch before nlinv_batch_profile_cg");
  if (b->prm.cg_iters < 2) return fail(nullptr, NLINV_EINVAL, "the batch's schedule has fewer than two CG iterations");
  cudaError_t e = cudaStreamSynchronize(b->stream);
  for (nlinv_ctx* c : b->frames)
    if (e == cudaSuccess) e = mark_running(c, 0);
  if (e != cudaSuccess) return fail(nullptr, NLINV_ECUDA, std::string("nlinv_batch_profile_cg: ") + cudaGetErrorString(e));
  // the six passes of the second CG iteration of the first Newton step, in every group
  std::vector<std::vector<size_t>> pass(kProfileSteps);
  for (size_t l = 0; l < b->launches.size(); ++l)
    if (b->launches[l].step > 0) pass[b->launches[l].step - 1].push_back(l);
  for (const std::vector<size_t>& v : pass)
    if (v.size() != b->groups.size()) return fail(nullptr, NLINV_EINVAL, "internal: CG launches not found");
  cudaEvent_t ev[2];
  for (int i = 0; i < 2; ++i)
    if ((e = cudaEventCreate(&ev[i])) != cudaSuccess)
      return fail(nullptr, NLINV_ECUDA, std::string("event create: ") + cudaGetErrorString(e));
  for (int k = 0; k < kProfileSteps && e == cudaSuccess; ++k) {
    e = cudaEventRecord(ev[0], b->stream);
    for (int it = 0; it < reps && e == cudaSuccess; ++it)
      for (size_t l : pass[k])
        if (e == cudaSuccess) e = launch_batched(b, b->launches[l], b->stream);
    if (e == cudaSuccess) e = cudaEventRecord(ev[1], b->stream);
    if (e == cudaSuccess) e = cudaEventSynchronize(ev[1]);
    float ms = 0.f;
    if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, ev[0], ev[1]);
    ms_out[k] = ms / reps;
  }
  for (int i = 0; i < 2; ++i) cudaEventDestroy(ev[i]);
  if (e != cudaSuccess) return fail(nullptr, NLINV_ECUDA, std::string("nlinv_batch_profile_cg: ") + cudaGetErrorString(e));
  return NLINV_OK;
}

nlinv_status nlinv_batch_destroy(nlinv_batch* b) {
  batch_free(b);
  return NLINV_OK;
}

const char* nlinv_last_error(const nlinv_ctx* c) { return c ? c->err.c_str() : g_create_error.c_str(); }

}  // extern "C"
