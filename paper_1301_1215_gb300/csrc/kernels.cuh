// NLINV pass kernels: batched row and column transforms over the coil planes with the pointwise steps of
// Eq. 2 and Eq. 3 fused into their loads and stores, CG vector updates, and deterministic FP64 reductions.
//
// Geometry.  A plane is N x N complex64, row-major, natural FFT order.  Omega (M_Omega of Eq. 2) is the square of
// indices e with e < f or e >= N - f in both axes (f = fov).  Image-domain intermediates only matter on Omega, so
// they are kept "compact": a T buffer holds J planes of N rows x Wc = 2f columns (the Omega columns), and the
// coil images c_j and the per-coil channel products hold J planes of Wc x Wc.  Compact index cc of natural
// index e: cc = e for e < f, cc = e - (N - 2f) for e >= N - f.
//
// Vectors of the unknown x = (rho, chat_1 .. chat_J) hold 1 + J planes: plane 0 is rho, planes 1..J chat_j.
#pragma once
#include <algorithm>
#include <cstdint>
#include <cuda_runtime.h>
#include <type_traits>
#include "fft_core.cuh"
#include "tc_dft.cuh"

namespace nlv {

// ------------------------------------------------------------------------------------------ arguments ----
enum Reduce : int {
  RED_NONE = 0,       // the block partials are summed into Scalars::last
  RED_RESID = 1,      // Scalars::resid[slot] = sqrt(sum)       (|y - F x_n|)
  RED_RR_INIT = 2,    // Scalars::rr = sum                      (|b|^2 at the start of CG)
};

constexpr int kMaxNewton = 64;

// An unevaluated sum of two floats (see pair_add).
struct Pair {
  float h, l;
};

// Scalars of the CG and Newton iterations, kept in device memory: those of CG as pairs, the residual norms in FP64.
// The values that one launch writes while its other blocks still read the value of the iteration before have two
// slots, indexed by the parity of the CG iteration.
struct Scalars {
  float unit;                    // of the current CG solve, see cg_unit: r, p, dx and the pairs below are in it
  Pair rr_pair;                  // |b|^2 of the current CG solve
  Pair rr_i[2];                  // |r_i|^2 of iteration i in slot i & 1 (batches: current and previous |r|^2)
  Pair beta_p;                   // beta of the current direction
  float step[2];                 // CG step length a_i of iteration i in slot i & 1
  double last;                   // result of a RED_NONE reduction
  double resid[kMaxNewton + 1];  // |y - F x_n| per Newton step
  int cg_stop[kMaxNewton + 1];   // per Newton step: the CG iteration that reached the rounding floor, -1 if none
                                 // (the last entry: the solve of the timing calls)
  int flags;                     // bit 0: CG breakdown (a non-finite |r|^2 or Re<p, A p>)
  unsigned ticket;               // completion counter of the last-block reduction
};

constexpr int kFlagBreakdown = 1;
// Rounding floor of CG: the solve stops once |r|^2 <= kCgFloor2 |b|^2, i.e. |r| at the FP32 unit roundoff 2^-24
// relative to |b| (further iterations cannot improve a single-precision solution; left to run, the recursive
// residual decays into the FP32 denormal range, where the step lengths lose their precision).
constexpr double kCgFloor2 = 0x1p-48;

struct alignas(16) KArgs {
  int N, J, f, Wc;          // grid side, coils, half-width of Omega, compact width 2f
  int nrows;                // row passes: rows of the coil planes (J*N); column passes: J
  int rows_per_cta;         // row passes: consecutive coil rows handled by one block
  int rho_per_cta;          // row passes with a rho part: consecutive rho-plane pixels handled by one block
  // Row passes of batches: the rows and the rho slice of such a block are shared by `sub` blocks of sub_lanes lanes, which
  // together stand for its group_threads threads (see rho_slice); sub = 0: single frames, no sharing.
  int sub, sub_lanes, group_threads;
  const float* wtab;        // Sobolev weight w(k) = (1 + a |k|^2)^(-l/2), N x N natural order
  float alpha;              // alpha_n of Eq. 3 for the normal operator and the right-hand side
  const float2* src;        // main input planes
  float2* dst;              // main output planes
  const float2* src2;       // passes with two inputs: the second (row passes: rows nrows1 .. nrows-1, into dst2)
  float2* dst2;
  int nrows1;
  float2* coil_out;         // column passes that form the coil maps: where they go (compact J x Wc x Wc), or NULL
  const float2* rho;        // rho of the linearisation point (natural N x N)
  const float2* drho;       // rho part of the direction (natural N x N)
  const float2* coil;       // c_j on Omega, compact J x Wc x Wc
  const float2* cimg;       // image-domain coils (natural J x N x N), forward simulation only
  float2* zsum;             // conj(c_j) z_j on Omega, compact J x Wc x Wc
  const uint8_t* mask;      // sampling pattern P, N x N
  const float2* y;          // data, J x N x N
  const float2* p;          // CG direction, (1+J) planes
  const float2* x;          // Newton iterate, (1+J) planes
  const float2* xref;       // regularisation centre, (1+J) planes
  float2* r;                // CG residual, (1+J) planes
  float2* dx;               // CG solution, (1+J) planes
  float2* U;                // CG direction pass: W^-1 p on Omega, compact J x Wc x Wc, carried from iteration to iteration
  const float2* twA;        // twiddles of the split (N1, N2)
  const float2* twB;        // twiddles of the split (N2, N1)
  double* partials;         // one double per block
  Scalars* sc;
  int reduce;               // Reduce
  int slot;                 // RED_RESID index; RED_RR_INIT and the CG passes: the Newton step
  int iter;                 // CG passes: index of the CG iteration; cg_finish: number of scheduled iterations
  int last;                 // CG update pass: the last scheduled iteration (its row transform would not be read)
  int scalars;              // DF^H column pass of a CG iteration: one more block forms the step length (cg_decide)
  const float2* q;          // vector passes: second operand; batch CG step: A p
  float2* pout;             // batches: CG direction written by the right-hand side pass
  // Batches: the normal-operator pass writes one partial of Re<p, A p> per block into pq_part (the CG step adds the n_pq
  // partials to form alpha), the CG step one of |r|^2 into brr_part (the first pass of the next iteration adds the n_rr
  // partials to form beta; NULL: beta from Scalars).
  Pair* pq_part;
  int n_pq;
  Pair* brr_part;
  long n2;                  // vector passes: number of float4 (two complex values each)
  // Sums without a last-block tail: a pass writes one partial per block and a later launch adds them.
  Pair* dd_part;            // PSF pass: partials of |P FFT(...)|^2 = |DF p|^2 (n_dd of them)
  int n_dd;
  Pair* rr_part;            // CG update pass: partials of |r|^2, then of Re<r, p>, then of |p|^2 (n_rr of each)
  int n_rr;
  float coef;               // vector passes: second coefficient of out = alpha X + coef Y
  const void* tcB;          // tensor-core passes: the B tiles of the radix-16 DFT stage (tc_dft.cuh)
  int skip;                 // a launch of the CG iteration: it returns at once when the solve stopped before CG
                            // iteration `skip` (0: never; see cg_stopped)
  int skip_after;           // a stop at iteration skip - 1 itself counts, read after the dependent-launch wait (the CG
                            // update pass; batches)
  int src_early;            // CG update pass: its rows of p, written two or more launches back, are staged before the
                            // dependent-launch wait
};

// ------------------------------------------------------------------------------- dependent launches ----
// Every kernel is launched with programmatic stream serialisation: it may be scheduled while the kernel before it
// in the stream is still running.  griddepcontrol.wait blocks until that kernel has completed and its memory is
// visible, so it must come before the first global memory access; launch_dependents then lets the next kernel be
// scheduled as soon as every block of this one has started.
__device__ __forceinline__ void pdl_enter() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// A pass of CG iteration i whose solve has stopped (Scalars::cg_stop) skips its work: the remaining iterations of a
// stopped solve are empty steps (the dx they would leave is the one already there).  Two passes of iteration i may
// record the stop, the direction pass and the DF^H column pass, while other blocks of theirs, or early blocks of the
// pass after, read it; what they record is i.  So the first three passes of an iteration skip for a stop before i
// (KArgs::skip = i) and take no notice of a stop at i -- what they then compute is not read --, and the update pass,
// after its wait, skips for a stop at i as well (skip = i + 1): all threads of a launch always decide alike.
//
// What a kernel may read before its wait: a kernel is scheduled only once every block of the kernel before it has
// passed its own wait (pdl_enter: wait, then launch_dependents), i.e. once the kernel two launches back has completed,
// so anything written two or more launches back (or before the stream reached the library's first kernel) is in
// place.  A stop before iteration i was recorded at least two launches before each pass of iteration i, so a single-frame
// pass reads it first thing, before its wait, and leaves at once, having staged nothing: a skipped iteration (four
// launches) took 9.8 us at 384 x 384 with 10 coils when its passes staged their side inputs before they looked, 8.0 us
// now; 14.8 and 9.3 us at 512 x 512 with 16, 5.4 and 4.6 us at 64 x 64 with 4.
__device__ __forceinline__ bool cg_stopped(const KArgs& A) {
  return A.skip > 0 && (unsigned)*(volatile const int*)&A.sc->cg_stop[A.slot] < (unsigned)A.skip;
}
// The stops that may be read before the wait.
__device__ __forceinline__ bool cg_stopped_early(const KArgs& A) {
  const int before = A.skip - (A.skip_after ? 1 : 0);
  return before > 0 && (unsigned)*(volatile const int*)&A.sc->cg_stop[A.slot] < (unsigned)before;
}

// ------------------------------------------------------------------------------------------- geometry ----
__device__ __forceinline__ bool in_omega(int e, int N, int f) { return e < f || e >= N - f; }
__device__ __forceinline__ int to_compact(int e, int N, int f) { return e < f ? e : e - (N - 2 * f); }
__device__ __forceinline__ int to_natural(int cc, int N, int f) { return cc < f ? cc : cc + (N - 2 * f); }

// ----------------------------------------------------------------------------------------- reductions ----
// Butterfly sum over the lanes of this warp that exist: lanes 0..cnt-1 (a block's last warp may be partial, and a
// row block can be narrower than a warp).  Only those lanes take part in the shuffles; a partner lane that does not
// exist counts as 0.  Valid in lane 0.
__device__ __forceinline__ double warp_sum(double v, int cnt = 32) {
  if (cnt >= 32) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
  }
  const unsigned mask = (1u << cnt) - 1u;
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const double w = __shfl_xor_sync(mask, v, o);
    if ((lane ^ o) < cnt) v += w;
  }
  return v;
}

// Lanes of the calling thread's warp that exist in this block.
__device__ __forceinline__ int warp_lanes() {
  const int rest = (int)blockDim.x - (int)(threadIdx.x & ~31u);
  return rest < 32 ? rest : 32;
}

// Deterministic block sum (fixed tree), result valid in thread 0.
__device__ __forceinline__ double block_sum(double v, double* red) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
  v = warp_sum(v, warp_lanes());
  __syncthreads();
  if (lane == 0) red[warp] = v;
  __syncthreads();
  double s = 0.0;
  if (warp == 0) {
    s = lane < nw ? red[lane] : 0.0;
    s = warp_sum(s, warp_lanes());
  }
  return s;
}

// Sums over the threads and blocks of a CG iteration are kept as an unevaluated pair of floats h + l: Knuth's two-sum
// gives the exact rounding error of every addition to h, which collects in l, so a sum of n terms is good to about
// n 2^-48.  The terms themselves are FP32 sums of at most 16 products, good to 2^-22 or so.  The scalars formed from the
// sums (beta, the step length) are pairs as well; the updates use them rounded to FP32.  FP64 runs at 1/90 of the FP32
// rate on sm_103a (1.4 additions a clock and SM), and a dependent chain at some hundred cycles an operation: a tree sum
// in FP64 cost the PSF pass 1.2 us of 7.4 at 384 x 384 with 10 coils, the update pass, with three, 3 us, and the
// scalars' two quotients of an iteration 4 us where nothing hides them.
__device__ __forceinline__ void pair_add(Pair& s, float x, float lo) {
  const float t = __fadd_rn(s.h, x);
  const float z = __fsub_rn(t, s.h);
  const float e = __fadd_rn(__fsub_rn(s.h, __fsub_rn(t, z)), __fsub_rn(x, z));
  s.h = t;
  s.l = __fadd_rn(s.l, __fadd_rn(e, lo));
}
// Arithmetic on pairs, relative error about 2^-45: products by fused multiply-add (exact low part), quotients by one
// correction of the FP32 quotient.
__device__ __forceinline__ Pair pair_norm(float h, float l) {            // |l| at most |h|
  const float t = __fadd_rn(h, l);
  return {t, __fsub_rn(l, __fsub_rn(t, h))};
}
__device__ __forceinline__ Pair pair_sum(Pair a, Pair b) {
  pair_add(a, b.h, b.l);
  return pair_norm(a.h, a.l);
}
__device__ __forceinline__ Pair pair_mul(Pair a, Pair b) {
  const float t = __fmul_rn(a.h, b.h);
  const float e = fmaf(a.h, b.h, -t);
  return pair_norm(t, fmaf(a.h, b.l, fmaf(a.l, b.h, e)));
}
__device__ __forceinline__ Pair pair_scale(Pair a, float s) { return {a.h * s, a.l * s}; }      // s a power of two
__device__ __forceinline__ Pair pair_div(Pair a, Pair b) {
  const float q = a.h / b.h;
  const float r = __fadd_rn(fmaf(-q, b.h, a.h), fmaf(-q, b.l, a.l));    // the first difference is exact
  return pair_norm(q, r / b.h);
}
__device__ __forceinline__ bool pair_gt(Pair a, Pair b) { return a.h > b.h || (a.h == b.h && a.l > b.l); }
// The unit of a CG solve: the power of two that takes |b| to between 1/2 and 1 (kept so small that its square and the
// inverse of that are ordinary floats).  A solve is linear in b: it runs on unit b, the first iteration's passes
// multiplying what the right-hand side pass left by it, and the result is divided by it.  Nothing is rounded by that, and
// neither the sums of squares nor the rounding floor of |r|^2, 2^-48 of its start, meet the ends of the FP32 range,
// whatever units the data are in: with raw data and a fixed factor of 2^-25 on the sums, a frame with |b| near 1e-12 never
// met its floor or met it two iterations early.
__device__ __forceinline__ float cg_unit(double bb) {
  if (!(bb > 0.0) || !isfinite(bb)) return 1.f;
  const int e = ((__double2hiint(bb) >> 20) & 0x7ff) - 1022;       // bb in [2^(e-1), 2^e)
  const int half = min(max((e + 1) >> 1, -62), 62);
  return __int_as_float((127 - half) << 23);
}
// |p|^2 of p = r + beta p_old from |r|^2, beta, Re<r, p_old> and |p_old|^2.
__device__ __forceinline__ Pair cg_direction_norm(Pair rr, Pair beta, Pair rp, Pair pp) {
  return pair_sum(rr, pair_mul(beta, pair_sum(pair_scale(rp, 2.f), pair_mul(beta, pp))));
}
// Butterfly sum over the existing lanes of the calling warp (all of them call it), valid in lane 0.
__device__ __forceinline__ Pair warp_sum(Pair s, int cnt) {
  const unsigned mask = cnt >= 32 ? 0xffffffffu : (1u << cnt) - 1u;
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float h = __shfl_xor_sync(mask, s.h, o), l = __shfl_xor_sync(mask, s.l, o);
    if ((lane ^ o) < cnt) pair_add(s, h, l);
  }
  return s;
}
// The sum of the n pairs at src (global or shared memory) by the calling warp, in a fixed order, valid in lane 0.
__device__ __forceinline__ Pair warp_sum_of(const Pair* src, int n) {
  constexpr int D = 12;            // loads in flight
  const int lane = threadIdx.x & 31, nl = warp_lanes();
  Pair s = {0.f, 0.f};
  for (int k0 = lane; k0 < n; k0 += D * nl) {
    Pair t[D];
#pragma unroll
    for (int d = 0; d < D; ++d) {
      const bool ok = k0 + d * nl < n;
      t[d].h = ok ? src[k0 + d * nl].h : 0.f;
      t[d].l = ok ? src[k0 + d * nl].l : 0.f;
    }
#pragma unroll
    for (int d = 0; d < D; ++d) pair_add(s, t[d].h, t[d].l);
  }
  return warp_sum(s, nl);
}
// Block sums of K pairs per thread that every thread has stored at sums[k * blockDim.x + threadIdx.x], a barrier ago:
// the block's last warps (in most splits they have no part in the layout-A steps) add one each and write out[k].
template <int K> __device__ __forceinline__ void block_pairs(const Pair* sums, Pair* const (&out)[K]) {
  const int nw = ((int)blockDim.x + 31) >> 5, warp = threadIdx.x >> 5;
#pragma unroll
  for (int k = 0; k < K; ++k)
    if (warp == nw - 1 - k % nw) {
      const Pair s = warp_sum_of(sums + k * blockDim.x, blockDim.x);
      if ((threadIdx.x & 31) == 0) *out[k] = s;
    }
}

__device__ __forceinline__ void finalize_scalar(Scalars* sc, int reduce, int slot, double total) {
  switch (reduce) {
    case RED_RESID: sc->resid[slot] = sqrt(total); break;
    case RED_RR_INIT:           // a new CG solve starts: nothing has stopped yet
      sc->beta_p = {0.f, 0.f};
      sc->unit = cg_unit(total);
      total *= (double)sc->unit * (double)sc->unit;
      sc->rr_pair.h = (float)total;
      sc->rr_pair.l = (float)(total - (double)sc->rr_pair.h);
      sc->rr_i[0] = sc->rr_pair;
      sc->cg_stop[slot] = -1;
      break;
    default: sc->last = total; break;
  }
}

// Every thread passes its partial; per-block sums in FP64 go to partials[], and the last block to finish
// adds them in block order (so the result does not depend on scheduling) and updates the scalars.
// bid / nblk: this block's index and the number of blocks working on the same problem (the whole grid, or one
// frame's share of a batched grid).
__device__ __forceinline__ void grid_reduce(double mine, const KArgs& A, int bid, int nblk) {
  __shared__ double red[32];
  __shared__ bool last;
  double s = block_sum(mine, red);
  if (threadIdx.x == 0) {
    A.partials[bid] = s;
    __threadfence();
    unsigned t = atomicAdd(&A.sc->ticket, 1u);
    last = (t == (unsigned)nblk - 1);
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  double acc = 0.0;
  for (int i = threadIdx.x; i < nblk; i += blockDim.x) acc += __ldcg(&A.partials[i]);
  double total = block_sum(acc, red);
  if (threadIdx.x == 0) {
    finalize_scalar(A.sc, A.reduce, A.slot, total);
    A.sc->ticket = 0u;
  }
}

// ------------------------------------------------------------------------------------ async staging ----
// Side inputs of a pass (sampling pattern, weights, CG vectors, coil maps, rho) and the twiddle tables are copied
// into shared memory with cp.async at the start of every pass, together with the main loads, so that all load
// latencies overlap once instead of stalling the pointwise steps between the transforms.
__device__ __forceinline__ void cp_async16(void* sdst, const void* gsrc) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(sdst);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(s), "l"(gsrc) : "memory");
}
__device__ __forceinline__ void cp_async8(void* sdst, const void* gsrc) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(sdst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(s), "l"(gsrc) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() {
  asm volatile("cp.async.commit_group;" ::: "memory");
  asm volatile("cp.async.wait_all;" ::: "memory");
}

// Copies nbytes (a multiple of 16, both addresses 16-byte aligned) with all threads of the block.
__device__ __forceinline__ void stage_bytes(void* sdst, const void* gsrc, int nbytes) {
  for (int i = threadIdx.x; i < nbytes / 16; i += blockDim.x)
    cp_async16((char*)sdst + 16 * i, (const char*)gsrc + 16 * i);
}

// Prefetches nbytes (a multiple of 16, 16-byte aligned) into L2.
__device__ __forceinline__ void prefetch_l2(const void* p, unsigned nbytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(nbytes) : "memory");
}
__host__ __device__ constexpr size_t align16(size_t v) { return (v + 15) / 16 * 16; }

// Rows R0 .. R0+nr-1 of rb bytes each (rb a multiple of 16) into consecutive rows of sdst: row R of gsrc, or row
// R mod N with `wrap` (tables of one plane shared by all coil planes); every run of consecutive source rows is one
// flat copy, so a thread issues about nr*rb / (16*blockDim.x) copies instead of one loop per row.
__device__ __forceinline__ void stage_rows(unsigned char* sdst, const void* gsrc, int R0, int nr, int rb, int N,
                                           bool wrap) {
  for (int l = 0; l < nr;) {
    const int R = R0 + l;
    const int e = wrap ? R % N : R;
    const int run = wrap ? min(nr - l, N - e) : nr - l;
    stage_bytes(sdst + (size_t)l * rb, (const unsigned char*)gsrc + (size_t)e * rb, run * rb);
    l += run;
  }
}

// ------------------------------------------------------------------------------------------ row passes ----
enum RowMode : int {
  ROW_W_IFFT = 0,        // T <- compact cols of FFT^-1_row(w * src / sqrt N)            (W^-1, first axis)
  ROW_PSF = 1,           // T <- compact cols of FFT^-1_row(P * FFT_row(T) / N)          (PSF step, Sec. 3.1)
  ROW_FFT_P_OUT = 2,     // dst <- P * FFT_row(T) / sqrt N                               (F, DF output)
  ROW_FFT_RESID = 3,     // dst <- y - P * FFT_row(T) / sqrt N, |dst|^2                  (Newton residual)
  ROW_P_IFFT = 4,        // T <- compact cols of FFT^-1_row(P * src / sqrt N)            (DF^H input)
  ROW_FFT_W_ADJ = 5,     // dst coil planes <- w FFT_row(T)/sqrt N; rho plane <- sum_j zsum_j (DF^H output)
  ROW_FFT_W_NORMAL = 6,  // as ADJ, plus alpha p                                          (normal operator)
  // single frames
  ROW_CG_RHS = 7,        // as ADJ, minus alpha (x - xref); r = b, |b|^2; T <- FFT^-1_row(w r)  (right-hand side)
  ROW_CG_UPDATE = 8,     // q = w FFT_row(T)/sqrt N + alpha p; the CG updates; T <- FFT^-1_row(w r)
  ROW_CG_PSF = 9,        // as PSF; |P FFT_row(T)|^2
  // batches
  ROW_BCG_RHS = 10,      // as ADJ, minus alpha (x - xref); r = p = b, dx = 0, |b|^2     (right-hand side)
  ROW_BCG_DIR = 11,      // p = r + beta p; T <- compact cols of FFT^-1_row(w p / sqrt N)
  ROW_BCG_NORMAL = 12,   // as NORMAL with the rho part of p = r + beta p; Re<p, q>
  // operators: two arrays in one launch
  ROW_W_W_IFFT = 13,     // T <- W_IFFT of src, T2 <- W_IFFT of src2
  ROW_W_P_IFFT = 14,     // T <- W_IFFT of src, T2 <- P_IFFT of src2
  NUM_ROW_MODES = 15
};

// Row passes run kRowCtasPerSM blocks per SM; a block holds up to kRowMaxThreads threads (whole lanes of TL
// threads) and loops over its share of rows when they do not fit at once.
constexpr int kRowMaxThreads = 320;
constexpr int kRowCtasPerSM = 2;
// Row passes of batches: where a block's rows divide evenly, the same warps per SM in twice the blocks of half the size.  A
// block of these passes waits for its loads, then for its exchanges; more and smaller blocks are more often at different
// points: 2 Newton steps of 15 iterations of 8 frames of 192^2/6 with 8 of 256^2/8 4.81 ms whole, 4.68 divided.  The 13
// rows of a block of side 384, the one side where they do not divide, would make parts of 5, 5 and 3 rows that hold a
// block of 5 each: 4 frames of 384^2/10 6.78 ms divided, 6.10 whole; 16 22.9 and 21.4; 8 with 8 of 320^2/8 16.8 and 15.0.
constexpr int kRowBatchThreads = 160;

template <int MODE> struct RowTraits {
  static constexpr bool both = (MODE == ROW_W_W_IFFT || MODE == ROW_W_P_IFFT);
  static constexpr bool inverse_first = (MODE == ROW_W_IFFT || MODE == ROW_P_IFFT || MODE == ROW_BCG_DIR || both);
  static constexpr bool load_compact = !inverse_first;
  static constexpr bool psf = (MODE == ROW_PSF || MODE == ROW_CG_PSF);
  static constexpr bool normal = (MODE == ROW_FFT_W_NORMAL || MODE == ROW_BCG_NORMAL);
  static constexpr bool rhs = (MODE == ROW_CG_RHS || MODE == ROW_BCG_RHS);
  static constexpr bool has_rho = (MODE == ROW_FFT_W_ADJ || normal || rhs);
  static constexpr bool reduces = (MODE == ROW_FFT_RESID || MODE == ROW_BCG_NORMAL || rhs);
  // a second transform follows the first one in the same pass
  static constexpr bool two = (psf || MODE == ROW_CG_RHS || MODE == ROW_CG_UPDATE);
  // side inputs staged per row: sampling-pattern row (bytes), weight row (floats), complex rows
  static constexpr bool s_mask = (psf || MODE == ROW_FFT_P_OUT || MODE == ROW_FFT_RESID);
  static constexpr bool s_w = has_rho || MODE == ROW_W_IFFT || MODE == ROW_BCG_DIR || MODE == ROW_CG_UPDATE || both;
};

// Shared-memory layout of a row pass (byte offsets), identical on host and device.
struct RowSmem {
  size_t xch, tw, mask, w, cplx, sums, total;
};
// Floats per staged weight row: w(g) = w(-g), so the CG update pass, short of shared memory, keeps g = 0 .. N/2.
__host__ __device__ constexpr int w_pitch(int mode, int N);
__host__ __device__ inline RowSmem row_smem(int mode, int N, int lanes, int sm_lane) {
  RowSmem L{};
  const bool m = (mode == ROW_PSF || mode == ROW_CG_PSF || mode == ROW_FFT_P_OUT || mode == ROW_FFT_RESID);
  const bool w = !m && mode != ROW_P_IFFT;
  L.xch = 0;
  L.tw = align16((size_t)lanes * sm_lane * 8);
  L.mask = L.tw + align16((size_t)2 * N * 8);
  L.w = L.mask + (m ? align16((size_t)lanes * N) : 0);
  L.cplx = L.w + (w ? align16((size_t)lanes * w_pitch(mode, N) * 4) : 0);
  L.sums = L.cplx + ((mode == ROW_FFT_RESID || mode == ROW_CG_UPDATE) ? (size_t)lanes * N * 8 : 0);
  L.total = L.sums + (mode == ROW_CG_UPDATE ? (size_t)3 * kRowMaxThreads * sizeof(Pair) : 0);
  return L;
}
__host__ __device__ constexpr int w_pitch(int mode, int N) { return mode == ROW_CG_UPDATE ? N / 2 + 4 : N; }

#ifndef NLV_COL_C
#define NLV_COL_C 8
#endif


// rho plane of the adjoint / normal / right-hand-side outputs: the sum of the channel products over the coils on
// Omega (the channel summation of Table 1) plus the mode's alpha term.  Every block takes an equal slice of the
// plane after its rows, all of its threads working on it.  A thread takes two pixels per step (o and
// o + blockDim.x) and issues every load of both before the first use; the coil sum of a pixel runs over even and
// odd coils in two partial sums added at the end.
// Dot-product partials: a thread sums at most 32 products in FP32 (one row round, or two pixels of the rho slice)
// before adding them to its FP64 or pair partial, so the FP32 summation length is bounded whatever the problem size.  In
// the single-frame CG passes the real and imaginary products of a thread go to two FP32 sums of at most 16 products each
// (one row round of at most 16 complex values, or one step of the rho slice) before they are added to its pair.
__device__ __forceinline__ void dot_acc(float2& acc, float2 a, float2 b) {     // acc += (Re a Re b, Im a Im b)
  acc.x = fmaf(a.x, b.x, acc.x);
  acc.y = fmaf(a.y, b.y, acc.y);
}

__device__ __forceinline__ void dot_flush(float2& acc, Pair& sum) {
  pair_add(sum, acc.x, 0.f);
  pair_add(sum, acc.y, 0.f);
  acc = make_float2(0.f, 0.f);
}

// The two pixels o0 and o0 + bd of a rho-plane step: which exist (ok), which lie on Omega (om, with their
// compact offset zo).  Pixel and channel-product offsets fit 32 bits: a plane has at most 1024^2 pixels, the J
// channel-product planes at most 64 x 512^2 entries.
template <int N>
__device__ __forceinline__ void rho_pixels(int o0, int bd, int e_end, int f, int Wc, bool (&ok)[2], bool (&om)[2],
                                           int (&zo)[2]) {
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const int o = o0 + k * bd;
    const int e1 = o / N, e2 = o - e1 * N;
    ok[k] = o < e_end;
    om[k] = ok[k] && in_omega(e1, N, f) && in_omega(e2, N, f);
    zo[k] = om[k] ? to_compact(e1, N, f) * Wc + to_compact(e2, N, f) : 0;
  }
}
// Channel sums of those two pixels, over even and odd coils in two partial sums added at the end.  Eight coils' loads of
// both pixels are in flight at once: with two, a frame of 10 coils paid the L2 latency five times.
__device__ __forceinline__ void rho_channel_sum(const KArgs& A, const bool (&om)[2], const int (&zo)[2], int stride,
                                                float2 (&z)[2]) {
  constexpr int D = 8;
  const float2 zero = make_float2(0.f, 0.f);
  float2 s[2][2] = {{zero, zero}, {zero, zero}};
  const float2* z0 = A.zsum + zo[0];
  const float2* z1 = A.zsum + zo[1];
  int j = 0;
  for (; j + D <= A.J; j += D) {
    float2 a[D], b[D];
#pragma unroll
    for (int d = 0; d < D; ++d) {
      a[d] = om[0] ? z0[d * stride] : zero;
      b[d] = om[1] ? z1[d * stride] : zero;
    }
#pragma unroll
    for (int d = 0; d < D; ++d) {
      s[0][d & 1] = cadd(s[0][d & 1], a[d]);
      s[1][d & 1] = cadd(s[1][d & 1], b[d]);
    }
    z0 += D * stride;
    z1 += D * stride;
  }
  if (j < A.J) {
    float2 a[D], b[D];
#pragma unroll
    for (int d = 0; d < D - 1; ++d) {
      a[d] = om[0] && j + d < A.J ? z0[d * stride] : zero;
      b[d] = om[1] && j + d < A.J ? z1[d * stride] : zero;
    }
#pragma unroll
    for (int d = 0; d < D - 1; ++d) {
      s[0][d & 1] = cadd(s[0][d & 1], a[d]);
      s[1][d & 1] = cadd(s[1][d & 1], b[d]);
    }
  }
  z[0] = cadd(s[0][0], s[0][1]);
  z[1] = cadd(s[1][0], s[1][1]);
}

// Adds a thread's FP32 partial to its FP64 sum or its pair.
__device__ __forceinline__ void acc_add(double& s, float v) { s += (double)v; }
__device__ __forceinline__ void acc_add(Pair& s, float v) { pair_add(s, v, 0.f); }

// t, bd: the thread's index in the block and the block's threads.  Blocks that share a slice (KArgs::sub) pass their
// threads' places in the undivided block, so that a thread's two pixels, whose products it adds in FP32, stay the same
// pair however the block is divided.
template <int N, int MODE, bool STDF, class Sum>
__device__ __forceinline__ void rho_slice(const KArgs& A, int bid, int t, int bd, Sum& sum) {
  const int f = STDF ? N / 4 : A.f, Wc = STDF ? N / 2 : A.Wc;
  constexpr int plane = N * N;
  const int e_begin = bid * A.rho_per_cta;
  const int e_end = min(e_begin + A.rho_per_cta, plane);
  const float beta = MODE == ROW_BCG_NORMAL ? A.sc->beta_p.h : 0.f;
  for (int o0 = e_begin + t; o0 < e_end; o0 += 2 * bd) {
    float acc = 0.f;
    float2 a[2], b[2], z[2];
    int zo[2];
    bool ok[2], om[2];
    rho_pixels<N>(o0, bd, e_end, f, Wc, ok, om, zo);
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const int o = o0 + k * bd;
      a[k] = b[k] = make_float2(0.f, 0.f);
      if (ok[k]) {
        if constexpr (RowTraits<MODE>::normal) a[k] = A.p[o];
        if constexpr (MODE == ROW_BCG_NORMAL) b[k] = A.r[o];
        if constexpr (RowTraits<MODE>::rhs) {
          a[k] = A.x[o];
          b[k] = A.xref[o];
        }
      }
    }
    rho_channel_sum(A, om, zo, Wc * Wc, z);
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      if (!ok[k]) continue;
      const int o = o0 + k * bd;
      if constexpr (MODE == ROW_FFT_W_ADJ) {
        A.dst[o] = z[k];
      } else if constexpr (RowTraits<MODE>::normal) {
        float2 pv = a[k];
        if constexpr (MODE == ROW_BCG_NORMAL) {
          if (A.iter == 0) b[k] = cscale(b[k], A.sc->unit);      // r holds b (the unit held in a register spilled 76 bytes
                                                                 // a thread at side 320)
          pv = make_float2(fmaf(beta, pv.x, b[k].x), fmaf(beta, pv.y, b[k].y));
          const_cast<float2*>(A.p)[o] = pv;
        }
        const float2 q = make_float2(fmaf(A.alpha, pv.x, z[k].x), fmaf(A.alpha, pv.y, z[k].y));
        A.dst[o] = q;
        if constexpr (MODE == ROW_BCG_NORMAL) acc += pv.x * q.x + pv.y * q.y;
      } else {
        const float2 bb = make_float2(z[k].x - A.alpha * (a[k].x - b[k].x), z[k].y - A.alpha * (a[k].y - b[k].y));
        A.r[o] = bb;
        if constexpr (MODE == ROW_BCG_RHS) {
          A.pout[o] = bb;
          A.dx[o] = make_float2(0.f, 0.f);
        }
        acc += bb.x * bb.x + bb.y * bb.y;
      }
    }
    if constexpr (RowTraits<MODE>::reduces) acc_add(sum, acc);
  }
}

// The scalars of one CG update (see cg_point).
struct CgStep {
  float a, a_prev, beta, alpha;
  float unit;                   // of the solve (iteration 0: r holds b)
  bool first, odd;              // iteration 0 (p = r); an odd iteration (the one that updates dx)
};
struct CgDots {                 // sums of |r|^2, Re<r, p> and |p|^2 of the new r and p
  float2 rr, rp, pp;
};
// One element of the CG update (in iteration 0 after r *= unit):  p = r + beta p_old;  q = z + alpha p (z: the element of DF^H DF p);  r -= a q.
// Returns the new r; p: in the old, out the new direction; g: what the pair of iterations adds to dx (odd
// iterations: a_prev p_old + a p).
__device__ __forceinline__ float2 cg_point(const CgStep& c, float2 z, float2 r, float2& p, float2& g, CgDots& acc) {
  const float2 po = p;
  if (c.first) r = cscale(r, c.unit);
  p = c.first ? r : make_float2(fmaf(c.beta, po.x, r.x), fmaf(c.beta, po.y, r.y));
  const float2 q = make_float2(fmaf(c.alpha, p.x, z.x), fmaf(c.alpha, p.y, z.y));
  r = make_float2(fmaf(-c.a, q.x, r.x), fmaf(-c.a, q.y, r.y));
  g = make_float2(fmaf(c.a_prev, po.x, c.a * p.x), fmaf(c.a_prev, po.y, c.a * p.y));
  dot_acc(acc.rr, r, r);
  dot_acc(acc.rp, r, p);
  dot_acc(acc.pp, p, p);
  return r;
}

// dx += g (odd iterations; the first one, iteration 1, writes it).  The addition happens in L2, so no thread waits for
// dx or holds it: read and written by the pass it cost 6 of 55 us at 512 x 512 with 16 coils and, held in registers
// across the second transform, spilled 300 bytes a thread.
__device__ __forceinline__ void cg_add_dx(float2* dx, float2 g, bool add) {
  if (add)
    asm volatile("red.global.add.v2.f32 [%0], {%1, %2};" ::"l"(dx), "f"(g.x), "f"(g.y) : "memory");
  else
    *dx = g;
}

// Adds a thread's products to its three sums at sums[k * blockDim.x]; first: they hold nothing yet.
__device__ __forceinline__ void cg_flush(CgDots& d, Pair* sums, bool first) {
  float2* v[3] = {&d.rr, &d.rp, &d.pp};
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    Pair s = {0.f, 0.f};
    if (!first) s = sums[k * blockDim.x];
    dot_flush(*v[k], s);
    sums[k * blockDim.x] = s;
  }
}

__device__ __forceinline__ void cg_flush(CgDots& d, Pair (&sums)[3]) {
  dot_flush(d.rr, sums[0]);
  dot_flush(d.rp, sums[1]);
  dot_flush(d.pp, sums[2]);
}

// The rho plane's slice of the CG update pass.
template <int N, bool STDF>
__device__ __forceinline__ void rho_cg_slice(const KArgs& A, int bid, const CgStep c, Pair* sums) {
  const int f = STDF ? N / 4 : A.f, Wc = STDF ? N / 2 : A.Wc;
  constexpr int plane = N * N;
  const int e_begin = bid * A.rho_per_cta;
  const int e_end = min(e_begin + A.rho_per_cta, plane);
  const int bd = blockDim.x;
  for (int o0 = e_begin + threadIdx.x; o0 < e_end; o0 += 2 * bd) {
    CgDots acc;
    acc.rr = acc.rp = acc.pp = make_float2(0.f, 0.f);
    float2 p[2], r[2], z[2];
    int zo[2];
    bool ok[2], om[2];
    rho_pixels<N>(o0, bd, e_end, f, Wc, ok, om, zo);
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const int o = o0 + k * bd;
      p[k] = r[k] = make_float2(0.f, 0.f);
      if (ok[k]) {
        r[k] = A.r[o];
        if (!c.first) p[k] = A.p[o];
      }
    }
    rho_channel_sum(A, om, zo, Wc * Wc, z);
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      if (!ok[k]) continue;
      const int o = o0 + k * bd;
      float2 g;
      A.r[o] = cg_point(c, z[k], r[k], p[k], g, acc);
      const_cast<float2*>(A.p)[o] = p[k];
      if (c.odd) cg_add_dx(A.dx + o, g, A.iter > 1);
    }
    cg_flush(acc, sums, false);
  }
}

// Side rows of the round starting at row R0 (sampling pattern, weights, data).  Every launch sequence writes these,
// if at all, two or more launches before the pass that stages them (the data rows of the gradient's second
// residual are the first residual, three launches back), never in the launch just before, so that a single-frame
// pass may stage them before its dependent-launch wait (see cg_stopped for why that suffices).
template <int N, int MODE>
__device__ __forceinline__ void row_stage_side(const KArgs& A, const RowSmem& L, int R0, int r_end, int LANES,
                                               unsigned char* smem_raw) {
  using T = RowTraits<MODE>;
  const int nr = min(LANES, r_end - R0);
  if constexpr (T::s_mask) stage_rows(smem_raw + L.mask, A.mask, R0, nr, N, N, true);
  if constexpr (MODE == ROW_CG_UPDATE) {
    constexpr int W = w_pitch(MODE, N), Q = W / 4;               // 16-byte chunks
    for (int i = threadIdx.x; i < nr * Q; i += blockDim.x) {
      const int l = i / Q, c = i - l * Q;
      cp_async16(smem_raw + L.w + (size_t)i * 16, A.wtab + (size_t)((R0 + l) % N) * N + 4 * c);
    }
  } else if constexpr (T::s_w) {
    stage_rows(smem_raw + L.w, A.wtab, R0, nr, N * 4, N, true);
  }
  if constexpr (MODE == ROW_FFT_RESID) stage_rows(smem_raw + L.cplx, A.y, R0, nr, N * 8, N, false);
}

// Rows of the CG direction p (coil planes) of the round starting at row R0; in iteration 0 p = r and none is read.
template <int N>
__device__ __forceinline__ void cg_stage_p(const KArgs& A, const RowSmem& L, int R0, int r_end, int LANES,
                                           unsigned char* smem_raw) {
  if (A.iter > 0) stage_rows(smem_raw + L.cplx, A.p + (size_t)N * N, R0, min(LANES, r_end - R0), N * 8, N, false);
}

// The twiddles and the first round's side rows of a single-frame row pass, issued before its dependent-launch
// wait (row_pass_body with PRE then skips them).
template <int N1, int N2, int MODE>
__device__ __forceinline__ void row_pass_prestage(const KArgs& A, int bid, unsigned char* smem_raw) {
  using S = Split<N1, N2>;
  constexpr int N = S::N;
  const int LANES = blockDim.x / S::TL;
  const RowSmem L = row_smem(MODE, N, LANES, S::SM_LANE);
  const int r_begin = bid * A.rows_per_cta;
  const int r_end = min(r_begin + A.rows_per_cta, A.nrows);
  stage_bytes(smem_raw + L.tw, A.twA, N * 8);
  stage_bytes(smem_raw + L.tw + N * 8, A.twB, N * 8);
  if (r_begin < r_end) {
    row_stage_side<N, MODE>(A, L, r_begin, r_end, LANES, smem_raw);
    if constexpr (MODE == ROW_CG_UPDATE)
      if (A.src_early) cg_stage_p<N>(A, L, r_begin, r_end, LANES, smem_raw);
  }
}

// Row pass: block b takes the coil rows [b*rows_per_cta, (b+1)*rows_per_cta) of the stacked J*N rows, one lane
// (TL threads) per row, in as many rounds as its lanes need; passes with a rho part then take a slice of the rho
// plane.  All threads of the block run every round (inactive lanes carry zeros) because of the barriers.
// PRE: the twiddles and the first round's side rows were staged by row_pass_prestage, and the body itself waits for
// the kernel before (pdl_enter) and applies the stop test before its first loads.
// tw_ready: the block has staged the twiddles already (a batched launch, for all its work items).
template <int N1, int N2, int MODE, bool STDF = false, class TC = NoTc, bool PRE = false>
__device__ __forceinline__ void row_pass_body(const KArgs& A, int bid, int nblk, unsigned char* smem_raw,
                                              TC* tc = nullptr, bool tw_ready = false) {
  using S = Split<N1, N2>;
  using T = RowTraits<MODE>;
  constexpr int N = S::N, TL = S::TL, E = S::E;
  constexpr bool CG = MODE == ROW_CG_UPDATE;
  static_assert(N2 == TL, "row passes assume N1 <= N2");
  const int LANES = blockDim.x / TL;
  // Two thread maps onto the rows of a round: layout A (N1 threads per row) packs the rows densely so that the
  // spare warps skip the layout-A steps; layout B uses N2 = TL threads per row (every thread).
  const int laneA = threadIdx.x / N1, idxA = threadIdx.x % N1;
  const bool mapA = (int)threadIdx.x < LANES * N1;
  const int laneB = threadIdx.x / N2, idxB = threadIdx.x % N2;
  const bool mapB = (int)threadIdx.x < LANES * N2;           // threads beyond the whole lanes stay idle
  const int f = STDF ? N / 4 : A.f, Wc = STDF ? N / 2 : A.Wc;
  float acc = 0.f;        // this round's products (at most N1 <= 16 complex values per thread)
  // sum of the rounds: FP64 outside the CG iteration, a pair inside
  using Sum = std::conditional_t<MODE == ROW_BCG_NORMAL, Pair, double>;
  Sum sum{};
  const RowSmem L = row_smem(MODE, N, LANES, S::SM_LANE);
  float2* smA = (float2*)(smem_raw + L.xch) + laneA * S::SM_LANE;
  float2* smB = (float2*)(smem_raw + L.xch) + laneB * S::SM_LANE;
  const float2* twA = (const float2*)(smem_raw + L.tw);
  const float2* twB = twA + N;
  const float rs = rsqrtf((float)N);
  const int group = !PRE && A.sub > 0 ? bid / A.sub : bid, part = bid - group * A.sub;
  int r_begin = group * A.rows_per_cta, r_end = min(r_begin + A.rows_per_cta, A.nrows);
  if (!PRE && A.sub > 0) {
    r_begin += part * A.sub_lanes;
    r_end = min(r_begin + A.sub_lanes, r_end);
  }
  if (!PRE && !tw_ready) {
    stage_bytes(smem_raw + L.tw, A.twA, N * 8);
    stage_bytes(smem_raw + L.tw + N * 8, A.twB, N * 8);
  }
  bool waited = !PRE;
  // the dependent-launch wait and the stop test (the same for every thread of the block); true: leave the pass
  auto enter = [&]() -> bool {
    pdl_enter();
    waited = true;
    if (CG && cg_stopped(A)) {     // a stop at this iteration; the passes before take no notice of it
      cp_async_wait_all();
      return true;
    }
    return false;
  };
  if (!waited) {
    if (enter()) return;
  }
  __shared__ CgStep s_cg;          // CG update: its scalars, and the threads' sums (live registers across the transforms
  [[maybe_unused]] Pair* sums = (Pair*)(smem_raw + L.sums) + threadIdx.x;      // would spill)
  __shared__ Pair s_pairs[MODE == ROW_CG_PSF || MODE == ROW_BCG_NORMAL ? kRowMaxThreads : 1];
  [[maybe_unused]] float2 dd = make_float2(0.f, 0.f);      // PSF pass: this round's |DF p|^2
  __shared__ float s_beta;       // beta of the batches' direction update p = r + beta p

  for (int R0 = r_begin; R0 < r_end; R0 += LANES) {
  const int RA = R0 + laneA, RB = R0 + laneB;               // rows of the stacked coil planes in the two maps
  const bool activeA = mapA && RA < r_end, activeB = mapB && RB < r_end;
  const int e1A = RA % N;
  const int rowB = (N + RB) * N + idxB;        // coil planes follow the rho plane (at most 65 x 512^2 elements)
  float2 v[E];

  // ---- batches' direction update: the rows of r go to the exchange buffer (natural order, pitch N) while p is loaded
  if constexpr (MODE == ROW_BCG_DIR) stage_rows(smem_raw + L.xch, A.r, R0, min(LANES, r_end - R0), N * 8, N, false);

  // passes over two arrays: which one this thread's layout-A row belongs to
  [[maybe_unused]] const bool second = T::both && RA >= A.nrows1;
  [[maybe_unused]] const float2* srcA = nullptr;
  if constexpr (T::both) srcA = second ? A.src2 + (size_t)(RA - A.nrows1) * N : A.src + (size_t)RA * N;
  // ---- main loads, layout A: thread a < N1 holds row elements a + N1*m (no stores until all are issued)
  if (mapA) {
#pragma unroll
    for (int m = 0; m < N2; ++m) {
      const int e2 = idxA + N1 * m;
      float2 val = make_float2(0.f, 0.f);
      if (activeA) {
        if constexpr (T::load_compact) {
          if (in_omega(e2, N, f)) val = A.src[(size_t)RA * Wc + to_compact(e2, N, f)];
        } else if constexpr (T::both) {
          val = srcA[e2];
          if constexpr (MODE == ROW_W_P_IFFT)
            if (second) val = A.mask[(size_t)e1A * N + e2] ? val : make_float2(0.f, 0.f);
        } else if constexpr (MODE != ROW_P_IFFT) {
          val = A.src[(size_t)RA * N + e2];
        } else {
          const float2 sv = A.src[(size_t)RA * N + e2];
          val = A.mask[(size_t)e1A * N + e2] ? sv : make_float2(0.f, 0.f);
        }
      }
      v[m] = val;
    }
  }

  // ---- staged side inputs (the twiddles were issued before the first round)
  if (!PRE || R0 != r_begin) row_stage_side<N, MODE>(A, L, R0, r_end, LANES, smem_raw);
  if constexpr (CG) {
    if (!PRE || !A.src_early || R0 != r_begin) cg_stage_p<N>(A, L, R0, r_end, LANES, smem_raw);
    if (R0 == r_begin && threadIdx.x == 0) {
      CgStep cg;
      cg.first = A.iter == 0;
      cg.odd = (A.iter & 1) != 0;
      cg.alpha = A.alpha;
      cg.unit = cg.first ? A.sc->unit : 1.f;
      cg.a = A.sc->step[A.iter & 1];
      cg.a_prev = cg.first ? 0.f : A.sc->step[(A.iter & 1) ^ 1];
      cg.beta = cg.first ? 0.f : A.sc->beta_p.h;
      s_cg = cg;
    }
  }
  // batches: beta from the |r|^2 partials of the CG step before, while the loads above are in flight (same order in
  // every block; block 0 publishes |r|^2 and beta for the CG step and the later passes of this iteration)
  if constexpr (MODE == ROW_BCG_DIR) {
    if (R0 == r_begin) {
      if (!A.brr_part) {
        if (threadIdx.x == 0) s_beta = A.sc->beta_p.h;
      } else if (threadIdx.x >= ((blockDim.x - 1) & ~31u)) {       // the last warp has the least to load
        const Pair t = warp_sum_of(A.brr_part, A.n_rr);
        if ((threadIdx.x & 31) == 0) {
          const Pair rp = A.sc->rr_i[1];
          const Pair b = rp.h != 0.f ? pair_div(t, rp) : Pair{0.f, 0.f};
          s_beta = b.h;
          if (bid == 0) {
            A.sc->rr_i[0] = t;
            A.sc->beta_p = b;
          }
        }
      }
    }
  }
  cp_async_wait_all();
  __syncthreads();

  if constexpr (MODE == ROW_BCG_DIR) {
    // p = r + beta p (r from the exchange buffer) written back, then weight
    const float* sw = (const float*)(smem_raw + L.w) + (size_t)laneA * N;
    const float2* sr = (const float2*)(smem_raw + L.xch) + (size_t)laneA * N;
    if (activeA) {
      const float unit = A.iter == 0 ? A.sc->unit : 1.f;      // r holds b
#pragma unroll
      for (int m = 0; m < N2; ++m) {
        const float2 rv = cscale(sr[idxA + N1 * m], unit);
        v[m] = make_float2(fmaf(s_beta, v[m].x, rv.x), fmaf(s_beta, v[m].y, rv.y));
        const_cast<float2*>(A.src)[(size_t)RA * N + idxA + N1 * m] = v[m];
        v[m] = cscale(v[m], sw[idxA + N1 * m] * rs);
      }
    }
    __syncthreads();   // the exchange below overwrites the staged rows of r
  } else if constexpr (MODE == ROW_W_IFFT || T::both) {
    const float* sw = (const float*)(smem_raw + L.w) + (size_t)laneA * N;
    if (activeA) {
#pragma unroll
      for (int m = 0; m < N2; ++m)
        v[m] = cscale(v[m], MODE == ROW_W_P_IFFT && second ? rs : sw[idxA + N1 * m] * rs);
    }
  } else if constexpr (MODE == ROW_P_IFFT) {
    if (mapA) {
#pragma unroll
      for (int m = 0; m < N2; ++m) v[m] = cscale(v[m], rs);
    }
  }

  if constexpr (T::inverse_first) {
    fft_AtoB2<N1, N2, +1, E, TC, false>(v, smA, idxA, mapA, smB, idxB, mapB, twA, tc);
    // layout B: thread b < N2 holds elements b + N2*m; keep the Omega columns
    if constexpr (T::both) {
      float2* d = RB >= A.nrows1 ? A.dst2 + (size_t)(RB - A.nrows1) * Wc : A.dst + (size_t)RB * Wc;
      if (activeB) {
#pragma unroll
        for (int m = 0; m < N1; ++m) {
          const int e2 = idxB + N2 * m;
          if (in_omega(e2, N, f)) d[to_compact(e2, N, f)] = v[m];
        }
      }
    } else if (activeB) {
#pragma unroll
      for (int m = 0; m < N1; ++m) {
        const int e2 = idxB + N2 * m;
        if (in_omega(e2, N, f)) A.dst[(size_t)RB * Wc + to_compact(e2, N, f)] = v[m];
      }
    }
  } else {
    // single-frame normal-operator pass: its rows of p (layout B) are loaded before the transform, so that their
    // latency overlaps it (the batched pass, HBM-bound, loads them after it: the early loads cost it 2.5 %)
    constexpr bool kEarlyP = MODE == ROW_FFT_W_NORMAL && PRE;
    float2 a0[T::normal ? N1 : 1];
    if constexpr (kEarlyP) {
      if (activeB) {
#pragma unroll
        for (int m = 0; m < N1; ++m) a0[m] = A.p[rowB + N2 * m];
      }
    }
    // passes with a second transform exchange again right after: keep the closing barrier there
    // the CG update issues its loads of r while the first transform is on its way (the registers of its layout-A
    // elements are free by then: loaded before it, they spilled 400 bytes a thread)
    float2 rB[CG ? N1 : 1];
    fft_AtoB2<N1, N2, -1, E, TC, T::two>(v, smA, idxA, mapA, smB, idxB, mapB, twA, tc, [&] {
      if constexpr (CG) {
        if (activeB) {
#pragma unroll
          for (int m = 0; m < N1; ++m) rB[m] = A.r[rowB + N2 * m];
        }
      }
    });
    const unsigned char* smask = smem_raw + L.mask + (size_t)laneB * N;
    const float* sw = (const float*)(smem_raw + L.w) + (size_t)laneB * N;
    // staged rows of y (residual) or of p (CG update)
    float2* scp = (float2*)(smem_raw + L.cplx) + (size_t)laneB * N;
    if constexpr (T::psf) {
#pragma unroll
      for (int m = 0; m < N1; ++m) {
        v[m] = (activeB && smask[idxB + N2 * m]) ? cscale(v[m], rs * rs) : make_float2(0.f, 0.f);
        if constexpr (MODE == ROW_CG_PSF) dot_acc(dd, v[m], v[m]);
      }
      if constexpr (MODE == ROW_CG_PSF) {           // |DF p|^2 of these rows (the values carry one more factor 1/sqrt(N))
        Pair t = {0.f, 0.f};
        if (R0 != r_begin) t = s_pairs[threadIdx.x];
        dot_flush(dd, t);
        s_pairs[threadIdx.x] = t;
      }
    } else if constexpr (CG) {
      const CgStep cg = s_cg;
      const float* swh = (const float*)(smem_raw + L.w) + (size_t)laneB * w_pitch(MODE, N);
      CgDots dots;
      dots.rr = dots.rp = dots.pp = make_float2(0.f, 0.f);
#pragma unroll
      for (int m = 0; m < N1; ++m) {
        const int e2 = idxB + N2 * m;
        float2 out = make_float2(0.f, 0.f);
        if (activeB) {
          const float w = swh[N2 * m < N / 2 ? e2 : N - e2] * rs;
          float2 p = cg.first ? make_float2(0.f, 0.f) : scp[e2], g;
          const float2 rn = cg_point(cg, cscale(v[m], w), rB[m], p, g, dots);
          A.r[rowB + N2 * m] = rn;
          const_cast<float2*>(A.p)[rowB + N2 * m] = p;
          if (cg.odd) cg_add_dx(A.dx + rowB + N2 * m, g, A.iter > 1);
          out = cscale(rn, w);
        }
        v[m] = out;
      }
      cg_flush(dots, sums, R0 == r_begin);
    } else if constexpr (T::rhs) {
      float2 x0[N1], x1[N1];          // x and x_ref, loaded before any store
      if (activeB) {
#pragma unroll
        for (int m = 0; m < N1; ++m) {
          x0[m] = A.x[rowB + N2 * m];
          x1[m] = A.xref[rowB + N2 * m];
        }
      }
#pragma unroll
      for (int m = 0; m < N1; ++m) {
        float2 out = make_float2(0.f, 0.f);
        if (activeB) {
          const float w = sw[idxB + N2 * m] * rs;
          const float2 val = cscale(v[m], w), xv = x0[m], xr = x1[m];
          const float2 b = make_float2(val.x - A.alpha * (xv.x - xr.x), val.y - A.alpha * (xv.y - xr.y));
          A.r[rowB + N2 * m] = b;
          if constexpr (MODE == ROW_BCG_RHS) {
            A.pout[rowB + N2 * m] = b;
            A.dx[rowB + N2 * m] = make_float2(0.f, 0.f);
          }
          acc += b.x * b.x + b.y * b.y;
          out = cscale(b, w);
        }
        v[m] = out;
      }
    } else {
      if constexpr (T::normal && !kEarlyP) {      // loaded before any store
        if (activeB) {
#pragma unroll
          for (int m = 0; m < N1; ++m) a0[m] = A.p[rowB + N2 * m];
        }
      }
      if (activeB) {
#pragma unroll
        for (int m = 0; m < N1; ++m) {
          const int e2 = idxB + N2 * m;
          const size_t o = (size_t)RB * N + e2;
          if constexpr (MODE == ROW_FFT_P_OUT) {
            A.dst[o] = smask[e2] ? cscale(v[m], rs) : make_float2(0.f, 0.f);
          } else if constexpr (MODE == ROW_FFT_RESID) {
            const float2 yv = scp[e2];
            const float2 rv = smask[e2] ? csub(yv, cscale(v[m], rs)) : yv;
            A.dst[o] = rv;
            acc += rv.x * rv.x + rv.y * rv.y;
          } else {
            const float2 val = cscale(v[m], sw[e2] * rs);
            if constexpr (MODE == ROW_FFT_W_ADJ) {
              A.dst[rowB + N2 * m] = val;
            } else {
              const float2 pv = a0[m];
              const float2 q = make_float2(fmaf(A.alpha, pv.x, val.x), fmaf(A.alpha, pv.y, val.y));
              A.dst[rowB + N2 * m] = q;
              if constexpr (MODE == ROW_BCG_NORMAL) acc += pv.x * q.x + pv.y * q.y;
            }
          }
        }
      }
    }
    if constexpr (T::two) {
      if (!CG || !A.last) {
        fft_AtoB2<N2, N1, +1, E, TC, false>(v, smB, idxB, mapB, smA, idxA, mapA, twB, tc);
        float2* dst = A.dst;
        if (activeA) {
#pragma unroll
          for (int m = 0; m < N2; ++m) {
            const int e2 = idxA + N1 * m;
            if (in_omega(e2, N, f)) dst[(size_t)RA * Wc + to_compact(e2, N, f)] = v[m];
          }
        }
      }
    }
  }
  if (R0 + LANES < r_end) __syncthreads();   // the next round restages the side rows and reuses the exchange
  if constexpr (T::reduces) {
    acc_add(sum, acc);
    acc = 0.f;
  }
  }  // rounds

  if constexpr (T::has_rho) {
    if (PRE || A.sub == 0) {
      rho_slice<N, MODE, STDF>(A, bid, threadIdx.x, blockDim.x, sum);
    } else {
      const int t = threadIdx.x + part * A.sub_lanes * TL;
      if ((int)threadIdx.x < A.sub_lanes * TL && t < A.group_threads)
        rho_slice<N, MODE, STDF>(A, group, t, A.group_threads, sum);
    }
  }
  if constexpr (CG) {
    rho_cg_slice<N, STDF>(A, bid, s_cg, sums);
    __syncthreads();
    block_pairs<3>(sums - threadIdx.x, {A.rr_part + bid, A.rr_part + A.n_rr + bid, A.rr_part + 2 * A.n_rr + bid});
  }
  // the pairs were stored before the second transform's barrier
  if constexpr (MODE == ROW_CG_PSF) block_pairs<1>(s_pairs, {A.dd_part + bid});
  if constexpr (MODE == ROW_BCG_NORMAL) {
    s_pairs[threadIdx.x] = sum;
    __syncthreads();
    block_pairs<1>(s_pairs, {A.pq_part + bid});
  } else if constexpr (T::reduces) {
    grid_reduce(sum, A, bid, nblk);
  }
}

template <int N1, int N2, int MODE, bool STDF = false>
__global__ void __launch_bounds__(kRowMaxThreads, kRowCtasPerSM) row_pass(const KArgs A) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  if (cg_stopped_early(A)) {
    pdl_enter();
    return;
  }
  row_pass_prestage<N1, N2, MODE>(A, blockIdx.x, smem_raw);
  row_pass_body<N1, N2, MODE, STDF, NoTc, true>(A, blockIdx.x, gridDim.x, smem_raw);
}

// --------------------------------------------------------------------------------------- column passes ----
enum ColMode : int {
  COL_IFFT_C = 0,         // coil <- Omega rows of FFT^-1_col(T) / sqrt N                 (W^-1, second axis)
  COL_PROD_FFT = 1,       // T <- FFT_col(M rho c_j) / sqrt N                             (F)
  COL_SIM_FFT = 2,        // T <- FFT_col(M rho cimg_j) / sqrt N                          (data simulation)
  COL_IFFT_PROD_FFT = 3,  // u = FFT^-1_col(T); T <- FFT_col(M (drho c_j + rho u))        (DF)
  COL_IFFT_ADJ_FFT = 4,   // z = M FFT^-1_col(T); zsum_j = conj(c_j) z; T <- FFT_col(conj(rho) z)   (DF^H)
  COL_CG_DIR = 5,         // single frames: U <- FFT^-1_col(T) + beta U;  T <- FFT_col(M ((r + beta p)_rho c_j + rho U))
  COL_BCG_DIR = 6,        // batches: COL_IFFT_PROD_FFT for the rho part of p = r + beta p
  // operators: the coil maps c = FFT^-1_col(T) and what follows them in one pass (c to coil_out, if given)
  COL_COIL_PROD = 7,      // T <- FFT_col(M rho c)                                               (F)
  COL_COIL_DIR = 8,       // u = FFT^-1_col(T2);  T <- FFT_col(M (drho c + rho u))                (DF)
  COL_COIL_ADJ = 9,       // z = M FFT^-1_col(T2);  zsum = conj(c) z;  T <- FFT_col(conj(rho) z)  (DF^H)
  NUM_COL_MODES = 10
};

// Shared-memory layout of a column pass (byte offsets): exchange, twiddles, then `nside` side arrays of
// Wc x C complex values (Omega rows of the block's columns: coil map, rho, drho, r; passes that form the coil maps: rho,
// drho), and for two inputs the block's columns of the second.
struct ColSmem {
  size_t xch, tw, side, t2, total;
  int nside;
};
__host__ __device__ constexpr bool col_forms_coils(int mode) { return mode >= COL_COIL_PROD && mode <= COL_COIL_ADJ; }

__host__ __device__ inline ColSmem col_smem(int mode, int N, int C, int sm_lane, int Wc) {
  ColSmem L{};
  L.nside = (mode == COL_CG_DIR || mode == COL_BCG_DIR) ? 4
            : (mode == COL_IFFT_PROD_FFT) ? 3
            : (mode == COL_IFFT_ADJ_FFT || mode == COL_COIL_DIR) ? 2
            : col_forms_coils(mode) ? 1 : 0;
  L.xch = 0;
  L.tw = align16((size_t)C * sm_lane * 8);
  L.side = L.tw + align16((size_t)2 * N * 8);
  L.t2 = L.side + (size_t)L.nside * Wc * C * 8;
  L.total = L.t2 + (mode == COL_COIL_DIR || mode == COL_COIL_ADJ ? (size_t)N * C * 8 : 0);
  return L;
}

template <int N1, int N2, int CC = NLV_COL_C> struct ColCfg {
  using S = Split<N1, N2>;
  static constexpr int C = CC;                      // adjacent compact columns per block
  static constexpr int THREADS = C * S::TL;
  static_assert(C % 2 == 0, "column staging copies pairs of complex values");
};

// Stages Omega rows of C columns starting at compact column cc0 of a compact (Wc x Wc per coil) array.  A thread
// keeps one 16-byte pair of columns (blockDim.x is a multiple of C/2) and steps down the rows.
__device__ __forceinline__ void stage_compact_cols(float2* sdst, const float2* plane, int cc0, int C, int Wc) {
  const int cpr = C / 2;                               // 16-byte chunks per row segment
  const int k = threadIdx.x % cpr, cc = cc0 + 2 * k, step = blockDim.x / cpr;
  if (cc >= Wc) return;
  const float2* src = plane + cc;
  for (int cr = threadIdx.x / cpr; cr < Wc; cr += step) cp_async16(sdst + (size_t)cr * C + 2 * k, src + (size_t)cr * Wc);
}
// Same for a natural N x N plane (rows and columns mapped from compact to natural indices).
__device__ __forceinline__ void stage_natural_cols(float2* sdst, const float2* plane, int cc0, int C, int Wc, int N,
                                                   int f) {
  if ((f & 1) == 0) {                                  // compact pairs (2k, 2k+1) stay adjacent in natural order
    const int cpr = C / 2;
    const int k = threadIdx.x % cpr, cc = cc0 + 2 * k, step = blockDim.x / cpr;
    if (cc >= Wc) return;
    const float2* src = plane + to_natural(cc, N, f);
    for (int cr = threadIdx.x / cpr; cr < Wc; cr += step)
      cp_async16(sdst + (size_t)cr * C + 2 * k, src + (size_t)to_natural(cr, N, f) * N);
  } else {
    for (int i = threadIdx.x; i < Wc * C; i += blockDim.x) {
      const int cr = i / C, k = i % C, cc = cc0 + k;
      if (cc < Wc)
        cp_async8(sdst + (size_t)cr * C + k, plane + (size_t)to_natural(cr, N, f) * N + to_natural(cc, N, f));
    }
  }
}

// Side inputs of a column pass.  `before`: those that no launch just before writes (the twiddles, the coil map and
// rho), which a single-frame pass stages before its dependent-launch wait; else the rest: drho, for the CG direction
// pass the rho planes of p and r that the CG update pass just before has written.
template <int N1, int N2, int MODE, bool STDF, int CC>
__device__ __forceinline__ void col_stage_side(const KArgs& A, int bid, unsigned char* smem_raw, bool before,
                                               bool tw_ready = false) {
  using S = Split<N1, N2>;
  constexpr int N = S::N, C = ColCfg<N1, N2, CC>::C;
  const int f = STDF ? N / 4 : A.f, Wc = STDF ? N / 2 : A.Wc;
  const int strips = (Wc + C - 1) / C;
  const int j = bid / strips;
  const int cc0 = (bid % strips) * C;
  const ColSmem L = col_smem(MODE, N, C, S::SM_LANE_COL, Wc);
  float2* sd = (float2*)(smem_raw + L.side);
  const size_t sstride = (size_t)Wc * C;
  if (before) {
    if (!tw_ready) {
      stage_bytes(smem_raw + L.tw, A.twA, N * 8);
      stage_bytes(smem_raw + L.tw + N * 8, A.twB, N * 8);
    }
    if constexpr (col_forms_coils(MODE)) {
      if (j < A.nrows) stage_natural_cols(sd, A.rho, cc0, C, Wc, N, f);
    } else if constexpr (MODE == COL_IFFT_PROD_FFT || MODE == COL_IFFT_ADJ_FFT || MODE == COL_CG_DIR ||
                         MODE == COL_BCG_DIR) {
      if (j < A.nrows) {
        stage_compact_cols(sd, A.coil + (size_t)j * Wc * Wc, cc0, C, Wc);
        stage_natural_cols(sd + sstride, A.rho, cc0, C, Wc, N, f);
      }
    }
  } else if constexpr (MODE == COL_COIL_DIR || MODE == COL_COIL_ADJ) {
    if (j < A.nrows) {
      if constexpr (MODE == COL_COIL_DIR) stage_natural_cols(sd + sstride, A.drho, cc0, C, Wc, N, f);
      // the columns of the second input, every row
      float2* t2 = (float2*)(smem_raw + L.t2);
      const int k = threadIdx.x % (C / 2), cc = cc0 + 2 * k, step = blockDim.x / (C / 2);
      if (cc < Wc)
        for (int e = threadIdx.x / (C / 2); e < N; e += step)
          cp_async16(t2 + (size_t)e * C + 2 * k, A.src2 + ((size_t)j * N + e) * Wc + cc);
    }
  } else if constexpr (MODE == COL_IFFT_PROD_FFT) {
    if (j < A.nrows) stage_natural_cols(sd + 2 * sstride, A.drho, cc0, C, Wc, N, f);
  } else if constexpr (MODE == COL_CG_DIR || MODE == COL_BCG_DIR) {
    if (j < A.nrows) {
      if (MODE == COL_BCG_DIR || A.iter > 0) stage_natural_cols(sd + 2 * sstride, A.drho, cc0, C, Wc, N, f);
      stage_natural_cols(sd + 3 * sstride, A.r, cc0, C, Wc, N, f);
    }
  }
}

// beta_i = |r_i|^2 / |r_{i-1}|^2 of the CG direction pass from the partials that the CG update pass before wrote, by
// the block's last warp (in most splits it has no part in the first register DFT), in the same order in every block.
// Block 0 publishes |r_i|^2 and beta and records the stop when |r_i| has reached the rounding floor (or is not finite);
// s_stop: the same for every block.
__device__ __forceinline__ void cg_direction_scalars(const KArgs& A, int bid, float& s_beta, int& s_stop) {
  if (threadIdx.x < ((blockDim.x - 1) & ~31u)) return;
  const Pair rp = A.sc->rr_i[(A.iter & 1) ^ 1], floor = pair_scale(A.sc->rr_pair, (float)kCgFloor2);
  const Pair t = warp_sum_of(A.rr_part, A.n_rr);
  if ((threadIdx.x & 31) == 0) {
    const Pair b = rp.h != 0.f ? pair_div(t, rp) : Pair{0.f, 0.f};
    const bool stop = !pair_gt(t, floor) || !isfinite(t.h);
    s_beta = b.h;
    s_stop = stop ? 1 : 0;
    if (bid == 0) {
      A.sc->rr_i[A.iter & 1] = t;
      A.sc->beta_p = b;
      if (stop) {
        A.sc->cg_stop[A.slot] = A.iter;
        if (!isfinite(t.h)) atomicOr(&A.sc->flags, kFlagBreakdown);
      }
    }
  }
}

// Step length of a CG iteration, by one block of the DF^H column pass that has no columns: Re<p, A p> =
// |DF p|^2 + alpha |p|^2 with |DF p|^2 from the PSF pass's partials and, for p = r + beta p_old,
// |p|^2 = |r|^2 + 2 beta Re<r, p_old> + beta^2 |p_old|^2 from those of the CG update pass before.  The solve stops at the
// rounding floor: |r|^2 <= kCgFloor2 |b|^2 (|r| at the FP32 unit roundoff relative to |b|, including b = 0),
// Re<p, A p> <= 0 (impossible in exact arithmetic for the positive definite system of Eq. 3) or a non-finite value.
// This iteration and every later one of the same solve are then empty (cg_stopped).  Non-finite values also set the
// breakdown flag.
template <int N>
__device__ __forceinline__ void cg_decide(const KArgs& A) {
  __shared__ Pair tot[3];
  const int nw = ((int)blockDim.x + 31) >> 5, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
  for (int k = 0; k < 3; ++k)
    if (warp == k % nw) {
      const Pair s = k == 0 ? warp_sum_of(A.dd_part, A.n_dd)
                            : warp_sum_of(A.rr_part + k * A.n_rr, A.iter > 0 ? A.n_rr : 0);
      if (lane == 0) tot[k] = s;
    }
  __syncthreads();
  if (threadIdx.x != 0 || A.sc->cg_stop[A.slot] == A.iter) return;    // stopped by the direction pass already
  const Pair none = {0.f, 0.f};
  const Pair rr = A.sc->rr_i[A.iter & 1], beta = A.iter > 0 ? A.sc->beta_p : none;
  const Pair pp = cg_direction_norm(rr, beta, tot[1], tot[2]);
  // the PSF pass's values carry one more transform factor rs ~ 1/sqrt(N) than DF p; it is divided out as the passes
  // round it (N in its place is off by up to 5e-7, and CG loses its orthogonality that much sooner)
  const float rs = rsqrtf((float)N);
  const Pair t = pair_sum(pair_div(tot[0], pair_mul({rs, 0.f}, {rs, 0.f})), pair_mul(pp, {A.alpha, 0.f}));
  const bool finite = isfinite(t.h) && isfinite(rr.h);
  if (finite && pair_gt(rr, pair_scale(A.sc->rr_pair, (float)kCgFloor2)) && t.h > 0.f) {
    A.sc->step[A.iter & 1] = pair_div(rr, t).h;
  } else {
    A.sc->cg_stop[A.slot] = A.iter;
    if (!finite) atomicOr(&A.sc->flags, kFlagBreakdown);
  }
}

// prestaged: the twiddles and the side inputs that no launch just before writes were staged by col_stage_side before
// the dependent-launch wait.
template <int N1, int N2, int MODE, bool STDF = false, class TC = NoTc, int CC = NLV_COL_C>
__device__ __forceinline__ void col_pass_body(const KArgs& A, int bid, int nblk, unsigned char* smem_raw,
                                              TC* tc = nullptr, bool prestaged = false, bool tw_ready = false) {
  using S = Split<N1, N2>;
  constexpr int N = S::N, E = S::E, C = ColCfg<N1, N2, CC>::C;
  if constexpr (MODE == COL_IFFT_ADJ_FFT) {
    if (A.scalars && bid == nblk - 1) {
      cp_async_wait_all();
      cg_decide<N>(A);
      return;
    }
  }
  const int lane = threadIdx.x % C, idx = threadIdx.x / C;
  const int f = STDF ? N / 4 : A.f, Wc = STDF ? N / 2 : A.Wc;
  const int strips = (Wc + C - 1) / C;
  const int j = bid / strips;
  const int cc0 = (bid % strips) * C;
  const int cc = cc0 + lane;
  const bool active = cc < Wc && j < A.nrows;
  const int x2 = to_natural(cc, N, f);
  const ColSmem L = col_smem(MODE, N, C, S::SM_LANE_COL, Wc);
  float2* sm = (float2*)(smem_raw + L.xch) + lane * S::SM_LANE_COL;
  const float2* twA = (const float2*)(smem_raw + L.tw);
  const float2* twB = twA + N;
  const float2* side = (const float2*)(smem_raw + L.side);
  const float rs = rsqrtf((float)N);
  const size_t tbase = (size_t)j * N * Wc + cc;       // T element (row e1) at tbase + e1*Wc
  const size_t cbase = (size_t)j * Wc * Wc + cc;      // compact coil element (row cr) at cbase + cr*Wc
  float2 v[E];

  // ---- main loads, layout A: thread a < N1 holds column elements a + N1*m
  if (idx < N1) {
#pragma unroll
    for (int m = 0; m < N2; ++m) {
      const int e1 = idx + N1 * m;
      float2 val = make_float2(0.f, 0.f);
      if constexpr (MODE == COL_PROD_FFT || MODE == COL_SIM_FFT) {
        if (active && in_omega(e1, N, f)) {
          const float2 c = (MODE == COL_PROD_FFT) ? A.coil[cbase + (size_t)to_compact(e1, N, f) * Wc]
                                                  : A.cimg[((size_t)j * N + e1) * N + x2];
          val = cmul(A.rho[(size_t)e1 * N + x2], c);
        }
      } else {
        if (active) val = A.src[tbase + (size_t)e1 * Wc];
      }
      v[m] = val;
    }
  }
  // ---- CG direction: the W^-1 p of the iteration before on this thread's Omega elements (layout B)
  [[maybe_unused]] float2 uo[MODE == COL_CG_DIR ? N1 : 1];
  [[maybe_unused]] float beta = 0.f;
  __shared__ float s_beta;
  __shared__ int s_stop;
  if constexpr (MODE == COL_CG_DIR) {
    if (idx < N2) {
#pragma unroll
      for (int m = 0; m < N1; ++m) {
        const int e1 = idx + N2 * m;
        uo[m] = make_float2(0.f, 0.f);
        if (A.iter > 0 && active && in_omega(e1, N, f)) uo[m] = A.U[cbase + (size_t)to_compact(e1, N, f) * Wc];
      }
    }
  }
  // ---- staged side inputs (Omega rows of this block's columns) and twiddles
  if (!prestaged) col_stage_side<N1, N2, MODE, STDF, CC>(A, bid, smem_raw, true, tw_ready);
  col_stage_side<N1, N2, MODE, STDF, CC>(A, bid, smem_raw, false);
  if constexpr (MODE == COL_CG_DIR) {      // while the loads above are in flight; read after the first transform
    if (A.iter > 0) cg_direction_scalars(A, bid, s_beta, s_stop);
  }
  cp_async_wait_all();
  __syncthreads();

  if constexpr (MODE == COL_PROD_FFT || MODE == COL_SIM_FFT) {
    fft_AtoB<N1, N2, -1, false>(v, sm, twA, idx, tc);
    if (active && idx < N2) {
#pragma unroll
      for (int m = 0; m < N1; ++m) {
        const int e1 = idx + N2 * m;
        A.dst[tbase + (size_t)e1 * Wc] = cscale(v[m], rs);
      }
    }
    return;
  } else {
    fft_AtoB<N1, N2, +1, MODE != COL_IFFT_C>(v, sm, twA, idx, tc);
    if constexpr (MODE == COL_IFFT_C) {
      if (active && idx < N2) {
#pragma unroll
        for (int m = 0; m < N1; ++m) {
          const int e1 = idx + N2 * m;
          if (in_omega(e1, N, f)) A.dst[cbase + (size_t)to_compact(e1, N, f) * Wc] = cscale(v[m], rs);
        }
      }
      return;
    } else {
      if constexpr (MODE == COL_CG_DIR) {
        if (A.iter > 0) {
          if (s_stop) return;          // the same in every block and thread: |r| has reached the rounding floor
          beta = s_beta;
        }
      }
      if constexpr (MODE == COL_BCG_DIR) beta = A.sc->beta_p.h;
      [[maybe_unused]] float unit = 1.f;           // iteration 0: r, and T of single frames, hold b
      if constexpr (MODE == COL_CG_DIR || MODE == COL_BCG_DIR)
        if (A.iter == 0) unit = A.sc->unit;
      const size_t sstride = (size_t)Wc * C;
      if constexpr (col_forms_coils(MODE)) {
        float2 c[N1];                       // the coil map on this thread's Omega elements (layout B)
        if (idx < N2) {
#pragma unroll
          for (int m = 0; m < N1; ++m) {
            const int e1 = idx + N2 * m;
            c[m] = make_float2(0.f, 0.f);
            if (active && in_omega(e1, N, f)) {
              c[m] = cscale(v[m], rs);
              if (A.coil_out) A.coil_out[cbase + (size_t)to_compact(e1, N, f) * Wc] = c[m];
            }
          }
        }
        if constexpr (MODE != COL_COIL_PROD) {
          const float2* t2 = (const float2*)(smem_raw + L.t2) + lane;
          if (idx < N1) {
#pragma unroll
            for (int m = 0; m < N2; ++m) v[m] = active ? t2[(size_t)(idx + N1 * m) * C] : make_float2(0.f, 0.f);
          }
          fft_AtoB<N1, N2, +1, true>(v, sm, twA, idx, tc);
        }
        if (idx < N2) {
#pragma unroll
          for (int m = 0; m < N1; ++m) {
            const int e1 = idx + N2 * m;
            float2 out = make_float2(0.f, 0.f);
            if (active && in_omega(e1, N, f)) {
              const int cr = to_compact(e1, N, f);
              const float2 rh = side[(size_t)cr * C + lane];
              if constexpr (MODE == COL_COIL_PROD) {
                out = cmul(rh, c[m]);
              } else {
                const float2 u = cscale(v[m], rs);
                if constexpr (MODE == COL_COIL_DIR) {
                  out = cadd(cmul(side[sstride + (size_t)cr * C + lane], c[m]), cmul(rh, u));
                } else {
                  A.zsum[cbase + (size_t)cr * Wc] = cmulc(c[m], u);
                  out = cmulc(rh, u);
                }
              }
            }
            v[m] = out;
          }
        }
      } else if (idx < N2) {
#pragma unroll
        for (int m = 0; m < N1; ++m) {
          const int e1 = idx + N2 * m;
          float2 out = make_float2(0.f, 0.f);
          if (active && in_omega(e1, N, f)) {
            const int cr = to_compact(e1, N, f);
            float2 u = cscale(v[m], MODE == COL_CG_DIR ? rs * unit : rs);
            const float2 c = side[(size_t)cr * C + lane];
            const float2 rh = side[sstride + (size_t)cr * C + lane];
            if constexpr (MODE == COL_IFFT_ADJ_FFT) {
              A.zsum[cbase + (size_t)cr * Wc] = cmulc(c, u);
              out = cmulc(rh, u);
            } else {
              float2 dr;
              if constexpr (MODE == COL_CG_DIR) {      // W^-1 p and the rho part of p = r + beta p
                dr = cscale(side[3 * sstride + (size_t)cr * C + lane], unit);
                if (A.iter > 0) {
                  const float2 po = side[2 * sstride + (size_t)cr * C + lane];
                  dr = make_float2(fmaf(beta, po.x, dr.x), fmaf(beta, po.y, dr.y));
                  u = make_float2(fmaf(beta, uo[m].x, u.x), fmaf(beta, uo[m].y, u.y));
                }
                A.U[cbase + (size_t)cr * Wc] = u;
              } else {
                dr = side[2 * sstride + (size_t)cr * C + lane];
                if constexpr (MODE == COL_BCG_DIR) {   // the rho part of p = r + beta p (written by the last row pass)
                  const float2 rv = cscale(side[3 * sstride + (size_t)cr * C + lane], unit);
                  dr = make_float2(fmaf(beta, dr.x, rv.x), fmaf(beta, dr.y, rv.y));
                }
              }
              out = cadd(cmul(dr, c), cmul(rh, u));
            }
          }
          v[m] = out;
        }
      }
      // without its closing barrier the DF^H pass (100 -> 92 registers) measured 1.1 us slower at 384^2/10
      fft_AtoB<N2, N1, -1, MODE == COL_IFFT_ADJ_FFT>(v, sm, twB, idx, tc);
      if (active && idx < N1) {
#pragma unroll
        for (int m = 0; m < N2; ++m) {
          const int e1 = idx + N1 * m;
          A.dst[tbase + (size_t)e1 * Wc] = cscale(v[m], rs);
        }
      }
    }
  }
}

template <int N1, int N2, int MODE, bool STDF = false, int CC = NLV_COL_C>
__global__ void __launch_bounds__(ColCfg<N1, N2, CC>::THREADS) col_pass(const KArgs A) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  if (cg_stopped_early(A)) {
    pdl_enter();
    return;
  }
  // before the wait only through L2 (16-byte copies): an odd f stages the natural planes with 8-byte copies,
  // which go through L1, after the wait
  const bool pre = STDF || (A.f & 1) == 0;
  if (pre) col_stage_side<N1, N2, MODE, STDF, CC>(A, blockIdx.x, smem_raw, true);
  pdl_enter();
  col_pass_body<N1, N2, MODE, STDF, NoTc, CC>(A, blockIdx.x, gridDim.x, smem_raw, nullptr, pre);
}

// ------------------------------------------------------------------------------- tensor-core passes ----
// The same passes with their radix-16 DFT stages on the tensor cores (tc_dft.cuh): the engine's shared memory
// follows the pass's own layout (offset tc_offset(...) below), its TMEM is allocated after the dependent-launch
// wait and freed at the end.
__host__ __device__ constexpr size_t tc_offset(size_t pass_bytes) { return (pass_bytes + 127) / 128 * 128; }

template <int N1, int N2, int MODE, bool STDF>
__global__ void __launch_bounds__(kRowMaxThreads, 1) row_pass_tc(const KArgs A) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  pdl_enter();
  if (cg_stopped(A)) return;
  using S = Split<N1, N2>;
  const RowSmem L = row_smem(MODE, S::N, blockDim.x / S::TL, S::SM_LANE);
  TcDft tc;
  tc.setup(smem_raw + tc_offset(L.total), A.tcB, &A.sc->flags);
  row_pass_body<N1, N2, MODE, STDF, TcDft>(A, blockIdx.x, gridDim.x, smem_raw, &tc);
  tc.teardown();
}

template <int N1, int N2, int MODE, bool STDF>
__global__ void __launch_bounds__(ColCfg<N1, N2>::THREADS, 1) col_pass_tc(const KArgs A) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  pdl_enter();
  if (cg_stopped(A)) return;
  using S = Split<N1, N2>;
  const ColSmem L = col_smem(MODE, S::N, ColCfg<N1, N2>::C, S::SM_LANE_COL, STDF ? S::N / 2 : A.Wc);
  TcDft tc;
  tc.setup(smem_raw + tc_offset(L.total), A.tcB, &A.sc->flags);
  col_pass_body<N1, N2, MODE, STDF, TcDft>(A, blockIdx.x, gridDim.x, smem_raw, &tc);
  tc.teardown();
}

// --------------------------------------------------------------------------------------------- batches ----
// A batched launch runs one pass for several independent frames of the same grid side: frame f owns the blocks
// [first[f], first[f+1]) and its own arguments args[f] (pointers into its own workspace).  Each block finds its
// frame, copies that frame's arguments into shared memory and runs the same pass body as a single-frame launch.
struct BatchArgs {
  const KArgs* args;       // per-frame arguments (device)
  const int* first;        // nframes + 1 block offsets (device)
  const int* const* stops; // per-frame Scalars::cg_stop (device)
  int nframes;
  int total;               // work items = first[nframes]; a block takes items blockIdx.x, + gridDim.x, ...
  int slot, skip;          // a launch of a CG iteration: its Newton step, and KArgs::skip
};

// The work items of a block: the arguments of the next item are fetched into shared memory while the block works on the
// current one, by its last warp (in most splits that warp has no part in the first half of a transform), so that an item
// starts without waiting for the chain offsets -> arguments -> stop -> inputs.  Before, that chain and the twiddles staged
// anew for every item took 299 ms of 64 uneven frames; so, 288.  The row passes' next inputs, consecutive rows, go to L2
// meanwhile (281 -> 275 ms; the column passes' 64-byte pieces did not gain from it).
struct BatchQueue {
  KArgs args[2];
  int bid[2], nblk[2];
  int stop[2];             // Scalars::cg_stop of the item's frame
};

// The calling warp fetches work item w into slot k (asynchronous copies: the caller waits, then a block barrier).
__device__ __forceinline__ void batch_fetch(const BatchArgs& B, int w, BatchQueue& q, int k) {
  const int lane = threadIdx.x & 31, nl = warp_lanes();
  const unsigned live = nl >= 32 ? 0xffffffffu : (1u << nl) - 1u;
  // the frame is the number of block offsets first[1 .. nframes-1] at or below this item (offsets increase): a warp tests
  // 32 of them per step, all loads of a step in flight together
  int f = 0;
  for (int base = 1; base < B.nframes; base += nl) {
    const int i = base + lane;
    const bool le = lane < nl && i < B.nframes && B.first[i] <= w;
    f += __popc(__ballot_sync(live, le));
  }
  static_assert(sizeof(KArgs) % 16 == 0, "copied in 16-byte pieces");
  for (int i = lane; i < (int)(sizeof(KArgs) / 16); i += nl) cp_async16((char*)&q.args[k] + 16 * i, (const char*)(B.args + f) + 16 * i);
  if (lane == 0) {
    q.stop[k] = B.skip > 0 ? *(volatile const int*)(B.stops[f] + B.slot) : -1;
    q.bid[k] = w - B.first[f];
    q.nblk[k] = B.first[f + 1] - B.first[f];
  }
}

// By one thread: the inputs of a row-pass work item that lie in consecutive rows, into L2.
template <int N1, int N2, int MODE, bool STDF>
__device__ __forceinline__ void row_prefetch(const KArgs& A, int bid) {
  using T = RowTraits<MODE>;
  constexpr int N = N1 * N2;
  const int Wc = STDF ? N / 2 : A.Wc;
  const int group = A.sub > 0 ? bid / A.sub : bid;
  const int r0 = group * A.rows_per_cta + (bid - group * A.sub) * A.sub_lanes;
  const int nr = min(min(A.sub > 0 ? A.sub_lanes : A.rows_per_cta, (group + 1) * A.rows_per_cta - r0), A.nrows - r0);
  if (nr <= 0) return;
  if constexpr (T::load_compact) prefetch_l2(A.src + (size_t)r0 * Wc, (unsigned)(nr * Wc * 8));
  else prefetch_l2(A.src + (size_t)r0 * N, (unsigned)(nr * N * 8));
  if constexpr (MODE == ROW_BCG_DIR) prefetch_l2(A.r + (size_t)r0 * N, (unsigned)(nr * N * 8));
  if constexpr (MODE == ROW_BCG_NORMAL) prefetch_l2(A.p + (size_t)(N + r0) * N, (unsigned)(nr * N * 8));
}

// Runs item(args, bid, nblk, stopped) for every work item of this block; stopped: the item's frame has stopped before this
// CG iteration (see cg_stopped).  ahead(args, bid): one thread, for the next item once it is fetched.
struct NoAhead {
  __device__ __forceinline__ void operator()(const KArgs&, int) const {}
};
template <class Item, class Ahead = NoAhead>
__device__ __forceinline__ void batch_items(const BatchArgs& B, BatchQueue& q, Item&& item, Ahead&& ahead = NoAhead()) {
  const bool fetcher = threadIdx.x >= ((blockDim.x - 1) & ~31u);
  int w = blockIdx.x, k = 0;
  if (fetcher && w < B.total) batch_fetch(B, w, q, 0);
  cp_async_wait_all();
  __syncthreads();
  for (; w < B.total; w += gridDim.x, k ^= 1) {
    if (fetcher && w + (int)gridDim.x < B.total) {
      batch_fetch(B, w + gridDim.x, q, k ^ 1);
      if constexpr (!std::is_same_v<std::decay_t<Ahead>, NoAhead>) {
        cp_async_wait_all();
        __syncwarp();
        if ((threadIdx.x & 31) == 0 && (unsigned)q.stop[k ^ 1] >= (unsigned)B.skip) ahead(q.args[k ^ 1], q.bid[k ^ 1]);
      }
    }
    item(q.args[k], q.bid[k], q.nblk[k], (unsigned)q.stop[k] < (unsigned)B.skip);
    cp_async_wait_all();
    __syncthreads();       // the next item is fetched, and this block is done with this one's shared memory
  }
}

template <int N1, int N2, int MODE, bool STDF = false>
__global__ void __launch_bounds__(kRowMaxThreads, kRowCtasPerSM) row_pass_batch(const BatchArgs B) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ BatchQueue q;
  using S = Split<N1, N2>;
  const RowSmem L = row_smem(MODE, S::N, blockDim.x / S::TL, S::SM_LANE);
  // the tables are the same for every frame of the side
  stage_bytes(smem_raw + L.tw, B.args[0].twA, S::N * 8);
  stage_bytes(smem_raw + L.tw + S::N * 8, B.args[0].twB, S::N * 8);
  pdl_enter();
  batch_items(B, q, [&](const KArgs& A, int bid, int nblk, bool stopped) {
    if (!stopped) row_pass_body<N1, N2, MODE, STDF>(A, bid, nblk, smem_raw, (NoTc*)nullptr, true);
  }, [&](const KArgs& A, int bid) { row_prefetch<N1, N2, MODE, STDF>(A, bid); });
}

// Column passes of batches are bound by the loads in flight: blocks per SM are asked for by the block's threads (left to
// the compiler, sides 320 and 384 took registers for 3 and 2).  64 frames (5 Newton steps of 12 iterations) 100.0 -> 98.7
// ms, three 384^2 frames 11.9 -> 11.7.
constexpr int col_batch_ctas(int threads) { return threads <= 128 ? 5 : threads <= 160 ? 4 : threads <= 192 ? 3 : 1; }
template <int N1, int N2, int MODE, bool STDF = false>
__global__ void __launch_bounds__(ColCfg<N1, N2>::THREADS, col_batch_ctas(ColCfg<N1, N2>::THREADS)) col_pass_batch(const BatchArgs B) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ BatchQueue q;
  using S = Split<N1, N2>;
  const ColSmem L = col_smem(MODE, S::N, ColCfg<N1, N2>::C, S::SM_LANE_COL, S::N / 2);
  stage_bytes(smem_raw + L.tw, B.args[0].twA, S::N * 8);
  stage_bytes(smem_raw + L.tw + S::N * 8, B.args[0].twB, S::N * 8);
  pdl_enter();
  batch_items(B, q, [&](const KArgs& A, int bid, int nblk, bool stopped) {
    if (!stopped) col_pass_body<N1, N2, MODE, STDF>(A, bid, nblk, smem_raw, (NoTc*)nullptr, false, true);
  });
}

// ------------------------------------------------------------------------- batches of several sides ----
// One launch per pass for frames of every grid side in kMultiSides: the block dispatches on its work item's grid
// side to that side's pass body.  Row passes run kRowMaxThreads threads (kRowMaxThreads / TL whole lanes of the
// side, the rest idle), column passes kMultiColThreads (NLV_COL_C columns x the largest lane width).
constexpr int kMultiSides[] = {128, 192, 256, 320, 384};
constexpr int kNumMultiSides = 5;
constexpr int kMultiColThreads = NLV_COL_C * 24;
__host__ __device__ constexpr bool multi_side(int n) {
  return n == 128 || n == 192 || n == 256 || n == 320 || n == 384;
}

// Each side's body is a separate (not inlined) function, so that registers are allocated per side rather than
// across all sides' branches at once.
template <int N1, int N2, int MODE, bool STDF>
__device__ __noinline__ void row_body_call(const KArgs& A, int bid, int nblk, unsigned char* smem) {
  row_pass_body<N1, N2, MODE, STDF>(A, bid, nblk, smem);
}
template <int N1, int N2, int MODE, bool STDF>
__device__ __noinline__ void col_body_call(const KArgs& A, int bid, int nblk, unsigned char* smem) {
  col_pass_body<N1, N2, MODE, STDF>(A, bid, nblk, smem);
}
template <int MODE, bool STDF>
__device__ __forceinline__ void row_body_of_side(const KArgs& A, int bid, int nblk, unsigned char* smem) {
  switch (A.N) {
    case 128: row_body_call<8, 16, MODE, STDF>(A, bid, nblk, smem); break;
    case 192: row_body_call<12, 16, MODE, STDF>(A, bid, nblk, smem); break;
    case 256: row_body_call<16, 16, MODE, STDF>(A, bid, nblk, smem); break;
    case 320: row_body_call<16, 20, MODE, STDF>(A, bid, nblk, smem); break;
    default: row_body_call<16, 24, MODE, STDF>(A, bid, nblk, smem); break;
  }
}
template <int MODE, bool STDF>
__device__ __forceinline__ void col_body_of_side(const KArgs& A, int bid, int nblk, unsigned char* smem) {
  switch (A.N) {
    case 128: col_body_call<8, 16, MODE, STDF>(A, bid, nblk, smem); break;
    case 192: col_body_call<12, 16, MODE, STDF>(A, bid, nblk, smem); break;
    case 256: col_body_call<16, 16, MODE, STDF>(A, bid, nblk, smem); break;
    case 320: col_body_call<16, 20, MODE, STDF>(A, bid, nblk, smem); break;
    default: col_body_call<16, 24, MODE, STDF>(A, bid, nblk, smem); break;
  }
}

template <int MODE, bool STDF>
__global__ void __launch_bounds__(kRowMaxThreads, kRowCtasPerSM) row_pass_multi(const BatchArgs B) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ BatchQueue q;
  pdl_enter();
  batch_items(B, q, [&](const KArgs& A, int bid, int nblk, bool stopped) {
    if (!stopped) row_body_of_side<MODE, STDF>(A, bid, nblk, smem_raw);
  });
}

template <int MODE, bool STDF>
__global__ void __launch_bounds__(kMultiColThreads) col_pass_multi(const BatchArgs B) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ BatchQueue q;
  pdl_enter();
  batch_items(B, q, [&](const KArgs& A, int bid, int nblk, bool stopped) {
    if (!stopped) col_body_of_side<MODE, STDF>(A, bid, nblk, smem_raw);
  });
}

// The multi-side kernels of every pass (defined in batch_multi.cu) and their dynamic shared memory (the largest
// over the sides).
struct MultiKernels {
  const void* row[NUM_ROW_MODES];
  const void* row_std[NUM_ROW_MODES];
  const void* col[NUM_COL_MODES];
  const void* col_std[NUM_COL_MODES];
  size_t row_smem[NUM_ROW_MODES];
  size_t col_smem[NUM_COL_MODES];
};
const MultiKernels* multi_kernels();

// ------------------------------------------------------------------------------- per-size kernel table ----
struct SizeKernels {
  int N1, N2;
  int tl;                   // threads per lane
  int col_lanes, col_threads;
  int sm_lane;              // shared float2 per lane for one exchange (row passes)
  int sm_lane_col;          // the same for column passes (bank-conflict padding)
  // Single-frame passes (no batch modes) and batched passes (no single-frame CG modes, no operator-only modes).
  const void* row[NUM_ROW_MODES];
  const void* col[NUM_COL_MODES];
  const void* row_batch[NUM_ROW_MODES];
  const void* col_batch[NUM_COL_MODES];
  // Passes of the CG iteration specialised for the standard field of view f = N/4 (a compile-time constant, so
  // the Omega tests of the register-held elements fold away); nullptr where the generic kernel is used.
  const void* row_std[NUM_ROW_MODES];
  const void* col_std[NUM_COL_MODES];
  const void* row_std_batch[NUM_ROW_MODES];
  const void* col_std_batch[NUM_COL_MODES];
  // Passes with their radix-16 DFT stages on the tensor cores (sides whose split has a factor 16); nullptr where
  // not compiled.  row_tc_std / col_tc_std: the standard-field-of-view forms, as row_std / col_std.
  const void* row_tc[NUM_ROW_MODES];
  const void* col_tc[NUM_COL_MODES];
  const void* row_tc_std[NUM_ROW_MODES];
  const void* col_tc_std[NUM_COL_MODES];
  // The whole CG solve of a small single frame as one cluster launch (cg_cluster.cuh); nullptr where not compiled.
  const void* cluster;
  int cluster_threads;
  size_t (*cluster_smem)(int J);
  size_t row_smem(int mode, int lanes) const { return nlv::row_smem(mode, N1 * N2, lanes, sm_lane).total; }
  size_t col_smem(int mode, int Wc) const { return nlv::col_smem(mode, N1 * N2, col_lanes, sm_lane_col, Wc).total; }
  size_t row_smem_tc(int mode, int lanes) const { return tc_offset(row_smem(mode, lanes)) + tc_smem_bytes(lanes * tl); }
  size_t col_smem_tc(int mode, int Wc) const { return tc_offset(col_smem(mode, Wc)) + tc_smem_bytes(col_threads); }
};

// Parts of a batch's row block of `rows` rows: as many as kRowBatchThreads asks for, if they come out equal.
inline int batch_row_split(const SizeKernels* k, int rows) {
  const int sub = (rows * k->tl + kRowBatchThreads - 1) / kRowBatchThreads;
  return rows % sub == 0 ? sub : 1;
}

// Launch geometry of a row pass: `blocks` blocks of `lanes` lanes, each taking rows_per_cta rows (and rho_per_cta
// pixels of the rho plane when the pass has one), so that the rows are split evenly over ctas_per_sm blocks per SM.
struct RowGrid {
  int blocks, lanes, rows_per_cta, rho_per_cta;
  int sub;       // batches: blocks that share one block's rows and slice (KArgs::sub)
};
inline RowGrid row_grid(const SizeKernels* k, int nrows, long rho_pixels, int sms, int ctas_per_sm) {
  RowGrid g{};
  const int max_lanes = kRowMaxThreads / k->tl;
  int want = sms * ctas_per_sm;
  if (want > nrows) want = nrows;
  // at least a warp of threads a block: narrower blocks only add partial sums for the next pass to read (64^2 with
  // 4 coils: 256 blocks of 8 threads)
  int per = (nrows + want - 1) / want;
  if (per * k->tl < 32) per = std::min((32 + k->tl - 1) / k->tl, nrows);
  const int rounds = (per + max_lanes - 1) / max_lanes;
  g.lanes = (per + rounds - 1) / rounds;
  g.rows_per_cta = per;
  g.blocks = (nrows + per - 1) / per;
  g.rho_per_cta = (int)((rho_pixels + g.blocks - 1) / g.blocks);
  return g;
}

// The operators' passes with two inputs or with the coil maps formed on the way (q_op_* in nlinv.cu).
template <int N1, int N2, int CC = NLV_COL_C> void add_op_cols(SizeKernels& k) {
  k.col[COL_COIL_PROD] = (const void*)col_pass<N1, N2, COL_COIL_PROD, false, CC>;
  k.col[COL_COIL_DIR] = (const void*)col_pass<N1, N2, COL_COIL_DIR, false, CC>;
  k.col[COL_COIL_ADJ] = (const void*)col_pass<N1, N2, COL_COIL_ADJ, false, CC>;
  k.col_std[COL_COIL_PROD] = (const void*)col_pass<N1, N2, COL_COIL_PROD, true, CC>;
  k.col_std[COL_COIL_DIR] = (const void*)col_pass<N1, N2, COL_COIL_DIR, true, CC>;
  k.col_std[COL_COIL_ADJ] = (const void*)col_pass<N1, N2, COL_COIL_ADJ, true, CC>;
}
template <int N1, int N2> void add_op_passes(SizeKernels& k) {
  k.row[ROW_W_W_IFFT] = (const void*)row_pass<N1, N2, ROW_W_W_IFFT>;
  k.row[ROW_W_P_IFFT] = (const void*)row_pass<N1, N2, ROW_W_P_IFFT>;
  k.row_std[ROW_W_W_IFFT] = (const void*)row_pass<N1, N2, ROW_W_W_IFFT, true>;
  k.row_std[ROW_W_P_IFFT] = (const void*)row_pass<N1, N2, ROW_W_P_IFFT, true>;
  add_op_cols<N1, N2>(k);
}
// The CG passes of single frames (q_cg_iter in nlinv.cu) and of batches (q_bcg_iter).
template <int N1, int N2, int CC = NLV_COL_C> void add_frame_cg_cols(SizeKernels& k) {
  k.col[COL_CG_DIR] = (const void*)col_pass<N1, N2, COL_CG_DIR, false, CC>;
  k.col_std[COL_CG_DIR] = (const void*)col_pass<N1, N2, COL_CG_DIR, true, CC>;
}
template <int N1, int N2> void add_frame_cg(SizeKernels& k) {
  k.row[ROW_CG_RHS] = (const void*)row_pass<N1, N2, ROW_CG_RHS>;
  k.row[ROW_CG_PSF] = (const void*)row_pass<N1, N2, ROW_CG_PSF>;
  k.row_std[ROW_CG_PSF] = (const void*)row_pass<N1, N2, ROW_CG_PSF, true>;
  k.row[ROW_CG_UPDATE] = (const void*)row_pass<N1, N2, ROW_CG_UPDATE>;
  k.row_std[ROW_CG_UPDATE] = (const void*)row_pass<N1, N2, ROW_CG_UPDATE, true>;
  add_frame_cg_cols<N1, N2>(k);
}
template <int N1, int N2> void add_batch_cg(SizeKernels& k) {
  k.row_batch[ROW_BCG_RHS] = (const void*)row_pass_batch<N1, N2, ROW_BCG_RHS>;
  k.row_std_batch[ROW_BCG_DIR] = (const void*)row_pass_batch<N1, N2, ROW_BCG_DIR, true>;
  k.row_std_batch[ROW_BCG_NORMAL] = (const void*)row_pass_batch<N1, N2, ROW_BCG_NORMAL, true>;
  k.col_std_batch[COL_BCG_DIR] = (const void*)col_pass_batch<N1, N2, COL_BCG_DIR, true>;
}

// Tuning variants of a side (nlinv_autotune): the default table with other column-strip widths, and the single-frame
// passes of an alternative four-step split.  They hold no batch or tensor-core kernels.
template <int N1, int N2, int CC> SizeKernels make_size_kernels_strip(const SizeKernels& base) {
  SizeKernels s = base;
  s.col_lanes = ColCfg<N1, N2, CC>::C;
  s.col_threads = ColCfg<N1, N2, CC>::THREADS;
  s.col[COL_IFFT_C] = (const void*)col_pass<N1, N2, COL_IFFT_C, false, CC>;
  s.col[COL_PROD_FFT] = (const void*)col_pass<N1, N2, COL_PROD_FFT, false, CC>;
  s.col[COL_SIM_FFT] = (const void*)col_pass<N1, N2, COL_SIM_FFT, false, CC>;
  s.col[COL_IFFT_PROD_FFT] = (const void*)col_pass<N1, N2, COL_IFFT_PROD_FFT, false, CC>;
  s.col[COL_IFFT_ADJ_FFT] = (const void*)col_pass<N1, N2, COL_IFFT_ADJ_FFT, false, CC>;
  for (int m = 0; m < NUM_COL_MODES; ++m) s.col_std[m] = nullptr;
  add_frame_cg_cols<N1, N2, CC>(s);
  add_op_cols<N1, N2, CC>(s);
  s.col_std[COL_IFFT_PROD_FFT] = (const void*)col_pass<N1, N2, COL_IFFT_PROD_FFT, true, CC>;
  for (int m = 0; m < NUM_ROW_MODES; ++m) s.row_batch[m] = s.row_std_batch[m] = s.row_tc[m] = s.row_tc_std[m] = nullptr;
  for (int m = 0; m < NUM_COL_MODES; ++m) s.col_batch[m] = s.col_std_batch[m] = s.col_tc[m] = s.col_tc_std[m] = nullptr;
  return s;
}

template <int N1, int N2> SizeKernels make_size_kernels_single() {
  SizeKernels s{};
  s.N1 = N1;
  s.N2 = N2;
  s.tl = Split<N1, N2>::TL;
  s.col_lanes = ColCfg<N1, N2>::C;
  s.col_threads = ColCfg<N1, N2>::THREADS;
  s.sm_lane = Split<N1, N2>::SM_LANE;
  s.sm_lane_col = Split<N1, N2>::SM_LANE_COL;
  s.row[ROW_W_IFFT] = (const void*)row_pass<N1, N2, ROW_W_IFFT>;
  s.row[ROW_PSF] = (const void*)row_pass<N1, N2, ROW_PSF>;
  s.row[ROW_FFT_P_OUT] = (const void*)row_pass<N1, N2, ROW_FFT_P_OUT>;
  s.row[ROW_FFT_RESID] = (const void*)row_pass<N1, N2, ROW_FFT_RESID>;
  s.row[ROW_P_IFFT] = (const void*)row_pass<N1, N2, ROW_P_IFFT>;
  s.row[ROW_FFT_W_ADJ] = (const void*)row_pass<N1, N2, ROW_FFT_W_ADJ>;
  s.row[ROW_FFT_W_NORMAL] = (const void*)row_pass<N1, N2, ROW_FFT_W_NORMAL>;
  s.col[COL_IFFT_C] = (const void*)col_pass<N1, N2, COL_IFFT_C>;
  s.col[COL_PROD_FFT] = (const void*)col_pass<N1, N2, COL_PROD_FFT>;
  s.col[COL_SIM_FFT] = (const void*)col_pass<N1, N2, COL_SIM_FFT>;
  s.col[COL_IFFT_PROD_FFT] = (const void*)col_pass<N1, N2, COL_IFFT_PROD_FFT>;
  s.col[COL_IFFT_ADJ_FFT] = (const void*)col_pass<N1, N2, COL_IFFT_ADJ_FFT>;
  s.row_std[ROW_W_IFFT] = (const void*)row_pass<N1, N2, ROW_W_IFFT, true>;
  s.row_std[ROW_PSF] = (const void*)row_pass<N1, N2, ROW_PSF, true>;
  s.row_std[ROW_FFT_W_NORMAL] = (const void*)row_pass<N1, N2, ROW_FFT_W_NORMAL, true>;
  s.col_std[COL_IFFT_PROD_FFT] = (const void*)col_pass<N1, N2, COL_IFFT_PROD_FFT, true>;
  add_frame_cg<N1, N2>(s);
  add_op_passes<N1, N2>(s);
  return s;
}

template <int N1, int N2> SizeKernels make_size_kernels() {
  SizeKernels s{};
  s.N1 = N1;
  s.N2 = N2;
  s.tl = Split<N1, N2>::TL;
  s.col_lanes = ColCfg<N1, N2>::C;
  s.col_threads = ColCfg<N1, N2>::THREADS;
  s.sm_lane = Split<N1, N2>::SM_LANE;
  s.sm_lane_col = Split<N1, N2>::SM_LANE_COL;
  s.row[ROW_W_IFFT] = (const void*)row_pass<N1, N2, ROW_W_IFFT>;
  s.row[ROW_PSF] = (const void*)row_pass<N1, N2, ROW_PSF>;
  s.row[ROW_FFT_P_OUT] = (const void*)row_pass<N1, N2, ROW_FFT_P_OUT>;
  s.row[ROW_FFT_RESID] = (const void*)row_pass<N1, N2, ROW_FFT_RESID>;
  s.row[ROW_P_IFFT] = (const void*)row_pass<N1, N2, ROW_P_IFFT>;
  s.row[ROW_FFT_W_ADJ] = (const void*)row_pass<N1, N2, ROW_FFT_W_ADJ>;
  s.row[ROW_FFT_W_NORMAL] = (const void*)row_pass<N1, N2, ROW_FFT_W_NORMAL>;
  s.col[COL_IFFT_C] = (const void*)col_pass<N1, N2, COL_IFFT_C>;
  s.col[COL_PROD_FFT] = (const void*)col_pass<N1, N2, COL_PROD_FFT>;
  s.col[COL_SIM_FFT] = (const void*)col_pass<N1, N2, COL_SIM_FFT>;
  s.col[COL_IFFT_PROD_FFT] = (const void*)col_pass<N1, N2, COL_IFFT_PROD_FFT>;
  s.col[COL_IFFT_ADJ_FFT] = (const void*)col_pass<N1, N2, COL_IFFT_ADJ_FFT>;
  s.row_batch[ROW_W_IFFT] = (const void*)row_pass_batch<N1, N2, ROW_W_IFFT>;
  s.row_batch[ROW_PSF] = (const void*)row_pass_batch<N1, N2, ROW_PSF>;
  s.row_batch[ROW_FFT_P_OUT] = (const void*)row_pass_batch<N1, N2, ROW_FFT_P_OUT>;
  s.row_batch[ROW_FFT_RESID] = (const void*)row_pass_batch<N1, N2, ROW_FFT_RESID>;
  s.row_batch[ROW_P_IFFT] = (const void*)row_pass_batch<N1, N2, ROW_P_IFFT>;
  s.row_batch[ROW_FFT_W_ADJ] = (const void*)row_pass_batch<N1, N2, ROW_FFT_W_ADJ>;
  s.row_batch[ROW_FFT_W_NORMAL] = (const void*)row_pass_batch<N1, N2, ROW_FFT_W_NORMAL>;
  s.col_batch[COL_IFFT_C] = (const void*)col_pass_batch<N1, N2, COL_IFFT_C>;
  s.col_batch[COL_PROD_FFT] = (const void*)col_pass_batch<N1, N2, COL_PROD_FFT>;
  s.col_batch[COL_SIM_FFT] = (const void*)col_pass_batch<N1, N2, COL_SIM_FFT>;
  s.col_batch[COL_IFFT_PROD_FFT] = (const void*)col_pass_batch<N1, N2, COL_IFFT_PROD_FFT>;
  s.col_batch[COL_IFFT_ADJ_FFT] = (const void*)col_pass_batch<N1, N2, COL_IFFT_ADJ_FFT>;
  // measured: the p-update, PSF and normal-operator row passes and the DF column pass gain from the constant
  // field of view (the batched p-update pass also stops spilling); the DF^H column pass does not
  s.row_std[ROW_W_IFFT] = (const void*)row_pass<N1, N2, ROW_W_IFFT, true>;
  s.row_std[ROW_PSF] = (const void*)row_pass<N1, N2, ROW_PSF, true>;
  s.row_std[ROW_FFT_W_NORMAL] = (const void*)row_pass<N1, N2, ROW_FFT_W_NORMAL, true>;
  s.col_std[COL_IFFT_PROD_FFT] = (const void*)col_pass<N1, N2, COL_IFFT_PROD_FFT, true>;
  s.row_std_batch[ROW_W_IFFT] = (const void*)row_pass_batch<N1, N2, ROW_W_IFFT, true>;
  s.row_std_batch[ROW_PSF] = (const void*)row_pass_batch<N1, N2, ROW_PSF, true>;
  s.row_std_batch[ROW_FFT_W_NORMAL] = (const void*)row_pass_batch<N1, N2, ROW_FFT_W_NORMAL, true>;
  s.col_std_batch[COL_IFFT_PROD_FFT] = (const void*)col_pass_batch<N1, N2, COL_IFFT_PROD_FFT, true>;
  add_frame_cg<N1, N2>(s);
  add_op_passes<N1, N2>(s);
  add_batch_cg<N1, N2>(s);
  return s;
}

// The kernel table of a side whose split has a factor 16, with the tensor-core passes added.
template <int N1, int N2> SizeKernels make_size_kernels_tc() {
  static_assert(N1 == 16 || N2 == 16, "the tensor-core stage is a radix-16 DFT");
  SizeKernels s = make_size_kernels<N1, N2>();
  s.row_tc[ROW_W_IFFT] = (const void*)row_pass_tc<N1, N2, ROW_W_IFFT, false>;
  s.row_tc[ROW_PSF] = (const void*)row_pass_tc<N1, N2, ROW_PSF, false>;
  s.row_tc[ROW_FFT_P_OUT] = (const void*)row_pass_tc<N1, N2, ROW_FFT_P_OUT, false>;
  s.row_tc[ROW_FFT_RESID] = (const void*)row_pass_tc<N1, N2, ROW_FFT_RESID, false>;
  s.row_tc[ROW_P_IFFT] = (const void*)row_pass_tc<N1, N2, ROW_P_IFFT, false>;
  s.row_tc[ROW_FFT_W_ADJ] = (const void*)row_pass_tc<N1, N2, ROW_FFT_W_ADJ, false>;
  s.row_tc[ROW_FFT_W_NORMAL] = (const void*)row_pass_tc<N1, N2, ROW_FFT_W_NORMAL, false>;
  s.row_tc[ROW_CG_RHS] = (const void*)row_pass_tc<N1, N2, ROW_CG_RHS, false>;
  s.row_tc[ROW_CG_PSF] = (const void*)row_pass_tc<N1, N2, ROW_CG_PSF, false>;
  s.row_tc[ROW_CG_UPDATE] = (const void*)row_pass_tc<N1, N2, ROW_CG_UPDATE, false>;
  s.col_tc[COL_IFFT_C] = (const void*)col_pass_tc<N1, N2, COL_IFFT_C, false>;
  s.col_tc[COL_PROD_FFT] = (const void*)col_pass_tc<N1, N2, COL_PROD_FFT, false>;
  s.col_tc[COL_SIM_FFT] = (const void*)col_pass_tc<N1, N2, COL_SIM_FFT, false>;
  s.col_tc[COL_IFFT_PROD_FFT] = (const void*)col_pass_tc<N1, N2, COL_IFFT_PROD_FFT, false>;
  s.col_tc[COL_IFFT_ADJ_FFT] = (const void*)col_pass_tc<N1, N2, COL_IFFT_ADJ_FFT, false>;
  s.col_tc[COL_CG_DIR] = (const void*)col_pass_tc<N1, N2, COL_CG_DIR, false>;
  s.row_tc_std[ROW_PSF] = (const void*)row_pass_tc<N1, N2, ROW_PSF, true>;
  s.row_tc_std[ROW_FFT_W_NORMAL] = (const void*)row_pass_tc<N1, N2, ROW_FFT_W_NORMAL, true>;
  s.row_tc_std[ROW_CG_PSF] = (const void*)row_pass_tc<N1, N2, ROW_CG_PSF, true>;
  s.row_tc_std[ROW_CG_UPDATE] = (const void*)row_pass_tc<N1, N2, ROW_CG_UPDATE, true>;
  s.col_tc_std[COL_IFFT_PROD_FFT] = (const void*)col_pass_tc<N1, N2, COL_IFFT_PROD_FFT, true>;
  s.col_tc_std[COL_CG_DIR] = (const void*)col_pass_tc<N1, N2, COL_CG_DIR, true>;
  return s;
}

}  // namespace nlv
