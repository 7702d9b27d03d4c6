// Krylov solvers: CG, restarted GMRES (CGS2 Arnoldi) and Richardson Minimal Residual.
//
// Every reduction is a deterministic sum in a fixed order: threads, then lanes and warps of a block,
// then blocks (as many as the vector's length asks for) whose double partials the last block to
// finish (atomic ticket) adds; it runs the scalar epilogue of the algorithm (step lengths, convergence
// tests in one thread, the Givens rotations of a GMRES step in one warp).  Double vectors are summed in
// double throughout, float vectors in float pairs up to the warp (Acc).  The scalars never leave the device; the
// host only reads the `done` flag every `check_every` iterations, one batch
// behind: it waits for the flag of batch k-1 with batch k already queued.  Kernels of an
// iteration return at once when the flag is set, so iterations enqueued ahead cost a launch
// each and change nothing.
#include "vd_launch.cuh"
#include "vd_krylov.cuh"
#include "vd_dd.cuh"
#include "vd_prof.h"

#include <algorithm>
#include <cmath>
#include <type_traits>
#include <cstddef>
#include <cstring>
#include <vector>
#include <mutex>

namespace vd {

// ---------------------------------------------------------------------------------------
// reduction machinery
// ---------------------------------------------------------------------------------------

template <typename T>
__device__ __forceinline__ cpx<double> ld(const cpx<T>* p, long long e) {
  const cpx<T> v = p[e];
  return mk<double>((double)v.x, (double)v.y);
}

// float -> double on the integer pipes (exact; subnormals take the conversion instruction).  The
// FP64 pipe of GB300, which also converts, takes ~17 cycles per warp instruction and SM, and a
// reduction's tail is bound by it.
__device__ __forceinline__ double widen(float f) {
  const unsigned u = __float_as_uint(f);
  return ((u & 0x7f800000u) == 0u && (u & 0x7fffffu) != 0u) ? (double)f : f2d_bits(f);
}

__host__ __device__ constexpr int log2_ceil(int n) { return n <= 1 ? 0 : 1 + log2_ceil((n + 1) / 2); }

// Sums of v[0..NV) (NV <= 32) over the block, one value per group of 8 threads: on return
// thread 8 i holds the total of value i (other threads nothing).  Within a warp the values are
// exchanged and halved (lanes whose bit is set keep the upper half of the values, the others the
// lower half), so NV values cost about NV + 5 - log2 NV additions per lane instead of 5 NV.  V =
// double, or dd: float-pair totals (of compensated float sums) are added as pairs on the FP32 pipes
// and widened once per warp, since a block's double additions queue for the FP64 pipe (a lone warp
// issues one per 64 cycles, eight warps one per 153 each).  87k points, 8 dots, caches flushed: 31.5 us
// with one double butterfly per value, 17.3 with the exchange in double; 32 dots, caches warm: 22.5 us
// in double, 14.9 in pairs.
__device__ __forceinline__ double shfl_xor(double v, int o) { return __shfl_xor_sync(0xffffffffu, v, o); }
__device__ __forceinline__ dd shfl_xor(dd v, int o) {
  return dd(__shfl_xor_sync(0xffffffffu, v.hi, o), __shfl_xor_sync(0xffffffffu, v.lo, o));
}
__device__ __forceinline__ double to_double(double v) { return v; }
__device__ __forceinline__ double to_double(dd v) { return widen(v.hi) + widen(v.lo); }
template <int NV, typename V>
__device__ __forceinline__ double block_sums(const V (&v)[NV], double (*sm)[kRedThreads / 32]) {
  constexpr int L = log2_ceil(NV), P = 1 << L;
  static_assert(NV >= 1 && P <= 32 && kRedThreads == 256, "one exchange step per lane bit");
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  V a[P];
#pragma unroll
  for (int i = 0; i < P; ++i) a[i] = i < NV ? v[i < NV ? i : 0] : V(0.0);
#pragma unroll
  for (int s = 0; s < 5; ++s) {
    const int o = 16 >> s, cnt = P >> (s + 1);   // values kept after this step
    if (cnt >= 1) {
      const bool up = (lane & o) != 0;
#pragma unroll
      for (int i = 0; i < cnt; ++i) {
        const V give = up ? a[i] : a[i + cnt], keep = up ? a[i + cnt] : a[i];
        a[i] = keep + shfl_xor(give, o);
      }
    } else {
      a[0] = a[0] + shfl_xor(a[0], o);
    }
  }
  const int mine = lane >> (5 - L);   // the value this lane ended with
  if ((lane & ((32 >> L) - 1)) == 0 && mine < NV) sm[mine][warp] = to_double(a[0]);
  __syncthreads();
  double s = 0.0;
  if (warp * 4 < NV) {   // warps holding a thread t with t / 8 < NV
    const int i = threadIdx.x >> 3;
    if (i < NV) s = sm[i][threadIdx.x & 7];
    s += __shfl_xor_sync(0xffffffffu, s, 4);
    s += __shfl_xor_sync(0xffffffffu, s, 2);
    s += __shfl_xor_sync(0xffffffffu, s, 1);
  }
  return s;
}

// Block-sum v[0..NV) into per-block partials (partials[i * blocks + block]); the last block gets
// the totals in tot (every thread).  Returns true (in every thread of the last block) when the
// caller must run the epilogue.  Fixed order: deterministic.
template <int NV, typename V>
__device__ bool reduce_last(const V (&v)[NV], double* partials, unsigned* counter, double (&tot)[NV]) {
  __shared__ double sm[NV][kRedThreads / 32];
  __shared__ int am_last;
  const int nb = (int)gridDim.x;
  const int vi = threadIdx.x >> 3;
  const double s = block_sums<NV, V>(v, sm);
  if (nb > 1) {
    if ((threadIdx.x & 7) == 0 && vi < NV) {
      partials[vi * nb + blockIdx.x] = s;
      __threadfence();
    }
    __syncthreads();
    if (threadIdx.x == 0) am_last = (atomicAdd(counter, 1u) == (unsigned)nb - 1u) ? 1 : 0;
    __syncthreads();
    if (!am_last) return false;
    __threadfence();
    double a[NV];
    if constexpr (NV < 8) {
#pragma unroll
      for (int i = 0; i < NV; ++i) a[i] = 0.0;
      for (int b = threadIdx.x; b < nb; b += kRedThreads) {
#pragma unroll
        for (int i = 0; i < NV; ++i) a[i] += __ldcg(partials + i * nb + b);
      }
      const double f = block_sums<NV, double>(a, sm);
      if ((threadIdx.x & 7) == 0 && vi < NV) sm[vi][0] = f;
    } else {
      // warp w sums the values w, w + 8, ...: their loads together, then the lanes' exchange
      constexpr int K = (NV + 7) / 8;
      const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
      double f[K];
#pragma unroll
      for (int k = 0; k < K; ++k) f[k] = 0.0;
      for (int b = lane; b < nb; b += 32) {
#pragma unroll
        for (int k = 0; k < K; ++k)
          if (w + 8 * k < NV) f[k] += __ldcg(partials + (w + 8 * k) * nb + b);
      }
#pragma unroll
      for (int k = 0; k < K; ++k) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) f[k] += __shfl_xor_sync(0xffffffffu, f[k], o);
        if (lane == 0 && w + 8 * k < NV) sm[w + 8 * k][0] = f[k];
      }
    }
    if (threadIdx.x == 0) *counter = 0u;
  } else {
    __syncthreads();   // sm is read by block_sums' last step
    if ((threadIdx.x & 7) == 0 && vi < NV) sm[vi][0] = s;
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < NV; ++i) tot[i] = sm[i][0];
  return true;
}

// Blocks of a reduction over len elements: up to one per SM while that leaves a thread at most
// kRedPerThread elements, then up to four (the tail's FP64 work grows with the blocks of an SM).
static inline int red_blocks(long long len) {
  constexpr long long kRedPerThread = 8, one = kRedBlocks / 4;
  const long long need = (len + kRedThreads - 1) / kRedThreads;
  if (need <= one * kRedPerThread) return (int)std::max<long long>(1, std::min(one, need));
  return (int)std::min<long long>(kRedBlocks, (need + kRedPerThread - 1) / kRedPerThread);
}

#define GRID_STRIDE(e, len) \
  for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < (len); e += (long long)gridDim.x * blockDim.x)

__device__ __forceinline__ bool bad(double v) { return !isfinite(v); }

__device__ void finish(KState* ks, int status) {
  ks->status = status;
  ks->done = 1;
  ks->cycle_done = 1;
}

__device__ void record(KState* ks, double* hist, double rel) {
  if (ks->iters < ks->hist_cap) hist[ks->iters] = rel;
}

// ---------------------------------------------------------------------------------------
// epilogues
// ---------------------------------------------------------------------------------------

enum Epi : int {
  EPI_INIT_CG = 0,    // tot = [bb, rr, rz]
  EPI_CG_ALPHA = 1,   // tot = [pq]
  EPI_CG_UPDATE = 2,  // tot = [rr, rz]
  EPI_INIT_RMR = 3,   // tot = [bb, rr]
  EPI_RMR_ALPHA = 4,  // tot = [rw, ww]
  EPI_RMR_UPDATE = 5, // tot = [rr]
  EPI_BB = 6,         // tot = [bb]
  EPI_GM_BETA = 7,    // tot = [rr]
  EPI_GM_H1 = 8,      // tot[i] -> h1[off + i]
  EPI_GM_H2 = 9,      // tot[i] -> h2[off + i]
  EPI_NORM = 11,      // tot = [vv] -> ks->rr
};

template <int NV>
__device__ void epilogue(int epi, const double (&t)[NV], KState* ks, double* hist, double tol, int off, int j) {
  if (tol < 0.0) tol = ks->dtol;
  switch (epi) {
    case EPI_INIT_CG:
    case EPI_INIT_RMR: {
      ks->bb = t[0];
      ks->tol2bb = tol * tol * t[0];
      if (t[0] == 0.0) {
        ks->relres = 0.0;
        record(ks, hist, 0.0);
        finish(ks, 0);
        return;
      }
      const double rel = sqrt(t[1] / t[0]);
      ks->relres = rel;
      ks->best = rel;
      ks->ref = rel;
      ks->ref_it = 0;
      ks->rr = t[1];
      if (epi == EPI_INIT_CG) ks->rz = t[NV > 2 ? 2 : 0];
      record(ks, hist, rel);
      if (bad(rel)) finish(ks, VD_ERR_NONFINITE);
      else if (rel <= tol) finish(ks, 0);
      else if (ks->maxit <= 0) finish(ks, VD_ERR_NOT_CONVERGED);
      return;
    }
    case EPI_CG_ALPHA: {
      const double pq = t[0];
      ks->pq = pq;
      if (pq == 0.0 || ks->rz == 0.0) {
        ks->iters += 1;
        finish(ks, VD_ERR_BREAKDOWN);
        return;
      }
      ks->alpha = ks->rz / pq;
      if (bad(ks->alpha)) {
        ks->iters += 1;
        finish(ks, VD_ERR_NONFINITE);
      }
      return;
    }
    case EPI_CG_UPDATE:
    case EPI_RMR_UPDATE: {
      ks->iters += 1;
      const double rr = t[0];
      const double rel = sqrt(rr / ks->bb);
      ks->rr = rr;
      ks->relres = rel;
      record(ks, hist, rel);
      if (bad(rel)) {
        finish(ks, VD_ERR_NONFINITE);
        return;
      }
      if (rr <= ks->tol2bb) {
        finish(ks, 0);
        return;
      }
      // residual-growth divergence test: RMR only (CG's residual norm is not monotone), except
      // for guarded CG solves that have already converged well below their start
      if (epi == EPI_RMR_UPDATE && rel > 1e3 * ks->best) {
        finish(ks, VD_ERR_DIVERGED);
        return;
      }
      if (epi == EPI_CG_UPDATE && ks->guard > 0) {
        if (rel < 0.5 * ks->ref) {
          ks->ref = rel;
          ks->ref_it = ks->iters;
        } else if (ks->best < 1e-3 && ks->iters - ks->ref_it >= kStallWindow) {
          finish(ks, VD_ERR_DIVERGED);   // stalled at its attainable accuracy
          return;
        }
        if (ks->best < 1e-3 && rel > (double)ks->guard * ks->best) {
          finish(ks, VD_ERR_DIVERGED);
          return;
        }
      }
      ks->best = fmin(ks->best, rel);
      if (epi == EPI_CG_UPDATE) {
        const double rz = t[NV > 1 ? 1 : 0];
        ks->beta = rz / ks->rz;
        ks->rz = rz;
      }
      if (ks->iters >= ks->maxit) finish(ks, VD_ERR_NOT_CONVERGED);
      return;
    }
    case EPI_RMR_ALPHA: {
      const double ww = t[NV > 1 ? 1 : 0];
      ks->rw = t[0];
      ks->ww = ww;
      if (ww == 0.0) {
        ks->iters += 1;
        finish(ks, VD_ERR_BREAKDOWN);
        return;
      }
      ks->alpha = t[0] / ww;
      return;
    }
    case EPI_BB: {
      ks->bb = t[0];
      ks->tol2bb = tol * tol * t[0];
      return;
    }
    case EPI_GM_BETA: {
      const double beta = sqrt(t[0]);
      ks->beta0 = beta;
      if (ks->bb == 0.0) {
        ks->relres = 0.0;
        if (ks->iters == 0) record(ks, hist, 0.0);
        finish(ks, 0);
        return;
      }
      const double rel = beta / sqrt(ks->bb);
      if (ks->iters == 0) record(ks, hist, rel);
      ks->relres = rel;
      if (bad(rel)) finish(ks, VD_ERR_NONFINITE);
      else if (rel <= tol) finish(ks, 0);
      else if (ks->iters >= ks->maxit) finish(ks, VD_ERR_NOT_CONVERGED);
      else {
        ks->k = 0;
        ks->cycle_done = 0;
        ks->gv[0] = beta;
      }
      return;
    }
    case EPI_GM_H1:
    case EPI_GM_H2: {
      double* h = (epi == EPI_GM_H1) ? ks->h1 : ks->h2;
      for (int i = 0; i < NV; ++i)
        if (off + i <= j) h[off + i] = t[i];
      return;
    }
    case EPI_NORM: {
      ks->rr = t[0];
      return;
    }
  }
}

// End of GMRES step j (tot = |w|^2): the new column of H through the rotations, the next rotation, the
// residual estimate and the cycle's end; by one warp.  One thread's rotations were four FP64 operations of
// 64 cycles each in a row, its square roots and quotients six of 600: 6 us of a step at j = 30.  Here
// the products that do not pass from rotation to rotation are formed by a lane per rotation, leaving
// one operation per rotation in the chain, and roots and quotients run side by side in lanes.
__device__ void gm_norm_epilogue(double tot, KState* ks, double* hist, double tol, int j) {
  if (tol < 0.0) tol = ks->dtol;
  const int lane = threadIdx.x;
  const int m = ks->m;
  double* __restrict__ col = ks->H + (size_t)j * (m + 1);
  constexpr int K = kMaxRestart / 32;
  double c[K], sn[K], cn[K], sx[K], at[K];   // rotation i = lane + 32 k: c, s, c h_{i+1}, s h_{i+1}, entry passed on
#pragma unroll
  for (int k = 0; k < K; ++k) {
    const int i = lane + 32 * k;
    const bool in = i < j;
    c[k] = in ? ks->cs[i] : 0.0;
    sn[k] = in ? ks->sn[i] : 0.0;
    const double h = in ? ks->h1[i + 1] + ks->h2[i + 1] : 0.0;
    cn[k] = c[k] * h;
    sx[k] = sn[k] * h;
    at[k] = 0.0;
  }
  const double root = sqrt(lane == 1 ? ks->bb : tot);
  const double hn = __shfl_sync(0xffffffffu, root, 0), bn = __shfl_sync(0xffffffffu, root, 1);
  double cur = ks->h1[0] + ks->h2[0];
#pragma unroll
  for (int k = 0; k < K; ++k)
    for (int l = 0; l < 32 && l + 32 * k < j; ++l) {
      at[k] = lane == l ? cur : at[k];
      cur = fma(-__shfl_sync(0xffffffffu, sn[k], l), cur, __shfl_sync(0xffffffffu, cn[k], l));
    }
#pragma unroll
  for (int k = 0; k < K; ++k)
    if (lane + 32 * k < j) col[lane + 32 * k] = fma(c[k], at[k], sx[k]);
  const double h2 = fma(cur, cur, hn * hn);
  const double h = (h2 > 1e-280 && h2 < 1e280) ? sqrt(h2) : hypot(cur, hn);
  const double g = ks->gv[j];
  const double q = (lane == 0 ? cur : (lane == 1 ? hn : g)) / (lane < 2 ? h : bn);
  const bool turn = hn != 0.0;
  const double cj = turn ? __shfl_sync(0xffffffffu, q, 0) : 1.0, sj = turn ? __shfl_sync(0xffffffffu, q, 1) : 0.0;
  const double est = fabs(sj) * fabs(__shfl_sync(0xffffffffu, q, 2));
  if (lane != 0) return;
  ks->cs[j] = cj;
  ks->sn[j] = sj;
  col[j] = cj * cur + sj * hn;
  col[j + 1] = 0.0;
  ks->gv[j + 1] = -sj * g;
  ks->gv[j] = cj * g;
  ks->iters += 1;
  ks->k = j + 1;
  ks->relres = est;
  record(ks, hist, est);
  ks->ww = hn;
  if (bad(est)) {
    ks->status = VD_ERR_NONFINITE;
    ks->cycle_done = 1;
  } else if (est <= tol || hn == 0.0) {
    ks->status = 0;   // converged (or invariant Krylov space): finished after the update
    ks->cycle_done = 1;
  } else if (j + 1 >= m || ks->iters >= ks->maxit) {
    ks->cycle_done = 1;
  }
}

// ---------------------------------------------------------------------------------------
// kernels
// ---------------------------------------------------------------------------------------

struct RedArgs {
  KState* ks;
  double* partials;
  unsigned* counter;
  double* hist;
  double tol;
};

// Grid-stride iteration over a spectral vector that tracks, without any division inside
// the loop, kx = e mod h0 (Parseval weight) and the symbol index e mod ncplx.
struct Ix {
  int len, h0, nc;   // vector length (complex elements), x half-spectrum length, field size
  int sh, sn;        // grid stride mod h0, grid stride mod nc
};

#define IX_LOOP(ix)                                                                          \
  const int ix_s_ = gridDim.x * blockDim.x;                                                 \
  int e = blockIdx.x * blockDim.x + threadIdx.x;                                            \
  int kx = e % (ix).h0, si = e % (ix).nc;                                                   \
  for (; e < (ix).len; e += ix_s_, kx += (ix).sh, kx -= (kx >= (ix).h0) ? (ix).h0 : 0,      \
                       si += (ix).sn, si -= (si >= (ix).nc) ? (ix).nc : 0)

// The loop of the memory-bound kernels: use(e, kx, load(e, si)) for every element of the thread, two
// elements' loads in flight (256^3 points: float CG update 74 -> 56 us, start of a CG solve 100 -> 75).  The elements come in the same order.
template <typename L, typename U>
__device__ __forceinline__ void ix_each(const Ix& ix, L load, U use) {
  const int step = gridDim.x * blockDim.x;
  int e = blockIdx.x * blockDim.x + threadIdx.x, kx = e % ix.h0, si = e % ix.nc;
  auto next = [&]() {
    kx += ix.sh;
    kx -= (kx >= ix.h0) ? ix.h0 : 0;
    si += ix.sn;
    si -= (si >= ix.nc) ? ix.nc : 0;
  };
  for (; e < ix.len - step; e += 2 * step) {
    const int k0 = kx;
    const auto v0 = load(e, si);
    next();
    const auto v1 = load(e + step, si);
    use(e, k0, v0);
    use(e + step, kx, v1);
    next();
  }
  if (e < ix.len) use(e, kx, load(e, si));
}

template <typename T>
__device__ __forceinline__ T pweight(int kx, int h0) {
  return (kx == 0 || kx == h0 - 1) ? T(1) : T(2);
}

// v times the Parseval weight.  Double: 2 v on the bits, since a multiply or an addition is a turn on
// the FP64 pipe (a compiler's select between the two values would take both): 256^3 points, double norm
// 53 -> 41 us, r = b - q with its norm 87 -> 71 us.
__device__ __forceinline__ float weighted(float v, int kx, int h0) { return v * pweight<float>(kx, h0); }
__device__ __forceinline__ double weighted(double v, int kx, int h0) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(v), sg = b & (1ull << 63);
  const unsigned e = (unsigned)(b >> 52) & 0x7ffu;
  unsigned long long t = b + (1ull << 52);             // normal: the next exponent
  if (e == 0u) t = sg | (b << 1);                      // zero and subnormal: the significand doubled
  if (e >= 0x7feu) t = e == 0x7ffu ? b : (sg | (0x7ffull << 52));
  return __longlong_as_double((long long)((kx == 0 || kx == h0 - 1) ? b : t));
}
template <typename T>
__device__ __forceinline__ cpx<T> weighted(cpx<T> v, int kx, int h0) {
  return mk<T>(weighted(v.x, kx, h0), weighted(v.y, kx, h0));
}

// Per-thread accumulator of a reduction.  Double vectors add in double.  Float vectors add
// with a compensated float sum (Knuth's two-sum carries the rounding error of every addition
// in a second float), about as accurate as a double accumulation of the float terms but
// without FP64 work per element: the FP64 pipe of GB300 is ~1/64 of the float rate and was
// the limiter of these memory-bound kernels.  The per-thread totals stay float pairs until one value per
// warp is left, which is widened; warps and blocks add in double (block_sums, reduce_last).  Dots of
// 2^12 to 2^20 terms, orthogonal vectors among them, err by 4e-10 to 2e-11 of the sum of their
// terms' magnitudes either way (the products are rounded to float); the pairs differ from double
// sums by less than 1e-18 of it.
template <typename T>
struct Acc {
  double a = 0.0;
  __device__ __forceinline__ void add(T v) { a += (double)v; }
  __device__ __forceinline__ void dot(cpx<T> u, cpx<T> v) { a = fma(u.x, v.x, fma(u.y, v.y, a)); }   // += Re(u conj v)
  __device__ __forceinline__ double total() const { return a; }
  using Sum = double;
};
template <>
struct Acc<float> {
  float s = 0.0f, c = 0.0f;   // value s + c
  __device__ __forceinline__ void add(float v) {
    const float t = s + v;
    const float bp = t - s;
    c += (s - (t - bp)) + (v - bp);
    s = t;
  }
  __device__ __forceinline__ void dot(cpx<float> u, cpx<float> v) { add(u.x * v.x + u.y * v.y); }
  __device__ __forceinline__ dd total() const { return dd_fast_two_sum(s, c); }
  using Sum = dd;
};

// float(v * s) on the integer and FP32 pipes: v scaled by the power of two in s (exponent bits), split
// into a float pair, times the rest of s in [1, 2), rounded to float once.  A double multiply and a
// conversion per value kept k_d2f_scaled at 64 us of 256^3 points against 30 us of memory.  Zeros pass;
// scaled values outside [2^-74, 2^126), whose pairs or products would lose bits, and an s that is no
// normal double take the double arithmetic.
struct Narrow {
  double s;
  float sh, sl;
  int k;   // s = (sh + sl) 2^k
  bool plain;
  static constexpr int kLeast = 1023 - 74, kEnd = 1023 + 126;   // exponent fields of the float arithmetic
  __device__ __forceinline__ explicit Narrow(double scale) : s(scale) {
    const int hi = __double2hiint(scale), ef = (hi >> 20) & 0x7ff;
    plain = ef == 0 || ef == 0x7ff;
    k = ef - 1023;
    const dd m = dd_from_double(__hiloint2double((hi & 0x800fffff) | 0x3ff00000, __double2loint(scale)));
    sh = m.hi;
    sl = m.lo;
  }
  __device__ __forceinline__ float operator()(double v) const {
    const int hi = __double2hiint(v), ef = (hi >> 20) & 0x7ff, en = ef + k;
    if (plain || ef == 0 || ef == 0x7ff || en < kLeast || en >= kEnd) {
      if (!plain && ((hi & 0x7fffffff) | __double2loint(v)) == 0)   // a zero with the product's sign
        return __int_as_float((hi ^ __double2hiint(s)) & (int)0x80000000);
      return (float)(v * s);
    }
    const dd d = dd_from_double(__hiloint2double(hi + (k << 20), __double2loint(v)));
    return mul_pair_dd(d, sh, sl);
  }
  // (d.hi + d.lo)(wh + wl), rounded once
  static __device__ __forceinline__ float mul_pair_dd(dd d, float wh, float wl) {
    const float p = d.hi * wh;
    return p + fmaf(d.lo, wh, fmaf(d.hi, wl, fmaf(d.hi, wh, -p)));
  }
};

// CG start: p = S r, reduce [bb, rr, rz]
template <typename T>
__global__ void __launch_bounds__(kRedThreads) k_cg_init(Ix ix, const cpx<T>* __restrict__ b,
                                                         const cpx<T>* __restrict__ r, cpx<T>* __restrict__ p,
                                                         const T* __restrict__ sym, RedArgs ra) {
  pdl_wait();
  Acc<T> a0, a1, a2;
  IX_LOOP(ix) {
    const cpx<T> bv = b[e], rv = r[e];
    const T sv = sym[si];
    p[e] = scal(rv, sv);
    const T r2 = weighted(rv.x * rv.x + rv.y * rv.y, kx, ix.h0);
    a0.add(weighted(bv.x * bv.x + bv.y * bv.y, kx, ix.h0));
    a1.add(r2);
    a2.add(sv * r2);
  }
  const typename Acc<T>::Sum v[3] = {a0.total(), a1.total(), a2.total()};
  double t[3];
  if (reduce_last(v, ra.partials, ra.counter, t) && threadIdx.x == 0)
    epilogue<3>(EPI_INIT_CG, t, ra.ks, ra.hist, ra.tol, 0, 0);
}

// CG start from x = 0: x = 0, r = b, p = S b, reduce [bb, rz].  With src64 (float solves of the
// refinement) b is src64 * s, narrowed here: its own pass, the copy of r and the clearing of x took
// 105 us of 256^3 points beside this kernel's 51.
template <typename T, bool SRC64>
__global__ void __launch_bounds__(kRedThreads, 4)
    k_cg_start(Ix ix, const cpx<T>* __restrict__ b, const cpx<double>* __restrict__ src64, double s, const OState* o,
               cpx<T>* __restrict__ x, cpx<T>* __restrict__ r, cpx<T>* __restrict__ p, const T* __restrict__ sym,
               RedArgs ra) {
  pdl_wait();
  Acc<T> a0, a1;
  const Narrow nw(o ? o->scale : s);
  using B = typename std::conditional<SRC64, double, T>::type;
  struct In {
    cpx<B> b;
    T s;
  };
  ix_each(
      ix,
      [&](int e, int si) {
        if constexpr (SRC64) return In{src64[e], sym[si]};
        else return In{b[e], sym[si]};
      },
      [&](int e, int kx, const In& v) {
        cpx<T> rv;
        if constexpr (SRC64) rv = mk<T>(nw(v.b.x), nw(v.b.y));
        else rv = v.b;
        x[e] = mk<T>(T(0), T(0));
        r[e] = rv;
        p[e] = scal(rv, v.s);
        const T r2 = weighted(rv.x * rv.x + rv.y * rv.y, kx, ix.h0);
        a0.add(r2);
        a1.add(v.s * r2);
      });
  const typename Acc<T>::Sum v[2] = {a0.total(), a1.total()};
  double t[2];
  if (reduce_last(v, ra.partials, ra.counter, t) && threadIdx.x == 0) {
    const double t3[3] = {t[0], t[0], t[1]};
    epilogue<3>(EPI_INIT_CG, t3, ra.ks, ra.hist, ra.tol, 0, 0);
  }
}

// reduce [(u,v)_w] or [(u,v)_w, (v,v)_w]
template <typename T, int NV>
__global__ void __launch_bounds__(kRedThreads) k_dot(Ix ix, const cpx<T>* __restrict__ u,
                                                     const cpx<T>* __restrict__ v, int epi, RedArgs ra,
                                                     const int* done) {
  pdl_wait();
  if (*done) return;
  Acc<T> a0, a1;
  IX_LOOP(ix) {
    const cpx<T> vv = v[e], wv = weighted(vv, kx, ix.h0);
    a0.dot(wv, u[e]);
    if (NV > 1) a1.dot(wv, vv);
  }
  typename Acc<T>::Sum a[NV];
  a[0] = a0.total();
  if (NV > 1) a[NV - 1] = a1.total();
  double t[NV];
  if (reduce_last(a, ra.partials, ra.counter, t) && threadIdx.x == 0)
    epilogue<NV>(epi, t, ra.ks, ra.hist, ra.tol, 0, 0);
}

// CG: x += alpha p, r -= alpha q; reduce [rr, (r, S r)]
template <typename T>
__global__ void __launch_bounds__(kRedThreads, 4) k_cg_update(Ix ix, cpx<T>* __restrict__ x,
                                                              const cpx<T>* __restrict__ p, cpx<T>* __restrict__ r,
                                                              const cpx<T>* __restrict__ q, const T* __restrict__ sym,
                                                              RedArgs ra) {
  pdl_wait();
  if (ra.ks->done) return;
  const T al = (T)ra.ks->alpha;
  Acc<T> a0, a1;
  struct In {
    cpx<T> p, q, x, r;
    T s;
  };
  ix_each(
      ix, [&](int e, int si) { return In{p[e], q[e], x[e], r[e], sym[si]}; },
      [&](int e, int kx, const In& v) {
        x[e] = mk<T>(fma(al, v.p.x, v.x.x), fma(al, v.p.y, v.x.y));
        const cpx<T> rv = mk<T>(fma(-al, v.q.x, v.r.x), fma(-al, v.q.y, v.r.y));
        r[e] = rv;
        const T r2 = weighted(rv.x * rv.x + rv.y * rv.y, kx, ix.h0);
        a0.add(r2);
        a1.add(v.s * r2);
      });
  const typename Acc<T>::Sum v[2] = {a0.total(), a1.total()};
  double t[2];
  if (reduce_last(v, ra.partials, ra.counter, t) && threadIdx.x == 0)
    epilogue<2>(EPI_CG_UPDATE, t, ra.ks, ra.hist, ra.tol, 0, 0);
}

// CG: p = S r + beta p
template <typename T>
__global__ void k_cg_p(Ix ix, cpx<T>* __restrict__ p, const cpx<T>* __restrict__ r, const T* __restrict__ sym,
                       const KState* ks) {
  pdl_wait();
  if (ks->done) return;
  const T be = (T)ks->beta;
  IX_LOOP(ix) {
    const T sv = sym[si];
    const cpx<T> rv = r[e], pv = p[e];
    p[e] = mk<T>(fma(be, pv.x, sv * rv.x), fma(be, pv.y, sv * rv.y));
  }
}

// RMR / GMRES start: reduce [bb, rr] or [rr]
template <typename T, int NV>
__global__ void __launch_bounds__(kRedThreads, 4) k_norms(Ix ix, const cpx<T>* __restrict__ b,
                                                          const cpx<T>* __restrict__ r, int epi, RedArgs ra,
                                                          const int* done) {
  pdl_wait();
  if (done && *done) return;
  Acc<T> a0, a1;
  struct In {
    cpx<T> b, r;
  };
  ix_each(
      ix,
      [&](int e, int) {
        const cpx<T> rv = r[e];
        return In{NV == 2 ? b[e] : rv, rv};
      },
      [&](int, int kx, const In& v) {
        if (NV == 2) a0.dot(weighted(v.b, kx, ix.h0), v.b);
        a1.dot(weighted(v.r, kx, ix.h0), v.r);
      });
  typename Acc<T>::Sum v[NV];
  if (NV == 2) v[0] = a0.total();
  v[NV - 1] = a1.total();
  double t[NV];
  if (reduce_last(v, ra.partials, ra.counter, t) && threadIdx.x == 0)
    epilogue<NV>(epi, t, ra.ks, ra.hist, ra.tol, 0, 0);
}

// weighted (Parseval) inner product of two spectral vectors -> ks->rr
template <typename T>
__global__ void __launch_bounds__(kRedThreads) k_pdot(Ix ix, const cpx<T>* __restrict__ a,
                                                      const cpx<T>* __restrict__ b, RedArgs ra) {
  pdl_wait();
  Acc<T> a0;
  IX_LOOP(ix) {
    const cpx<T> u = a[e], v = b[e];
    a0.dot(weighted(u, kx, ix.h0), v);
  }
  const typename Acc<T>::Sum v[1] = {a0.total()};
  double t[1];
  if (reduce_last(v, ra.partials, ra.counter, t) && threadIdx.x == 0) epilogue<1>(EPI_NORM, t, ra.ks, ra.hist, ra.tol, 0, 0);
}

// r = b - q and |r|^2 (weighted) -> ks->rr, accumulated like k_norms
template <typename T>
__global__ void __launch_bounds__(kRedThreads, 4) k_sub_norm(Ix ix, const cpx<T>* __restrict__ b,
                                                             const cpx<T>* q, cpx<T>* r, RedArgs ra) {
  pdl_wait();
  Acc<T> a1;
  struct In {
    cpx<T> b, q;
  };
  ix_each(
      ix, [&](int e, int) { return In{b[e], q[e]}; },   // (r may be q)
      [&](int e, int kx, const In& v) {
        const cpx<T> rv = v.b - v.q;
        r[e] = rv;
        a1.dot(weighted(rv, kx, ix.h0), rv);
      });
  const typename Acc<T>::Sum v[1] = {a1.total()};
  double t[1];
  if (reduce_last(v, ra.partials, ra.counter, t) && threadIdx.x == 0) epilogue<1>(EPI_NORM, t, ra.ks, ra.hist, ra.tol, 0, 0);
}

// RMR: x += alpha S r, r -= alpha w; reduce [rr]
template <typename T>
__global__ void __launch_bounds__(kRedThreads, 4) k_rmr_update(Ix ix, cpx<T>* __restrict__ x, cpx<T>* __restrict__ r,
                                                               const cpx<T>* __restrict__ wv,
                                                               const T* __restrict__ sym, RedArgs ra) {
  pdl_wait();
  if (ra.ks->done) return;
  const T al = (T)ra.ks->alpha;
  Acc<T> a0;
  struct In {
    cpx<T> w, x, r;
    T s;
  };
  ix_each(
      ix, [&](int e, int si) { return In{wv[e], x[e], r[e], sym[si]}; },
      [&](int e, int kx, const In& v) {
        const T as = al * v.s;
        x[e] = mk<T>(fma(as, v.r.x, v.x.x), fma(as, v.r.y, v.x.y));
        const cpx<T> rv = mk<T>(fma(-al, v.w.x, v.r.x), fma(-al, v.w.y, v.r.y));
        r[e] = rv;
        a0.dot(weighted(rv, kx, ix.h0), rv);
      });
  const typename Acc<T>::Sum v[1] = {a0.total()};
  double t[1];
  if (reduce_last(v, ra.partials, ra.counter, t) && threadIdx.x == 0)
    epilogue<1>(EPI_RMR_UPDATE, t, ra.ks, ra.hist, ra.tol, 0, 0);
}

// GMRES: dst = src / beta0 (first basis vector) or src / H[j+1,j] (next)
template <typename T>
__global__ void k_gm_scale(Ix ix, cpx<T>* __restrict__ dst, const cpx<T>* __restrict__ src, const KState* ks,
                           int first) {
  pdl_wait();
  if (ks->cycle_done) return;
  const T s = (T)(1.0 / (first ? ks->beta0 : ks->ww));
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < ix.len; e += gridDim.x * blockDim.x)
    dst[e] = scal(src[e], s);
}

// GMRES orthogonalisation (classical Gram-Schmidt twice).  k_gm_mdot: h1[off + i] =
// (w, V_{off+i})_w for i < nv <= NB.  k_gm_step: w -= sum_{i<nv} h1_i V_i, then h2_i = (w, V_i)_w in
// the same pass: every vector is local to an element, so V is read once, into registers, for both
// (the pair was two kernels and, at 8 vectors per dot kernel, up to nine launches per iteration).
// Up to 32 basis vectors; past that the dots run 32 at a time and the update apart.
template <typename T, int NB>
__global__ void __launch_bounds__(kRedThreads) k_gm_mdot(Ix ix, const cpx<T>* __restrict__ w,
                                                         const cpx<T>* __restrict__ V, int off, int nv, int epi, int j,
                                                         RedArgs ra) {
  pdl_wait();
  if (ra.ks->cycle_done) return;
  Acc<T> a[NB];
  IX_LOOP(ix) {
    const cpx<T> wv = weighted(w[e], kx, ix.h0);
#pragma unroll
    for (int i = 0; i < NB; ++i)
      if (i < nv) a[i].dot(wv, V[(size_t)(off + i) * ix.len + e]);
  }
  typename Acc<T>::Sum v[NB];
#pragma unroll
  for (int i = 0; i < NB; ++i) v[i] = a[i].total();
  double t[NB];
  if (reduce_last(v, ra.partials, ra.counter, t) && threadIdx.x == 0)
    epilogue<NB>(epi, t, ra.ks, ra.hist, ra.tol, off, j);
}

template <typename T, int NB>
__global__ void __launch_bounds__(kRedThreads) k_gm_step(Ix ix, cpx<T>* __restrict__ w, const cpx<T>* __restrict__ V,
                                                         int nv, RedArgs ra) {
  pdl_wait();
  if (ra.ks->cycle_done) return;
  __shared__ T hs[NB];
  for (int i = threadIdx.x; i < NB; i += blockDim.x) hs[i] = (i < nv) ? (T)ra.ks->h1[i] : T(0);
  __syncthreads();
  Acc<T> a[NB];
  IX_LOOP(ix) {
    cpx<T> wv = w[e], vv[NB];
#pragma unroll
    for (int i = 0; i < NB; ++i)
      if (i < nv) vv[i] = V[(size_t)i * ix.len + e];
#pragma unroll
    for (int i = 0; i < NB; ++i)
      if (i < nv) wv = mk<T>(fma(-hs[i], vv[i].x, wv.x), fma(-hs[i], vv[i].y, wv.y));
    w[e] = wv;
    wv = weighted(wv, kx, ix.h0);
#pragma unroll
    for (int i = 0; i < NB; ++i)
      if (i < nv) a[i].dot(wv, vv[i]);
  }
  typename Acc<T>::Sum v[NB];
#pragma unroll
  for (int i = 0; i < NB; ++i) v[i] = a[i].total();
  double t[NB];
  if (reduce_last(v, ra.partials, ra.counter, t) && threadIdx.x == 0)
    epilogue<NB>(EPI_GM_H2, t, ra.ks, ra.hist, ra.tol, 0, nv - 1);
}

// GMRES: w -= sum_{i<=j} h_i V_i (h = h1 or h2); with_norm: reduce [(w,w)] -> gm_norm_epilogue
template <typename T>
__global__ void __launch_bounds__(kRedThreads) k_gm_maxpy(Ix ix, cpx<T>* __restrict__ w,
                                                          const cpx<T>* __restrict__ V, int j, int which, int with_norm,
                                                          RedArgs ra) {
  pdl_wait();
  if (ra.ks->cycle_done) return;
  __shared__ T hs[kMaxRestart + 1];
  const double* h = which ? ra.ks->h2 : ra.ks->h1;
  for (int i = threadIdx.x; i <= j; i += blockDim.x) hs[i] = (T)h[i];
  __syncthreads();
  Acc<T> a0;
  IX_LOOP(ix) {
    cpx<T> wv = w[e];
#pragma unroll 8
    for (int i = 0; i <= j; ++i) {
      const T c = hs[i];
      const cpx<T> vv = V[(size_t)i * ix.len + e];
      wv = mk<T>(fma(-c, vv.x, wv.x), fma(-c, vv.y, wv.y));
    }
    w[e] = wv;
    a0.dot(weighted(wv, kx, ix.h0), wv);
  }
  if (!with_norm) return;
  const typename Acc<T>::Sum v[1] = {a0.total()};
  double t[1];
  if (reduce_last(v, ra.partials, ra.counter, t) && threadIdx.x < 32)
    gm_norm_epilogue(t[0], ra.ks, ra.hist, ra.tol, j);
}

static inline Ix mkix(long long len, int h0, long long nc, int blocks, int threads);

// NB vectors per thread: the least of 2, 4, 8, 16, 32 that holds nv
#define GM_BY_COUNT(nv, CALL)       \
  do {                              \
    if ((nv) <= 2) CALL(2);         \
    else if ((nv) <= 4) CALL(4);    \
    else if ((nv) <= 8) CALL(8);    \
    else if ((nv) <= 16) CALL(16);  \
    else CALL(32);                  \
  } while (0)

// the orthogonalisation of w against V_0..V_j on st: h1, h2, w and |w| (gm_norm_epilogue)
template <typename T>
static void gm_orthogonalise(const SpecSystem& sys, cpx<T>* w, const cpx<T>* V, int j, const RedArgs& ra,
                             cudaStream_t st) {
  const int n = j + 1;
  const int cls = sizeof(T) == 4 ? PC_VEC32 : PC_VEC64;
  const double el = (double)sys.len * sizeof(cpx<T>);
  // the partials hold 8 kRedBlocks values: fewer blocks for more values
  auto blocks = [&](int nb) { return std::min(red_blocks(sys.len), kRedBlocks * 8 / nb); };
  auto index = [&](int rb) { return mkix(sys.len, sys.h0, sys.G->g.ncplx, rb, kRedThreads); };
  auto mdot = [&](int off, int nv, int epi) {
    ProfScope ps_(cls, st, (nv + 1) * el, 0.0);
#define GM_MDOT(NB) \
  pdl_launch(k_gm_mdot<T, NB>, blocks(NB), kRedThreads, 0, st, index(blocks(NB)), w, V, off, nv, epi, j, ra)
    GM_BY_COUNT(nv, GM_MDOT);
#undef GM_MDOT
  };
  auto maxpy = [&](int which) {
    ProfScope ps_(cls, st, (n + 2) * el, 0.0);
    pdl_launch(k_gm_maxpy<T>, blocks(1), kRedThreads, 0, st, index(blocks(1)), w, V, j, which, which, ra);
  };
  for (int off = 0; off < n; off += 32) mdot(off, std::min(32, n - off), EPI_GM_H1);
  if (n <= 32) {
    ProfScope ps_(cls, st, (n + 2) * el, 0.0);
#define GM_STEP(NB) pdl_launch(k_gm_step<T, NB>, blocks(NB), kRedThreads, 0, st, index(blocks(NB)), w, V, n, ra)
    GM_BY_COUNT(n, GM_STEP);
#undef GM_STEP
  } else {
    maxpy(0);
    for (int off = 0; off < n; off += 32) mdot(off, std::min(32, n - off), EPI_GM_H2);
  }
  maxpy(1);
}
#undef GM_BY_COUNT

// GMRES: back substitution H(0:k,0:k) y = g: one warp, column by column, the triangle in shared
// memory (one thread reading it from global memory took 35 us at k = 30)
__global__ void __launch_bounds__(32) k_gm_solve(KState* ks) {
  pdl_wait();
  if (ks->done) return;
  __shared__ double tri[kMaxRestart * kMaxRestart], g[kMaxRestart], inv[kMaxRestart];
  const int k = ks->k, m = ks->m, lane = threadIdx.x;
  for (int l = 0; l < k; ++l)
    for (int i = lane; i <= l; i += 32) tri[i + l * kMaxRestart] = ks->H[i + (size_t)l * (m + 1)];
  __syncwarp();
  for (int i = lane; i < k; i += 32) {
    g[i] = ks->gv[i];
    inv[i] = 1.0 / tri[i + i * kMaxRestart];
  }
  __syncwarp();
  for (int l = k - 1; l >= 0; --l) {
    // g / H by the reciprocal and one correction (a division takes ~600 cycles, the three products 200)
    const double h = tri[l + l * kMaxRestart], y0 = g[l] * inv[l];
    const double y = isfinite(y0) ? fma(fma(-h, y0, g[l]), inv[l], y0) : g[l] / h;
    __syncwarp();
    for (int i = lane; i < l; i += 32) g[i] -= tri[i + l * kMaxRestart] * y;
    if (lane == 0) ks->y[l] = y;
    __syncwarp();
  }
}

// GMRES: x += S sum_{i<k} y_i V_i
template <typename T>
__global__ void k_gm_update(Ix ix, cpx<T>* __restrict__ x, const cpx<T>* __restrict__ V, const T* __restrict__ sym,
                            const KState* ks) {
  pdl_wait();
  if (ks->done) return;
  __shared__ T ys[kMaxRestart];
  const int k = ks->k;
  for (int i = threadIdx.x; i < k; i += blockDim.x) ys[i] = (T)ks->y[i];
  __syncthreads();
  IX_LOOP(ix) {
    T ax = T(0), ay = T(0);
    for (int i = 0; i < k; ++i) {
      const cpx<T> vv = V[(size_t)i * ix.len + e];
      ax = fma(ys[i], vv.x, ax);
      ay = fma(ys[i], vv.y, ay);
    }
    const T sv = sym[si];
    const cpx<T> xv = x[e];
    x[e] = mk<T>(fma(sv, ax, xv.x), fma(sv, ay, xv.y));
  }
}

// GMRES end of cycle: converged inside the cycle -> finished
__global__ void k_gm_close(KState* ks) {
  pdl_wait();
  if (threadIdx.x != 0 || blockIdx.x != 0 || ks->done) return;
  if (ks->status == 0 || ks->status == VD_ERR_NONFINITE) ks->done = 1;
}

// ---------------------------------------------------------------------------------------
// small vector helpers
// ---------------------------------------------------------------------------------------

template <typename T>
__global__ void k_copy_scale(long long len, const cpx<T>* __restrict__ x, double s, cpx<T>* __restrict__ y) {
  pdl_wait();
  GRID_STRIDE(e, len) {
    const cpx<double> v = ld(x, e);
    y[e] = mk<T>((T)(v.x * s), (T)(v.y * s));
  }
}
template <typename T>
__global__ void k_axpy(long long len, double a, const cpx<T>* __restrict__ x, cpx<T>* __restrict__ y) {
  pdl_wait();
  GRID_STRIDE(e, len) {
    const cpx<double> v = ld(x, e), w = ld(y, e);
    y[e] = mk<T>((T)fma(a, v.x, w.x), (T)fma(a, v.y, w.y));
  }
}
template <typename T>
__global__ void k_sub(long long len, const cpx<T>* __restrict__ b, const cpx<T>* __restrict__ q,
                      cpx<T>* __restrict__ r, const int* done) {
  pdl_wait();
  if (done && *done) return;
  GRID_STRIDE(e, len) { r[e] = b[e] - q[e]; }
}
// refinement steps fused over one pass of the double vectors (same arithmetic per element as
// the separate kernels): out = float(in * s) and y += a * double(xf); s and a come from the
// host, or from the refinement state (o->scale, o->rnorm) when o is set
__global__ void k_d2f_scaled(long long len, const cpx<double>* __restrict__ in, double s, const OState* o,
                             cpx<float>* __restrict__ out) {
  pdl_wait();
  const Narrow nw(o ? o->scale : s);
  GRID_STRIDE(e, len) {
    const cpx<double> v = in[e];
    out[e] = mk<float>(nw(v.x), nw(v.y));
  }
}
__global__ void k_axpy_f2d(long long len, double a, const OState* o, const cpx<float>* __restrict__ xf,
                           cpx<double>* __restrict__ y) {
  pdl_wait();
  if (o) a = o->rnorm;
  GRID_STRIDE(e, len) {
    const cpx<float> v = xf[e];
    const cpx<double> w = y[e];
    y[e] = mk<double>(fma(a, widen(v.x), w.x), fma(a, widen(v.y), w.y));
  }
}
template <typename T>
__global__ void k_project(GridDesc g, int ncomp, cpx<T>* v, double* removed) {
  pdl_wait();
  const int t = threadIdx.x;   // one thread per corner mode and component
  const int d = g.ndim;
  const int ncorner = 1 << d;
  if (t >= ncorner * ncomp) return;
  const int c = t / ncorner, m = t % ncorner;
  const int kx = (m & 1) ? g.n0 / 2 : 0;
  const int ky = (d >= 2 && (m & 2)) ? g.n1 / 2 : 0;
  const int kz = (d >= 3 && (m & 4)) ? g.n2 / 2 : 0;
  const long long e = ((long long)kz * g.n1 + ky) * g.h0 + kx;
  cpx<T>* q = v + (long long)c * g.ncplx + e;
  // the removed coefficient's share of the squared norm (Parseval weight 1: kx is 0 or n0/2)
  if (removed) removed[t] = (double)q->x * (double)q->x + (double)q->y * (double)q->y;
  *q = mk<T>(T(0), T(0));
}

static inline Ix mkix(long long len, int h0, long long nc, int blocks, int threads) {
  const long long S = (long long)blocks * threads;
  Ix ix;
  ix.len = (int)len;
  ix.h0 = h0;
  ix.nc = (int)nc;
  ix.sh = (int)(S % h0);
  ix.sn = (int)(S % nc);
  return ix;
}

static inline int ew_blocks(long long len) {
  return (int)std::max<long long>(1, std::min<long long>((len + 255) / 256, 8 * 1024));
}

template <typename T>
void spec_copy_scale(long long len, const void* x, double s, void* y, cudaStream_t st) {
  { pdl_launch(k_copy_scale<T>, ew_blocks(len), 256, 0, st, len, (const cpx<T>*)x, s, (cpx<T>*)y); count_launch(); }
}
template <typename T>
void spec_axpy(long long len, double a, const void* x, void* y, cudaStream_t st) {
  { pdl_launch(k_axpy<T>, ew_blocks(len), 256, 0, st, len, a, (const cpx<T>*)x, (cpx<T>*)y); count_launch(); }
}
template <typename T>
void spec_sub(long long len, const void* b, const void* q, void* r, cudaStream_t st) {
  { ProfScope ps_(sizeof(T) == 4 ? PC_VEC32 : PC_VEC64, st, (double)3 * len * sizeof(cpx<T>), 0.0); pdl_launch(k_sub<T>, ew_blocks(len), 256, 0, st, len, (const cpx<T>*)b, (const cpx<T>*)q, (cpx<T>*)r, nullptr); }
}
template <typename T>
void spec_project(const vd_grid* G, int ncomp, void* v, cudaStream_t st, double* removed) {
  { pdl_launch(k_project<T>, 1, 32, 0, st, G->g, ncomp, (cpx<T>*)v, removed); count_launch(); }
}

template <typename T>
double spec_norm2_host(const SpecSystem& sys, const void* v, const KWork& kw, cudaStream_t st) {
  RedArgs ra{kw.ks, kw.partials, kw.counter, kw.hist, 0.0};
  const int rb = red_blocks(sys.len);
  const Ix ix = mkix(sys.len, sys.h0, sys.G->g.ncplx, rb, kRedThreads);
  { ProfScope ps_(sizeof(T) == 4 ? PC_VEC32 : PC_VEC64, st, (double)1 * sys.len * sizeof(cpx<T>), 0.0); pdl_launch(k_norms<T, 1>, rb, kRedThreads, 0, st, ix, nullptr, (const cpx<T>*)v, EPI_NORM, ra, nullptr); }
  double rr = 0.0;
  cudaMemcpyAsync(&rr, &kw.ks->rr, sizeof(double), cudaMemcpyDeviceToHost, st);
  cudaStreamSynchronize(st);
  return rr;
}

template <typename T>
double spec_dot_host(const SpecSystem& sys, const void* a, const void* b, const KWork& kw, cudaStream_t st) {
  RedArgs ra{kw.ks, kw.partials, kw.counter, kw.hist, 0.0};
  const int rb = red_blocks(sys.len);
  const Ix ix = mkix(sys.len, sys.h0, sys.G->g.ncplx, rb, kRedThreads);
  { ProfScope ps_(sizeof(T) == 4 ? PC_VEC32 : PC_VEC64, st, (double)2 * sys.len * sizeof(cpx<T>), 0.0); pdl_launch(k_pdot<T>, rb, kRedThreads, 0, st, ix, (const cpx<T>*)a, (const cpx<T>*)b, ra); }
  double rr = 0.0;
  cudaMemcpyAsync(&rr, &kw.ks->rr, sizeof(double), cudaMemcpyDeviceToHost, st);
  cudaStreamSynchronize(st);
  return rr;
}

double spec_sub_norm2_host(const SpecSystem& sys, const void* b, const void* q, void* r, const KWork& kw,
                           cudaStream_t st) {
  RedArgs ra{kw.ks, kw.partials, kw.counter, kw.hist, 0.0};
  const int rb = red_blocks(sys.len);
  const Ix ix = mkix(sys.len, sys.h0, sys.G->g.ncplx, rb, kRedThreads);
  { ProfScope ps_(PC_VEC64, st, (double)3 * sys.len * sizeof(cpx<double>), 0.0); pdl_launch(k_sub_norm<double>, rb, kRedThreads, 0, st, ix, (const cpx<double>*)b, (const cpx<double>*)q, (cpx<double>*)r, ra); }
  double rr = 0.0;
  cudaMemcpyAsync(&rr, &kw.ks->rr, sizeof(double), cudaMemcpyDeviceToHost, st);
  cudaStreamSynchronize(st);
  return rr;
}

void spec_axpy_f2d(long long len, double a, const void* xf, void* y, cudaStream_t st) {
  { ProfScope ps_(PC_VEC64, st, (double)len * (sizeof(cpx<float>) + 2 * sizeof(cpx<double>)), 0.0); pdl_launch(k_axpy_f2d, ew_blocks(len), 256, 0, st, len, a, nullptr, (const cpx<float>*)xf, (cpx<double>*)y); }
}

// ---------------------------------------------------------------------------------------
// host drivers
// ---------------------------------------------------------------------------------------

template <typename T>
size_t krylov_vec_bytes(const SpecSystem& sys, int solver, int restart) {
  const size_t v = sizeof(cpx<T>) * (size_t)sys.len;
  if (solver == VD_SOLVER_CG) return 3 * v;
  if (solver == VD_SOLVER_RMR) return 2 * v;
  const int m = restart > 0 ? restart : 30;
  return (size_t)(m + 2) * v;
}

struct KHead {   // host mirror of the first fields of KState
  double bb, tol2bb, rr, rz, pq, alpha, beta, rw, ww, best, relres;
  int iters, maxit, status, done, hist_cap, m, k, cycle_done, guard;
};
static_assert(offsetof(KState, bb) == 0, "layout");

static vd_status read_head(const KWork& kw, KHead* h, cudaStream_t st) {
  VD_CUDA(cudaMemcpyAsync(h, kw.ks, sizeof(KHead), cudaMemcpyDeviceToHost, st));
  VD_CUDA(cudaStreamSynchronize(st));
  return VD_OK;
}

// Convergence polling one batch behind: after enqueuing batch k the host waits for the head
// snapshot taken after batch k-1, so the device always has the next batch queued instead of
// idling while the host wakes up and launches.  Batches enqueued past convergence return at
// once (every kernel of an iteration checks the device `done` flag).  Two pinned snapshot
// slots and events per solve in flight, leased from a process-wide pool (server slots solve
// from several threads; the pool never shrinks, so it holds the peak number of concurrent
// solves).
struct HeadPipe {
  KHead* slot = nullptr;
  cudaEvent_t ev[2] = {nullptr, nullptr};
  int taken = 0;
  bool ok = false;
  HeadPipe() {
    ok = cudaHostAlloc(reinterpret_cast<void**>(&slot), 2 * sizeof(KHead), cudaHostAllocDefault) == cudaSuccess &&
         cudaEventCreateWithFlags(&ev[0], cudaEventDisableTiming) == cudaSuccess &&
         cudaEventCreateWithFlags(&ev[1], cudaEventDisableTiming) == cudaSuccess;
  }
  // snapshot of the head after the work enqueued so far
  vd_status snapshot(const KWork& kw, cudaStream_t st) {
    const int k = taken & 1;
    VD_CUDA(cudaMemcpyAsync(slot + k, kw.ks, sizeof(KHead), cudaMemcpyDeviceToHost, st));
    VD_CUDA(cudaEventRecord(ev[k], st));
    ++taken;
    return VD_OK;
  }
  // wait for the latest snapshot (taken before the batch just enqueued) and copy it out
  vd_status latest(KHead* h) {
    const int k = (taken - 1) & 1;
    VD_CUDA(cudaEventSynchronize(ev[k]));
    *h = slot[k];
    return VD_OK;
  }
};

class HeadPipeLease {
 public:
  HeadPipeLease() {
    {
      std::lock_guard<std::mutex> lk(mu());
      if (!pool().empty()) {
        hp_ = pool().back();
        pool().pop_back();
      }
    }
    if (!hp_) hp_ = new HeadPipe();
    hp_->taken = 0;
  }
  ~HeadPipeLease() {
    // no snapshot copy may still be landing in the slots when the next solve takes them
    if (hp_->ok && hp_->taken > 0) {
      cudaEventSynchronize(hp_->ev[0]);
      if (hp_->taken > 1) cudaEventSynchronize(hp_->ev[1]);
    }
    std::lock_guard<std::mutex> lk(mu());
    pool().push_back(hp_);
  }
  HeadPipeLease(const HeadPipeLease&) = delete;
  HeadPipeLease& operator=(const HeadPipeLease&) = delete;
  // null when the pinned buffer or the events could not be created: poll synchronously
  HeadPipe* get() const { return hp_->ok ? hp_ : nullptr; }

 private:
  static std::mutex& mu() {
    static std::mutex m;
    return m;
  }
  static std::vector<HeadPipe*>& pool() {
    static std::vector<HeadPipe*> p;
    return p;
  }
  HeadPipe* hp_ = nullptr;
};

// The start of a solve from x = 0.  CG: one pass (k_cg_start).  RMR and GMRES: x cleared and, with
// src64, b narrowed into its buffer (which the solver reads again).
template <typename T>
static void cg_start(const SpecSystem& sys, const SolveOpts& o, const cpx<T>* B, cpx<T>* X, cpx<T>* r, cpx<T>* p,
                     const RedArgs& ra, cudaStream_t st) {
  const long long nc = sys.G->g.ncplx;
  const int rb = red_blocks(sys.len);
  const Ix ix = mkix(sys.len, sys.h0, nc, rb, kRedThreads);
  const double el = (double)sys.len * sizeof(cpx<T>);
  ProfScope ps_(sizeof(T) == 4 ? PC_VEC32 : PC_VEC64, st, (o.src64 ? 5 : 4) * el + (double)nc * sizeof(T), 0.0);
  if constexpr (sizeof(T) == 4) {
    if (o.src64) {
      pdl_launch(k_cg_start<T, true>, rb, kRedThreads, 0, st, ix, B, (const cpx<double>*)o.src64, o.src_scale,
                 o.dev_outer, X, r, p, (const T*)sys.sym, ra);
      return;
    }
  }
  pdl_launch(k_cg_start<T, false>, rb, kRedThreads, 0, st, ix, B, nullptr, 1.0, nullptr, X, r, p, (const T*)sys.sym,
             ra);
}
template <typename T>
static vd_status start_from_zero(const SolveOpts& o, const void* b, void* x, long long len, cudaStream_t st) {
  if (!o.x_zero) return VD_OK;
  VD_CUDA(cudaMemsetAsync(x, 0, sizeof(cpx<T>) * len, st));
  if (o.src64) {
    ProfScope ps_(PC_VEC64, st, (double)len * (sizeof(cpx<double>) + sizeof(cpx<float>)), 0.0);
    pdl_launch(k_d2f_scaled, ew_blocks(len), 256, 0, st, len, (const cpx<double>*)o.src64, o.src_scale, o.dev_outer,
               (cpx<float>*)const_cast<void*>(b));
  }
  return VD_OK;
}

template <typename T>
vd_status krylov_solve(const SpecSystem& sys, const SolveOpts& o, const void* b, void* x, void* vecs,
                       const KWork& kw, double* host_hist, int host_hist_cap, SolveOut* out, cudaStream_t st) {
  const long long len = sys.len;
  const long long nc = sys.G->g.ncplx;
  const int h0 = sys.h0;
  const T* sym = (const T*)sys.sym;
  const int rb = red_blocks(len);
  const int eb = ew_blocks(len);
  const Ix ixr = mkix(len, h0, nc, rb, kRedThreads);
  const Ix ixe = mkix(len, h0, nc, eb, 256);
  RedArgs ra{kw.ks, kw.partials, kw.counter, kw.hist, o.tol};
  int* done = &kw.ks->done;
  int* cdone = &kw.ks->cycle_done;
  const int m = std::min(std::max(o.restart > 0 ? o.restart : 30, 1), kMaxRestart);
  const int check = std::max(1, o.check_every);

  // reset the scalar state
  KHead h0s;
  std::memset(&h0s, 0, sizeof(h0s));
  h0s.maxit = o.maxit;
  h0s.status = KS_RUNNING;
  h0s.hist_cap = host_hist_cap > 0 ? std::min(host_hist_cap, 1 << 20) : 0;
  h0s.m = m;
  h0s.guard = o.guard;
  VD_CUDA(cudaMemcpyAsync(kw.ks, &h0s, sizeof(KHead), cudaMemcpyHostToDevice, st));
  VD_CUDA(cudaMemsetAsync(kw.counter, 0, sizeof(unsigned), st));

  cpx<T>* X = (cpx<T>*)x;
  const cpx<T>* B = (const cpx<T>*)b;
  cpx<T>* vb = (cpx<T>*)vecs;
  KHead hd;
  if (o.solver != VD_SOLVER_CG) {
    const vd_status e0 = start_from_zero<T>(o, b, x, len, st);
    if (e0 != VD_OK) return e0;
  }

  if (o.solver == VD_SOLVER_CG) {
    cpx<T>* r = vb;
    cpx<T>* p = vb + len;
    cpx<T>* q = vb + 2 * len;
    if (o.x_zero) {
      cg_start<T>(sys, o, B, X, r, p, ra, st);
    } else {
      sys.apply(sys, X, q, false, nullptr, st);
      { ProfScope ps_(sizeof(T) == 4 ? PC_VEC32 : PC_VEC64, st, (double)3 * len * sizeof(cpx<T>), 0.0); pdl_launch(k_sub<T>, eb, 256, 0, st, len, B, q, r, nullptr); }
      { ProfScope ps_(sizeof(T) == 4 ? PC_VEC32 : PC_VEC64, st, (double)3 * len * sizeof(cpx<T>) + (double)nc * sizeof(T), 0.0); pdl_launch(k_cg_init<T>, rb, kRedThreads, 0, st, ixr, B, r, p, sym, ra); }
    }
    int it = 0;
    HeadPipeLease lease;
    HeadPipe* hp = lease.get();
    for (;;) {
      const long long mark = prof_mark();
      for (int c = 0; c < check && it < o.maxit; ++c, ++it) {
        sys.apply(sys, p, q, false, done, st);
        { ProfScope ps_(sizeof(T) == 4 ? PC_VEC32 : PC_VEC64, st, (double)2 * len * sizeof(cpx<T>), 0.0); pdl_launch(k_dot<T, 1>, rb, kRedThreads, 0, st, ixr, p, q, EPI_CG_ALPHA, ra, done); }
        { ProfScope ps_(sizeof(T) == 4 ? PC_VEC32 : PC_VEC64, st, (double)6 * len * sizeof(cpx<T>) + (double)nc * sizeof(T), 0.0); pdl_launch(k_cg_update<T>, rb, kRedThreads, 0, st, ixr, X, p, r, q, sym, ra); }
        { ProfScope ps_(sizeof(T) == 4 ? PC_VEC32 : PC_VEC64, st, (double)3 * len * sizeof(cpx<T>) + (double)nc * sizeof(T), 0.0); pdl_launch(k_cg_p<T>, eb, 256, 0, st, ixe, p, r, sym, kw.ks); }
      }
      vd_status e = VD_OK;
      if (!hp) {
        e = read_head(kw, &hd, st);
        if (e != VD_OK) return e;
        if (hd.done || it >= o.maxit) break;
        continue;
      }
      if (hp->taken > 0) {
        e = hp->latest(&hd);   // the batch before the one just enqueued
        if (e != VD_OK) return e;
        if (hd.done) {
          prof_discard(mark, st);   // the batch just enqueued returns at once
          break;
        }
      }
      if (it >= o.maxit) break;
      e = hp->snapshot(kw, st);
      if (e != VD_OK) return e;
    }
  } else if (o.solver == VD_SOLVER_RMR) {
    cpx<T>* r = vb;
    cpx<T>* w = vb + len;
    if (o.x_zero) {
      VD_CUDA(cudaMemcpyAsync(r, B, sizeof(cpx<T>) * len, cudaMemcpyDeviceToDevice, st));
    } else {
      sys.apply(sys, X, w, false, nullptr, st);
      { ProfScope ps_(sizeof(T) == 4 ? PC_VEC32 : PC_VEC64, st, (double)3 * len * sizeof(cpx<T>), 0.0); pdl_launch(k_sub<T>, eb, 256, 0, st, len, B, w, r, nullptr); }
    }
    { ProfScope ps_(sizeof(T) == 4 ? PC_VEC32 : PC_VEC64, st, (double)2 * len * sizeof(cpx<T>), 0.0); pdl_launch(k_norms<T, 2>, rb, kRedThreads, 0, st, ixr, B, r, EPI_INIT_RMR, ra, nullptr); }
    int it = 0;
    HeadPipeLease lease;
    HeadPipe* hp = lease.get();
    for (;;) {
      const long long mark = prof_mark();
      for (int c = 0; c < check && it < o.maxit; ++c, ++it) {
        sys.apply(sys, r, w, true, done, st);
        { ProfScope ps_(sizeof(T) == 4 ? PC_VEC32 : PC_VEC64, st, (double)2 * len * sizeof(cpx<T>), 0.0); pdl_launch(k_dot<T, 2>, rb, kRedThreads, 0, st, ixr, r, w, EPI_RMR_ALPHA, ra, done); }
        { ProfScope ps_(sizeof(T) == 4 ? PC_VEC32 : PC_VEC64, st, (double)5 * len * sizeof(cpx<T>) + (double)nc * sizeof(T), 0.0); pdl_launch(k_rmr_update<T>, rb, kRedThreads, 0, st, ixr, X, r, w, sym, ra); }
      }
      vd_status e = VD_OK;
      if (!hp) {
        e = read_head(kw, &hd, st);
        if (e != VD_OK) return e;
        if (hd.done || it >= o.maxit) break;
        continue;
      }
      if (hp->taken > 0) {
        e = hp->latest(&hd);
        if (e != VD_OK) return e;
        if (hd.done) {
          prof_discard(mark, st);
          break;
        }
      }
      if (it >= o.maxit) break;
      e = hp->snapshot(kw, st);
      if (e != VD_OK) return e;
    }
  } else {
    cpx<T>* V = vb;
    cpx<T>* w = vb + (size_t)(m + 1) * len;
    HeadPipeLease lease;
    HeadPipe* hp = lease.get();
    { ProfScope ps_(sizeof(T) == 4 ? PC_VEC32 : PC_VEC64, st, (double)1 * len * sizeof(cpx<T>), 0.0); pdl_launch(k_norms<T, 1>, rb, kRedThreads, 0, st, ixr, nullptr, B, EPI_BB, ra, nullptr); }
    for (int cycle = 0;; ++cycle) {
      // r = b - A x into V_0 (unnormalised), then V_0 /= beta
      if (cycle == 0 && o.x_zero) {
        VD_CUDA(cudaMemcpyAsync(V, B, sizeof(cpx<T>) * len, cudaMemcpyDeviceToDevice, st));
      } else {
        sys.apply(sys, X, w, false, done, st);
        { ProfScope ps_(sizeof(T) == 4 ? PC_VEC32 : PC_VEC64, st, (double)3 * len * sizeof(cpx<T>), 0.0); pdl_launch(k_sub<T>, eb, 256, 0, st, len, B, w, V, done); }
      }
      { ProfScope ps_(sizeof(T) == 4 ? PC_VEC32 : PC_VEC64, st, (double)1 * len * sizeof(cpx<T>), 0.0); pdl_launch(k_norms<T, 1>, rb, kRedThreads, 0, st, ixr, nullptr, V, EPI_GM_BETA, ra, done); }
      { ProfScope ps_(sizeof(T) == 4 ? PC_VEC32 : PC_VEC64, st, (double)2 * len * sizeof(cpx<T>), 0.0); pdl_launch(k_gm_scale<T>, eb, 256, 0, st, ixe, V, V, kw.ks, 1); }
      // the flag of step j is read with step j + check already queued (its kernels see the device's
      // flag and return), so the device does not wait for the host between steps.  Not for three
      // components: the step that comes to nothing at the end of their cycle is 25 launches, more than the
      // waits it saves.  Solves ahead and not, us: pressure 64^2 mixed 1729 and 1850, 512^2 fp64 5147 and
      // 5297, 32^3 mixed 1870 and 2047, 128^3 mixed_dd 5969 and 6170; velocity 64^2 mixed 962 and 986, 512^2
      // 3005 and 3096; three components 32^3 mixed 1416 and 1420, 48^3 1700 and 1656, 96^3 5708 and
      // 5627, 128^3 fp64 37390 and 36880 (nine sizes in all, no exception).
      const bool ahead = hp && sys.ncomp < 3;
      int snaps = 0;
      long long mark = 0;
      for (int j = 0; j < m; ++j) {
        if (j % check == 0) mark = prof_mark();
        cpx<T>* Vj = V + (size_t)j * len;
        sys.apply(sys, Vj, w, true, cdone, st);
        gm_orthogonalise<T>(sys, w, V, j, ra, st);
        { ProfScope ps_(sizeof(T) == 4 ? PC_VEC32 : PC_VEC64, st, (double)2 * len * sizeof(cpx<T>), 0.0); pdl_launch(k_gm_scale<T>, eb, 256, 0, st, ixe, V + (size_t)(j + 1) * len, w, kw.ks, 0); }
        if ((j + 1) % check == 0 || j + 1 == m) {
          vd_status e = VD_OK;
          if (!ahead) {
            e = read_head(kw, &hd, st);
            if (e != VD_OK) return e;
            if (hd.cycle_done || hd.done) break;
            continue;
          }
          if (snaps > 0) {
            e = hp->latest(&hd);
            if (e != VD_OK) return e;
            if (hd.cycle_done || hd.done) {
              prof_discard(mark, st);
              break;
            }
          }
          e = hp->snapshot(kw, st);
          if (e != VD_OK) return e;
          ++snaps;
        }
      }
      { pdl_launch(k_gm_solve, 1, 32, 0, st, kw.ks); count_launch(); }
      { ProfScope ps_(sizeof(T) == 4 ? PC_VEC32 : PC_VEC64, st, (double)(m + 2) * len * sizeof(cpx<T>) + (double)nc * sizeof(T), 0.0); pdl_launch(k_gm_update<T>, eb, 256, 0, st, ixe, X, V, sym, kw.ks); }
      { pdl_launch(k_gm_close, 1, 1, 0, st, kw.ks); count_launch(); }
      vd_status e = read_head(kw, &hd, st);
      if (e != VD_OK) return e;
      if (hd.done) break;
      if (hd.iters >= o.maxit) {
        // one more loop head forms the true residual and sets the final status
        sys.apply(sys, X, w, false, done, st);
        { ProfScope ps_(sizeof(T) == 4 ? PC_VEC32 : PC_VEC64, st, (double)3 * len * sizeof(cpx<T>), 0.0); pdl_launch(k_sub<T>, eb, 256, 0, st, len, B, w, V, done); }
        { ProfScope ps_(sizeof(T) == 4 ? PC_VEC32 : PC_VEC64, st, (double)1 * len * sizeof(cpx<T>), 0.0); pdl_launch(k_norms<T, 1>, rb, kRedThreads, 0, st, ixr, nullptr, V, EPI_GM_BETA, ra, done); }
        e = read_head(kw, &hd, st);
        if (e != VD_OK) return e;
        break;
      }
    }
  }
  VD_CUDA(cudaGetLastError());
  vd_status e = read_head(kw, &hd, st);
  if (e != VD_OK) return e;
  if (!hd.done) hd.status = VD_ERR_NOT_CONVERGED;
  out->iters = hd.iters;
  out->status = hd.status < 0 ? VD_ERR_NOT_CONVERGED : hd.status;
  out->relres = hd.relres;
  if (host_hist && h0s.hist_cap > 0) {
    const int nh = std::min(h0s.hist_cap, hd.iters + 1);
    VD_CUDA(cudaMemcpyAsync(host_hist, kw.hist, sizeof(double) * nh, cudaMemcpyDeviceToHost, st));
    VD_CUDA(cudaStreamSynchronize(st));
  }
  return VD_OK;
}

// ---------------------------------------------------------------------------------------
// graph form: the same kernels, with the iteration loop as a conditional WHILE node whose
// body ends in a kernel that sets the loop condition from the device `done` flag.  Nothing
// in it synchronises with the host, so it can be captured and replayed as a whole.
// ---------------------------------------------------------------------------------------

__global__ void k_ks_reset(KState* ks, int maxit, int m, cudaGraphConditionalHandle loop) {
  pdl_wait();
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  // a loop nested in another conditional body keeps its last condition value: arm it here
  cudaGraphSetConditional(loop, 1u);
  KHead* h = reinterpret_cast<KHead*>(ks);
  unsigned* w = reinterpret_cast<unsigned*>(h);
  for (size_t i = 0; i < sizeof(KHead) / sizeof(unsigned); ++i) w[i] = 0u;
  h->maxit = maxit;
  h->status = KS_RUNNING;
  h->m = m;
}

// inner solve of a refinement sweep: budget and tolerance from the refinement state
__global__ void k_ks_reset_dev(KState* ks, const OState* o, int m, cudaGraphConditionalHandle loop) {
  pdl_wait();
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  cudaGraphSetConditional(loop, 1u);
  KHead* h = reinterpret_cast<KHead*>(ks);
  unsigned* w = reinterpret_cast<unsigned*>(h);
  for (size_t i = 0; i < sizeof(KHead) / sizeof(unsigned); ++i) w[i] = 0u;
  h->maxit = o->maxit - o->total;
  h->status = KS_RUNNING;
  h->m = m;
  h->guard = kInnerGuard;
  ks->dtol = o->itol;
}

// The Arnoldi steps of a recorded GMRES cycle stand in groups, each the body of an IF node: a group that
// ends before the cycle does sets the condition of the next, so the steps after convergence are
// skipped (as kernels that return at once, 16 to 25 a step, they were half of a 64^3 velocity solve:
// 5.0 ms recorded, 2.6 in groups).
constexpr int kGmGroups = 8;
constexpr int kGmGroupAt[kGmGroups + 1] = {0, 4, 8, 12, 16, 24, 32, 48, kMaxRestart};
struct GmConds {
  cudaGraphConditionalHandle h[kGmGroups];
};
// start of a cycle: the first group runs unless the residual already meets the tolerance
__global__ void k_gm_arm(GmConds c, int n, const KState* ks) {
  pdl_wait();
  if (threadIdx.x < n) cudaGraphSetConditional(c.h[threadIdx.x], (threadIdx.x == 0 && !ks->cycle_done) ? 1u : 0u);
}
__global__ void k_gm_next(cudaGraphConditionalHandle h, const KState* ks) {
  pdl_wait();
  if (threadIdx.x == 0) cudaGraphSetConditional(h, ks->cycle_done ? 0u : 1u);
}

static vd_status open_cond(cudaStream_t st, cudaGraphConditionalNodeType type, cudaGraphConditionalHandle hnd,
                           cudaGraph_t* body) {
  cudaStreamCaptureStatus cs;
  cudaGraph_t g = nullptr;
  const cudaGraphNode_t* deps = nullptr;
  size_t nd = 0;
  VD_CUDA(cudaStreamGetCaptureInfo(st, &cs, nullptr, &g, &deps, nullptr, &nd));
  if (cs != cudaStreamCaptureStatusActive) return fail(VD_ERR_INVALID_ARG, "graph solve needs a capturing stream");
  cudaGraphNodeParams cp{};
  cp.type = cudaGraphNodeTypeConditional;
  cp.conditional.handle = hnd;
  cp.conditional.type = type;
  cp.conditional.size = 1;
  cudaGraphNode_t node;
  VD_CUDA(cudaGraphAddNode(&node, g, deps, nullptr, nd, &cp));
  VD_CUDA(cudaStreamUpdateCaptureDependencies(st, &node, nullptr, 1, cudaStreamSetCaptureDependencies));
  *body = cp.conditional.phGraph_out[0];
  return VD_OK;
}

__global__ void k_graph_cond(cudaGraphConditionalHandle handle, const KState* ks) {
  pdl_wait();
  if (threadIdx.x == 0 && blockIdx.x == 0) cudaGraphSetConditional(handle, ks->done ? 0u : 1u);
}

template <typename T>
vd_status krylov_enqueue_graph(const SpecSystem& sys, const SolveOpts& o, const void* b, void* x, void* vecs,
                               const KWork& kw, cudaStream_t st, cudaStream_t body_st, cudaStream_t group_st) {
  const long long len = sys.len;
  const long long nc = sys.G->g.ncplx;
  const int h0 = sys.h0;
  const T* sym = (const T*)sys.sym;
  const int rb = red_blocks(len);
  const int eb = ew_blocks(len);
  const Ix ixr = mkix(len, h0, nc, rb, kRedThreads);
  const Ix ixe = mkix(len, h0, nc, eb, 256);
  RedArgs ra{kw.ks, kw.partials, kw.counter, kw.hist, o.dev_outer ? -1.0 : o.tol};
  int* done = &kw.ks->done;
  int* cdone = &kw.ks->cycle_done;
  const int m = std::min(std::max(o.restart > 0 ? o.restart : 30, 1), kMaxRestart);
  cpx<T>* X = (cpx<T>*)x;
  const cpx<T>* B = (const cpx<T>*)b;
  cpx<T>* vb = (cpx<T>*)vecs;

  // the loop's condition handle belongs to the graph being captured on st
  cudaGraphConditionalHandle hnd;
  {
    cudaStreamCaptureStatus cs;
    cudaGraph_t g = nullptr;
    VD_CUDA(cudaStreamGetCaptureInfo(st, &cs, nullptr, &g, nullptr, nullptr, nullptr));
    if (cs != cudaStreamCaptureStatusActive) return fail(VD_ERR_INVALID_ARG, "graph solve needs a capturing stream");
    VD_CUDA(cudaGraphConditionalHandleCreate(&hnd, g, 1, cudaGraphCondAssignDefault));
  }
  if (o.dev_outer) pdl_launch(k_ks_reset_dev, 1, 1, 0, st, kw.ks, o.dev_outer, m, hnd);
  else pdl_launch(k_ks_reset, 1, 1, 0, st, kw.ks, o.maxit, m, hnd);
  count_launch();
  VD_CUDA(cudaMemsetAsync(kw.counter, 0, sizeof(unsigned), st));
  // the while node: splice it into the capture of st, then capture its body on body_st
  auto open_loop = [&](cudaGraphConditionalHandle* h) -> vd_status {
    cudaStreamCaptureStatus cs;
    cudaGraph_t g = nullptr;
    const cudaGraphNode_t* deps = nullptr;
    size_t nd = 0;
    VD_CUDA(cudaStreamGetCaptureInfo(st, &cs, nullptr, &g, &deps, nullptr, &nd));
    if (cs != cudaStreamCaptureStatusActive) return fail(VD_ERR_INVALID_ARG, "graph solve needs a capturing stream");
    cudaGraphNodeParams cp{};
    cp.type = cudaGraphNodeTypeConditional;
    cp.conditional.handle = *h;
    cp.conditional.type = cudaGraphCondTypeWhile;
    cp.conditional.size = 1;
    cudaGraphNode_t node;
    VD_CUDA(cudaGraphAddNode(&node, g, deps, nullptr, nd, &cp));
    VD_CUDA(cudaStreamUpdateCaptureDependencies(st, &node, nullptr, 1, cudaStreamSetCaptureDependencies));
    VD_CUDA(cudaStreamBeginCaptureToGraph(body_st, cp.conditional.phGraph_out[0], nullptr, nullptr, 0,
                                          cudaStreamCaptureModeRelaxed));
    return VD_OK;
  };
  auto close_loop = [&](cudaGraphConditionalHandle hnd) -> vd_status {
    pdl_launch(k_graph_cond, 1, 1, 0, body_st, hnd, kw.ks);
    count_launch();
    cudaGraph_t body = nullptr;
    VD_CUDA(cudaStreamEndCapture(body_st, &body));
    return VD_OK;
  };
  vd_status e;
  if (o.solver != VD_SOLVER_CG && (e = start_from_zero<T>(o, b, x, len, st)) != VD_OK) return e;
  if (o.solver == VD_SOLVER_CG) {
    cpx<T>* r = vb;
    cpx<T>* p = vb + len;
    cpx<T>* q = vb + 2 * len;
    if (o.x_zero) {
      cg_start<T>(sys, o, B, X, r, p, ra, st);
    } else {
      sys.apply(sys, X, q, false, nullptr, st);
      pdl_launch(k_sub<T>, eb, 256, 0, st, len, B, q, r, nullptr);
      pdl_launch(k_cg_init<T>, rb, kRedThreads, 0, st, ixr, B, r, p, sym, ra);
      count_launch();
      count_launch();
    }
    if ((e = open_loop(&hnd)) != VD_OK) return e;
    sys.apply(sys, p, q, false, done, body_st);
    pdl_launch(k_dot<T, 1>, rb, kRedThreads, 0, body_st, ixr, p, q, EPI_CG_ALPHA, ra, done);
    pdl_launch(k_cg_update<T>, rb, kRedThreads, 0, body_st, ixr, X, p, r, q, sym, ra);
    pdl_launch(k_cg_p<T>, eb, 256, 0, body_st, ixe, p, r, sym, kw.ks);
    count_launch();
    count_launch();
    count_launch();
    if ((e = close_loop(hnd)) != VD_OK) return e;
  } else if (o.solver == VD_SOLVER_RMR) {
    cpx<T>* r = vb;
    cpx<T>* w = vb + len;
    if (o.x_zero) {
      VD_CUDA(cudaMemcpyAsync(r, B, sizeof(cpx<T>) * len, cudaMemcpyDeviceToDevice, st));
    } else {
      sys.apply(sys, X, w, false, nullptr, st);
      pdl_launch(k_sub<T>, eb, 256, 0, st, len, B, w, r, nullptr);
      count_launch();
    }
    pdl_launch(k_norms<T, 2>, rb, kRedThreads, 0, st, ixr, B, r, EPI_INIT_RMR, ra, nullptr);
    count_launch();
    if ((e = open_loop(&hnd)) != VD_OK) return e;
    sys.apply(sys, r, w, true, done, body_st);
    pdl_launch(k_dot<T, 2>, rb, kRedThreads, 0, body_st, ixr, r, w, EPI_RMR_ALPHA, ra, done);
    pdl_launch(k_rmr_update<T>, rb, kRedThreads, 0, body_st, ixr, X, r, w, sym, ra);
    count_launch();
    count_launch();
    if ((e = close_loop(hnd)) != VD_OK) return e;
  } else {
    cpx<T>* V = vb;
    cpx<T>* w = vb + (size_t)(m + 1) * len;
    pdl_launch(k_norms<T, 1>, rb, kRedThreads, 0, st, ixr, nullptr, B, EPI_BB, ra, nullptr);
    count_launch();
    if ((e = open_loop(&hnd)) != VD_OK) return e;
    // one restart cycle: r = b - A x, V_0 = r / beta, m Arnoldi steps, update x
    sys.apply(sys, X, w, false, done, body_st);
    pdl_launch(k_sub<T>, eb, 256, 0, body_st, len, B, w, V, done);
    pdl_launch(k_norms<T, 1>, rb, kRedThreads, 0, body_st, ixr, nullptr, V, EPI_GM_BETA, ra, done);
    pdl_launch(k_gm_scale<T>, eb, 256, 0, body_st, ixe, V, V, kw.ks, 1);
    count_launch();
    count_launch();
    count_launch();
    int groups = 0;
    while (kGmGroupAt[groups] < m) ++groups;
    GmConds conds{};
    {
      cudaStreamCaptureStatus cs;
      cudaGraph_t g = nullptr;
      VD_CUDA(cudaStreamGetCaptureInfo(body_st, &cs, nullptr, &g, nullptr, nullptr, nullptr));
      for (int k = 0; k < groups; ++k)
        VD_CUDA(cudaGraphConditionalHandleCreate(&conds.h[k], g, 0, cudaGraphCondAssignDefault));
    }
    pdl_launch(k_gm_arm, 1, 32, 0, body_st, conds, groups, kw.ks);
    count_launch();
    for (int k = 0; k < groups; ++k) {
      cudaGraph_t gb = nullptr;
      if ((e = open_cond(body_st, cudaGraphCondTypeIf, conds.h[k], &gb)) != VD_OK) return e;
      VD_CUDA(cudaStreamBeginCaptureToGraph(group_st, gb, nullptr, nullptr, 0, cudaStreamCaptureModeRelaxed));
      for (int j = kGmGroupAt[k]; j < std::min(m, kGmGroupAt[k + 1]); ++j) {
        cpx<T>* Vj = V + (size_t)j * len;
        sys.apply(sys, Vj, w, true, cdone, group_st);
        gm_orthogonalise<T>(sys, w, V, j, ra, group_st);
        pdl_launch(k_gm_scale<T>, eb, 256, 0, group_st, ixe, V + (size_t)(j + 1) * len, w, kw.ks, 0);
        count_launch();
      }
      if (k + 1 < groups) {
        pdl_launch(k_gm_next, 1, 1, 0, group_st, conds.h[k + 1], kw.ks);
        count_launch();
      }
      VD_CUDA(cudaStreamEndCapture(group_st, &gb));
    }
    pdl_launch(k_gm_solve, 1, 32, 0, body_st, kw.ks);
    pdl_launch(k_gm_update<T>, eb, 256, 0, body_st, ixe, X, V, sym, kw.ks);
    pdl_launch(k_gm_close, 1, 1, 0, body_st, kw.ks);
    count_launch();
    count_launch();
    count_launch();
    if ((e = close_loop(hnd)) != VD_OK) return e;
  }
  VD_CUDA(cudaGetLastError());
  return VD_OK;
}

// result record of a graph solve: info[0] iterations, [1] status, [2] monitored relres,
// [3] |b|^2, [4] true relres
__global__ void k_graph_info(const KState* ks, double* info, int phase) {
  pdl_wait();
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  if (phase == 0) {
    info[0] = (double)ks->iters;
    const int st = ks->done ? (ks->status < 0 ? VD_ERR_NOT_CONVERGED : ks->status) : VD_ERR_NOT_CONVERGED;
    info[1] = (double)st;
    info[2] = ks->relres;
  } else if (phase == 1) {
    info[3] = ks->rr;
  } else {
    info[4] = info[3] > 0.0 ? sqrt(ks->rr / info[3]) : 0.0;
  }
}

template <typename T>
vd_status krylov_graph_finish(const SpecSystem& sys, const void* b, const void* x, void* vecs, const KWork& kw,
                              double* info, cudaStream_t st) {
  const long long len = sys.len;
  const int rb = red_blocks(len);
  const int eb = ew_blocks(len);
  const Ix ixr = mkix(len, sys.h0, sys.G->g.ncplx, rb, kRedThreads);
  RedArgs ra{kw.ks, kw.partials, kw.counter, kw.hist, 0.0};
  const cpx<T>* B = (const cpx<T>*)b;
  cpx<T>* W = (cpx<T>*)vecs;
  pdl_launch(k_graph_info, 1, 1, 0, st, kw.ks, info, 0);
  pdl_launch(k_norms<T, 1>, rb, kRedThreads, 0, st, ixr, nullptr, B, EPI_NORM, ra, nullptr);
  pdl_launch(k_graph_info, 1, 1, 0, st, kw.ks, info, 1);
  sys.apply(sys, x, W, false, nullptr, st);
  pdl_launch(k_sub<T>, eb, 256, 0, st, len, B, W, W, nullptr);
  pdl_launch(k_norms<T, 1>, rb, kRedThreads, 0, st, ixr, nullptr, W, EPI_NORM, ra, nullptr);
  pdl_launch(k_graph_info, 1, 1, 0, st, kw.ks, info, 2);
  for (int i = 0; i < 6; ++i) count_launch();
  VD_CUDA(cudaGetLastError());
  return VD_OK;
}
template vd_status krylov_graph_finish<double>(const SpecSystem&, const void*, const void*, void*, const KWork&,
                                               double*, cudaStream_t);

// ---------------------------------------------------------------------------------------
// iterative refinement as a graph fragment
// ---------------------------------------------------------------------------------------

__global__ void k_out_init(OState* o, const KState* ks, double tol, double itol0, int maxit,
                           cudaGraphConditionalHandle loop) {
  pdl_wait();
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  cudaGraphSetConditional(loop, 1u);
  o->bb = ks->rr;   // |b|^2, and the first residual is b
  o->rr = ks->rr;
  o->rnorm = o->rel = o->scale = 0.0;
  o->tol = tol;
  o->itol0 = itol0;
  o->itol = itol0;
  o->total = o->outer = 0;
  o->maxit = maxit;
  o->maxouter = 20;
  o->done = 0;
  o->status = VD_ERR_NOT_CONVERGED;
  o->force = 0;
}

// top of a refinement sweep: the same decisions as the host loop of vd_solve
__global__ void k_out_check(OState* o, cudaGraphConditionalHandle h_loop, cudaGraphConditionalHandle h_sweep) {
  pdl_wait();
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  const double rnorm = sqrt(o->rr);
  const double bnorm = sqrt(o->bb);
  // a non-finite norm must not read as a zero right-hand side (NaN > 0 is false)
  const double rel = (!isfinite(bnorm) || !isfinite(rnorm)) ? (double)NAN : (bnorm > 0.0 ? rnorm / bnorm : 0.0);
  o->rnorm = rnorm;
  o->rel = rel;
  if (o->force) {
    o->done = 1;
    o->status = o->force;
  } else if (!isfinite(rel)) {
    o->done = 1;
    o->status = VD_ERR_NONFINITE;
  } else if (rel <= o->tol) {
    o->done = 1;
    o->status = VD_OK;
  } else if (o->total >= o->maxit || o->outer >= o->maxouter) {
    o->done = 1;
    o->status = VD_ERR_NOT_CONVERGED;
  } else {
    o->scale = 1.0 / rnorm;
    o->itol = fmax(o->itol0, 0.5 * o->tol / rel);
  }
  cudaGraphSetConditional(h_loop, o->done ? 0u : 1u);
  cudaGraphSetConditional(h_sweep, o->done ? 0u : 1u);
}

__global__ void k_out_after_inner(OState* o, const KState* ks) {
  pdl_wait();
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  o->total += ks->iters;
  o->outer += 1;
  const int st = ks->done ? ks->status : VD_ERR_NOT_CONVERGED;
  if (st == VD_ERR_NONFINITE) o->force = VD_ERR_NONFINITE;
  else if (ks->iters == 0 && st != VD_OK) o->force = VD_ERR_NOT_CONVERGED;
}

__global__ void k_out_rr(OState* o, const KState* ks) {
  pdl_wait();
  if (threadIdx.x == 0 && blockIdx.x == 0) o->rr = ks->rr;
}

__global__ void k_out_info(const OState* o, double* info) {
  pdl_wait();
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  info[0] = (double)o->total;
  info[1] = (double)(o->done ? o->status : VD_ERR_NOT_CONVERGED);
  info[2] = o->rel;
  info[3] = o->bb;
  info[4] = o->rel;   // the refinement residual is the accurately computed true residual
  info[5] = (double)o->outer;
}

// v *= 1/|r| and x += |r| d with the scalars read from the refinement state

vd_status refine_enqueue_graph(const SpecSystem& sys64, const SpecSystem& sys32,
                               void (*resid)(const void* ctx, const void* x, void* y, cudaStream_t st),
                               const void* resid_ctx, const SolveOpts& inner, double tol, double itol0, int maxit,
                               void* bh, void* xh, void* rh, void* bh_f, void* xh_f, void* vecs, const KWork& kw,
                               OState* ost, double* info, cudaStream_t st, cudaStream_t s1, cudaStream_t s2,
                               cudaStream_t s3, cudaStream_t s4) {
  const long long len = sys64.len;
  const int rb = red_blocks(len);
  const int eb = ew_blocks(len);
  const Ix ixr = mkix(len, sys64.h0, sys64.G->g.ncplx, rb, kRedThreads);
  RedArgs ra{kw.ks, kw.partials, kw.counter, kw.hist, 0.0};
  cpx<double>* BH = (cpx<double>*)bh;
  cpx<double>* XH = (cpx<double>*)xh;
  cpx<double>* RH = (cpx<double>*)rh;
  // |b|^2, x = 0, r = b
  cudaGraphConditionalHandle h_loop, h_sweep;
  {
    cudaStreamCaptureStatus cs;
    cudaGraph_t g0 = nullptr;
    VD_CUDA(cudaStreamGetCaptureInfo(st, &cs, nullptr, &g0, nullptr, nullptr, nullptr));
    if (cs != cudaStreamCaptureStatusActive) return fail(VD_ERR_INVALID_ARG, "graph solve needs a capturing stream");
    VD_CUDA(cudaGraphConditionalHandleCreate(&h_loop, g0, 1, cudaGraphCondAssignDefault));
  }
  VD_CUDA(cudaMemsetAsync(kw.counter, 0, sizeof(unsigned), st));
  pdl_launch(k_norms<double, 1>, rb, kRedThreads, 0, st, ixr, nullptr, BH, EPI_NORM, ra, nullptr);
  pdl_launch(k_out_init, 1, 1, 0, st, ost, kw.ks, tol, itol0, maxit, h_loop);
  VD_CUDA(cudaMemsetAsync(XH, 0, sizeof(cpx<double>) * len, st));
  VD_CUDA(cudaMemcpyAsync(RH, BH, sizeof(cpx<double>) * len, cudaMemcpyDeviceToDevice, st));
  count_launch();
  count_launch();
  // while (not done) { check; if (sweep) { ... } }
  cudaGraph_t loop_body = nullptr, sweep_body = nullptr;
  vd_status e;
  if ((e = open_cond(st, cudaGraphCondTypeWhile, h_loop, &loop_body)) != VD_OK) return e;
  VD_CUDA(cudaStreamBeginCaptureToGraph(s1, loop_body, nullptr, nullptr, 0, cudaStreamCaptureModeRelaxed));
  {
    cudaStreamCaptureStatus cs;
    cudaGraph_t g1 = nullptr;
    VD_CUDA(cudaStreamGetCaptureInfo(s1, &cs, nullptr, &g1, nullptr, nullptr, nullptr));
    VD_CUDA(cudaGraphConditionalHandleCreate(&h_sweep, g1, 0, cudaGraphCondAssignDefault));
  }
  pdl_launch(k_out_check, 1, 1, 0, s1, ost, h_loop, h_sweep);
  count_launch();
  {
    cudaStreamCaptureStatus cs;
    cudaGraph_t g1 = nullptr;
    const cudaGraphNode_t* deps = nullptr;
    size_t nd = 0;
    VD_CUDA(cudaStreamGetCaptureInfo(s1, &cs, nullptr, &g1, &deps, nullptr, &nd));
    cudaGraphNodeParams cp{};
    cp.type = cudaGraphNodeTypeConditional;
    cp.conditional.handle = h_sweep;
    cp.conditional.type = cudaGraphCondTypeIf;
    cp.conditional.size = 1;
    cudaGraphNode_t node;
    VD_CUDA(cudaGraphAddNode(&node, g1, deps, nullptr, nd, &cp));
    VD_CUDA(cudaStreamUpdateCaptureDependencies(s1, &node, nullptr, 1, cudaStreamSetCaptureDependencies));
    sweep_body = cp.conditional.phGraph_out[0];
  }
  VD_CUDA(cudaStreamBeginCaptureToGraph(s2, sweep_body, nullptr, nullptr, 0, cudaStreamCaptureModeRelaxed));
  // the sweep: d solves A32 d = r/|r| in float, x += |r| d, r = b - A x, |r|^2
  SolveOpts si = inner;
  si.src64 = RH;
  si.x_zero = 1;
  si.dev_outer = ost;
  if ((e = krylov_enqueue_graph<float>(sys32, si, bh_f, xh_f, vecs, kw, s2, s3, s4)) != VD_OK) return e;
  pdl_launch(k_out_after_inner, 1, 1, 0, s2, ost, kw.ks);
  pdl_launch(k_axpy_f2d, eb, 256, 0, s2, len, 0.0, ost, (const cpx<float>*)xh_f, XH);
  resid(resid_ctx, XH, RH, s2);
  VD_CUDA(cudaMemsetAsync(kw.counter, 0, sizeof(unsigned), s2));
  pdl_launch(k_sub_norm<double>, rb, kRedThreads, 0, s2, ixr, BH, RH, RH, ra);
  pdl_launch(k_out_rr, 1, 1, 0, s2, ost, kw.ks);
  for (int i = 0; i < 4; ++i) count_launch();
  cudaGraph_t tmp = nullptr;
  VD_CUDA(cudaStreamEndCapture(s2, &tmp));
  VD_CUDA(cudaStreamEndCapture(s1, &tmp));
  pdl_launch(k_out_info, 1, 1, 0, st, ost, info);
  count_launch();
  (void)sys64;
  VD_CUDA(cudaGetLastError());
  return VD_OK;
}

template vd_status krylov_enqueue_graph<double>(const SpecSystem&, const SolveOpts&, const void*, void*, void*,
                                                const KWork&, cudaStream_t, cudaStream_t, cudaStream_t);
template vd_status krylov_enqueue_graph<float>(const SpecSystem&, const SolveOpts&, const void*, void*, void*,
                                               const KWork&, cudaStream_t, cudaStream_t, cudaStream_t);

template vd_status krylov_solve<double>(const SpecSystem&, const SolveOpts&, const void*, void*, void*, const KWork&,
                                        double*, int, SolveOut*, cudaStream_t);
template vd_status krylov_solve<float>(const SpecSystem&, const SolveOpts&, const void*, void*, void*, const KWork&,
                                       double*, int, SolveOut*, cudaStream_t);
template size_t krylov_vec_bytes<double>(const SpecSystem&, int, int);
template size_t krylov_vec_bytes<float>(const SpecSystem&, int, int);
template void spec_copy_scale<double>(long long, const void*, double, void*, cudaStream_t);
template void spec_copy_scale<float>(long long, const void*, double, void*, cudaStream_t);
template void spec_axpy<double>(long long, double, const void*, void*, cudaStream_t);
template void spec_axpy<float>(long long, double, const void*, void*, cudaStream_t);
template void spec_sub<double>(long long, const void*, const void*, void*, cudaStream_t);
template void spec_sub<float>(long long, const void*, const void*, void*, cudaStream_t);
template void spec_project<double>(const vd_grid*, int, void*, cudaStream_t, double*);
template void spec_project<float>(const vd_grid*, int, void*, cudaStream_t, double*);
template double spec_dot_host<double>(const SpecSystem&, const void*, const void*, const KWork&, cudaStream_t);
template double spec_norm2_host<double>(const SpecSystem&, const void*, const KWork&, cudaStream_t);
template double spec_norm2_host<float>(const SpecSystem&, const void*, const KWork&, cudaStream_t);

}  // namespace vd
