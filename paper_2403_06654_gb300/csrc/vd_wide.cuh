// Transform passes of any supported length in float and double: Stockham stages of radices up to
// 16 whose first stage loads from global memory and whose last one stores to it.
//
// A line of length n = R_0 ... R_{s-1} (radices up to 5, 8 or 16 by the size of the field, wide_class;
// 256 points in four, three or two stages) makes one shared-memory round trip per stage boundary only.  A thread transforms whole butterflies: in
// the first stage butterfly i of radix R reads elements i + r n/R, in the last one it writes
// elements i + r n/R, so both stages' rows are the thread's own registers.  In the fused x pass
// the forward transform runs its radices in reverse order: the last inverse butterfly's outputs
// are, after the weights, the inputs of the first forward butterfly of the same thread.
//
// What bounds it.  Float: the issue rate and the latency of the chain load - stages - store; the
// wide radices took the instructions per point of a 160-point y pass from 130 to about 70.
// Double: the FP64 pipe, which takes ~17 cycles of the SM per warp instruction whether its lanes
// are busy or not.  So butterflies and (un)packing items are numbered over all the lines of a
// block (no idle lanes at a line's end: the 64-point x pass ran 8 butterflies on 16 threads per
// line), y-pass lines are numbered across planes (no ragged tiles), the two halves of a real
// transform's spectrum are (un)packed in pairs (12 operations a pair instead of 20), and a unit
// scale is not multiplied.
#pragma once

#include "vd_launch.cuh"
#include "vd_passes.cuh"
#include "vd_fft.cuh"

#include <algorithm>
#include <type_traits>

namespace vd {

// ---------------------------------------------------------------------------------------
// codelets of the composite radices (S = -1 forward, +1 inverse)
// ---------------------------------------------------------------------------------------

// prime-factor form for coprime N1, N2 (no twiddles): input N2 n1 + N1 n2, output A k1 + B k2 (mod
// N1 N2), A = N2 (1/N2 mod N1), B = N1 (1/N1 mod N2)
template <typename T, int S, int N1, int N2, int A, int B>
__device__ __forceinline__ void dft_pfa(cpx<T>* u) {
  constexpr int N = N1 * N2;
  cpx<T> v[N2][N1];
#pragma unroll
  for (int b = 0; b < N2; ++b) {
#pragma unroll
    for (int a = 0; a < N1; ++a) v[b][a] = u[(N2 * a + N1 * b) % N];
    dftR<T, S, N1>(v[b]);
  }
#pragma unroll
  for (int a = 0; a < N1; ++a) {
    cpx<T> t[N2];
#pragma unroll
    for (int b = 0; b < N2; ++b) t[b] = v[b][a];
    dftR<T, S, N2>(t);
#pragma unroll
    for (int b = 0; b < N2; ++b) u[(A * a + B * b) % N] = t[b];
  }
}

// 9 = 3 x 3 with the twiddles W9^{bc}
template <typename T, int S>
__device__ __forceinline__ void dft9(cpx<T>* u) {
  const T c1 = T(0.76604444311897803520239265055542), s1 = T(0.64278760968653932632264340990726);
  const T c2 = T(0.17364817766693034885171662676931), s2 = T(0.98480775301220805936674302458952);
  const T c4 = T(-0.93969262078590838405410927732473), s4 = T(0.34202014332566873304409961468226);
  cpx<T> v[3][3];
#pragma unroll
  for (int b = 0; b < 3; ++b) {
    v[b][0] = u[b];
    v[b][1] = u[3 + b];
    v[b][2] = u[6 + b];
    dftR<T, S, 3>(v[b]);
  }
  v[1][1] = cmul(v[1][1], mk<T>(c1, T(S) * s1));
  v[1][2] = cmul(v[1][2], mk<T>(c2, T(S) * s2));
  v[2][1] = cmul(v[2][1], mk<T>(c2, T(S) * s2));
  v[2][2] = cmul(v[2][2], mk<T>(c4, T(S) * s4));
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    cpx<T> t[3] = {v[0][c], v[1][c], v[2][c]};
    dftR<T, S, 3>(t);
#pragma unroll
    for (int d = 0; d < 3; ++d) u[c + 3 * d] = t[d];
  }
}

template <typename T, int S, int R>
__device__ __forceinline__ void dft_wide(cpx<T>* u) {
  if constexpr (R == 6) dft_pfa<T, S, 2, 3, 3, 4>(u);
  else if constexpr (R == 9) dft9<T, S>(u);
  else if constexpr (R == 10) dft_pfa<T, S, 2, 5, 5, 6>(u);
  else if constexpr (R == 12) dft_pfa<T, S, 4, 3, 9, 4>(u);
  else if constexpr (R == 15) dft_pfa<T, S, 3, 5, 10, 6>(u);
  else dftR<T, S, R>(u);
}

// CALL(R) for the run-time radix
#define VD_WIDE_RADIX(RAD, CALL) \
  switch (RAD) {                 \
    case 2: CALL(2); break;      \
    case 3: CALL(3); break;      \
    case 4: CALL(4); break;      \
    case 5: CALL(5); break;      \
    case 6: CALL(6); break;      \
    case 8: CALL(8); break;      \
    case 9: CALL(9); break;      \
    case 10: CALL(10); break;    \
    case 12: CALL(12); break;    \
    case 15: CALL(15); break;    \
    default: CALL(16); break;    \
  }

template <typename T, int S>
__device__ __forceinline__ cpx<T> twiddled(cpx<T> v, cpx<T> w) {
  return (S < 0) ? cmul(v, w) : cmulc(v, w);
}

template <typename T>
__device__ __forceinline__ T wide_kfac(const GridDesc& g, int a) {
  if constexpr (sizeof(T) == 4) return g.kfac_f[a];
  else return g.kfac[a];
}

// ---------------------------------------------------------------------------------------
// y and z passes
// ---------------------------------------------------------------------------------------

// Block: W = 2^lw lines side by side, tpl threads per line.  Shared memory: the twiddle table, one
// (two stages) or two (more) tiles of W x n, and k~ of every index along the axis.
// PAD: rows of narrow tiles are padded (tiles of 128-byte rows need none).
template <typename T, int S, bool PAD>
__global__ void __launch_bounds__(kWideThreads, (sizeof(T) == 8 ? 2 : 3))
    k_axis_w(const __grid_constant__ AxisProg P, const __grid_constant__ GridDesc g, const cpx<T>* __restrict__ twg,
             int lw, int tpl, int ps, int cls) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int axis = P.axis;
  const WidePlan& pl = (axis == 2) ? g.wz[cls] : g.wy[cls];
  const int n = pl.n, nst = pl.nst, W = 1 << lw;
  cpx<T>* tw = reinterpret_cast<cpx<T>*>(smem_raw);
  cpx<T>* A = tw + n;
  const int tile = W * (PAD ? n + (n >> ps) : n);
  cpx<T>* B = A + (nst > 2 ? tile : 0);
  T* katab = reinterpret_cast<T*>(B + tile);
  auto at = [&](int j) { return (PAD ? j + (j >> ps) : j) << lw; };   // row of element j of the lines
  const T kfa = wide_kfac<T>(g, axis);
  for (int j = threadIdx.x; j < n; j += blockDim.x) {
    tw[j] = twg[pl.tw_off + j];
    katab[j] = kfa * (T)freq_tilde(j, n);
  }
  // lines are numbered over the whole field: z pass, the (y, x) plane; y pass, x within z
  const int line = (int)blockIdx.x * W + ((int)threadIdx.x & (W - 1));
  const int ib = (int)threadIdx.x >> lw;
  const int w = threadIdx.x & (W - 1);
  const int ls = (axis == 2) ? g.n1 * g.h0 : g.h0;
  const int o = (axis == 2) ? 0 : line / g.h0;
  const int col = (axis == 2) ? line : line - o * g.h0;
  const bool ok = line < ((axis == 2) ? ls : g.n2 * g.h0);
  const int g0 = o * g.n1 * g.h0 + col;
  const T* __restrict__ symarr = reinterpret_cast<const T*>(P.symarr);
  auto kperp2 = [&]() -> T {   // |k~|^2 of the other axes, for the multipliers that need it
    if (axis == 2) {
      const int kyi = col / g.h0;
      const T kx = wide_kfac<T>(g, 0) * (T)freq_tilde(col - kyi * g.h0, g.n0);
      const T ky = wide_kfac<T>(g, 1) * (T)freq_tilde(kyi, g.n1);
      return kx * kx + ky * ky;
    }
    const T kx = wide_kfac<T>(g, 0) * (T)freq_tilde(col, g.n0);
    T k2 = kx * kx;
    if (g.ndim == 3) {
      const T kz = wide_kfac<T>(g, 2) * (T)freq_tilde(o, g.n2);
      k2 += kz * kz;
    }
    return k2;
  };
  pdl_wait();
  if (P.done && *P.done) return;
  __syncthreads();   // the tables are complete

  // (blocks of one y index take every gridDim.y-th transform: independent ones only, see split_axis)
  for (int t = blockIdx.y; t < P.nxf; t += gridDim.y) {
    const Xf xf = P.xf[t];
    const cpx<T>* src = reinterpret_cast<const cpx<T>*>(P.in[xf.src]);
    cpx<T>* dst = reinterpret_cast<cpx<T>*>(P.out[xf.dst]);
    const T scale = (T)((sizeof(T) == 4) ? xf.scale_hi : xf.scale);
    const bool unit = scale == T(1);
    const T kp2 = ((xf.pre | xf.post) & MUL_NEGK2) ? kperp2() : T(0);
    auto mult = [&](int flags, int i, T base) -> T {
      const T ka = katab[i];
      T c = base;
      if (flags & MUL_IK) c *= ka;
      if (flags & MUL_IK2) c *= -ka * ka;
      if (flags & MUL_SYM) c *= symarr[g0 + i * ls];
      if (flags & MUL_NEGK2) c *= -(ka * ka + kp2);
      return c;
    };
    // an even number of stages ends reading A, which the next transform's first stage writes
    if (t >= (int)gridDim.y && !(nst & 1)) __syncthreads();
    auto first_stage = [&](auto rc) {
      constexpr int R = decltype(rc)::value;
      const int nb = n / R;
      for (int i = ib; i < nb; i += tpl) {
        cpx<T> u[R];
#pragma unroll
        for (int r = 0; r < R; ++r) u[r] = ok ? src[g0 + (i + r * nb) * ls] : mk<T>(T(0), T(0));
        if (xf.pre == MUL_IK) {
#pragma unroll
          for (int r = 0; r < R; ++r) u[r] = mul_ik(u[r], katab[i + r * nb]);
        } else if (xf.pre && ok) {
#pragma unroll
          for (int r = 0; r < R; ++r) {
            u[r] = scal(u[r], mult(xf.pre, i + r * nb, T(1)));
            if (xf.pre & MUL_IK) u[r] = mul_i(u[r]);
          }
        }
        dft_wide<T, S, R>(u);
#pragma unroll
        for (int r = 0; r < R; ++r) A[at(i * R + r) + w] = u[r];
      }
    };
    auto mid_stage = [&](auto rc, const cpx<T>* a, cpx<T>* b, int p) {
      constexpr int R = decltype(rc)::value;
      const int nb = n / R, tws = nb / p;
      const int mask = (p & (p - 1)) ? -1 : p - 1;
      for (int i = ib; i < nb; i += tpl) {
        const int k = mask >= 0 ? (i & mask) : i % p;
        cpx<T> u[R];
#pragma unroll
        for (int r = 0; r < R; ++r) u[r] = a[at(i + r * nb) + w];
#pragma unroll
        for (int r = 1; r < R; ++r) u[r] = twiddled<T, S>(u[r], tw[r * k * tws]);
        dft_wide<T, S, R>(u);
        const int j = (i - k) * R + k;
#pragma unroll
        for (int r = 0; r < R; ++r) b[at(j + r * p) + w] = u[r];
      }
    };
    // p = n / R = nb: k = i, rows i + r nb, twiddle index r i
    auto last_stage = [&](auto rc, const cpx<T>* a) {
      constexpr int R = decltype(rc)::value;
      const int nb = n / R;
      for (int i = ib; i < nb; i += tpl) {
        cpx<T> u[R];
        if (a) {
#pragma unroll
          for (int r = 0; r < R; ++r) u[r] = a[at(i + r * nb) + w];
#pragma unroll
          for (int r = 1; r < R; ++r) u[r] = twiddled<T, S>(u[r], tw[r * i]);
        } else {   // the only stage of the line
#pragma unroll
          for (int r = 0; r < R; ++r) {
            u[r] = ok ? src[g0 + r * ls] : mk<T>(T(0), T(0));
            if (xf.pre && ok) {
              u[r] = scal(u[r], mult(xf.pre, r, T(1)));
              if (xf.pre & MUL_IK) u[r] = mul_i(u[r]);
            }
          }
        }
        dft_wide<T, S, R>(u);
        if (!ok) continue;
        // the multiplier of the output, the common cases (none, i k~, with a unit scale) in code of
        // their own, then the stores; partial sums (written by this thread) are read in batches ahead of them
        if (xf.post == MUL_IK && unit) {
#pragma unroll
          for (int r = 0; r < R; ++r) u[r] = mul_ik(u[r], katab[i + r * nb]);
        } else if (xf.post) {
#pragma unroll
          for (int r = 0; r < R; ++r) {
            u[r] = scal(u[r], mult(xf.post, i + r * nb, scale));
            if (xf.post & MUL_IK) u[r] = mul_i(u[r]);
          }
        } else if (!unit) {
#pragma unroll
          for (int r = 0; r < R; ++r) u[r] = scal(u[r], scale);
        }
        cpx<T>* q = dst + g0 + i * ls;
        const int qs = nb * ls;
        if (xf.first) {
#pragma unroll
          for (int r = 0; r < R; ++r) q[r * qs] = u[r];
        } else {
          constexpr int PB = R < 4 ? R : 4;
#pragma unroll
          for (int r0 = 0; r0 < R; r0 += PB) {
            cpx<T> prev[PB];
#pragma unroll
            for (int b = 0; b < PB; ++b)
              if (r0 + b < R) prev[b] = q[(r0 + b) * qs];
#pragma unroll
            for (int b = 0; b < PB; ++b)
              if (r0 + b < R) q[(r0 + b) * qs] = prev[b] + u[r0 + b];
          }
        }
      }
    };
    const cpx<T>* cur = nullptr;
    if (nst > 1) {
#define VD_CALL(R) first_stage(std::integral_constant<int, R>{})
      VD_WIDE_RADIX(pl.rad[0], VD_CALL)
#undef VD_CALL
      cur = A;
      int p = pl.rad[0];
      for (int s = 1; s + 1 < nst; ++s) {
        __syncthreads();
        cpx<T>* nxt = (cur == A) ? B : A;
#define VD_CALL(R) mid_stage(std::integral_constant<int, R>{}, cur, nxt, p)
        VD_WIDE_RADIX(pl.rad[s], VD_CALL)
#undef VD_CALL
        cur = nxt;
        p *= pl.rad[s];
      }
      __syncthreads();
    }
#define VD_CALL(R) last_stage(std::integral_constant<int, R>{}, cur)
    VD_WIDE_RADIX(pl.rad[nst - 1], VD_CALL)
#undef VD_CALL
  }
}

// ---------------------------------------------------------------------------------------
// contiguous x pass
// ---------------------------------------------------------------------------------------

// walk over the items (line l, index k < per) of a block, blockDim.x apart, without a division per
// item: item index = l per + k
struct ItemWalk {
  int l, k, per, dl, dk;
  __device__ __forceinline__ ItemWalk(int per_) : per(per_) {
    l = (int)threadIdx.x / per;
    k = (int)threadIdx.x - l * per;
    dl = (int)blockDim.x / per;
    dk = (int)blockDim.x - dl * per;
  }
  __device__ __forceinline__ void next() {
    l += dl;
    k += dk;
    if (k >= per) {
      k -= per;
      ++l;
    }
  }
};

// MODE as XProg::mode.  Block: L = 2^llpc lines.  Element j of a line lies at j + (j >> ps) of its
// buffer (line stride ls): a first stage's stores, radix apart, then fall on different banks.
template <typename T, int MODE>
__global__ void __launch_bounds__(kWideThreads, (sizeof(T) == 8 ? 2 : 3))
    k_xpass_w(const __grid_constant__ XProg P, const __grid_constant__ GridDesc g, const cpx<T>* __restrict__ twg,
              int llpc, int ps, int ls, int cls) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const WidePlan& pl = g.wx[cls];
  const int m = pl.n, nst = pl.nst, h0 = g.h0, half = m / 2 + 1, L = 1 << llpc;
  cpx<T>* tw = reinterpret_cast<cpx<T>*>(smem_raw);   // W_m^j
  cpx<T>* pk = tw + m;                                // W_{n0}^k, k <= m / 2
  cpx<T>* A = pk + half;
  cpx<T>* B = A + L * ls;
  T* kt = reinterpret_cast<T*>(B + L * ls);           // k~ along x
  const T kfx = wide_kfac<T>(g, 0);
  for (int j = threadIdx.x; j < m; j += blockDim.x) tw[j] = twg[pl.tw_off + j];
  for (int j = threadIdx.x; j < half; j += blockDim.x) pk[j] = twg[g.pk_off + j];
  for (int j = threadIdx.x; j < h0; j += blockDim.x) kt[j] = kfx * (T)freq_tilde(j, g.n0);
  const int line0 = (int)blockIdx.x << llpc;
  const int nl = min(L, g.n1 * g.n2 - line0);
  const T scale = (T)((sizeof(T) == 4) ? P.scale_hi : P.scale);
  const T* __restrict__ symarr = reinterpret_cast<const T*>(P.symarr);
  auto at = [&](int l, int j) { return l * ls + j + (j >> ps); };
  auto factor = [&](int flags, int k, int go, T base) -> T {
    T c = base;
    if (flags & MUL_IK) c *= kt[k];
    if (flags & MUL_SYM) c *= symarr[go];
    if (flags & (MUL_NEGK2 | MUL_IK2)) c *= -kt[k] * kt[k];
    return c;
  };
  const ItemWalk wh(half);
  pdl_wait();
  if (P.done && *P.done) return;

  for (int c = blockIdx.y; c < P.ncomp; c += gridDim.y) {
    __syncthreads();   // the tables are complete; the previous component's buffers are free
    cpx<T>*cur = A, *oth = B;
    if constexpr (MODE != 1) {
      // half spectrum -> length-m spectrum, the entries k and m - k of a line together:
      // Z_k = S + i C, Z_{m-k} = conj(S - i C), S = X_k + conj X_{m-k}, C = (X_k - conj X_{m-k}) conj W^k
      const cpx<T>* src = reinterpret_cast<const cpx<T>*>(P.in[c]);
      const int pre = P.pre[c];
      ItemWalk it = wh;
#pragma unroll 2
      for (; it.l < nl; it.next()) {
        const int k = it.k, go = (line0 + it.l) * h0;
        cpx<T> X = src[go + k], Y = src[go + m - k];
        if (pre == MUL_IK) {
          X = mul_ik(X, kt[k]);
          Y = mul_ik(Y, kt[m - k]);
        } else if (pre) {
          X = scal(X, factor(pre, k, go + k, T(1)));
          Y = scal(Y, factor(pre, m - k, go + m - k, T(1)));
          if (pre & MUL_IK) {
            X = mul_i(X);
            Y = mul_i(Y);
          }
        }
        Y = conjg(Y);
        const cpx<T> s = X + Y, ic = mul_i(cmulc(X - Y, pk[k]));
        A[at(it.l, k)] = s + ic;
        if (k > 0 && 2 * k != m) A[at(it.l, m - k)] = conjg(s - ic);
      }
      __syncthreads();
    }
    // one stage from src to dst, both in shared memory
    auto stage = [&](auto rc, auto sc, const cpx<T>* src, cpx<T>* dst, int p) {
      constexpr int R = decltype(rc)::value, S = decltype(sc)::value;
      const int nb = m / R, tws = nb / p;
      const int mask = (p & (p - 1)) ? -1 : p - 1;
      for (ItemWalk it(nb); it.l < nl; it.next()) {
        const int i = it.k, k = mask >= 0 ? (i & mask) : i % p;
        cpx<T> u[R];
#pragma unroll
        for (int r = 0; r < R; ++r) u[r] = src[at(it.l, i + r * nb)];
        if (p > 1) {
#pragma unroll
          for (int r = 1; r < R; ++r) u[r] = twiddled<T, S>(u[r], tw[r * k * tws]);
        }
        dft_wide<T, S, R>(u);
        const int j = (i - k) * R + k;
#pragma unroll
        for (int r = 0; r < R; ++r) dst[at(it.l, j + r * p)] = u[r];
      }
    };
    // The stage that meets physical space, radix R = the last of the plan: its elements are i + r nb.
    // MODE 0: last inverse stage, weights, first forward stage; MODE 1: first forward stage from the
    // real line; MODE 2: last inverse stage to the real line.
    auto outer_stage = [&](auto rc, const cpx<T>* src, cpx<T>* dst) {
      constexpr int R = decltype(rc)::value;
      const int nb = m / R;
      const cpx<T>* __restrict__ wf = reinterpret_cast<const cpx<T>*>(P.wfield);
      for (ItemWalk it(nb); it.l < nl; it.next()) {
        const int i = it.k, rb = (line0 + it.l) * m + i;
        cpx<T> u[R];
        if constexpr (MODE == 1) {
          const cpx<T>* in = reinterpret_cast<const cpx<T>*>(P.in[c]);
#pragma unroll
          for (int r = 0; r < R; ++r) u[r] = in[rb + r * nb];
        } else {
#pragma unroll
          for (int r = 0; r < R; ++r) u[r] = src[at(it.l, i + r * nb)];
          if (nb > 1) {
#pragma unroll
            for (int r = 1; r < R; ++r) u[r] = twiddled<T, 1>(u[r], tw[r * i]);
          }
          dft_wide<T, 1, R>(u);
        }
        if constexpr (MODE == 2) {
          cpx<T>* out = reinterpret_cast<cpx<T>*>(P.out[c]);
#pragma unroll
          for (int r = 0; r < R; ++r) out[rb + r * nb] = scal(u[r], scale);
        } else {
          if (MODE == 0 && wf) {
            bool pairs = false;
            if constexpr (sizeof(T) == 4) {
              if (P.wf_dd) {
                pairs = true;
                const float4* __restrict__ wf4 = reinterpret_cast<const float4*>(P.wfield);
#pragma unroll
                for (int r = 0; r < R; ++r) {
                  const float4 q = wf4[rb + r * nb];
                  u[r] = mk<T>(mul_pair(u[r].x, q.x, q.y), mul_pair(u[r].y, q.z, q.w));
                }
              }
            }
            if (!pairs) {
#pragma unroll
              for (int r = 0; r < R; ++r) {
                const cpx<T> q = wf[rb + r * nb];
                u[r] = mk<T>(u[r].x * q.x, u[r].y * q.y);
              }
            }
          }
          dft_wide<T, -1, R>(u);
#pragma unroll
          for (int r = 0; r < R; ++r) dst[at(it.l, i * R + r)] = u[r];
        }
      }
    };
    auto swap = [&]() {
      cpx<T>* q = cur;
      cur = oth;
      oth = q;
    };
    if constexpr (MODE != 1) {
      int p = 1;
      for (int s = 0; s + 1 < nst; ++s) {
#define VD_CALL(R) stage(std::integral_constant<int, R>{}, std::integral_constant<int, 1>{}, cur, oth, p)
        VD_WIDE_RADIX(pl.rad[s], VD_CALL)
#undef VD_CALL
        p *= pl.rad[s];
        swap();
        __syncthreads();
      }
    }
#define VD_CALL(R) outer_stage(std::integral_constant<int, R>{}, cur, oth)
    VD_WIDE_RADIX(pl.rad[nst - 1], VD_CALL)
#undef VD_CALL
    if (MODE == 2) continue;
    swap();
    int p = pl.rad[nst - 1];
    for (int s = nst - 2; s >= 0; --s) {
      __syncthreads();
#define VD_CALL(R) stage(std::integral_constant<int, R>{}, std::integral_constant<int, -1>{}, cur, oth, p)
      VD_WIDE_RADIX(pl.rad[s], VD_CALL)
#undef VD_CALL
      p *= pl.rad[s];
      swap();
    }
    __syncthreads();
    // length-m spectrum -> half spectrum: X_k = S - i C, X_{m-k} = conj(S + i C), S = Z_k + conj Z_{m-k},
    // C = (Z_k - conj Z_{m-k}) W^k
    cpx<T>* dst = reinterpret_cast<cpx<T>*>(P.out[c]);
    const int post = P.post[c];
    ItemWalk it = wh;
#pragma unroll 2
    for (; it.l < nl; it.next()) {
      const int k = it.k, go = (line0 + it.l) * h0;
      const cpx<T> Z = cur[at(it.l, k)], Y = conjg(cur[at(it.l, k == 0 ? 0 : m - k)]);
      const cpx<T> s = Z + Y, ic = mul_i(cmul(Z - Y, pk[k]));
      cpx<T> lo = s - ic, hi = conjg(s + ic);
      lo = scal(lo, factor(post, k, go + k, scale));
      if (post & MUL_IK) lo = mul_i(lo);
      dst[go + k] = lo;
      if (2 * k != m) {
        hi = scal(hi, factor(post, m - k, go + m - k, scale));
        if (post & MUL_IK) hi = mul_i(hi);
        dst[go + m - k] = hi;
      }
    }
  }
}

// ---------------------------------------------------------------------------------------
// launches
// ---------------------------------------------------------------------------------------

template <typename T, int S>
static void wide_axis_launch(const AxisProg& P, const GridDesc& g, const cpx<T>* tw, int W, int groups,
                             cudaStream_t st) {
  const int cls = wide_class(sizeof(T), (long long)g.ncplx);
  const WidePlan& pl = (P.axis == 2 ? g.wz : g.wy)[cls];
  const long long lines = (long long)g.h0 * (P.axis == 2 ? g.n1 : g.n2);
  const int l = wide_log2(W), tpl = pl.tpl[l] > 0 ? pl.tpl[l] : wide_threads(pl, W);
  const size_t smem = wide_axis_smem(pl, W, sizeof(T));
  const bool pad = W * (int)sizeof(cpx<T>) < 128;
  auto kernel = pad ? k_axis_w<T, S, true> : k_axis_w<T, S, false>;
  ensure_smem(reinterpret_cast<const void*>(kernel), smem);
  pdl_launch(kernel, dim3((unsigned)((lines + W - 1) / W), groups), W * tpl, smem, st, P, g, tw, l, tpl,
             wide_pad_shift(pl), cls);
}

template <typename T>
void wide_axis(const AxisProg& P, int dir, const GridDesc& g, const void* tw, int W, int groups, cudaStream_t st) {
  if (dir < 0) wide_axis_launch<T, -1>(P, g, reinterpret_cast<const cpx<T>*>(tw), W, groups, st);
  else wide_axis_launch<T, 1>(P, g, reinterpret_cast<const cpx<T>*>(tw), W, groups, st);
}

template <typename T, int MODE>
static void wide_xpass_launch(const XProg& P, const GridDesc& g, const cpx<T>* tw, int L, int groups,
                              cudaStream_t st) {
  const int cls = wide_class(sizeof(T), (long long)g.ncplx);
  const WidePlan& pl = g.wx[cls];
  const int ps = wide_pad_shift(pl), ls = wide_line_stride(pl);
  const size_t smem = wide_xpass_smem(pl, L, sizeof(T));
  const long long lines = (long long)g.n1 * g.n2;
  int nb = 1;
  for (int s = 0; s < pl.nst; ++s) nb = std::max(nb, pl.n / pl.rad[s]);
  const int threads = std::min(kWideThreads, (int)std::max<long long>(32, ((long long)L * nb + 31) / 32 * 32));
  ensure_smem(reinterpret_cast<const void*>(k_xpass_w<T, MODE>), smem);
  pdl_launch(k_xpass_w<T, MODE>, dim3((unsigned)((lines + L - 1) / L), groups), threads, smem, st, P, g, tw, wide_log2(L), ps, ls, cls);
}

template <typename T>
void wide_xpass(const XProg& P, const GridDesc& g, const void* tw, int L, int groups, cudaStream_t st) {
  const cpx<T>* twp = reinterpret_cast<const cpx<T>*>(tw);
  if (P.mode == 0) wide_xpass_launch<T, 0>(P, g, twp, L, groups, st);
  else if (P.mode == 1) wide_xpass_launch<T, 1>(P, g, twp, L, groups, st);
  else wide_xpass_launch<T, 2>(P, g, twp, L, groups, st);
}

}  // namespace vd
