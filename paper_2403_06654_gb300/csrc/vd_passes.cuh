// Transform passes of the spectral operators (host-side declarations).
//
// A 3D operator apply in spectral space is a chain of passes, each reading and writing
// half-spectrum fields in HBM once:
//   z pass (lines along z) -> y pass (lines along y) -> fused x pass (inverse real
//   transform, pointwise physical-space work, forward real transform) -> y pass -> z pass.
// 2D chains drop the z passes and 1D chains are a single fused x pass.  Multipliers that
// are diagonal in Fourier space (derivatives i k~_j, -|k~|^2, preconditioner symbols)
// are applied while a pass loads or stores, so they cost no extra memory traffic.
#pragma once

#include "vd_common.cuh"

namespace vd {

// pre/post multiplier flags (combinable)
enum MulFlags : int {
  MUL_IK = 1,      // i k~ of the pass axis
  MUL_SYM = 2,     // the program's diagonal symbol (needs every axis in spectral space)
  MUL_NEGK2 = 4,   // -|k~|^2 (needs every axis in spectral space)
  MUL_IK2 = 8,     // (i k~)^2 = -k~^2 of the pass axis
};

constexpr int kMaxXf = 16;
constexpr int kMaxIO = 16;

// One transform of an axis pass: out[dst] (=|+=) scale * post( FFT( pre( in[src] ) ) ).
// Every transform writes out[dst] (an accumulating one adds to what an earlier transform of
// the same program wrote there), so a program must not read a buffer after one of its
// transforms has overwritten it; `last` is informative only.
// MUL_SYM reads the program's symbol array at the element's spectral index, so it is only
// meaningful where every axis is in spectral space (first inverse / last forward pass).
struct Xf {
  int8_t src, dst, pre, post;
  int8_t first;   // start a new accumulation for dst
  int8_t last;    // write dst after this transform
  double scale;
  float scale_hi, scale_lo;   // float-pair split of scale (set on the host)
};

struct AxisProg {
  int nxf;
  Xf xf[kMaxXf];
  const void* in[kMaxIO];
  void* out[kMaxIO];
  const void* symarr;   // real symbol array (ncplx, same layout as the spectral fields)
  const int* done;      // if non-null and *done != 0 the kernel returns at once
  int axis;   // 1 = y, 2 = z
  int conv_in;          // float-pair kernels: bit i set -> in[i] holds doubles (split on load)
  int conv_out;         // float-pair kernels: bit i set -> out[i] holds doubles (summed on store)
};

// Fused x pass: for every component c, in[c] (half spectrum) -> pre -> inverse real FFT ->
// multiply by wfield (real, n0 per line; nullptr = 1) -> forward real FFT -> post -> out[c].
// mode 0: fused as described; mode 1: real in (in[c] is T*), forward only; mode 2: inverse
// only, real out (out[c] is T*).  scale multiplies the result.
constexpr int kMaxXComp = 6;

struct XProg {
  int ncomp;   // <= kMaxXComp
  int mode;
  const void* in[kMaxXComp];
  void* out[kMaxXComp];
  int pre[kMaxXComp];
  int post[kMaxXComp];
  const void* wfield;
  // float programs only: wfield holds a float pair (hi, lo) per real point, and the multiply
  // z * (hi + lo) is carried in float-pair arithmetic, rounded to float once
  int wf_dd;
  double scale;
  float scale_hi, scale_lo;   // float-pair split of scale (set by launch_xpass)
  const void* symarr;
  const int* done;
  int conv_in;          // float-pair kernels: bit c set -> in[c] holds doubles
  int conv_out;         // float-pair kernels: bit c set -> out[c] holds doubles
  // mode 0 only: if aux_out is set, component 0 is also transformed inverse-only (no pre
  // multiplier, as mode 2) into the real field aux_out, scaled by aux_scale (doubles when
  // aux_conv is set); that output equals a separate mode-2 pass over in[0] bit for bit
  void* aux_out;
  double aux_scale;
  float aux_scale_hi, aux_scale_lo;
  int aux_conv;
};

template <typename T>
void launch_axis(const AxisProg& P, int dir, const GridDesc& g, const void* tw, cudaStream_t st);

template <typename T>
void launch_xpass(const XProg& P, const GridDesc& g, const void* tw, cudaStream_t st);

// launch-shape table (vd_passes.cu).  kind 0: y/z pass (key: type, length, axis, direction);
// kind 1: x pass (key: type, n0/2, axis 0, mode).  type: 0 double, 1 float, 2 float-pair.
// choice: 0 register four-step kernel, > 0 lines per block, < 0 (get) absent / (set) erase.
// Entries set by hand (tune_set) hold for every field; the tuner's (tune_put) for fields of the tuned one's
// scope: the same radix class and a line count within the same power of two.  The bytes of a shape
// depend on the class and the better shape on the line count: the 16-line blocks and register kernels
// that win on 256^3 leave most SMs idle on a 256^2 field.  A scoped entry goes before one set by hand.
// kind 0 choice kChoiceStaged: the register kernel with TMA-staged input (float y/z passes of
// length 128 / 256).  Type 2 choice kChoiceUnpacked (either kind): the Stockham engine on
// unpacked float pairs with the default lines per block, instead of the packed engine that the
// float-pair passes use for lengths whose radices are 2, 4 and 8 (same results, bit for bit).
constexpr int kChoiceStaged = 128;
constexpr int kChoiceUnpacked = 256;
int tune_get(int kind, int type, int n, int axis, int dir, int scope);
void tune_set(int kind, int type, int n, int axis, int dir, int choice);   // replaces the scoped ones too
// builtin: the built-in shape is the best of this scope (choice: which one that was, for the listing)
void tune_put(int kind, int type, int n, int axis, int dir, int scope, int choice, bool builtin);
inline int tune_scope(int cls, long long lines) {
  int l = 0;
  while ((lines >> (l + 1)) > 0) ++l;
  return 1 + 32 * cls + l;   // 0: every field
}
int tune_table(int* out, int max);   // 6 ints per entry; returns the entry count
// the built-in choice for a pass of `lines` lines in all (kind 1: n = n0/2)
int default_shape(int kind, int type, const FftPlan& pl, const WidePlan& wide, int axis, long long lines);
void tune_save();                    // write the table to $VD_TUNE_FILE (if set)

// most dynamic shared memory of a block (227 KB)
constexpr size_t kSmemMost = 227 * 1024;
// opt a kernel into more than 48 KB of dynamic shared memory (once per size)
void ensure_smem(const void* func, size_t smem);
int sm_count();

// the float and double passes of any length (vd_wide.cuh): W / L lines per block, powers of two; the
// transforms / components shared out over `groups` blocks per tile
template <typename T>
void wide_axis(const AxisProg& P, int dir, const GridDesc& g, const void* tw, int W, int groups, cudaStream_t st);
template <typename T>
void wide_xpass(const XProg& P, const GridDesc& g, const void* tw, int L, int groups, cudaStream_t st);
// the plan of length n in a radix class, its table at tw_off, without threads per line
bool make_wide_plan(int n, int tw_off, int cls, WidePlan* p);
// threads per line of a y/z pass with W lines per block
int wide_threads(const WidePlan& pl, int W);
// the threads per line of the shapes that launches of double y/z passes on g take: descriptions made
// for a single call form no others (all of a length's, 21 searches, take up to 114 us)
void wide_axis_threads(GridDesc* g);
// The radix class of a pass over a field of ncplx points.  Wide radices make fewer trips through
// shared memory, narrow ones more and shorter threads.  Double: a warp issues one FP64 instruction
// per 64 cycles however independent, four warps per SM saturate the pipe, so a small field wants
// many threads of few operations (pressure apply in radices up to 5, 8 and 16, us: 96 x 96 59, 70, 85;
// 320 x 320 103, 108, 138; 512 x 1024 281, 277, 275; 80^3 366, 335, 342; 128^3 1351, 1292, 1148).  Float:
// latency until the field is large (forward transform in radices up to 8 and 16: 512 x 1024 13.8 and
// 14.7, 128 x 120 x 128 20.6 and 16.9, 320 x 256 x 160 137 and 92).
inline int wide_class(size_t el, long long ncplx) {
  if (el == sizeof(float)) return ncplx >= (1 << 20) ? 2 : 1;
  return ncplx >= (1 << 21) ? 2 : (ncplx >= (1 << 17) ? 1 : 0);
}
inline int wide_log2(int v) {
  int l = 0;
  while ((1 << (l + 1)) <= v) ++l;
  return l;
}
// Stockham buffers pad one element in 2^shift, so that the stores of a first stage (a radix apart)
// spread over the banks: 17 elements apart for radix 16, 9 for 8
inline int wide_pad_shift(const WidePlan& pl) {
  int r = 0;
  for (int s = 0; s < pl.nst; ++s) r = r > pl.rad[s] ? r : pl.rad[s];
  return r > 10 ? 4 : 3;
}
inline int wide_line_stride(const WidePlan& pl) { return (pl.n + (pl.n >> wide_pad_shift(pl)) + 1) | 1; }
// shared memory of a block of W y/z lines or L x lines; el: bytes of a real
inline size_t wide_axis_smem(const WidePlan& pl, int W, size_t el) {
  const size_t rows = (size_t)pl.n + (size_t)(pl.n >> wide_pad_shift(pl));
  return 2 * el * ((size_t)pl.n + (pl.nst > 2 ? 2 : 1) * (size_t)W * rows) + el * (size_t)pl.n;
}
inline size_t wide_xpass_smem(const WidePlan& pl, int L, size_t el) {
  return 2 * el * ((size_t)pl.n + pl.n / 2 + 1 + 2 * (size_t)L * wide_line_stride(pl)) + el * (size_t)(pl.n + 1);
}
// dynamic shared memory a launch of `lines` lines per block takes in type code `type`
size_t shape_smem(int kind, int type, const FftPlan& pl, const WidePlan& wide, int lines);

}  // namespace vd
