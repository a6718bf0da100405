// Batched DFT of lines of any length (the transforms of eqs. step1FFTfcoeff /
// step3IFFTz3coeff where the length is not a power of two): Stockham auto-sort
// passes with the butterflies of a pass in registers.
//
// A length is split into radices 2 .. 10 (register DFTs: 6 and 10 by Good's
// prime-factor maps, odd primes with the products halved by pairing inputs r
// and R - r) with as few passes as possible, since a pass costs an exchange
// through shared memory; primes 11 .. 61 are passes of their own, whose outputs
// are shared out over the threads (a thread per butterfly would leave most of
// a CTA idle on the short lines they occur in).  The
// first pass reads global memory, the last one writes it.  Lengths with a
// prime above 64 use Bluestein's chirp-z transform on a convolution length m
// that is the cheapest 7-smooth number in [2n - 1, 2^k], not always 2^k;
// the second of its transforms runs the first one's radices backwards, so the
// last pass of the one, the product with the chirp's spectrum and the first
// pass of the other stay in registers.
//
// The inverse transform is conj(DFT(conj x)), so only forward butterflies
// exist.  Bound: complex64 lines by HBM for smooth lengths (up to 10 points in
// flight per thread), by FP32 issue and shared memory for Bluestein;
// complex128 by the FP64 pipe, which is why the twiddles are table loads and
// the odd radices are paired.
#pragma once

#include <algorithm>
#include <cmath>

#include "helm_dft_mix.h"
#include "helm_dft_radix.cuh"

namespace helm {

constexpr int kPairGroup = 3;     // output pairs of a prime pass per thread
constexpr int kAccumBatch = 4;    // old values read ahead by the accumulating stores

// b / d by the multiplier floor(2^32 / d) + 1 (exact for b d < 2^32; 0: d = 1)
__device__ __forceinline__ int fast_div(int b, uint32_t mul) { return mul ? (int)__umulhi((uint32_t)b, mul) : b; }

// v, not known to be the same in the next loop iteration: keeps the multiples
// of a pass's strides from being formed ahead of its loop, where one per point
// and radix would be spilled
__device__ __forceinline__ int fresh(int v) {
  asm volatile("" : "+r"(v));
  return v;
}

template <typename C>
__device__ __forceinline__ C conj_if(C v, bool c) {
  if (c) v.y = -v.y;
  return v;
}

// Results lo <= q < hi of R to p + g0 + off + q * doff; the accumulating modes
// read kAccumBatch old values before they use one (more would spill).
template <typename C, int R>
__device__ __forceinline__ void store_many(void* p, int mode, int64_t g0, int off, int doff, const C (&v)[R], int lo,
                                           int hi, double accum_scale) {
  if (mode == kOutC64) {
    float2* o = reinterpret_cast<float2*>(p) + g0;
#pragma unroll
    for (int q = 0; q < R; ++q) {
      if (q >= hi) break;
      if (q >= lo) o[off + q * doff] = make_float2((float)v[q].x, (float)v[q].y);
    }
  } else if (mode == kOutC128) {
    double2* o = reinterpret_cast<double2*>(p) + g0;
#pragma unroll
    for (int q = 0; q < R; ++q) {
      if (q >= hi) break;
      if (q >= lo) o[off + q * doff] = make_double2(widen(v[q].x), widen(v[q].y));
    }
  } else if (mode == kOutAccumC128) {
    double2* o = reinterpret_cast<double2*>(p) + g0;
#pragma unroll
    for (int q0 = 0; q0 < R; q0 += kAccumBatch) {
      if (q0 >= hi) break;
      double2 u[kAccumBatch];
#pragma unroll
      for (int i = 0; i < kAccumBatch; ++i)
        if (q0 + i < R && q0 + i >= lo && q0 + i < hi) u[i] = o[off + (q0 + i) * doff];
#pragma unroll
      for (int i = 0; i < kAccumBatch; ++i)
        if (q0 + i < R && q0 + i >= lo && q0 + i < hi)
          o[off + (q0 + i) * doff] = make_double2(u[i].x + accum_scale * widen(v[(q0 + i) % R].x),
                                                  u[i].y + accum_scale * widen(v[(q0 + i) % R].y));
    }
  } else if (mode == kOutFF) {
    float4* o = reinterpret_cast<float4*>(p) + g0;
#pragma unroll
    for (int q = 0; q < R; ++q) {
      if (q >= hi) break;
      if (q >= lo) o[off + q * doff] = make_float4((float)v[q].x, (float)v[q].y, 0.f, 0.f);
    }
  } else {
    float4* o = reinterpret_cast<float4*>(p) + g0;
#pragma unroll
    for (int q0 = 0; q0 < R; q0 += kAccumBatch) {
      if (q0 >= hi) break;
      float4 u[kAccumBatch];
#pragma unroll
      for (int i = 0; i < kAccumBatch; ++i)
        if (q0 + i < R && q0 + i >= lo && q0 + i < hi) u[i] = o[off + (q0 + i) * doff];
#pragma unroll
      for (int i = 0; i < kAccumBatch; ++i)
        if (q0 + i < R && q0 + i >= lo && q0 + i < hi) {
          ff_add_f(u[i].x, u[i].z, (float)accum_scale * (float)v[(q0 + i) % R].x);
          ff_add_f(u[i].y, u[i].w, (float)accum_scale * (float)v[(q0 + i) % R].y);
          o[off + (q0 + i) * doff] = u[i];
        }
    }
  }
}

// What the passes of one CTA share.  Lines: ROWS, `lines` lines of m.n points
// [line][padded point] (a padding point per 128 bytes keeps the strided writes
// of a pass off each other's banks); columns, 2^lt neighbouring columns
// [point][column], the lanes of a warp on consecutive columns.  TIGHT: rows
// without padding, see run_mix.
template <typename T, bool COLS, bool BS, bool TIGHT>
struct Ctx {
  using C = typename cpx<T>::type;
  static constexpr int kPad = TIGHT ? 31 : sizeof(T) == 4 ? 4 : 3;
  // points from one line to the next
  static __host__ __device__ constexpr int pitch_of(int n) { return TIGHT ? n : n + (n >> kPad) + 1; }
  const void* in;
  void* out;
  int kind;      // of `in` (kIn*)
  int out_mode;
  int len;       // points of a line in memory (m.n without Bluestein)
  int lines;     // lines or columns of this CTA
  int lt;        // log2 of the column slots (COLS)
  int pitch;     // shared-memory points per line (rows)
  int64_t g0;    // first point of the CTA's first line
  int inner;     // distance of a line's points (COLS)
  bool cj;       // inverse: conjugate on the way in and out
  T scale;
  double accum_scale;
  const C *sc_in, *sc_out, *tw, *bw, *bf;
  C *buf0, *buf1;

  __device__ __forceinline__ C* buf(int s) const { return s & 1 ? buf1 : buf0; }  // pass s writes it

  __device__ __forceinline__ int sidx(int c, int k) const {
    return COLS ? (k << lt) + c : c * pitch + k + (k >> kPad);
  }
  // point k of line c from the CTA's first point (below 2^31: one slab, or one
  // CTA's lines)
  __device__ __forceinline__ int gidx(int c, int k) const { return COLS ? k * inner + c : c * len + k; }
  // work item b of a pass with nb butterflies a line -> (line, butterfly)
  __device__ __forceinline__ void split(int b, int nb, uint32_t mnb, int& c, int& j) const {
    if (COLS) {
      c = b & ((1 << lt) - 1);
      j = b >> lt;
    } else {
      c = fast_div(b, mnb);
      j = b - c * nb;
    }
  }
  __device__ __forceinline__ int items(int nb) const { return COLS ? nb << lt : nb * lines; }
  // points k0 + r dk of line c from global memory (zero past a line's end), 8
  // (16-byte points) or all loads issued before the first value is used
  template <int R>
  __device__ __forceinline__ void gload(C (&v)[R], int c, int k0, int dk) const {
    const int off = gidx(c, k0), doff = COLS ? dk * inner : dk;
    const int top = BS ? gidx(c, len - 1) : 0;  // Bluestein: points past the end read the last one, times a zero chirp
    auto at = [&](int r) { return BS ? min(off + r * doff, top) : off + r * doff; };
    if (sizeof(T) == 8 || (!COLS && kind == kInC128)) {
      const double2* p = reinterpret_cast<const double2*>(in) + g0;
#pragma unroll
      for (int r0 = 0; r0 < R; r0 += 8) {
        double2 t[8];
#pragma unroll
        for (int i = 0; i < 8; ++i)
          if (r0 + i < R) t[i] = p[at(r0 + i)];
#pragma unroll
        for (int i = 0; i < 8; ++i)
          if (r0 + i < R) v[(r0 + i) % R] = cvt<C>(t[i]);
      }
    } else {
      // a float-float point's hi part is the first half of its float4
      const int w = !COLS && kind == kInFF ? 1 : 0;
      const float2* p = reinterpret_cast<const float2*>(in) + (g0 << w);
#pragma unroll
      for (int r = 0; r < R; ++r) v[r] = cvt<C>(p[(uint32_t)at(r) << w]);
    }
    if (sc_in) {
#pragma unroll
      for (int r = 0; r < R; ++r) v[r] = cmul(v[r], __ldg(&sc_in[BS ? min(k0 + r * dk, len - 1) : k0 + r * dk]));
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
      v[r] = conj_if(v[r], cj);
      if (BS) v[r] = cmulc(v[r], __ldg(&bw[k0 + r * dk]));
    }
  }
  // v_r *= e^{-2 pi i r k / (ns R)}: complex64 from the pass's own table
  // [k][R] (one address, two twiddles a load for even R), complex128 from the
  // length's table of roots
  template <int R>
  __device__ __forceinline__ void twiddle(C (&v)[R], const MixStage& st, int k) const {
    if constexpr (sizeof(T) == 4) {
      const C* t = tw + st.toff + k * R;
      if constexpr (R % 2 == 0) {
#pragma unroll
        for (int r = 0; r < R; r += 2) {
          const float4 w = __ldg(reinterpret_cast<const float4*>(t + r));
          if (r) v[r] = cmul(v[r], mk<C>(w.x, w.y));
          v[r + 1] = cmul(v[r + 1], mk<C>(w.z, w.w));
        }
      } else {
#pragma unroll
        for (int r = 1; r < R; ++r) v[r] = cmul(v[r], __ldg(t + r));
      }
    } else {
      int e = 0;
#pragma unroll
      for (int r = 1; r < R; ++r) {
        e += k * st.st;
        v[r] = cmul(v[r], __ldg(&tw[e]));
      }
    }
  }
  // the same for one r of a prime pass
  __device__ __forceinline__ C twiddle_one(const MixStage& st, int k, int r) const {
    return __ldg(&tw[sizeof(T) == 4 ? st.toff + k * st.r + r : r * k * st.st]);
  }
  // results q (lo <= q < hi) to points k0 + q dk of line c
  template <int R>
  __device__ __forceinline__ void gstore(C (&v)[R], int c, int k0, int dk, int lo, int hi) const {
    if (BS) hi = k0 < len ? min(hi, (len - k0 + dk - 1) / dk) : 0;
#pragma unroll
    for (int q = 0; q < R; ++q) {
      // Bluestein: the second transform was run on conjugated data
      if (BS) v[q] = cmulc(conj_if(v[q], true), __ldg(&bw[min(k0 + q * dk, len - 1)]));
      v[q] = cscale(conj_if(v[q], cj), scale);
    }
    if (sc_out) {
#pragma unroll
      for (int q = 0; q < R; ++q) {
        if (q >= hi) break;
        if (q >= lo) v[q] = cmul(v[q], __ldg(&sc_out[k0 + q * dk]));
      }
    }
    store_many<C, R>(out, out_mode, g0, gidx(c, k0), COLS ? dk * inner : dk, v, lo, hi, accum_scale);
  }
};

// One pass of radix R <= 10: thread per butterfly.
template <int R, typename T, bool COLS, bool BS, bool TIGHT>
__device__ __forceinline__ void pass_reg(const Ctx<T, COLS, BS, TIGHT>& x, const MixStage& st, int s, bool last, bool mid) {
  using C = typename cpx<T>::type;
  const int total = x.items(st.nb);
  const C* src = x.buf(s + 1);
  C* dst = x.buf(s);
  for (int b = threadIdx.x; b < total; b += blockDim.x) {
    int c, j;
    x.split(b, st.nb, st.mnb, c, j);
    if (COLS && c >= x.lines) continue;
    C v[R];
    const int nb = fresh(st.nb);
    if (s == 0) {
      x.template gload<R>(v, c, j, nb);
    } else {
#pragma unroll
      for (int r = 0; r < R; ++r) v[r] = src[x.sidx(c, j + r * nb)];
    }
    const int k = j - fast_div(j, st.mns) * st.ns;
    if (st.ns > 1) x.template twiddle<R>(v, st, k);
    int base = (j - k) * R + k, step = fresh(st.ns);
#pragma unroll 1
    for (bool more = BS && mid;; more = false) {
      dft_fwd<C, R>(v);
      if (!more) break;
      // times the chirp's spectrum, conjugated, then the first pass of the
      // second transform, whose inputs are this thread's outputs
#pragma unroll
      for (int q = 0; q < R; ++q) v[q] = conj_if(cmul(v[q], __ldg(&x.bf[base + q * step])), true);
      base = j * R;
      step = fresh(1);
    }
    if (!BS && last) {
      x.template gstore<R>(v, c, base, step, 0, R);
    } else {
#pragma unroll
      for (int q = 0; q < R; ++q) dst[x.sidx(c, base + q * step)] = v[q];
    }
  }
}

// Bluestein: the convolution's first len points (in buf) to global memory.
// The last pass does not store them itself: with the lines ending inside its
// butterflies, their bounds cost more registers than this exchange's time.
template <typename T, bool COLS, bool BS, bool TIGHT>
__device__ __forceinline__ void copy_out(const Ctx<T, COLS, BS, TIGHT>& x, const typename cpx<T>::type* buf) {
  using C = typename cpx<T>::type;
  const int dk = COLS ? (int)blockDim.x >> x.lt : (int)blockDim.x;  // 2^lt divides the thread count
  for (int c0 = 0; c0 < (COLS ? 1 : x.lines); ++c0) {
    const int c = COLS ? (int)threadIdx.x & ((1 << x.lt) - 1) : c0;
    if (COLS && c >= x.lines) return;
    for (int k0 = COLS ? (int)threadIdx.x >> x.lt : (int)threadIdx.x; k0 < x.len; k0 += kAccumBatch * dk) {
      C v[kAccumBatch];
#pragma unroll
      for (int i = 0; i < kAccumBatch; ++i) v[i] = buf[x.sidx(c, min(k0 + i * dk, x.len - 1))];
      x.template gstore<kAccumBatch>(v, c, k0, dk, 0, kAccumBatch);
    }
  }
}

// One pass of a prime radix R in 11 .. 61.  First the inputs' pair sums and
// differences s_r = v_r + v_{R-r}, d_r = v_r - v_{R-r} (twiddled) replace
// them in shared memory; then every thread forms kPairGroup output pairs
// y_q, y_{R-q} = a -+ i b of one butterfly (see dft_odd; q = 0 is y_0).
template <typename T, bool COLS, bool BS, bool TIGHT>
__device__ void pass_prime(const Ctx<T, COLS, BS, TIGHT>& x, const MixStage& st, int s, bool last,
                           typename cpx<T>::type* root) {
  using C = typename cpx<T>::type;
  const int R = st.r, H = (R - 1) / 2, nb = st.nb;
  C* src = x.buf(s + 1);
  C* dst = x.buf(s);
  const auto root_in = [&](int e) -> int { return sizeof(T) == 4 ? st.roff + e : e * (x.len / R); };  // e^{-2 pi i e / R} in tw
  if (!TIGHT)
    for (int e = threadIdx.x; e < R; e += blockDim.x) root[e] = x.tw[root_in(e)];
  const int per = x.items(nb);  // items of one value of r
  for (int b = threadIdx.x; b < per * (H + 1); b += blockDim.x) {
    const int r = b / per;
    int c, j;
    x.split(b - r * per, nb, st.mnb, c, j);
    if (COLS && c >= x.lines) continue;
    const int ka = j + r * nb, kb = j + (R - r) * nb;
    if (r == 0) {
      if (s == 0) {
        C v[1];
        x.template gload<1>(v, c, ka, 0);
        src[x.sidx(c, ka)] = v[0];
      }
      continue;
    }
    C v[2];
    if (s == 0) {
      x.template gload<2>(v, c, ka, kb - ka);
    } else {
      v[0] = src[x.sidx(c, ka)];
      v[1] = src[x.sidx(c, kb)];
      const int k = j - fast_div(j, st.mns) * st.ns;
      if (st.ns > 1) {
        v[0] = cmul(v[0], x.twiddle_one(st, k, r));
        v[1] = cmul(v[1], x.twiddle_one(st, k, R - r));
      }
    }
    src[x.sidx(c, ka)] = cadd(v[0], v[1]);
    src[x.sidx(c, kb)] = csub(v[0], v[1]);
  }
  __syncthreads();
  const int groups = (H + kPairGroup) / kPairGroup;  // H + 1 pairs (q = 0 .. H)
  for (int b = threadIdx.x; b < per * groups; b += blockDim.x) {
    const int gq = b / per;
    int c, j;
    x.split(b - gq * per, nb, st.mnb, c, j);
    if (COLS && c >= x.lines) continue;
    const C v0 = src[x.sidx(c, j)];
    C a[kPairGroup], bb[kPairGroup];
    int e[kPairGroup], q[kPairGroup];
#pragma unroll
    for (int g = 0; g < kPairGroup; ++g) {
      a[g] = v0;
      bb[g] = mk<C>(0, 0);
      e[g] = 0;
      q[g] = gq * kPairGroup + g;
    }
    for (int r = 1; r <= H; ++r) {
      const C sv = src[x.sidx(c, j + r * nb)], dv = src[x.sidx(c, j + (R - r) * nb)];
#pragma unroll
      for (int g = 0; g < kPairGroup; ++g) {
        e[g] += q[g];
        if (e[g] >= R) e[g] -= R;
        const C w = TIGHT ? __ldg(&x.tw[root_in(e[g])]) : root[e[g]];  // (cos, -sin); pairs past H read in range and are not stored
        a[g].x = fma(w.x, sv.x, a[g].x);
        a[g].y = fma(w.x, sv.y, a[g].y);
        bb[g].x = fma(w.y, dv.x, bb[g].x);
        bb[g].y = fma(w.y, dv.y, bb[g].y);
      }
    }
    const int k = j - fast_div(j, st.mns) * st.ns;
    const int base = (j - k) * R + k;
    C y[kPairGroup], z[kPairGroup];  // y_q and y_{R-q}
#pragma unroll
    for (int g = 0; g < kPairGroup; ++g) {
      // bb = -sum sin d: y_q = a + i bb, y_{R-q} = a - i bb
      y[g].x = a[g].x - bb[g].y;
      y[g].y = a[g].y + bb[g].x;
      z[g].x = a[g].x + bb[g].y;
      z[g].y = a[g].y - bb[g].x;
    }
    const int ky = base + q[0] * st.ns, kz = base + (R - q[0]) * st.ns;
    const int lo = q[0] == 0 ? 1 : 0, hi = min(kPairGroup, H + 1 - q[0]);
    if (last) {
      x.template gstore<kPairGroup>(y, c, ky, st.ns, 0, hi);
      x.template gstore<kPairGroup>(z, c, kz, -st.ns, lo, hi);
    } else {
#pragma unroll
      for (int g = 0; g < kPairGroup; ++g) {
        if (g < hi) dst[x.sidx(c, ky + g * st.ns)] = y[g];
        if (g >= lo && g < hi) dst[x.sidx(c, kz - g * st.ns)] = z[g];
      }
    }
  }
}

// Registers: radices up to 10 fit 80 in complex64 and 128 in complex128.
// Radices up to 16 (fewer passes) need 128 in complex64 too and were slower:
// 223 x 127 planes (Bluestein, 448 and 256 points) 109 / 134 us against 100 /
// 109, 1021-point lines 31.6 against 28.0, 300- and 150-point lines equal.
template <typename T>
constexpr int mix_min_ctas() {
  return sizeof(T) == 4 ? 3 : 2;
}

// ROWS: CTA = L consecutive lines.  COLS: CTA = 2^lt neighbouring columns of
// one slab of [outer][len][inner].
template <typename T, bool COLS, bool BS, bool TIGHT>
__global__ void __launch_bounds__(kMixThreads, mix_min_ctas<T>())
    k_dft_mix(const void* in, int kind, void* out, int out_mode, int64_t nlines, int inner, int L, int lt, int len, MixArgs a,
              int inverse, T scale, double accum_scale, const typename cpx<T>::type* __restrict__ sc_in,
              const typename cpx<T>::type* __restrict__ sc_out, const int* __restrict__ skip) {
  using C = typename cpx<T>::type;
  if (skip && *skip) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* root = nullptr;
  if constexpr (!TIGHT && !BS) {
    __shared__ C roots[kMixRoots];
    root = roots;
  }
  Ctx<T, COLS, BS, TIGHT> x;
  x.in = in;
  x.out = out;
  x.kind = kind;
  x.out_mode = out_mode;
  x.len = len;
  x.lt = lt;
  x.inner = inner;
  x.pitch = x.pitch_of(a.m.n);
  if (COLS) {
    const int tiles = (inner + (1 << lt) - 1) >> lt;
    const int slab = blockIdx.x / tiles, c0 = (blockIdx.x - slab * tiles) << lt;
    x.lines = min(1 << lt, inner - c0);
    x.g0 = (int64_t)slab * len * inner + c0;
  } else {
    const int64_t row0 = (int64_t)blockIdx.x * L;
    x.lines = (int)min((int64_t)L, nlines - row0);
    x.g0 = row0 * len;
  }
  x.cj = inverse != 0;
  x.scale = scale;
  x.accum_scale = accum_scale;
  x.sc_in = sc_in;
  x.sc_out = sc_out;
  x.tw = reinterpret_cast<const C*>(a.tw);
  x.bw = reinterpret_cast<const C*>(a.bw);
  x.bf = reinterpret_cast<const C*>(a.bf);
  x.buf0 = reinterpret_cast<C*>(smem_raw);
  x.buf1 = x.buf0 + (COLS ? (a.m.n << lt) : x.pitch * L);
  for (int s = 0; s < a.m.nstages; ++s) {
    const MixStage& st = a.m.s[s];
    const bool last = s == a.m.nstages - 1, mid = BS && s == a.m.mid;
    if (s) __syncthreads();  // the previous pass's outputs are in buf(s + 1)
    switch (st.r) {
#define HELM_PASS(R) \
  case R: pass_reg<R>(x, st, s, last, mid); break;
      HELM_PASS(2)
      HELM_PASS(3)
      HELM_PASS(4)
      HELM_PASS(5)
      HELM_PASS(6)
      HELM_PASS(7)
      HELM_PASS(8)
      HELM_PASS(9)
      HELM_PASS(10)
#undef HELM_PASS
      default:
        if constexpr (!BS) pass_prime(x, st, s, last, root);
    }
  }
  if constexpr (BS) {
    __syncthreads();
    copy_out(x, x.buf(a.m.nstages + 1));
  }
}

template <typename T, bool COLS, bool BS>
cudaError_t run_mix(const MixArgs& a, int len, const void* in, int kind, void* out, int out_mode, int64_t nlines,
                    int64_t outer, int64_t inner, int sign, double scale, double accum_scale, const void* sc_in,
                    const void* sc_out, const int* skip, cudaStream_t st) {
  using C = typename cpx<T>::type;
  const MixShape h = mix_shape(a.m, COLS, sizeof(C), nlines, outer, inner);
  const int64_t grid = COLS ? outer * ((inner + (int64_t(1) << h.lt) - 1) >> h.lt) : (nlines + h.L - 1) / h.L;
  if (grid == 0) return cudaSuccess;
  auto go = [&](auto kern, size_t line) -> cudaError_t {
    const size_t smem = line * h.L * h.nbuf * sizeof(C);
    if (smem > 40 * 1024) {
      const cudaError_t e = allow_dynamic_smem((const void*)kern, smem);
      if (e != cudaSuccess) return e;
    }
    kern<<<(unsigned)grid, h.threads, smem, st>>>(in, kind, out, out_mode, nlines, (int)inner, h.L, h.lt, len, a,
                                                  sign > 0 ? 1 : 0, (T)scale, accum_scale, (const C*)sc_in,
                                                  (const C*)sc_out, skip);
    return cudaGetLastError();
  };
  if (COLS) return go(k_dft_mix<T, COLS, BS, false>, a.m.n);  // L = 2^lt columns
  const size_t padded = Ctx<T, COLS, BS, false>::pitch_of(a.m.n);
  // The longest rows (6428 .. 7264 points in complex128, 13643 .. 14528 in
  // complex64, one line a CTA) leave no room for padding or roots: these are
  // read from global memory.
  if constexpr (!COLS && !BS)
    if ((padded * h.L * h.nbuf + kMixRoots) * sizeof(C) > kMixSmem)
      return go(k_dft_mix<T, COLS, BS, true>, Ctx<T, COLS, BS, true>::pitch_of(a.m.n));
  return go(k_dft_mix<T, COLS, BS, false>, padded);
}

}  // namespace helm
