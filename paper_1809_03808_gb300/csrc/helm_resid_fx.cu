// The FP64 refinement residual r = f - A u of eqs. A2D (9-point) and A3D
// (27-point) in 64-bit fixed point on the integer pipe.
//
// An FP64 instruction costs this GPU's SM the issue time of about 64 FP32 or
// integer ones, and the stencil needs 26 (3D) or 14 (2D) of them per unknown:
// in FP64 the residual of 512^3 took 8.1 ms where its 40 bytes per unknown take
// 0.8 ms.  Its sums do not need a floating exponent per value, though: inside
// a tile every term is compared with the tile's largest one.  So a tile's u
// (and f) are converted to integers with one common exponent, the neighbour
// sums become exact 64-bit integer adds, and a product with a coefficient
// three 32 x 32 -> 64-bit multiply-adds.
//
// Formats.  K is a key of the tile: |u| < 2^(K - eS - 1022) and
// |f| < 2^(K - 1022) for all values seen so far, where sum |c| over the 27 (9)
// coefficients of any point is below 2^eS.
//   u -> integer u 2^60 / 2^(K - eS - 1022): below 2^60, the monomials
//        P_bc = Sy^b Sz^c u (exact sums of 1, 2, 2, 4 values) below 2^62;
//   c -> integer c 2^(62 - eS) = ch 2^32 + cl, |cl| <= 2^31;
//   P c / 2^64 -> ph ch + (ph cl + pl ch) / 2^32 with P = ph 2^32 + pl,
//        |pl| <= 2^31; the middle sums of a monomial set stay below
//        9 2^59 + 2^61 < 2^63.  Dropped: pl cl / 2^64 < 1/4 per product;
//   f -> integer in the result's unit 2^(K - 1022 - 58).
// Values within 2^-7 of the tile's largest are converted exactly, and the
// sum's error is about one unit, 2^-58 of sum |c| max |u|: FP64 rounds to
// 2^-53 of its terms at every addition.  So a loud tile's residuals are more
// accurate than in FP64, and those of nodes below about 2^-5 of the loudest are
// less so; their errors stay under the ones that FP64 makes at the loud nodes,
// and a correction sweep spreads all of them over the grid.  K only grows along
// a tile's planes (rows in 2D); carried sums are shifted when it does.  A NaN or
// an infinity makes the rest of its tile's residuals NaN.
//
// The stencil is split as in helm_resid.cu: Q(x) = sum_bc C_0bc P_bc(x),
// R(x) = sum_bc C_1bc P_bc(x), r(x) = f(x) - Q(x) - R(x-1) - R(x+1); points on
// a face take the complex coefficients of their class, by warps that hold one.
#include <algorithm>
#include <cmath>

#include "helm_async.cuh"
#include "helm_fx.h"
#include "helm_kernels.cuh"
#include "helm_resid.h"

namespace helm {

namespace {

typedef long long ll;

struct FxArgs {
  int nx, ny, nz;
  int es;  // eS
  // the coefficients' negatives: real ones inside (class 0), then all classes
  Limb q[4], r[4];
  LimbC c0[8][4];
  LimbC c1[4][4];
};

constexpr int kBadKey = 1 << 20;  // key of a NaN or an infinity

struct cll {
  ll x, y;
};

__device__ __forceinline__ cll operator+(cll a, cll b) { return {a.x + b.x, a.y + b.y}; }

// The largest magnitude among high words of doubles, and the biased exponent
// of it (kBadKey beyond the finite ones).
__device__ __forceinline__ int mag_max(int m, int hi) { return max(m, hi & 0x7fffffff); }
__device__ __forceinline__ int key_of(int mag) { return mag >= 0x7ff00000 ? kBadKey : mag >> 20; }

// High word of a b, plus c.  On the integer multiplier, which has slots left
// here: additions, logic and shifts share another pipe, the kernels' bound.
__device__ __forceinline__ uint32_t mul_hi(uint32_t a, uint32_t b) {
  uint32_t d;
  asm("mul.hi.u32 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
  return d;
}
__device__ __forceinline__ uint32_t mad_hi(uint32_t a, uint32_t b, uint32_t c) {
  uint32_t d;
  asm("mad.hi.u32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
  return d;
}

// v as an integer, mantissa << L >> (kb - e): kb >= e, and kb >= 64 so that
// zeros and subnormals (e = 0) vanish.
template <int L>
__device__ __forceinline__ ll to_fx(double v, int kb) {
  const uint32_t hi = (uint32_t)__double2hiint(v), lo = (uint32_t)__double2loint(v);
  const int e = (int)mul_hi(hi * 2u, 1u << 11);  // the exponent field
  const uint32_t mh = (hi & 0xfffffu) | 0x100000u;
  const uint64_t m = (uint64_t)mad_hi(lo, 1u << L, mh << L) << 32 | (lo << L);
  const ll w = (ll)(m >> min(kb - e, 63));
  const ll s = (int)hi >> 31;
  return (w ^ s) - s;
}

// P = h 2^32 + l, l signed
__device__ __forceinline__ void split32(ll p, int& h, int& l) {
  l = (int)p;
  h = (int)mad_hi((uint32_t)p, 2u, (uint32_t)((uint64_t)p >> 32));
}

// s + a b.  Residuals of one solve at 512^3 and at 8192 x 4096: 9.80 and 1.11 ms
// in this form; 9.98 and 1.18 by mad.wide, 11.4 and 1.22 by s + (ll)a * b.
__device__ __forceinline__ ll mad_wide(int a, int b, ll s) {
  ll d;
  asm("mul.wide.s32 %0, %1, %2;" : "=l"(d) : "r"(a), "r"(b));
  return s + d;
}

// (hh, mm) += p c
__device__ __forceinline__ void mac(ll& hh, ll& mm, int ph, int pl, Limb c) {
  hh = mad_wide(ph, c.h, hh);
  mm = mad_wide(ph, c.l, mm);
  mm = mad_wide(pl, c.h, mm);
}

// hh + (mm >> 32); the middle sums begin at kHalf, so this rounds to nearest
constexpr ll kHalf = 1ll << 31;
__device__ __forceinline__ ll fold(ll hh, ll mm) { return mad_wide((int)(mm >> 32), 1, hh); }

// Q + sum_k q_k P_k and sum_k r_k P_k with real coefficients
template <int NK>
__device__ __forceinline__ void dot_real(const cll (&P)[NK], const Limb* q, const Limb* r, cll& Q, cll& R) {
  cll qm = {kHalf, kHalf}, rh = {0, 0}, rm = {kHalf, kHalf};
#pragma unroll
  for (int k = 0; k < NK; ++k) {
    int xh, xl, yh, yl;
    split32(P[k].x, xh, xl);
    split32(P[k].y, yh, yl);
    mac(Q.x, qm.x, xh, xl, q[k]);
    mac(Q.y, qm.y, yh, yl, q[k]);
    mac(rh.x, rm.x, xh, xl, r[k]);
    mac(rh.y, rm.y, yh, yl, r[k]);
  }
  Q = {fold(Q.x, qm.x), fold(Q.y, qm.y)};
  R = {fold(rh.x, rm.x), fold(rh.y, rm.y)};
}

// s + sum_k c_k P_k with complex coefficients c_k = (re, im); the products
// with the real and with the imaginary parts have a middle sum each (its bound)
template <int NK>
__device__ __forceinline__ cll dot_cplx(cll s, const cll (&P)[NK], const LimbC* c) {
  ll ax = kHalf, ay = kHalf, bx = kHalf, by = kHalf;
#pragma unroll
  for (int k = 0; k < NK; ++k) {
    int xh, xl, yh, yl;
    split32(P[k].x, xh, xl);
    split32(P[k].y, yh, yl);
    mac(s.x, ax, xh, xl, c[k].re);
    mac(s.x, bx, yh, yl, c[k].nim);
    mac(s.y, ay, yh, yl, c[k].re);
    mac(s.y, by, xh, xl, c[k].im);
  }
  return {fold(fold(s.x, ax), bx), fold(fold(s.y, ay), by)};
}

// v / 2^32 for v = h 2^32 + l with l signed (h = 0 whenever v fits l): two
// 32-bit conversions (one of 64 bits would run on the FP64 pipe).
__device__ __forceinline__ float fx_to_float(ll v) {
  const int l = (int)v, h = (int)(v >> 32) + (int)((uint32_t)l >> 31);
  return fmaf((float)l, 0x1p-32f, (float)h);
}

// Factors of 2^32 units of the result, 2^(K - 1048) (two: K may leave a
// float's exponents), NaN from a bad key on.
struct Unit {
  float a, b;
};
__device__ __forceinline__ Unit unit_of(int K) {
  if (K >= kBadKey / 2) return {__int_as_float(0x7fffffff), 1.0f};
  const int s = K - 1048;
  const int s1 = max(-126, min(127, s)), s2 = max(-126, min(127, s - s1));
  return {__int_as_float((s1 + 127) << 23), __int_as_float((s2 + 127) << 23)};
}

// What a thread carries along its column: -R(x-1), f - Q - R(x-2) at x-1, and
// the sums of |r|^2 (in 2^32 units: 64 x 32 of them stay in a float's range)
// and |f|^2.  The latter is of f itself, which may lie far below the tile's
// terms of A u, and in FP64: two instructions on a pipe that is idle here.
struct Column {
  cll A = {0, 0}, R = {0, 0};
  float r2 = 0.f;
  double f2 = 0.0;
  __device__ __forceinline__ void add_f(double2 f) { f2 = fma(f.x, f.x, fma(f.y, f.y, f2)); }
  // r at x-1 from -R(x)
  __device__ __forceinline__ float2 finish(cll Rn, Unit un) {
    const float x = fx_to_float(A.x + Rn.x), y = fx_to_float(A.y + Rn.y);
    r2 = fmaf(x, x, fmaf(y, y, r2));
    return make_float2(x * un.a * un.b, y * un.a * un.b);
  }
  // a unit 2^d times larger
  __device__ __forceinline__ void grow(int d) {
    const float g = __int_as_float((127 - min(d, 126)) << 23);
    r2 = r2 * g * g;
    d = min(d, 63);
    A = {A.x >> d, A.y >> d};
    R = {R.x >> d, R.y >> d};
  }
};

// Block sums of |r|^2 and |f|^2 in fixed order; K: the warp's last key.
template <int NT>
__device__ __forceinline__ void fx_norms(const Column& c, int K, double* sums, int64_t bid) {
  __shared__ double sr[NT / 32], sf[NT / 32];
  float r2 = c.r2;
  double f2 = c.f2;
  for (int off = 16; off > 0; off >>= 1) {
    r2 += __shfl_down_sync(0xffffffffu, r2, off);
    f2 += __shfl_down_sync(0xffffffffu, f2, off);
  }
  const int tid = threadIdx.y * blockDim.x + threadIdx.x;
  if ((tid & 31) == 0) {
    sr[tid >> 5] = K >= kBadKey / 2 ? (double)__int_as_float(0x7fffffff) : scalbn((double)r2, 2 * (K - 1048));
    sf[tid >> 5] = f2;
  }
  __syncthreads();
  if (tid == 0) {
    double a2 = 0, b2 = 0;
    for (int i = 0; i < NT / 32; ++i) {
      a2 += sr[i];
      b2 += sf[i];
    }
    sums[2 * bid] = a2;
    sums[2 * bid + 1] = b2;
  }
}

// ---- 3D -------------------------------------------------------------------
// CTA = 16 x 32 columns (y, z) x up to FX planes, a thread per column.  Planes of
// u (18 x 34 halo box) and f arrive by TMA in a ring of four: while plane i is
// combined, plane i + 1 is converted in place, the key of plane i + 2 is taken
// and plane i + 3 is in flight, with one barrier per plane.
constexpr int FZ = 32, FY = 16, FX = 64, FT = FZ * FY;
constexpr int FW = FZ + 2;                                            // row of the halo box
constexpr int FHALO = (FY + 2) * FW;                                  // its points
constexpr int FUB = FHALO * (int)sizeof(double2);                     // its bytes
constexpr int FUS = (FUB + 127) / 128 * 128;                          // stride of the ring
constexpr int FFB = FY * FZ * (int)sizeof(double2);                   // f tile
constexpr int FNB = 4;                                                // ring
constexpr size_t kFxSmem = (size_t)FNB * (FUS + FFB) + FNB * (sizeof(uint64_t) + sizeof(int));

__global__ void __launch_bounds__(FT, 2)
    k_residual3d_fx(const __grid_constant__ CUtensorMap umap, const __grid_constant__ CUtensorMap fmap,
                    const __grid_constant__ FxArgs a, float2* __restrict__ r, double* __restrict__ sums,
                    const int* __restrict__ skip, int* err) {
  if (skip && *skip) return;
  extern __shared__ __align__(128) unsigned char fsm[];
  unsigned char* sU = fsm;                                    // [FNB][FUS]
  unsigned char* sF = sU + FNB * FUS;                         // [FNB][FFB]
  uint64_t* bar = reinterpret_cast<uint64_t*>(sF + FNB * FFB);  // [FNB]
  int* keys = reinterpret_cast<int*>(bar + FNB);              // [FNB]
  const int tz = threadIdx.x, ty = threadIdx.y, tid = ty * FZ + tz;
  const int z0 = blockIdx.x * FZ, y0 = blockIdx.y * FY;
  const int xs = blockIdx.z * FX, xe = min(xs + FX, a.nx);
  const int np = xe - xs + 2;  // planes xs-1 .. xe
  const int gz = z0 + tz;
  const int kmin = max(a.es, 0) + 64;
  if (tid == 0) {
    for (int b = 0; b < FNB; ++b) {
      mbar_init(&bar[b], 1);
      keys[b] = kmin;
    }
    fence_mbar_init();
  }
  __syncthreads();
  auto issue = [&](int i) {  // plane xs - 1 + i into buffer i % FNB (thread 0; zeros outside the grid)
    const int b = i % FNB;
    mbar_arrive_expect_tx(&bar[b], (uint32_t)(FUB + FFB));
    tma_load_3d(sU + b * FUS, &umap, 2 * (z0 - 1), y0 - 1, xs - 1 + i, &bar[b]);
    tma_load_3d(sF + b * FFB, &fmap, 2 * z0, y0, xs - 1 + i, &bar[b]);
  };
  int issued = 0;
  if (tid == 0)
    for (; issued < 3; ++issued) issue(issued);  // np >= 3
  auto wait = [&](int i) { return mbar_wait_bounded(&bar[i % FNB], (uint32_t)((i / FNB) & 1), err); };
  // largest key of plane i into keys[i % FNB]
  auto take_key = [&](int i) {
    const int4* U = reinterpret_cast<const int4*>(sU + (i % FNB) * FUS);
    const int4* F = reinterpret_cast<const int4*>(sF + (i % FNB) * FFB);
    int ku = 0, kf = 0;
#pragma unroll
    for (int k = 0; k < (FHALO + FT - 1) / FT; ++k) {
      const int e = tid + k * FT;
      if (e < FHALO) {
        const int4 v = U[e];
        ku = mag_max(mag_max(ku, v.y), v.w);
      }
    }
#pragma unroll
    for (int k = 0; k < FY * FZ / FT; ++k) {
      const int4 v = F[tid + k * FT];
      kf = mag_max(mag_max(kf, v.y), v.w);
    }
    const int key = __reduce_max_sync(0xffffffffu, max(key_of(ku) + a.es, key_of(kf)));
    if (tz == 0) atomicMax(&keys[i % FNB], key);
  };
  // plane i of u to integers, in place
  auto convert = [&](int i, int K) {
    double2* U = reinterpret_cast<double2*>(sU + (i % FNB) * FUS);
#pragma unroll
    for (int k = 0; k < (FHALO + FT - 1) / FT; ++k) {
      const int e = tid + k * FT;
      if (e < FHALO) {
        const double2 v = U[e];
        const cll w = {to_fx<7>(v.x, K - a.es), to_fx<7>(v.y, K - a.es)};
        reinterpret_cast<cll*>(U)[e] = w;
      }
    }
    // the buffer's next contents come by TMA: order these writes before it
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  };

  bool ok = wait(0);
  take_key(0);
  ok = wait(1) && ok;
  take_key(1);
  bool failed = __syncthreads_or(!ok);
  int K = max(kmin, keys[0]);
  if (!failed) convert(0, K);
  Unit un = unit_of(K);

  const int gy = y0 + ty;
  const bool own = gz < a.nz && gy < a.ny;
  const int cyz = own ? 2 * (gy == 0 || gy == a.ny - 1 ? 1 : 0) + (gz == 0 || gz == a.nz - 1 ? 1 : 0) : 0;
  const bool face = __any_sync(0xffffffffu, cyz != 0);
  Column col;
  float2* rp = r + ((int64_t)xs * a.ny + gy) * a.nz + gz;  // of the plane to complete
  ok = true;
  int i = 0;
  for (; !failed && i < np; ++i) {
    // plane i converted and key i + 1 complete; everyone is past plane i - 1
    if (__syncthreads_or(!ok)) {
      failed = true;
      break;
    }
    const int Kn = max(K, keys[(i + 1) % FNB]);
    if (tid == 0 && i + 3 < np) {
      issue(i + 3);
      issued = i + 4;
    }
    const int ip = xs - 1 + i;
    const bool outp = ip >= xs && ip < xe;
    const cll* U = reinterpret_cast<const cll*>(sU + (i % FNB) * FUS) + ty * FW + tz;
    cll P[4];
    P[0] = U[FW + 1];
    P[1] = U[FW] + U[FW + 2];
    P[2] = U[1] + U[2 * FW + 1];
    P[3] = (U[0] + U[2]) + (U[2 * FW] + U[2 * FW + 2]);
    const double2 fv = reinterpret_cast<const double2*>(sF + (i % FNB) * FFB)[tid];
    cll A = {to_fx<5>(fv.x, K), to_fx<5>(fv.y, K)}, Rn;  // f - Q, -R
    if (outp) col.add_f(fv);  // zeros outside the grid
    const bool cx = ip == 0 || ip == a.nx - 1;
    if (!face && !cx) {
      dot_real<4>(P, a.q, a.r, A, Rn);
    } else {
      A = dot_cplx<4>(A, P, a.c0[(cx ? 4 : 0) + cyz]);
      Rn = dot_cplx<4>({0, 0}, P, a.c1[cyz]);
    }
    if (ip > xs) {  // plane ip - 1 is complete
      if (own) *rp = col.finish(Rn, un);
      rp += (int64_t)a.ny * a.nz;
    }
    col.A = A + col.R;
    col.R = Rn;
    ok = true;
    if (tid == 0) keys[(i + 3) % FNB] = kmin;  // (i - 1) % FNB, read before this plane's barrier
    if (i + 2 < np) {
      ok = wait(i + 2);
      take_key(i + 2);
    }
    if (i + 1 < np) {
      if (Kn > K) {
        col.grow(Kn - K);
        K = Kn;
        un = unit_of(K);
      }
      convert(i + 1, K);
    }
  }
  if (failed && tid == 0)
    for (int j = 0; j < issued; ++j)
      if (j + FNB >= issued) mbar_wait_bounded(&bar[j % FNB], (uint32_t)((j / FNB) & 1), nullptr);
  fx_norms<FT>(col, K, sums, ((int64_t)blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x);
}

// ---- 2D -------------------------------------------------------------------
// A warp takes 30 columns (y) and one on each side, and `rows` rows of x,
// which it walks with a key of its own: no barrier, no shared memory, the
// neighbours' integers by shuffles.
constexpr int kFx2Warps = 8;
constexpr int kFx2Cols = 30;
__global__ void __launch_bounds__(32 * kFx2Warps, 3)
    k_residual2d_fx(const __grid_constant__ FxArgs a, int rows, const double2* __restrict__ f,
                    const double2* __restrict__ u, float2* __restrict__ r, double* __restrict__ sums,
                    const int* __restrict__ skip) {
  if (skip && *skip) return;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int y = ((int)blockIdx.x * kFx2Warps + warp) * kFx2Cols + lane - 1;
  const int xs = (int)blockIdx.y * rows, xe = min(xs + rows, a.nx);
  const bool in = y >= 0 && y < a.ny;
  const bool own = in && lane >= 1 && lane <= kFx2Cols;
  const int cy = own && (y == 0 || y == a.ny - 1) ? 1 : 0;
  const bool face = __any_sync(0xffffffffu, cy != 0);
  int K = max(a.es, 0) + 64;
  Unit un = unit_of(K);
  Column col;
  const double2 zero = make_double2(0.0, 0.0);
  const double2* up = u + (int64_t)(xs - 1) * a.ny + y;
  const double2* fp = f + (int64_t)(xs - 1) * a.ny + y;
  float2* rp = r + (int64_t)xs * a.ny + y;
  constexpr int AHEAD = 3;  // rows in flight
  double2 ub[AHEAD], fb[AHEAD];
  auto fetch = [&](int ip, double2& uv, double2& fv) {
    uv = fv = zero;
    if (in && ip >= 0 && ip < a.nx && ip <= xe) uv = __ldg(up);
    if (own && ip >= xs && ip < xe) fv = __ldg(fp);
    up += a.ny;
    fp += a.ny;
  };
#pragma unroll
  for (int k = 0; k < AHEAD; ++k) fetch(xs - 1 + k, ub[k], fb[k]);
  for (int i0 = xs - 1; i0 <= xe; i0 += AHEAD) {
#pragma unroll
    for (int k = 0; k < AHEAD; ++k) {
      const int ip = i0 + k;
      if (ip > xe) break;
      const double2 uv = ub[k], fv = fb[k];
      fetch(ip + AHEAD, ub[k], fb[k]);
      const int ku = key_of(mag_max(mag_max(0, __double2hiint(uv.x)), __double2hiint(uv.y)));
      const int kf = key_of(mag_max(mag_max(0, __double2hiint(fv.x)), __double2hiint(fv.y)));
      const int Kn = __reduce_max_sync(0xffffffffu, max(ku + a.es, kf));
      if (Kn > K) {  // warp-uniform
        col.grow(Kn - K);
        K = Kn;
        un = unit_of(K);
      }
      cll P[2];
      P[0] = {to_fx<7>(uv.x, K - a.es), to_fx<7>(uv.y, K - a.es)};
      P[1].x = __shfl_up_sync(0xffffffffu, P[0].x, 1) + __shfl_down_sync(0xffffffffu, P[0].x, 1);
      P[1].y = __shfl_up_sync(0xffffffffu, P[0].y, 1) + __shfl_down_sync(0xffffffffu, P[0].y, 1);
      cll A = {to_fx<5>(fv.x, K), to_fx<5>(fv.y, K)}, Rn;  // f - Q, -R
      col.add_f(fv);  // zero where the lane has no output here
      const bool cx = ip == 0 || ip == a.nx - 1;
      if (!face && !cx) {
        dot_real<2>(P, a.q, a.r, A, Rn);
      } else {
        A = dot_cplx<2>(A, P, a.c0[(cx ? 2 : 0) + cy]);
        Rn = dot_cplx<2>({0, 0}, P, a.c1[cy]);
      }
      if (ip > xs) {  // row ip - 1 is complete
        if (own) *rp = col.finish(Rn, un);
        rp += a.ny;
      }
      col.A = A + col.R;
      col.R = Rn;
    }
  }
  fx_norms<32 * kFx2Warps>(col, K, sums, (int64_t)blockIdx.y * gridDim.x + blockIdx.x);
}

// Rows per warp of the 2D kernel: 64 (two halo rows in 66), fewer while the
// grid leaves an SM without 16 warps.
int fx2_rows(const int64_t* n) {
  const int64_t cols = (n[1] + kFx2Cols - 1) / kFx2Cols;
  int rows = 64;
  while (rows > 2 && cols * ((n[0] + rows - 1) / rows) < kSMs * 16) rows /= 2;
  return rows;
}

dim3 fx_grid(int dim, const int64_t* n) {
  if (dim == 2) {
    const int rows = fx2_rows(n);
    return dim3((unsigned)((n[1] + kFx2Warps * kFx2Cols - 1) / (kFx2Warps * kFx2Cols)),
                (unsigned)((n[0] + rows - 1) / rows));
  }
  return dim3((unsigned)((n[2] + FZ - 1) / FZ), (unsigned)((n[1] + FY - 1) / FY), (unsigned)((n[0] + FX - 1) / FX));
}

FxArgs fx_args(int dim, const ResidQArgs& q) {
  FxArgs a{};
  a.nx = (int)q.n[0];
  a.ny = (int)q.n[1];
  a.nz = dim == 3 ? (int)q.n[2] : 1;
  const int nk = dim == 3 ? 4 : 2, n0 = dim == 3 ? 8 : 4, n1 = dim == 3 ? 4 : 2;
  const double mult[4] = {1, 2, 2, 4};
  auto mag = [](double2 c) { return std::fabs(c.x) + std::fabs(c.y); };
  double S = 0;
  for (int c = 0; c < n0; ++c) {
    double s = 0;
    for (int k = 0; k < nk; ++k) s += mult[k] * (mag(q.c0[c][k]) + 2 * mag(q.c1[c % n1][k]));
    S = std::max(S, s);
  }
  if (!std::isfinite(S) || S <= 0) S = 1;
  std::frexp(S * (1 + 1e-12), &a.es);  // S < 2^es
  auto neg = [&](double2 c) { return fx_limb_c(-c.x, -c.y, a.es); };
  for (int k = 0; k < nk; ++k) {
    a.q[k] = neg(q.c0[0][k]).re;
    a.r[k] = neg(q.c1[0][k]).re;
    for (int c = 0; c < n0; ++c) a.c0[c][k] = neg(q.c0[c][k]);
    for (int c = 0; c < n1; ++c) a.c1[c][k] = neg(q.c1[c][k]);
  }
  return a;
}

}  // namespace

int64_t residual_fx_blocks(int dim, const int64_t* n) {
  const dim3 g = fx_grid(dim, n);
  return (int64_t)g.x * g.y * g.z;
}

cudaError_t launch_residual_fx(int dim, const ResidQArgs& q, const double2* f, const double2* u, float2* r,
                               double* sums, int64_t* nblocks, const int* skip, int* err, cudaStream_t st) {
  const dim3 grid = fx_grid(dim, q.n);
  *nblocks = (int64_t)grid.x * grid.y * grid.z;
  const FxArgs a = fx_args(dim, q);
  if (dim == 2) {
    k_residual2d_fx<<<grid, 32 * kFx2Warps, 0, st>>>(a, fx2_rows(q.n), f, u, r, sums, skip);
    return cudaGetLastError();
  }
  CUtensorMap um, fm;
  if (allow_dynamic_smem((const void*)k_residual3d_fx, kFxSmem) != cudaSuccess ||
      !residual_map(&um, u, q.n, FZ + 2, FY + 2) || !residual_map(&fm, f, q.n, FZ, FY)) {
    cudaGetLastError();
    return cudaErrorNotSupported;
  }
  k_residual3d_fx<<<grid, dim3(FZ, FT / FZ), kFxSmem, st>>>(um, fm, a, r, sums, skip, err);
  return cudaGetLastError();
}

}  // namespace helm
