// Planner and launchers of the mixed-radix transforms (kernels:
// helm_dft_mix.cuh): the radices of a length, Bluestein's convolution length,
// and the shape of a launch.
#include <algorithm>
#include <cmath>

#include "helm_dft_mix.h"

namespace helm {

namespace {

// Arithmetic of one point in a radix-R butterfly (fused operations).
double radix_cost(int R) {
  static const double c[11] = {0, 0, 2, 5.3, 4, 8, 7.3, 11, 6.5, 9, 10};
  return R <= 10 ? c[R] : (double)(R - 1) * (R - 1) / R + 6.0;
}

// Cost of a pass per point beside its butterfly: twiddle and exchange (on
// the FP64 pipe only the twiddle's four operations show).
double pass_cost(int prec) { return prec == kPrecF64 ? 4.5 : 9.0; }

struct MixSearch {
  int prec;
  explicit MixSearch(int p) : prec(p) {}
  int best[kMixStages], cur[kMixStages];
  int nbest = 0;
  double cost = 1e300;
  void go(int n, int from, int depth, double c) {
    if (c >= cost) return;
    if (n == 1) {
      cost = c;
      nbest = depth;
      std::copy(cur, cur + depth, best);
      return;
    }
    if (depth == kMixStages) return;
    for (int r = std::min(from, n); r >= 2; --r)
      if (n % r == 0) {
        cur[depth] = r;
        go(n / r, r, depth + 1, c + radix_cost(r) + pass_cost(prec));
      }
  }
};

// Radices of n (descending; primes above 10 lead), 0 passes if a prime
// factor exceeds 64.
MixSearch mix_radices(int64_t n, int prec) {
  MixSearch f(prec);
  int lead = 0;
  double c = 0;
  int m = (int)n;
  for (int q = 61; q >= 11; --q) {
    bool prime = true;
    for (int d = 2; d * d <= q; ++d) prime = prime && q % d;
    while (prime && m % q == 0 && lead < kMixStages) {
      f.cur[lead++] = q;
      m /= q;
      c += radix_cost(q) + pass_cost(prec);
    }
  }
  f.go(m, 10, lead, c);
  return f;
}

// Where each pass's tables begin (mix_tables): 16-byte aligned, -1: none.
void place_tables(MixPlan* m) {
  int at = 0;
  for (int s = 0; s < m->nstages; ++s) {
    MixStage& t = m->s[s];
    t.toff = t.ns > 1 ? at : -1;
    if (t.ns > 1) at += t.ns * t.r;
    t.roff = t.r > 10 ? at : -1;
    if (t.r > 10) at += t.r;
    at += at & 1;
  }
}

void put_stage(MixStage& s, int n, int r, int ns) {
  auto mul = [](int d) -> uint32_t { return d > 1 ? (uint32_t)((uint64_t(1) << 32) / (uint64_t)d) + 1u : 0u; };
  s.r = r;
  s.nb = n / r;
  s.ns = ns;
  s.st = n / (ns * r);
  s.mnb = mul(s.nb);
  s.mns = mul(ns);
}

}  // namespace

MixShape mix_shape(const MixPlan& m, bool cols, size_t es, int64_t nlines, int64_t outer, int64_t inner) {
  MixShape h{1, 0, 64, 1};
  bool prime = false;
  for (int s = 0; s < m.nstages; ++s) prime = prime || m.s[s].r > 10;
  h.nbuf = prime || m.nstages > 2 ? 2 : (m.nstages > 1 ? 1 : 0);
  const int nbuf = std::max(1, h.nbuf);
  const size_t line = (size_t)m.n * es * nbuf;
  // a CTA takes lines of about 48 KB of shared memory (four CTAs an SM), fewer
  // while the grid leaves SMs without two CTAs
  if (cols) {
    int tc = es == 8 ? 16 : 8;  // 128-byte rows
    while (tc > 4 && tc * line > 48 * 1024) tc /= 2;
    while (tc > 1 && tc * line > 160 * 1024) tc /= 2;
    while (tc > 1 && tc / 2 >= inner) tc /= 2;
    while (tc > 2 && outer * ((inner + tc - 1) / tc) < 2 * kSMs) tc /= 2;
    while ((1 << h.lt) < tc) ++h.lt;
    h.L = tc;
  } else {
    int64_t l = std::min<int64_t>(4096 / m.n, (int64_t)(48 * 1024 / line));
    l = std::min<int64_t>(l, nlines / (2 * kSMs));
    h.L = (int)std::max<int64_t>(1, l);
  }
  // threads: the fewest thread slots over all passes (idle slots of the last
  // round of each pass count)
  double best = 1e300;
  for (int t = 64; t <= kMixThreads; t += 32) {
    double c = 0;
    for (int s = 0; s < m.nstages; ++s) {
      const int r = m.s[s].r;
      int64_t items = (int64_t)h.L * m.s[s].nb;
      double w = (radix_cost(r) + pass_cost(es == 16 ? kPrecF64 : kPrecF32)) * r;
      if (r > 10) {
        items *= (r + 1) / 2;
        w = w / ((r + 1) / 2);
      }
      const double rounds = (double)((items + t - 1) / t);
      c += rounds * (t + 64.0) * w;  // 64: a longer chain of rounds is latency
    }
    if (c < best) {
      best = c;
      h.threads = t;
    }
  }
  return h;
}

namespace {

template <bool COLS>
cudaError_t launch_mix(int prec, const void* in, int kind, void* out, int out_mode, int64_t nlines, int64_t outer,
                       int64_t inner, const DftPlan& p, const void* tw, int sign, double scale, double accum_scale,
                       const void* sc_in, const void* sc_out, const int* skip, cudaStream_t st) {
  const bool f64 = prec == kPrecF64, bs = p.bm != 0;
  // complex128 reads complex128; complex64 columns read complex64
  if (!p.mix.nstages || (!f64 && !p.mtw) || (f64 && kind != kInC128) || (!f64 && COLS && kind != kInC64)) return cudaErrorInvalidValue;
  // the kernels index one slab, or one CTA's lines, with 32 bits
  if (COLS && (int64_t)p.n * inner > INT32_MAX / 2) return cudaErrorInvalidValue;
  const MixArgs a{p.mix, !f64 ? p.mtw : bs ? p.btw : tw, p.bw, p.bf};
  auto go = [&](auto f) {
    return f(a, p.n, in, kind, out, out_mode, nlines, outer, inner, sign, scale, accum_scale, sc_in, sc_out, skip, st);
  };
  if (f64) return bs ? go(run_mix<double, COLS, true>) : go(run_mix<double, COLS, false>);
  return bs ? go(run_mix<float, COLS, true>) : go(run_mix<float, COLS, false>);
}

}  // namespace

void mix_plan(int64_t n, int prec, MixPlan* m) {
  *m = MixPlan{};
  m->n = (int)n;
  m->mid = -1;
  if (n < 2) return;
  const MixSearch f = mix_radices(n, prec);
  int ns = 1;
  for (int s = 0; s < f.nbest; ++s) {
    put_stage(m->s[s], (int)n, f.best[s], ns);
    ns *= f.best[s];
  }
  m->nstages = f.nbest;
  place_tables(m);
}

int64_t mix_bluestein(int64_t n, int64_t top, int prec, MixPlan* m) {
  double best = 1e300;
  int64_t pick = 0;
  MixSearch pf(prec);
  for (int64_t k = 2 * n - 1; k <= top; ++k) {
    int64_t r = k;
    for (int q : {2, 3, 5, 7})
      while (r % q == 0) r /= q;
    if (r != 1) continue;
    const MixSearch f = mix_radices(k, prec);
    if (!f.nbest || 2 * f.nbest - 1 > kMixStages) continue;
    const double c = (double)k * (f.cost - 0.5 * pass_cost(prec));  // the middle pass is shared
    if (c < best) {
      best = c;
      pick = k;
      pf = f;
    }
  }
  *m = MixPlan{};
  if (!pick) return 0;
  m->n = (int)pick;
  const int P = pf.nbest;
  m->mid = P - 1;
  m->nstages = 2 * P - 1;
  int ns = 1;
  for (int s = 0; s < P; ++s) {
    put_stage(m->s[s], (int)pick, pf.best[s], ns);
    ns *= pf.best[s];
  }
  ns = pf.best[P - 1];
  for (int s = P - 2; s >= 0; --s) {
    put_stage(m->s[2 * P - 2 - s], (int)pick, pf.best[s], ns);
    ns *= pf.best[s];
  }
  place_tables(m);
  return pick;
}

void mix_tables(const MixPlan& m, std::vector<std::complex<double>>* out) {
  std::vector<double> re(m.n), im(m.n);
  unit_roots(m.n, re.data(), im.data());
  out->clear();
  for (int s = 0; s < m.nstages; ++s) {
    const MixStage& t = m.s[s];
    const bool tw = t.toff >= 0;
    for (int k = 0; tw && k < t.ns; ++k)
      for (int q = 0; q < t.r; ++q) {
        const int64_t e = (int64_t)q * k * t.st;
        out->push_back({re[e], im[e]});
      }
    for (int q = 0; t.roff >= 0 && q < t.r; ++q) out->push_back({re[(int64_t)q * t.nb], im[(int64_t)q * t.nb]});
    if (out->size() % 2) out->push_back(0.0);
  }
}

cudaError_t launch_dft_rows_mix(int prec, const void* in, int in_is_double, void* out, int out_mode, int64_t nrows,
                                const DftPlan& p, const void* tw, int sign, double scale, double accum_scale,
                                const void* sc_in, const void* sc_out, const int* skip, cudaStream_t st) {
  return launch_mix<false>(prec, in, in_is_double, out, out_mode, nrows, 1, 1, p, tw, sign, scale, accum_scale, sc_in,
                           sc_out, skip, st);
}

cudaError_t launch_dft_cols_mix(int prec, const void* in, int in_is_double, void* out, int out_mode, int64_t outer,
                                int64_t inner, const DftPlan& p, const void* tw, int sign, double scale,
                                double accum_scale, const void* sc_in, const void* sc_out, const int* skip,
                                cudaStream_t st) {
  return launch_mix<true>(prec, in, in_is_double, out, out_mode, outer * inner, outer, inner, p, tw, sign, scale,
                          accum_scale, sc_in, sc_out, skip, st);
}

}  // namespace helm
