// Host side of the run-time FFT engine (fft.cuh): plans, and the launch shapes of the passes that use it.
#include "qg_kernels.h"

#include <atomic>
#include <cmath>
#include <utility>

namespace qg {

FftPlan fft_plan(int n, int el) {
  FftPlan p;
  p.n = n;
  p.el = el;
  const Radices r = fft_radices(n, p.el);
  p.tt = n / p.el;
  p.npass = r.np;
  for (int i = 0; i < p.npass; ++i)
    p.pass[i] = {r.radix[i], r.ns[i], r.ns[i] > 1 ? (unsigned)((1ull << 32) / (unsigned)r.ns[i] + 1) : 0u, r.off[i]};
  p.table = r.table;
  p.buf = n + n / 16 + 1;
  return p;
}

// ---- twiddle tables.  A table's rounding errors are the same in every transform, so they add up from step to step;
// the entries are formed in double-double arithmetic (a value as the unevaluated sum h + l) and rounded once.
namespace {
struct DD {
  double h, l;
};
DD norm(double a, double b) {  // |a| >= |b|
  const double s = a + b;
  return {s, b - (s - a)};
}
DD add(DD a, DD b) {
  const double s = a.h + b.h, t = s - a.h;
  return norm(s, (a.h - (s - t)) + (b.h - t) + (a.l + b.l));
}
DD neg(DD a) { return {-a.h, -a.l}; }
DD mul(DD a, DD b) {
  const double p = a.h * b.h;
  return norm(p, std::fma(a.h, b.h, -p) + std::fma(a.h, b.l, a.l * b.h));
}
DD div(DD a, double b) {
  const double q = a.h / b;
  return norm(q, (std::fma(-q, b, a.h) + a.l) / b);
}
struct Rot {
  DD c, s;
};
Rot turn(const Rot& a, const Rot& b) {
  return {add(mul(a.c, b.c), neg(mul(a.s, b.s))), add(mul(a.s, b.c), mul(a.c, b.s))};
}
}  // namespace

std::vector<double> fft_table(const FftPlan& p, int esz) {
  // cos and sin of 2 pi i / (4 n) for angles up to pi / 4: the smallest by its Taylor series, the others by addition
  const long n = p.n;
  std::vector<Rot> rot(n / 2 + 1);
  rot[0] = {{1.0, 0.0}, {0.0, 0.0}};
  const DD x = div(DD{1.5707963267948966, 6.123233995736766e-17}, (double)n);
  Rot r = rot[0];
  DD term = {1.0, 0.0};
  for (int k = 1; k < 24; ++k) {
    term = div(mul(term, x), k);
    DD& sum = k & 1 ? r.s : r.c;
    sum = add(sum, k & 2 ? neg(term) : term);
  }
  rot[1] = r;
  for (long i = 2; i <= n / 2; ++i) rot[i] = turn(rot[i / 2], rot[i - i / 2]);
  std::vector<double> t(2 * (size_t)p.table);
  for (int e = 0; e < p.table; ++e) {
    const FftEntry f = fft_table_entry(p, e);
    const long q4 = 4L * f.j, quad = q4 / n, rem = q4 - quad * n;  // the angle within its quadrant is (pi / 2) rem / n
    const bool low = 2 * rem <= n;
    const Rot& w = rot[low ? rem : n - rem];
    DD c = low ? w.c : w.s, s = low ? w.s : w.c;
    if (quad & 1) std::swap(c, s);
    if (quad == 1 || quad == 2) c = neg(c);
    if (quad < 2) s = neg(s);  // exp(-i angle)
    t[2 * e] = c.h;
    t[2 * e + 1] = s.h;
    if (ratio_twiddle(f.radix, esz)) {
      if (std::fabs(c.h) < kRatioMinCos) t[2 * e] = kRatioMinCos;
      t[2 * e + 1] = div(s, t[2 * e]).h;
    }
  }
  return t;
}

int device_sms() {
  static std::atomic<int> sms[64];
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev < 0 || dev >= 64) return 1;
  int n = sms[dev].load(std::memory_order_relaxed);
  if (!n) {
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n < 1) n = 1;
    sms[dev].store(n, std::memory_order_relaxed);
  }
  return n;
}

// dynamic shared memory a CTA can have: 227 KB less the passes' static part (under 768 bytes)
constexpr size_t kSmemCap = 227 * 1024 - 768;

static size_t tw_bytes(const FftPlan& p, int esz) { return tw_shared(p.table) ? (size_t)p.table * 2 * esz : 0; }

RowConfig row_config(const FftPlan& p, const RowDesc& d, int esz) {
  RowConfig c{};
  const bool direct = d.prog == RP_SCALE || d.prog == RP_COPY;
  int nin = d.nin, nout = d.nout;
  if (direct) nin = nout = d.npair > 0 ? 2 * d.npair : d.in_phys ? d.nout : d.nin;
  c.nslot = direct ? 0 : (nin > nout ? nin : nout);
  auto tasks = [](int rows, int nf) { return rows * (nf / 2) + (nf & 1 ? (rows + 1) / 2 : 0); };
  auto bytes = [&](int rows, int groups, int nbuf) {
    return (tw_bytes(p, esz) + (size_t)groups * nbuf * p.buf * 2 * esz) + (size_t)rows * c.nslot * p.n * esz;
  };
  const bool odd = (nin & 1) || (nout & 1);
  c.rows = odd && (direct || (p.n >= 256 && bytes(2, 1, 2) <= kSmemCap / 2)) ? 2 : 1;
  const int most = tasks(c.rows, nin) > tasks(c.rows, nout) ? tasks(c.rows, nin) : tasks(c.rows, nout);
  const int target = esz == 4 ? 256 : 192;
  int groups = target / p.tt;
  if (groups < 1) groups = 1;
  if (groups > most) groups = most;
  // even rounds
  const int rounds = (most + groups - 1) / groups;
  groups = (most + rounds - 1) / rounds;
  while (groups > 1 && bytes(c.rows, groups, 2) > kSmemCap / 2) --groups;
  c.groups = groups;
  c.one_buf = bytes(c.rows, groups, 2) > kSmemCap;
  if (c.rows == 2 && bytes(2, groups, 1) > kSmemCap) c.rows = 1;
  c.smem = bytes(c.rows, groups, c.one_buf ? 1 : 2);
  c.threads = (groups * p.tt + 31) / 32 * 32;
  // FP64 is bound by its operations, so the last, partial round of row pairs goes out as single rows where that
  // leaves no SM with two of them (1024^2: 3 pairs and a row per SM against 4 pairs)
  const int pairs = p.n / c.rows, sms = device_sms(), rest = pairs % sms;
  c.full = pairs;
  if (esz == 8 && c.rows == 2 && !direct && pairs > sms && rest > 0 && 2 * rest <= sms) c.full = pairs - rest;
  c.warp = p.tt <= 32 && 32 % p.tt == 0;
  return c;
}

int col_width(const FftPlan& p, int esz) {
  if (p.n <= 512) return 1;
  return esz == 4 && 2 * p.tt <= pass_threads(p.el, esz) ? 2 : 1;
}

ColConfig col_config(const Geom& g, const FftPlan& p, const ColDesc& d, int W, int esz) {
  ColConfig c{};
  c.w = W;
  c.pitch = (p.buf + 15) / 16 * 16 + (W > 1 ? (esz == 4 ? 16 : 8) / W : 0);
  const int most = d.nfwd > d.nder ? d.nfwd : d.nder;
  auto bytes = [&](int f, int nbuf) {
    return tw_bytes(p, esz) + ((size_t)f * W * nbuf * c.pitch + 2 * (size_t)W * g.Ny) * 2 * esz;
  };
  const int target = esz == 4 ? 256 : 192;
  int f = target / (p.tt * W);
  if (f < 1) f = 1;
  if (f > most) f = most > 0 ? most : 1;
  const int rounds = most > 0 ? (most + f - 1) / f : 1;
  f = most > 0 ? (most + rounds - 1) / rounds : 1;
  while (f > 1 && bytes(f, 2) > kSmemCap / 2) --f;
  c.fields = f;
  c.one_buf = bytes(f, 2) > kSmemCap;
  c.smem = bytes(f, c.one_buf ? 1 : 2);
  c.threads = (f * W * p.tt + 31) / 32 * 32;
  // FP64: the columns beyond a whole number of rounds over the SMs share out their outgoing fields, one CTA per SM,
  // at the price of transforming the incoming ones in each (1024^2: 342 columns, 38 of them in four parts; with the
  // single rows of row_config 1508 -> 1374 us per step).  Not with less than a round: 128^2, 43 columns in three
  // parts each, 140 us against 136.  Not where an op reads what it writes: a column's parts run at the same time.
  const int tiles = g.Kcp / W, sms = device_sms(), rest = tiles % sms;
  bool reads_own = d.op == CO_AB2CN || d.op == CO_AB2CN_COMBINE ||
                   ((d.op == CO_STAGE_STATIC || d.op == CO_DYN_COMBINE) && d.store_w0);
  for (int i = 0; i < d.nfwd; ++i)
    for (int q = 0; q < d.nder; ++q) reads_own = reads_own || d.fin[i] == d.dout[q];
  c.full = tiles;
  c.split = 1;
  if (esz == 8 && !reads_own && d.nder > 1 && rest > 0 && tiles > sms) {
    const int s = sms / rest < d.nder ? sms / rest : d.nder;
    if (s > 1) {
      c.split = s;
      c.full = tiles - rest;
    }
  }
  c.grid = c.full + (tiles - c.full) * c.split;
  c.warp = p.tt * W <= 32 && 32 % (p.tt * W) == 0;
  return c;
}

}  // namespace qg
