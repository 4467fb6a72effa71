// The FP64 dslash of one site in block fixed point, on the integer pipe.
//
// An SM quarter of GB300 takes one FP64 warp instruction every 67 cycles
// (measured), but a 32 x 32 + 64-bit integer multiply-add every 4.2 and an
// integer add, logic or shift instruction every 2.4.  The FP64 stencil takes 614
// FP64 instructions a site and is bound by that pipe alone (24^3 x 64, temporal
// gauge, 18 reals: 471 us).  Here every number of a hop is a 64-bit integer, and a
// product of two takes three integer multiply-adds: 149 us (its bytes take 81);
// M_hat with 12-real general links of 20 x 14 x 22 x 38 132 us; 8^3 x 16, four
// warps per 32 sites, 6.0 us.  No pipe is full: 12 warps per SM (168 registers)
// leave the latencies of 6300 dependent integer instructions per 32 sites in sight.
//
//  * A link element u, |u| <= 1, is the integer u 2^61 (converted once, when
//    the links are loaded).  A double of at least 2^-9 is exact in it, a
//    smaller one is off by at most 2^-62.
//  * The spinors of a site's neighbours share one exponent E (|x| < 2^(E-1023)
//    for all of their components): x is the integer x 2^(59-(E-1023)), so a
//    projected component, a sum of two, is below 2^60.
//  * Both are kept as two signed 32-bit limbs, a = ah 2^32 + al with al in
//    [-2^31, 2^31).  Of a product's limbs ah bh, (ah bl + al bh) 2^-32 and
//    al bl 2^-64, the last is left out: at most a quarter of the unit 2^(E-1079)
//    in which the sums are kept.
//  * The 24 sums are 64-bit integers of that unit, rounded once, to the double they
//    become.
//
// Accuracy.  B = 2^(E-1023) is one to four times the largest neighbour component.
// The sums are off by 25 units of 2^-56 B at most (a hop: 1.5 dropped limbs, 0.5 the
// middle sums' rounding, 1.0 the cut numbers; one the shifts to a larger E) and by
// one unit as a rule; FP64 rounds each component relative to what feeds it, sum |u|
// |psi|, which is more than B in ordinary fields but may be far less.  So each spin
// collects the smallest colour of every row that feeds it (fixed_weight), and a site
// with a spin that gets less than 2^-6 B is computed in FP64 (dslash_site_weak).
// What is left is right to 2^-44 of sum |u| |psi| in every complex component, and as
// a rule to 2^-50, inside the 2^-49 that FP64's 15 roundings may add up to.  No site
// of Gaussian fields goes that way, 5e-4 of a point source's solution at kappa 0.12,
// and the fronts of its first iterates.  The weights take 3 % of the dslash (144.5 ->
// 149.1 us at 24^3 x 64, 5.7 -> 6.0 at 8^3 x 16), the FP64 sites 0.3 % of twelve point
// sources' batch on 16^3 x 32 (4 % when each was left to its own thread).
// (A third row rebuilt from 12 reals is right to a few 2^-53 of 1 in FP64.)
//
// E is known only when all neighbours are, so it is a running maximum: a hop
// that raises it shifts the sums down.  Starting one above the first hop's
// exponent makes that rare.  Sums cannot overflow: where the parts of a row add up
// to 3.5 (kFixedLinkSum, a rule by which links take this form), each of the eight
// hops adds at most 3.5 x 2^57, and a middle sum stays below 3.5 x 2^60 + 6 x 2^59.
//
// Sites whose neighbours hold an infinity, a NaN, or only numbers outside
// 2^-830 .. 2^870 are computed by dslash_site in FP64 as well.
#pragma once

#include "wd_async.cuh"
#include "wd_device.cuh"

namespace wd {

constexpr int kFixedMinExp = 192, kFixedMaxExp = 1892;  // biased exponents E of the fixed-point path
// Weak sites of a warp that its lanes compute together, one after the other; more
// are computed by their own threads at a time.  8^3 x 16, 18 (12) reals: 3.1 us (3.9)
// a site against 27 us (33) for all of a warp's; 24^3 x 64 with every site weak 1614
// us (2180) against 632 (797), which crosses at ten.
constexpr int kFixedShared = 8;
constexpr int kFixedWeak = 1 << 21;  // 2^-6 of the common exponent, in the unit of the high words (fixed_weight)

struct Fx {
  int h, l;  // h * 2^32 + l
};

__device__ __forceinline__ Fx fx_split(long long v) {
  const unsigned lo = (unsigned)v;
  return Fx{(int)(v >> 32) + (int)(lo >> 31), (int)lo};
}
__device__ __forceinline__ long long fx_join(Fx a) { return ((long long)a.h << 32) + a.l; }
// a b + c.  The product is opaque to the compiler's algebra, which would split
// one with a negated factor; with the sum left to it, the two become one
// multiply-add (a mad.wide in its place took 0.7 more instructions)
__device__ __forceinline__ long long fx_mad(int a, int b, long long c) {
  long long p;
  asm("mul.wide.s32 %0, %1, %2;" : "=l"(p) : "r"(a), "r"(b));
  return c + p;
}

// shifts that give 0 (or the sign) for any count of 64 and more
__device__ __forceinline__ unsigned long long fx_shr(unsigned long long v, int s) {
  unsigned long long r;
  asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(s));
  return r;
}
__device__ __forceinline__ int fx_shr32(int v, int s) {  // v >= 0; 0 for any count of 32 and more
  int r;
  asm("shr.u32 %0, %1, %2;" : "=r"(r) : "r"(v), "r"(s));
  return r;
}
// v 2^-s rounded to nearest, |v| < 2^62
__device__ __forceinline__ long long fx_round_sar(long long v, int s) {
  s = min(s, 62);
  return (v + ((1ll << s) >> 1)) >> s;
}

// v 2^e by the conversion of the FP64 pipe (otherwise idle here) and an
// addition to its exponent
__device__ __forceinline__ double fx_sum_value(long long v, int e) {
  const double d = __ll2double_rn(v);
  const int hi = __double2hiint(d);
  return __hiloint2double(hi ? hi + (e << 20) : 0, __double2loint(d));
}

// The FP64 links in this form: the words of GaugeF64, each double replaced by
// its two limbs (h first), and the doubles themselves for the sites left to FP64.
struct GaugeX64 {
  using real = double;
  static constexpr bool kScaled = false;
  const int4* p;
  int stride;
  int recon;
  const double2* d;
  __device__ __forceinline__ GaugeF64 f64() const { return GaugeF64{d, stride, recon, nullptr}; }
};

// Staging of one hop per thread, as in wd_async.cuh: the neighbour's spinor and
// the link, each refilled by cp.async for the next hop as soon as this hop has
// read it (the spinor while the SU(3) product runs, the link while the next
// spinor is converted), so the loads hold no registers.
constexpr int kFixedBlock = 128;
struct FixedSlots {
  uint4 sp[12][kFixedBlock];
  int4 lk[9][kFixedBlock];
};

// a b + c d - e f - g q of link elements, as a link element
__device__ __forceinline__ long long fx_minor(Fx a, Fx b, Fx c, Fx d, Fx e, Fx f, Fx g, Fx q) {
  long long hp = fx_mad(a.h, b.h, 0), mp = fx_mad(a.h, b.l, 1ll << 28);
  mp = fx_mad(a.l, b.h, mp);
  hp = fx_mad(c.h, d.h, hp);
  mp = fx_mad(c.h, d.l, mp);
  mp = fx_mad(c.l, d.h, mp);
  long long hq = fx_mad(e.h, f.h, 0), mq = fx_mad(e.h, f.l, 0);
  mq = fx_mad(e.l, f.h, mq);
  hq = fx_mad(g.h, q.h, hq);
  mq = fx_mad(g.h, q.l, mq);
  mq = fx_mad(g.l, q.h, mq);
  return ((hp - hq) << 3) + ((mp - mq) >> 29);
}

// row c = (a x b)^* of a 12-real link, written to its slots
__device__ __forceinline__ void fx_row3(FixedSlots& sm) {
  const int tid = threadIdx.x;
  Fx r[6], i[6];
#pragma unroll
  for (int c = 0; c < 6; ++c) {
    const int4 w = sm.lk[c][tid];
    r[c] = Fx{w.x, w.y};
    i[c] = Fx{w.z, w.w};
  }
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const int j = (c + 1) % 3, k = (c + 2) % 3;
    const Fx re = fx_split(fx_minor(r[j], r[3 + k], i[k], i[3 + j], i[j], i[3 + k], r[k], r[3 + j]));
    const Fx im = fx_split(fx_minor(r[k], i[3 + j], i[k], r[3 + j], r[j], i[3 + k], i[j], r[3 + k]));
    sm.lk[6 + c][tid] = make_int4(re.h, re.l, im.h, im.l);
  }
}

// The double (low word x, high word y) in the unit of the
// common exponent, e4 = E + 4: |x| 2^(59-(E-1023)) cut to an integer, 0 for a
// denormal or a zero, times the sign of x and of the mask `flip` (0 or -1).  A
// negative number is the one's complement of its magnitude, one unit (2^-59 of
// the largest component, an eighth of the unit of the sums) too low; a zero
// stays zero in the sums, which round.
__device__ __forceinline__ unsigned fx_xor3(unsigned a, unsigned b, unsigned c) {
  unsigned r;
  asm("lop3.b32 %0, %1, %2, %3, 0x96;" : "=r"(r) : "r"(a), "r"(b), "r"(c));
  return r;
}
__device__ __forceinline__ long long fx_number(unsigned x, unsigned y, int e4, int flip) {
  const int s = e4 - (int)((y >> 20) & 0x7ffu);
  const unsigned mh = __funnelshift_l(x, y, 11) | 0x80000000u;
  unsigned ml;  // x << 11 by the funnel shifter: the compiler's choice is the multiplier, which bounds the kernel
  asm("shf.l.clamp.b32 %0, 0, %1, 11;" : "=r"(ml) : "r"(x));
  const unsigned long long a = fx_shr(((unsigned long long)mh << 32) | ml, s);
  const int m = (int)y >> 31;
  const unsigned lo = fx_xor3((unsigned)a, m, flip), hi = fx_xor3((unsigned)(a >> 32), m, flip);
  return (long long)(((unsigned long long)hi << 32) | lo);
}

// largest of m and |a|, |b| read as floats: the high words of doubles order like
// floats, and an exponent above 2039 (infinities and NaN among them) reads as a
// NaN, which stays
__device__ __forceinline__ float fx_max(float m, unsigned a, unsigned b) {
  float r;
  asm("max.NaN.abs.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(m), "f"(__uint_as_float(a)), "f"(__uint_as_float(b)));
  return r;
}
// the biased exponent of the double whose high word gave m, plus 1
__device__ __forceinline__ int fx_exponent(float m) { return (int)(__float_as_uint(m) >> 20) + 1; }

// ------------------------------------------------------ products of two sites
// Inner products of a site's 24 doubles in integers, for kernels that the FP64
// pipe bounds.  A vector becomes integers of 58 bits in the unit of its largest
// exponent, each split into two signed halves; a product is three 32-bit
// multiply-adds (12 cycles or so of an SM quarter, an FP64 one 67), the product of
// the low halves dropped, and a site's 24 products are added exactly.
//
// Cutting (48), dropping (6) and rounding are at most 55 units of 2^-114 to 2^-116
// of 2^58 x 2^58, the two vectors' units; 24 FP64 multiply-adds may be off by 24 x
// 2^-53 of the sum of |w| |a|.  So the integers are no worse wherever that sum is
// 2^54.2 units or more, as a norm's always is (2^56), and the products of vectors
// whose large components do not meet are left to FP64 (fx_products).
constexpr int kFxSiteMinExp = 600, kFxSiteMaxExp = 1500;  // (biased) squares and scales stay normal doubles
constexpr int kFxDense = 5 << 18;  // 2^54.3 units as products of the halves' upper 12 bits
// biased exponent of the largest of 24 doubles; 24 zeros, as most sites of a point
// source are, count as in range, with an exponent of their own
__device__ __forceinline__ int fx_site_exp(const double (&x)[24]) {
  float m = 0.f;
#pragma unroll
  for (int k = 0; k < 24; k += 2) m = fx_max(m, (unsigned)__double2hiint(x[k]), (unsigned)__double2hiint(x[k + 1]));
  if (__float_as_uint(m) == 0u) {
    unsigned lo = 0u;
#pragma unroll
    for (int k = 0; k < 24; ++k) lo |= (unsigned)__double2loint(x[k]);
    return lo ? 0 : kFxSiteMinExp;
  }
  const int e = (int)(__float_as_uint(m) >> 20);
  return e == kFxSiteMinExp ? 0 : e;
}
__device__ __forceinline__ bool fx_site_ok(int e) { return e >= kFxSiteMinExp && e <= kFxSiteMaxExp; }
struct FxSite {
  int h[24], l[24];  // x 2^(1080-e) = h 2^29 + l
  int e;
  __device__ __forceinline__ FxSite(const double (&x)[24], int e) : e(e) {
#pragma unroll
    for (int k = 0; k < 24; ++k) {
      const long long v =
          fx_number((unsigned)__double2loint(x[k]), (unsigned)__double2hiint(x[k]), e + 6, 0) + (1 << 28);
      h[k] = (int)(v >> 29);
      l[k] = ((int)v & ((1 << 29) - 1)) - (1 << 28);
    }
  }
};
struct FxSum {
  long long hh = 0, hl = 0;
  __device__ __forceinline__ void add(int ah, int al, int bh, int bl) {
    hh = fx_mad(ah, bh, hh);
    hl = fx_mad(ah, bl, hl);
    hl = fx_mad(al, bh, hl);
  }
  __device__ __forceinline__ double value(int ea, int eb) const {
    const long long t = hh + ((hl + (1 << 28)) >> 29);
    return (double)t * __hiloint2double((ea + eb - 1079) << 20, 0);  // 2^(ea+eb-2102)
  }
};
// |a|^2 and <w, a> = sum conj(w) a
__device__ __forceinline__ double fx_norm2(const FxSite& a) {
  FxSum n;
#pragma unroll
  for (int k = 0; k < 24; ++k) n.add(a.h[k], a.l[k], a.h[k], a.l[k]);
  return n.value(a.e, a.e);
}
__device__ __forceinline__ double2 fx_dot(const FxSite& w, const FxSite& a) {
  FxSum re, im;
#pragma unroll
  for (int k = 0; k < 24; k += 2) {
    re.add(w.h[k], w.l[k], a.h[k], a.l[k]);
    re.add(w.h[k + 1], w.l[k + 1], a.h[k + 1], a.l[k + 1]);
    im.add(w.h[k], w.l[k], a.h[k + 1], a.l[k + 1]);
    im.add(-w.h[k + 1], -w.l[k + 1], a.h[k], a.l[k]);
  }
  return make_double2(re.value(w.e, a.e), im.value(w.e, a.e));
}

// the larger part of complex number k, the upper 12 bits of its upper half
__device__ __forceinline__ int fx_part(const FxSite& a, int k) { return max(abs(a.h[2 * k]), abs(a.h[2 * k + 1])) >> 17; }
// |a|^2 and <w, a>, or false where FP64 has to form them
__device__ __forceinline__ bool fx_products(const double (&wv)[24], const double (&av)[24], double& norm2, double2& dot) {
  const int ea = fx_site_exp(av), ew = fx_site_exp(wv);
  if (!fx_site_ok(ea) || !fx_site_ok(ew)) return false;
  const FxSite a(av, ea), w(wv, ew);
  int met = 0;
#pragma unroll
  for (int k = 0; k < 12; ++k) met += fx_part(w, k) * fx_part(a, k);
  norm2 = fx_norm2(a);
  dot = fx_dot(w, a);
  return met >= kFxDense || ea == kFxSiteMinExp || ew == kFxSiteMinExp;
}

__device__ __forceinline__ int fixed_neighbour(const Geom& g, int h, int x, int y, int z, int t, int k) {
  switch (k) {
    case 0: return (x == g.X - 1) ? h - (g.Xh - 1) : h + (x & 1);
    case 1: return (x == 0) ? h + (g.Xh - 1) : h - ((x & 1) ^ 1);
    case 2: return (y == g.Y - 1) ? h - g.wy : h + g.Xh;
    case 3: return (y == 0) ? h + g.wy : h - g.Xh;
    case 4: return (z == g.Z - 1) ? h - g.wz : h + g.XhY;
    case 5: return (z == 0) ? h + g.wz : h - g.XhY;
    case 6: return (t == g.T - 1) ? h - g.wt : h + g.XhYZ;
    default: return (t == 0) ? h + g.wt : h - g.XhYZ;
  }
}

// copies of hop k: the neighbour's spinor (the half a temporal hop reads), and
// the link (none for the unit links of the temporal gauge)
template <bool DAGGER>
__device__ __forceinline__ void fixed_issue_spinor(FixedSlots& sm, const SpinorF64& in, int n, int k) {
  const int tid = threadIdx.x;
  const bool lower = (k == 6) != DAGGER;  // the temporal hop's projector keeps spins 2, 3
  const double2* p = in.p + (size_t)((k >= 6 && lower) ? 6 : 0) * in.stride + n;
#pragma unroll
  for (int c = 0; c < 6; ++c) cp16_cg(&sm.sp[c][tid], p + (size_t)c * in.stride);
  if (k < 6) {
#pragma unroll
    for (int c = 6; c < 12; ++c) cp16_cg(&sm.sp[c][tid], p + (size_t)c * in.stride);
  }
}
__device__ __forceinline__ void fixed_issue_link(FixedSlots& sm, const GaugeX64& gauge, int parity, int h, int n,
                                                 int k) {
  const int tid = threadIdx.x;
  const int nc = gauge.recon >> 1;
  const int slot = ((k & 1) ? 1 - parity : parity) * 4 + (k >> 1);
  const int4* p = gauge.p + (size_t)slot * nc * gauge.stride + ((k & 1) ? n : h);
  const uint64_t pol = l2_evict_first();
#pragma unroll
  for (int c = 0; c < 6; ++c) cp16_cg_ef(&sm.lk[c][tid], p + (size_t)c * gauge.stride, pol);
  if (nc == 9) {
#pragma unroll
    for (int c = 6; c < 9; ++c) cp16_cg_ef(&sm.lk[c][tid], p + (size_t)c * gauge.stride, pol);
  }
}

// reconstruct() of row s: the upper row s of a hop, and the lower row that the
// projector makes of it.  CONJ: the row is that of the conjugate (backward hops,
// see dslash_site_fixed)
// weak[s] collects the weight (fixed_weight) of the rows that feed output spin s.
template <int MU, int S_, bool CONJ, int ROW>
__device__ __forceinline__ void fixed_add(const long long (&gr)[3], const long long (&gi)[3], int weight,
                                          long long (&a)[24], int (&weak)[4]) {
  constexpr int S = (MU == 1) ? -S_ : S_;
  constexpr int up = (MU == 3 && S_ < 0) ? 12 + 6 * ROW : 6 * ROW;
  constexpr int lo = (MU == 2) ? 12 + 6 * ROW : 18 - 6 * ROW;
  // lower row = t g (y) or t i g (x, z): x: -S for both rows, y: -S, S, z: -S, S
  constexpr int t = (MU == 0 || ROW == 0) ? -S : S;
  constexpr int ci = CONJ ? -1 : 1;
  weak[up / 6] += weight;
  if constexpr (MU != 3) weak[lo / 6] += weight;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    a[up + 2 * c] += gr[c];
    a[up + 2 * c + 1] += ci * gi[c];
    if constexpr (MU == 1) {
      a[lo + 2 * c] += t * gr[c];
      a[lo + 2 * c + 1] += t * ci * gi[c];
    } else if constexpr (MU != 3) {
      a[lo + 2 * c] += -t * ci * gi[c];
      a[lo + 2 * c + 1] += t * gr[c];
    }
  }
}

// The smallest colour of a row of h, by its larger part, in the unit of the high
// words: whatever the row of the link, no less than that (times sum |u| >= 1)
// goes into each colour that the row feeds.
__device__ __forceinline__ int fixed_weight(const long long (&hr)[3], const long long (&hi)[3]) {
  int w[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) w[c] = max(abs((int)(hr[c] >> 32)), abs((int)(hi[c] >> 32)));
  return __vimin3_s32(w[0], w[1], w[2]);
}
__device__ __forceinline__ bool fixed_is_outside(int top) { return top < kFixedMinExp || top > kFixedMaxExp; }
// An output spin that so little feeds that the unit of the sums may show in it
__device__ __forceinline__ bool fixed_is_weak(const int (&weak)[4]) {
  return min(min(weak[0], weak[1]), min(weak[2], weak[3])) < kFixedWeak;
}

// A site whose neighbours are zero (out = 0), or hold numbers the fixed-point form
// does not take (out = (D in)(h) in FP64).  Not inlined: the FP64
// arithmetic would be in every kernel that has the fixed-point one.
template <bool DAGGER, bool TFIX, bool PAIR>
__device__ __noinline__ void dslash_site_outside(Geom g, SpinorF64 in, GaugeX64 gauge, int h,
                                                 int parity, int top, double (&out)[24]) {
  if (top < kFixedMinExp) {
    int x, y, z, t;
    site_coords(g, h, parity, x, y, z, t);
    int nb[8];
    neighbours(g, h, x, y, z, t, nb);
    unsigned long long any = 0;
#pragma unroll
    for (int k = 0; k < 8; ++k)
#pragma unroll 1
      for (int c = 0; c < 12; ++c) {
        const ulonglong2 v = __ldg(reinterpret_cast<const ulonglong2*>(in.p + (size_t)c * in.stride + nb[k]));
        any |= (v.x | v.y) & 0x7fffffffffffffffull;
      }
    if (any == 0) {
#pragma unroll
      for (int k = 0; k < 24; ++k) out[k] = 0.0;
      return;
    }
  }
  dslash_site<DAGGER, TFIX, false, PAIR>(g, in, gauge.f64(), h, parity, out);
}

// Site h in FP64 by the warp's lanes 0 .. n - 1, all of which call this with the
// same site (a site with a spin that little feeds): one part (re, im) of one row of
// one hop per lane, 24 FP64 instructions each (56 with a third row to rebuild) and
// 7 for the sums, against some 614 in a row by the site's own thread, 20 us that
// the others of a launch then wait for.  The parts pass through the warp's spinor
// slots (216 doubles, 64 to a row of slots).  Not inlined: its registers would be in
// every kernel.
struct FixedScratch {
  FixedSlots& sm;
  int first;  // the warp's first thread
  __device__ __forceinline__ double& operator[](int i) const {
    return reinterpret_cast<double*>(&sm.sp[i >> 6][first])[i & 63];
  }
};
template <bool DAGGER, bool TFIX>
__device__ __noinline__ void dslash_site_weak(Geom g, SpinorF64 in, GaugeF64 gauge, FixedSlots& sm, int h, int parity,
                                              int n) {
  const int lane = threadIdx.x & 31;
  const unsigned lanes = 0xffffffffu >> (32 - n);
  const FixedScratch sc{sm, (int)threadIdx.x - lane};
  const int nc = gauge.recon >> 1;
  int x, y, z, t;
  site_coords(g, h, parity, x, y, z, t);
  __syncwarp(lanes);  // the slots are read
#pragma unroll 1
  for (int role = lane; role < 32; role += n) {
    const int k = role >> 2, row = (role >> 1) & 1, part = role & 1, mu = k >> 1;
    const bool fwd = (k & 1) == 0;
    const bool minus = fwd != DAGGER;  // S = -1
    const int nb = fixed_neighbour(g, h, x, y, z, t, k);
    // h = p + s q (y) or p + s i q (x, z), or twice p: its two parts in the order
    // that this part of the product takes them
    const int up = mu < 3 ? row : row + (minus ? 2 : 0);
    const int lo = mu == 2 ? 2 + row : 3 - row;  // the spin that joins a row, and that it gives
    const bool edge = mu == 3 && (fwd ? t == g.T - 1 : t == 0);
    const double s = minus != (row == 1 && mu != 0) ? -1.0 : 1.0;
    const double sr = mu == 1 ? s : -s, f = (edge && g.tbc_anti) ? -2.0 : 2.0;
    double a[3], b[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const double2 p = __ldg(in.p + (size_t)(3 * up + c) * in.stride + nb);
      double hr, hi;
      if (mu < 3) {
        const double2 q = __ldg(in.p + (size_t)(3 * lo + c) * in.stride + nb);
        hr = fma(sr, mu == 1 ? q.x : q.y, p.x);
        hi = fma(s, mu == 1 ? q.y : q.x, p.y);
      } else {
        hr = f * p.x;
        hi = f * p.y;
      }
      a[c] = part ? hi : hr;
      b[c] = part ? hr : -hi;
    }
    double v[3];
    if (TFIX && mu == 3 && !edge) {
#pragma unroll
      for (int c = 0; c < 3; ++c) v[c] = a[c];
    } else {
      const double2* l = gauge.p + (size_t)((fwd ? parity : 1 - parity) * 4 + mu) * nc * gauge.stride + (fwd ? h : nb);
      double u[18];
#pragma unroll
      for (int e = 0; e < 9; ++e) {
        const double2 d = e < nc ? __ldg(l + (size_t)e * gauge.stride) : make_double2(0.0, 0.0);
        u[2 * e] = d.x;
        u[2 * e + 1] = d.y;
      }
      if (nc == 6) reconstruct_row3(u);
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        v[c] = 0.0;
#pragma unroll
        for (int j = 0; j < 3; ++j) {
          const int e = 2 * (3 * c + j), et = 2 * (3 * j + c);  // U, or U^dag
          v[c] = fma(fwd ? u[e] : u[et], a[j], v[c]);
          v[c] = fma(fwd ? u[e + 1] : -u[et + 1], b[j], v[c]);
        }
      }
    }
    // to its own spin, and (spatial hops) to the other: s' v (y), or s' i v (x, z)
    const bool m1 = mu == 0 ? !minus : mu == 1 ? minus == (row == 0) : minus != (row == 0);
    const int to = mu == 1 ? part : 1 - part;
    const bool m2 = m1 != (mu != 1 && part == 1);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      sc[24 * k + 6 * up + 2 * c + part] = v[c];
      if (mu < 3) sc[24 * k + 6 * lo + 2 * c + to] = m2 ? -v[c] : v[c];
    }
  }
  __syncwarp(lanes);
  for (int q = lane; q < 24; q += n) {
    double v = sc[24 * ((q >= 12) != DAGGER ? 6 : 7) + q];
#pragma unroll
    for (int k = 0; k < 6; ++k) v += sc[24 * k + q];
    sc[192 + q] = v;
  }
  __syncwarp(lanes);
}

// out of the lanes in `todo`, whose sites are weakly fed, computed in FP64; the
// warp's lanes 0 .. n - 1 have consecutive sites
template <bool DAGGER, bool TFIX, bool PAIR>
__device__ __forceinline__ void dslash_weak_sites(const Geom& g, const SpinorF64& in, const GaugeX64& gauge,
                                                  FixedSlots& sm, int h, int parity, int n, unsigned todo,
                                                  double (&out)[24]) {
  const int lane = threadIdx.x & 31;
  if (__popc(todo) > kFixedShared) {
    if (todo >> lane & 1u) {
      double slow[24];
      dslash_site_outside<DAGGER, TFIX, PAIR>(g, in, gauge, h, parity, kFixedMinExp, slow);
#pragma unroll
      for (int k = 0; k < 24; ++k) out[k] = slow[k];
    }
    return;
  }
  while (todo) {
    const int l = __ffs(todo) - 1;
    todo &= todo - 1;
    dslash_site_weak<DAGGER, TFIX>(g, in, gauge.f64(), sm, h - lane + l, parity, n);
    if (lane == l) {
      const FixedScratch sc{sm, (int)threadIdx.x - lane};
#pragma unroll
      for (int k = 0; k < 24; ++k) out[k] = sc[192 + k];
    }
    __syncwarp(0xffffffffu >> (32 - n));
  }
}

// U h: the limbs of the two rows of h, the link in its slots read by rows (step
// 3, 1) or columns (1, 3); g in the unit of the sums
__device__ __forceinline__ void fixed_su3(const FixedSlots& sm, int step_i, int step_j, const long long (&hr)[2][3],
                                          const long long (&hi)[2][3], long long (&gr)[2][3], long long (&gi)[2][3]) {
  const int tid = threadIdx.x;
  Fx r[2][3], i[2][3], ni[2][3];
#pragma unroll
  for (int s = 0; s < 2; ++s)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      r[s][j] = fx_split(hr[s][j]);
      i[s][j] = fx_split(hi[s][j]);
      ni[s][j] = Fx{-i[s][j].h, ~i[s][j].l};  // -hi, one unit of 2^-59 low
    }
  const long long half = 1ll << 31;  // the middle sums are rounded to their high words
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    long long rh[2], ih[2], rm[2], im[2];
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      const int4 w = sm.lk[c * step_i + j * step_j][tid];
#pragma unroll
      for (int s = 0; s < 2; ++s) {
        rh[s] = fx_mad(w.x, r[s][j].h, j ? rh[s] : 0);
        rm[s] = fx_mad(w.x, r[s][j].l, j ? rm[s] : half);
        ih[s] = fx_mad(w.x, i[s][j].h, j ? ih[s] : 0);
        im[s] = fx_mad(w.x, i[s][j].l, j ? im[s] : half);
      }
#pragma unroll
      for (int s = 0; s < 2; ++s) {
        rm[s] = fx_mad(w.y, r[s][j].h, rm[s]);
        im[s] = fx_mad(w.y, i[s][j].h, im[s]);
        rh[s] = fx_mad(w.z, ni[s][j].h, rh[s]);
        ih[s] = fx_mad(w.z, r[s][j].h, ih[s]);
      }
#pragma unroll
      for (int s = 0; s < 2; ++s) {
        rm[s] = fx_mad(w.z, ni[s][j].l, rm[s]);
        im[s] = fx_mad(w.z, r[s][j].l, im[s]);
        rm[s] = fx_mad(w.w, ni[s][j].h, rm[s]);
        im[s] = fx_mad(w.w, r[s][j].h, im[s]);
      }
    }
#pragma unroll
    for (int s = 0; s < 2; ++s) {
      gr[s][c] = rh[s] + (int)(rm[s] >> 32);
      gi[s][c] = ih[s] + (int)(im[s] >> 32);
    }
  }
}

// the sums move to the exponent of a hop that needs a larger one
__device__ __forceinline__ void fixed_raise(float m, int& E, int& top, long long (&acc)[24], int (&weak)[4]) {
  const int e = fx_exponent(m);
  top = max(top, e);
  if (e > E) {
#pragma unroll
    for (int q = 0; q < 24; ++q) acc[q] = fx_round_sar(acc[q], e - E);
#pragma unroll
    for (int s = 0; s < 4; ++s) weak[s] = fx_shr32(weak[s], e - E);
    E = e;
  }
}

// dslash_site in fixed point.  Two loops, over the six spatial and the two
// temporal hops: unrolled, a site is 7600 instructions that the instruction
// caches do not hold, and the warps wait for instructions longer than for
// anything else.  The directions differ in which lower spin row joins which
// upper one (a choice of slots), in signs (masks of the conversion) and in the
// rows that the sums go to (a branch that all threads take alike).
//
// A backward hop takes U^dag h as the conjugate of U^T h^*: the same product
// with the link read by columns, the projection's imaginary parts negated as
// they are converted, and the result's as they are added.
//
// The hops k0 .. k1 - 1 of a site (0, 8: all), in the unit of E; top: the largest
// exponent met; weak: what feeds each output spin.
template <bool DAGGER, bool TFIX>
__device__ __forceinline__ void fixed_hops(const Geom& g, const SpinorF64& in, const GaugeX64& gauge, FixedSlots& sm,
                                           int h, int parity, int k0, int k1, int& E, int& top,
                                           long long (&acc)[24], int (&weak)[4]) {
  constexpr int SF = DAGGER ? +1 : -1;  // the projector sign of the forward hops
  const int tid = threadIdx.x;
  int x, y, z, t;
  site_coords(g, h, parity, x, y, z, t);
  const bool last = (t == g.T - 1), first = (t == 0);
#pragma unroll
  for (int k = 0; k < 24; ++k) acc[k] = 0;
#pragma unroll
  for (int s = 0; s < 4; ++s) weak[s] = 0;
  E = kFixedMinExp;
  top = 0;
  const int n = fixed_neighbour(g, h, x, y, z, t, k0);
  fixed_issue_spinor<DAGGER>(sm, in, n, k0);
  cp_commit();
  if (!(TFIX && k0 == 6 && !last)) fixed_issue_link(sm, gauge, parity, h, n, k0);
  cp_commit();
#pragma unroll 1
  for (int k = k0; k < min(k1, 6); ++k) {
    const int mu = k >> 1;
    const bool fwd = (k & 1) == 0;
    cp_wait<1>();  // the spinor of hop k
    {
      float m = 0.f;
#pragma unroll
      for (int c = 0; c < 12; ++c) {
        const uint4 w = sm.sp[c][tid];
        m = fx_max(m, w.y, w.w);
      }
      if (k == k0) E = max(fx_exponent(m), kFixedMinExp) + 1;
      fixed_raise(m, E, top, acc, weak);
    }
    // rows 0, 1 and their partners: row 0 joins spin 3 (x, y) or 2 (z), row 1
    // the other; a real part joins a real one (y) or an imaginary one (x, z)
    const uint2* p = reinterpret_cast<const uint2*>(&sm.sp[0][tid]);
    const int qr = (mu == 1) ? 0 : 1, qi = 1 - qr;
    // sign masks.  cj: imaginary parts of a backward hop; sp: the sign S of the
    // projector; x: h0 = p0 + S i p3, h1 = p1 + S i p2; y: h0 = p0 + S p3,
    // h1 = p1 - S p2; z: h0 = p0 + S i p2, h1 = p1 - S i p3
    const int cj = fwd ? 0 : -1;
    const int sp = (fwd != DAGGER) ? -1 : 0;
    const int e4 = E + 4;
    const int step_i = fwd ? 3 : 1, step_j = fwd ? 1 : 3;
    long long hr[2][3], hi[2][3];
#pragma unroll
    for (int s = 0; s < 2; ++s) {
      const int q = ((mu == 2) == (s == 1) ? 9 : 6) * (2 * kFixedBlock);
      const int fr = s ? ((mu == 2) ? sp : ~sp) : ((mu == 1) ? sp : ~sp);
      const int fi = (s && mu != 0) ? ~sp ^ cj : sp ^ cj;
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const uint4 w = sm.sp[3 * s + c][tid];
        const uint2 vr = p[q + c * 2 * kFixedBlock + qr], vi = p[q + c * 2 * kFixedBlock + qi];
        hr[s][c] = fx_number(w.x, w.y, e4, 0) + fx_number(vr.x, vr.y, e4, fr);
        hi[s][c] = fx_number(w.z, w.w, e4, cj) + fx_number(vi.x, vi.y, e4, fi);
      }
    }
    const int w0 = fixed_weight(hr[0], hi[0]), w1 = fixed_weight(hr[1], hi[1]);
    // the next hop's spinor takes the slots just read
    int nn = 0;
    if (k + 1 < k1) {
      nn = fixed_neighbour(g, h, x, y, z, t, k + 1);
      fixed_issue_spinor<DAGGER>(sm, in, nn, k + 1);
    }
    cp_commit();
    cp_wait<1>();  // the link of hop k
    if (gauge.recon == 12) fx_row3(sm);
    long long gr[2][3], gi[2][3];
    fixed_su3(sm, step_i, step_j, hr, hi, gr, gi);
    if (k + 1 < k1 && !(TFIX && k == 5 && !last)) fixed_issue_link(sm, gauge, parity, h, nn, k + 1);
    cp_commit();
#define WD_FIXED_ADD(MU, S, CONJ)                                \
  fixed_add<MU, S, CONJ, 0>(gr[0], gi[0], w0, acc, weak);        \
  fixed_add<MU, S, CONJ, 1>(gr[1], gi[1], w1, acc, weak)
    switch (k) {
      case 0: WD_FIXED_ADD(0, SF, false); break;
      case 1: WD_FIXED_ADD(0, -SF, true); break;
      case 2: WD_FIXED_ADD(1, SF, false); break;
      case 3: WD_FIXED_ADD(1, -SF, true); break;
      case 4: WD_FIXED_ADD(2, SF, false); break;
      default: WD_FIXED_ADD(2, -SF, true); break;
    }
  }
#pragma unroll 1
  for (int k = max(k0, 6); k < k1; ++k) {
    const bool fwd = k == 6;
    cp_wait<1>();
    {
      float m = 0.f;
#pragma unroll
      for (int c = 0; c < 6; ++c) {
        const uint4 w = sm.sp[c][tid];
        m = fx_max(m, w.y, w.w);
      }
      if (k == k0) E = max(fx_exponent(m), kFixedMinExp) + 1;
      fixed_raise(m, E, top, acc, weak);
    }
    const bool unit = TFIX && (fwd ? !last : !first);
    const int fm = (g.tbc_anti && (fwd ? last : first)) ? -1 : 0;
    const int cj = (fwd || unit) ? fm : ~fm;
    long long hr[2][3], hi[2][3];
#pragma unroll
    for (int q = 0; q < 6; ++q) {  // twice the component: the projector is 2
      const uint4 w = sm.sp[q][tid];
      hr[q / 3][q % 3] = fx_number(w.x, w.y, E + 3, fm);
      hi[q / 3][q % 3] = fx_number(w.z, w.w, E + 3, cj);
    }
    const int w0 = fixed_weight(hr[0], hi[0]), w1 = fixed_weight(hr[1], hi[1]);
    int nn = 0;
    if (fwd) {
      nn = fixed_neighbour(g, h, x, y, z, t, 7);
      fixed_issue_spinor<DAGGER>(sm, in, nn, 7);
    }
    cp_commit();
    cp_wait<1>();
    long long gr[2][3], gi[2][3];
    if (unit) {
#pragma unroll
      for (int q = 0; q < 6; ++q) {
        gr[q / 3][q % 3] = (hr[q / 3][q % 3] + 4) >> 3;
        gi[q / 3][q % 3] = (hi[q / 3][q % 3] + 4) >> 3;
      }
    } else {
      if (gauge.recon == 12) fx_row3(sm);
      fixed_su3(sm, fwd ? 3 : 1, fwd ? 1 : 3, hr, hi, gr, gi);
      if (!fwd) {
#pragma unroll
        for (int q = 0; q < 6; ++q) gi[q / 3][q % 3] = -gi[q / 3][q % 3];
      }
    }
    if (fwd && !(TFIX && !first)) fixed_issue_link(sm, gauge, parity, h, nn, 7);
    cp_commit();
    if (fwd) {
      WD_FIXED_ADD(3, SF, false);
    } else {
      WD_FIXED_ADD(3, -SF, false);
    }
  }
#undef WD_FIXED_ADD
}

// out = (D in)(h) for this thread's site; the warp's lanes 0 .. n - 1 have one
template <bool DAGGER, bool TFIX, bool PAIR>
__device__ __forceinline__ void dslash_site_fixed(const Geom& g, const SpinorF64& in, const GaugeX64& gauge,
                                                  FixedSlots& sm, int h, int parity, int n, double (&out)[24]) {
  int E, top, weak[4];
  long long acc[24];
  fixed_hops<DAGGER, TFIX>(g, in, gauge, sm, h, parity, 0, 8, E, top, acc, weak);
  const bool outside = fixed_is_outside(top);
  if (outside) {
    double slow[24];  // its address is taken on this path only
    dslash_site_outside<DAGGER, TFIX, PAIR>(g, in, gauge, h, parity, top, slow);
#pragma unroll
    for (int k = 0; k < 24; ++k) out[k] = slow[k];
  } else {
#pragma unroll
    for (int k = 0; k < 24; ++k) out[k] = fx_sum_value(acc[k], E - 1079);
  }
  const unsigned todo = __ballot_sync(0xffffffffu >> (32 - n), !outside && fixed_is_weak(weak));
  dslash_weak_sites<DAGGER, TFIX, PAIR>(g, in, gauge, sm, h, parity, n, todo, out);
}

// The same with four warps for 32 sites, warp w taking the two hops of direction
// w: a lattice that gives an SM no more than a warp or two per quarter is bound
// by the latency of one thread's eight hops.  The partial sums pass through the
// slots; warp w adds and converts spin w, and the threads of warp 0 get the
// result (true) of sites below h_end.
template <bool DAGGER, bool TFIX, bool PAIR>
__device__ __forceinline__ bool dslash_site_fixed_split(const Geom& g, const SpinorF64& in, const GaugeX64& gauge,
                                                        FixedSlots& sm, int h0, int h_end, int parity,
                                                        double (&out)[24]) {
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5, h = h0 + lane;
  const bool ok = h < h_end;
  if (ok) {
    int E, top, weak[4];
    long long acc[24];
    fixed_hops<DAGGER, TFIX>(g, in, gauge, sm, h, parity, 2 * w, 2 * w + 2, E, top, acc, weak);
#pragma unroll
    for (int c = 0; c < 12; ++c)
      *reinterpret_cast<longlong2*>(&sm.sp[c][tid]) = make_longlong2(acc[2 * c], acc[2 * c + 1]);
    sm.lk[0][tid] = make_int4(E, top, 0, 0);
    sm.lk[4][tid] = make_int4(weak[0], weak[1], weak[2], weak[3]);
  }
  __syncthreads();
  double* fin = reinterpret_cast<double*>(&sm.lk[1][0]);  // [24][32]
  const int n = min(32, h_end - h0);
  int top = 0;
  if (ok) {
    int e[4], E = 0;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int4 v = sm.lk[0][lane + 32 * q];
      e[q] = v.x;
      E = max(E, v.x);
      top = max(top, v.y);
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      long long r = 0, i = 0;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const longlong2 v = *reinterpret_cast<const longlong2*>(&sm.sp[3 * w + c][lane + 32 * q]);
        r += fx_round_sar(v.x, E - e[q]);
        i += fx_round_sar(v.y, E - e[q]);
      }
      fin[(6 * w + 2 * c) * 32 + lane] = fx_sum_value(r, E - 1079);
      fin[(6 * w + 2 * c + 1) * 32 + lane] = fx_sum_value(i, E - 1079);
    }
    int feeds = 0;
#pragma unroll
    for (int q = 0; q < 4; ++q) feeds += fx_shr32(reinterpret_cast<const int*>(&sm.lk[4][lane + 32 * q])[w], E - e[q]);
    const unsigned weak_w = __ballot_sync(0xffffffffu >> (32 - n), feeds < kFixedWeak && !fixed_is_outside(top));
    if (lane == 0) reinterpret_cast<unsigned*>(&sm.lk[5][0])[w] = weak_w;
  }
  __syncthreads();
  if (!ok || w != 0) return false;
  if (fixed_is_outside(top)) {
    double slow[24];
    dslash_site_outside<DAGGER, TFIX, PAIR>(g, in, gauge, h, parity, top, slow);
#pragma unroll
    for (int k = 0; k < 24; ++k) out[k] = slow[k];
  } else {
#pragma unroll
    for (int k = 0; k < 24; ++k) out[k] = fin[k * 32 + lane];
  }
  const int4 f = sm.lk[5][0];
  dslash_weak_sites<DAGGER, TFIX, PAIR>(g, in, gauge, sm, h, parity, n, (unsigned)(f.x | f.y | f.z | f.w), out);
  return true;
}

// epi on (D in)(h) for the sites [h_begin, h_end) of a launch
template <bool DAGGER, bool TFIX, bool SPLIT, class Epi>
__device__ __forceinline__ void dslash_sites_fixed(const Geom& g, const SpinorF64& in, const GaugeX64& gauge,
                                                   int h_begin, int h_end, int parity, const Epi& epi, double* red) {
  __shared__ FixedSlots sm;
  constexpr bool kPair = Epi::NRED == 0;
  double acc[24];
  if constexpr (SPLIT) {
    for (int h0 = h_begin + blockIdx.x * 32; h0 < h_end; h0 += gridDim.x * 32) {
      if (dslash_site_fixed_split<DAGGER, TFIX, kPair>(g, in, gauge, sm, h0, h_end, parity, acc))
        epi(h0 + (int)threadIdx.x, acc, red);
      __syncthreads();  // the slots are read: the next tile's copies may start
    }
  } else {
    for (int h = h_begin + blockIdx.x * blockDim.x + threadIdx.x; h < h_end; h += gridDim.x * blockDim.x) {
      dslash_site_fixed<DAGGER, TFIX, kPair>(g, in, gauge, sm, h, parity, min(32, h_end - h + (int)(threadIdx.x & 31)),
                                             acc);
      epi(h, acc, red);
    }
  }
}

}  // namespace wd
