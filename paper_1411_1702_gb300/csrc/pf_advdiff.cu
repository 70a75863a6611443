// pf_advdiff.cu -- stage kernels of the epoch for the paper's 2D
// advection-diffusion system (Sec. 4): U' = L U on the periodic nt x nt grid,
//   L = -{k1^2 B1'B1 + k1 k3 (B1'B2 + B2'B1) + (k2^2 + k3^2) B2'B2} + c1 B1 + c2 B2,
// B1 = I (x) ell, B2 = ell (x) I, (ell u)_j = u_j - u_{j-1} (periodic), state
// U[iy*nt + ix], theta = (k1, k2, k3, c1, c2).
//
// L is built from circulant difference matrices, so the 2D DFT diagonalises
// it: with a(m) = 1 - exp(-2 pi i m / nt) the symbol of ell,
//   lambda(mx, my) = -(k1^2 |a_x|^2 + 2 k1 k3 Re(conj(a_x) a_y) + (k2^2 + k3^2) |a_y|^2)
//                    + c1 a_x + c2 a_y.
// The system is linear, so Newton's method with the exact Jacobian L solves
// each implicit BDF step in one iteration (Sec. 2.1), and the solution of
//   x_{n+1} - rho1 x_n - rho2 x_{n-1} = gamma L x_{n+1}
// is, mode by mode, X_{n+1} = (rho1 X_n + rho2 X_{n-1}) / (1 - gamma lambda).
// Every quantity of an interval's S substeps is a fixed linear combination of
// the modes of (x_n, x_{n-1}, x_{n-2}): the predictor pi0 X_n + pi1 X_{n-1} +
// pi2 X_{n-2}, the explicit-Euler predictor (1 + h lambda) X_n of a cold
// start, the corrector, and Milne's estimate mu (X_{n+1} - X_p).  So each
// particle's history is transformed once at the interval's start and stays in
// the Fourier basis, each thread stepping its own modes in registers through
// all S substeps; only what is needed in physical space is transformed back:
// the final states, and in stage 2 each substep's local error, whose squares
// are summed per grid point (Step 4b: Gamma = kappa diag(sum_s e_s^2)).
//
// What FP64 is needed for (an FP64 instruction costs the time of 64 FP32 ones on
// GB300, a 32x32-bit integer multiply-add into 64 bits that of five or six):
//  - the mode steps X_{n+1} = W (X_n + kappa X_{n-1}), W = rho1/(1 - gamma lambda)
//    complex, kappa = rho2/rho1: 8 FP64 instructions a mode.  The substeps of a
//    uniform grid have gammas that differ in their last bits; W is formed for the
//    first and the others' difference applied to first order in FP32.
//  - Milne's estimate mu (X_{n+1} - X_p) while it is not small beside the state:
//    the first three or four substeps of an interval, whose innovation left noise in
//    the stiff modes.  Afterwards it is formed in pairs of floats (pf_ff.cuh) from
//    the differences D of the states, to 2^-48 of itself.
// The transforms, most of the arithmetic, are integer sums in block floating point:
// a field is scaled by its largest value to 54-bit integers, split in two parts
// of 28 bits, and so is the twiddle table; three products a term (the product of the
// low parts, 2^-56 of the scale, is dropped), exact sums.  That is as accurate as
// FP64 sums, whose roundings are of the same size, at a quarter of their time.  The
// history is transformed as x_n and the differences D1 = x_n - x_{n-1}, D2 = x_{n-1} -
// x_{n-2}, each at its own scale.
//
// Transforms.  nt is odd and the state real, so the half spectrum mx =
// 0..H-1, H = (nt+1)/2, carries everything.  The transforms are direct sums
// over a cos/sin table (nt is small and prime or nearly so), organised by
// the symmetry of the twiddles: the terms of indices m and nt - m share their
// cosine and have opposite sines, so
//   sum_m z_m e^{+i phi m k} = z_0 + sum_{m=1}^{H-1} [(z_m + z_{nt-m}) cos(phi m k)
//                                              + i (z_m - z_{nt-m}) sin(phi m k)],
// and the outputs k and nt - k differ only in the sign of the sine part.
// The forward transform of a real field folds both axes as it is loaded: of
// u(+-iy, +-ix) the four sums and differences, H^2 of each.
// One work unit computes an output pair from the sum and difference
// of an input pair: 4 (H-1) products for two complex outputs instead of 8 nt.
// A thread owns the mode pairs (my, mx) and (nt - my, mx) of its units, in
// registers, so the forward transform ends and the inverse begins in the
// owning thread.
//
// A block advances PB particles (1, 2 or 4: on small grids several
// particles fill the block's warps), all in step through the same substeps.
// Shared memory holds the substep tables and the twiddle tables, and per
// particle the folded fields, the pair buffers of the transforms and in
// stage 2 the error sums.  Global memory is touched once per particle per
// stage.
#include "pf_epoch.cuh"
#include "pf_fast.cuh"
#include "pf_kernels.h"

namespace pfg {

constexpr int kAdMaxSide = 45;
constexpr int kAdMaxUnitsPerThread = 2;  // mode-pair units a thread steps in registers

__host__ __device__ inline int ad_side(int d) {
  for (int nt = 3; nt <= kAdMaxSide; nt += 2)
    if (nt * nt == d) return nt;
  return 0;
}

// What a substep adds to its StepCoef: kappa = rho2/rho1, the differences of
// gamma and rho1 from the substep whose W serves (StepCoef::ref), and the
// estimate's weights, mu with the inverse transform's 1/d.
struct AdCoef {
  double kappa;
  float dgamma, drho;  // gamma - gamma_ref, rho1/rho1_ref - 1
  ff pa, pb, mu;
};

// Shared-memory layout of one block, in doubles: the substep tables and the
// twiddle tables, then one region per particle of the block.
struct AdLayout {
  int nt, d, H, PB;
  int sc;    // step table, S entries
  int ac;    // its AdCoef entries
  int tw;    // cos(2 pi k / nt), then sin(2 pi k / nt), k < nt
  int twx;   // the same as integers of scale 2^54
  int base;  // particle 0's region; particle q's is at base + q * per
  int per;   // doubles per particle region
  // offsets within a particle's region:
  int F[3];  // folded x_n, D1, D2 (4 H^2 each); afterwards x + v by grid point; the FP64
             // error sums, then the running state; the ff error sums, then v
  int ps;    // pair sums [p][mx] (complex), p < H; p = 0 holds the unpaired entry
  int pd;    // pair differences [p][mx] (complex)
  int cy;    // inverse columns [iy][mx] (complex), iy < nt
  int total;
};

__host__ __device__ inline AdLayout ad_layout(int d, int S, int PB) {
  AdLayout L;
  L.nt = ad_side(d);
  L.d = d;
  L.H = (L.nt + 1) / 2;
  L.PB = PB;
  int off = 0;
  L.sc = off;
  off += S * (int)(sizeof(StepCoef) / sizeof(double));
  L.ac = off;
  off += S * (int)(sizeof(AdCoef) / sizeof(double));
  L.tw = off;
  off += 2 * L.nt;
  L.twx = off;
  off += 2 * L.nt;
  L.base = off;
  int r = 0;
  for (int k = 0; k < 3; ++k) {
    L.F[k] = r;
    r += 4 * L.H * L.H;  // at least d
  }
  L.ps = r;
  r += 2 * L.H * L.H;
  L.pd = r;
  r += 2 * L.H * L.H;
  L.cy = r;
  r += 2 * L.nt * L.H;
  L.per = r;
  L.total = off + PB * r;
  return L;
}

// The operator's Fourier symbol for one parameter vector.
struct AdOp {
  double kxx, kxy, kyy, c1, c2;  // k1^2, k1 k3, k2^2 + k3^2, c1, c2
};

__device__ __forceinline__ AdOp ad_op(const double* th) {
  const double k1 = th[0], k2 = th[1], k3 = th[2];
  AdOp o;
  o.kxx = k1 * k1;
  o.kxy = k1 * k3;
  o.kyy = fma(k2, k2, k3 * k3);
  o.c1 = th[3];
  o.c2 = th[4];
  return o;
}

// lambda(mx, my)
__device__ __forceinline__ void ad_lambda(const AdLayout& L, const AdOp& o, const double* tw, int my,
                                          int mx, double& lr, double& li) {
  const int nt = L.nt;
  const double axr = 1.0 - tw[mx], axi = tw[nt + mx];
  const double ayr = 1.0 - tw[my], ayi = tw[nt + my];
  const double ax2 = fma(axr, axr, axi * axi), ay2 = fma(ayr, ayr, ayi * ayi);
  const double cr = fma(axr, ayr, axi * ayi);
  lr = fma(o.c1, axr, o.c2 * ayr) - fma(o.kxx, ax2, fma(2.0 * o.kxy, cr, o.kyy * ay2));
  li = fma(o.c1, axi, o.c2 * ayi);
}

// ------------------------------------------------ block floating point
// Z = h 2^28 + l, |l| <= 2^27
struct Fx {
  int32_t h, l;
};
__device__ __forceinline__ Fx fx_split(long long Z) {
  const int32_t h = (int32_t)((Z + (1ll << 27)) >> 28);
  return Fx{h, (int32_t)Z - (h << 28)};
}
__device__ __forceinline__ long long fx_join(Fx z) { return ((long long)z.h << 28) + z.l; }

// A field's scale: every |value| < 2^e, from the largest high word (without
// sign) of its doubles.
__device__ __forceinline__ int fx_scale(unsigned hi_max) {
  const int e = (int)(hi_max >> 20) - 1022;
  return e < -900 ? -900 : e;
}
// 2^(e + k) of it, NaN if a value was not finite
__device__ __forceinline__ double fx_unit(unsigned hi_max, int k) {
  return hi_max >= 0x7ff00000u ? CUDART_NAN : d_from((uint32_t)(fx_scale(hi_max) + k + 1023) << 20, 0u);
}
__device__ __forceinline__ unsigned hi_abs(double v) { return d_hi(v) & 0x7fffffffu; }

// round(v 2^(B - e)) on the integer pipe
template <int B>
__device__ __forceinline__ long long fx_of(double v, int e) {
  const uint32_t hi = d_hi(v);
  const int E = (int)((hi >> 20) & 0x7ffu);
  const unsigned long long m = ((((unsigned long long)((hi & 0xfffffu) | 0x100000u)) << 32) | d_lo(v)) << (B - 53);
  int rs = e + 1022 - E;
  rs = rs < 0 ? 0 : rs > 63 ? 63 : rs;
  const long long r = (long long)((m + ((1ull << rs) >> 1)) >> rs);
  return (int32_t)hi < 0 ? -r : r;
}
// round(v 2^(57 - e)) of a pair of floats (to its own 48 bits), s = 2^(26 - e)
template <int B>
__device__ __forceinline__ long long fx_of(ff v, float s) {
  static_assert(B == 57, "the inverse's scale");
  const int32_t h = __float2int_rn(f_mul(v.h, s));
  const float r = f_add(f_fma(v.h, s, -(float)h), f_mul(v.l, s));
  return (((long long)h << 28) + __float2int_rn(f_mul(r, 0x1.0p28f))) << 3;
}

// A sum of products z c with the twiddles c (scale 2^54): a collects the high
// parts, m the mixed ones at 2^-28 of them.  The sum is a + m 2^-28 in units of
// four of z's.  Bounds: |z| <= 2^58.5 (see ad_inverse), |c| <= 2^54 and at most 22
// terms keep a below 2^61 and m below 2^62.
struct FxSum {
  long long a, m;
};
__device__ __forceinline__ FxSum fx_start(Fx z) { return FxSum{(long long)z.h << 26, (long long)z.l << 26}; }
__device__ __forceinline__ void accumulate(FxSum& s, Fx z, Fx c) {
  s.a += (long long)z.h * c.h;
  s.m += (long long)z.h * c.l;
  s.m += (long long)z.l * c.h;
}
__device__ __forceinline__ long long fx_round(const FxSum& s) { return s.a + ((s.m + (1ll << 27)) >> 28); }
// in units of two of z's
__device__ __forceinline__ long long fx_round2(const FxSum& s) { return 2 * s.a + ((s.m + (1ll << 26)) >> 27); }

// A thread's modes: work item t = q * H^2 + p * H + mx (particle q of the
// block) holds mode A = (my = p, mx) and, for p >= 1, mode B = (my = nt - p,
// mx).  Index [j][0] is A, [j][1] is B, for the items t = tid + j T (one particle's:
// U = 2 only with one particle a block).
template <class V, int U>
struct Modes {
  V re[U][2], im[U][2];
};
__device__ __forceinline__ int ad_own(int tid, int units, int PB) {
  const int q = tid / units;
  return q < PB ? q : PB - 1;
}

// Folded field at (p, k), p, k < H, from u(iy, ix), iy = +-p, ix = +-k: the sums
// and differences over the axes, [0] even-even, [1] even in y, odd in x, [2] odd in
// y, even in x, [3] odd-odd, in four arrays of H^2.
// a = u(p, k), b = u(p, -k), c = u(-p, k), d = u(-p, -k)
__device__ __forceinline__ void ad_fold(Fx* F, int units, int v, bool y0, bool x0, int e, double a, double b, double c,
                                        double d) {
  const long long A = fx_of<54>(a, e), B = x0 ? 0 : fx_of<54>(b, e), C = y0 ? 0 : fx_of<54>(c, e),
                  D = x0 || y0 ? 0 : fx_of<54>(d, e);
  F[v] = fx_split((A + B) + (C + D));
  F[units + v] = x0 ? Fx{0, 0} : fx_split((A - B) + (C - D));
  F[2 * units + v] = y0 ? Fx{0, 0} : fx_split((A + B) - (C + D));
  F[3 * units + v] = x0 || y0 ? Fx{0, 0} : fx_split((A - B) - (C - D));
}

__device__ __forceinline__ void ad_fold(double* F, int units, int v, bool y0, bool x0, double a, double b, double c,
                                        double d) {
  const double s = x0 ? a : a + b, t = x0 ? 0.0 : a - b, w = x0 ? c : c + d, z = x0 ? 0.0 : c - d;
  F[v] = y0 ? s : s + w;
  F[units + v] = y0 ? t : t + z;
  F[2 * units + v] = y0 ? 0.0 : s - w;
  F[3 * units + v] = y0 ? 0.0 : t - z;
}

// The forward transform's two arithmetics: integers for the differences, FP64 for
// the state itself (a field with a few high peaks has most of its points far
// below the scale, where integers would lose what FP64 keeps: the cold start's
// estimate multiplies the state's high modes by h lambda).
struct InFx {
  using V = Fx;
  using S = FxSum;
  __device__ __forceinline__ static S start(V z) { return fx_start(z); }
  __device__ __forceinline__ static S none() { return S{0, 0}; }
  __device__ __forceinline__ static V keep(const S& s) { return fx_split(fx_round(s)); }
  __device__ __forceinline__ static V keep_neg(const S& s) { return fx_split(-fx_round(s)); }
  __device__ __forceinline__ static double sum(const S& a, const S& b, double unit) {
    return (double)(fx_round2(a) + fx_round2(b)) * unit;
  }
  __device__ __forceinline__ static double diff(const S& a, const S& b, double unit) {
    return (double)(fx_round2(a) - fx_round2(b)) * unit;
  }
};
__device__ __forceinline__ void accumulate(double& s, double z, double c) { s = fma(z, c, s); }
struct InFp64 {
  using V = double;
  using S = double;
  __device__ __forceinline__ static S start(V z) { return z; }
  __device__ __forceinline__ static S none() { return 0.0; }
  __device__ __forceinline__ static V keep(S s) { return s; }
  __device__ __forceinline__ static V keep_neg(S s) { return -s; }
  __device__ __forceinline__ static double sum(S a, S b, double) { return a + b; }
  __device__ __forceinline__ static double diff(S a, S b, double) { return a - b; }
};

// Forward real 2D DFT of a folded field (region `field`; in integers unit is 2^(e -
// 51) of the thread's own particle) of every particle of the block into the
// calling thread's own modes:
//   X(my, mx) = sum_{iy,ix} u[iy][ix] exp(-i phi (mx ix + my iy)).
// Ends with a barrier.
template <class P, int U>
__device__ void ad_forward(const AdLayout& L, double* sm, int field, int table, double unit, Modes<double, U>& out) {
  using V = typename P::V;
  using Sum = typename P::S;
  const int nt = L.nt, H = L.H, T = blockDim.x, tid = threadIdx.x, units = H * H;
  const int items = L.PB * units;
  const V* tw = reinterpret_cast<const V*>(sm + table);
  // along x: row pairs' sums (cosines of the even part, minus sines of the odd) and
  // differences
  for (int t = tid; t < items; t += T) {
    const int q = t / units, v = t - q * units;
    double* R = sm + L.base + q * L.per;
    const V* F = reinterpret_cast<const V*>(R + field);
    V* ps = reinterpret_cast<V*>(R + L.ps);
    V* pd = reinterpret_cast<V*>(R + L.pd);
    const int py = v / H, mx = v - py * H;
    const V *ee = F + py * H, *eo = ee + units, *oe = eo + units, *oo = oe + units;
    Sum r1 = P::start(ee[0]), i1 = P::none(), r2 = P::start(oe[0]), i2 = P::none();
    int k = mx;
    for (int ix = 1; ix < H; ++ix) {
      const V cs = tw[k], sn = tw[nt + k];
      accumulate(r1, ee[ix], cs);
      accumulate(i1, eo[ix], sn);
      accumulate(r2, oe[ix], cs);
      accumulate(i2, oo[ix], sn);
      k += mx;
      if (k >= nt) k -= nt;
    }
    ps[2 * v] = P::keep(r1);
    ps[2 * v + 1] = P::keep_neg(i1);
    pd[2 * v] = P::keep(r2);
    pd[2 * v + 1] = P::keep_neg(i2);
  }
  __syncthreads();
  // columns: X(my) = R0 + sum_{iy=1}^{H-1} [s_iy cos(phi my iy) - i d_iy sin(phi my iy)]
  // for my = p, and the conjugate sine part for my = nt - p
#pragma unroll
  for (int j = 0; j < U; ++j) {
    const int t = tid + j * T;
    Sum cr = P::none(), ci = P::none(), dr = P::none(), di = P::none();
    if (t < items) {
      const int q = t / units, v = t - q * units;
      const double* R = sm + L.base + q * L.per;
      const V* ps = reinterpret_cast<const V*>(R + L.ps);
      const V* pd = reinterpret_cast<const V*>(R + L.pd);
      const int p = v / H, mx = v - p * H;
      cr = P::start(ps[2 * mx]);
      ci = P::start(ps[2 * mx + 1]);
      int k = p;
      for (int iy = 1; iy < H; ++iy) {
        const int o = 2 * (iy * H + mx);
        const V cs = tw[k], sn = tw[nt + k];
        accumulate(cr, ps[o], cs);
        accumulate(ci, ps[o + 1], cs);
        accumulate(dr, pd[o], sn);
        accumulate(di, pd[o + 1], sn);
        k += p;
        if (k >= nt) k -= nt;
      }
    }
    // A: C - i D, B: C + i D (no B, whose size would count in the scales, where my = 0
    // is unpaired)
    const bool pair = t % units >= H;
    out.re[j][0] = P::sum(cr, di, unit);
    out.im[j][0] = P::diff(ci, dr, unit);
    out.re[j][1] = pair ? P::diff(cr, di, unit) : 0.0;
    out.im[j][1] = pair ? P::sum(ci, dr, unit) : 0.0;
  }
  __syncthreads();
}

// Scale factors of the inverse's input: doubles by their exponent, pairs of
// floats by a float power of two.
__device__ __forceinline__ int fx_key(double, int e) { return e; }
__device__ __forceinline__ float fx_key(ff, int e) { return f_from_bits((uint32_t)(127 + 26 - e) << 23); }
__device__ __forceinline__ unsigned fx_top(double a, double b) { return max(hi_abs(a), hi_abs(b)); }
// the high word that the double of a float would have (a value that is not finite: a NaN's)
__device__ __forceinline__ unsigned fx_top(ff a, ff b) {
  const unsigned m = max(f_bits(a.h) & 0x7fffffffu, f_bits(b.h) & 0x7fffffffu);
  return m >= 0x7f800000u ? 0x7ff80000u : m < 0x0d800000u ? 0x39b00000u : (m >> 3) + 0x38000000u;
}

// 2^k; kAdNaN: a value was not finite
constexpr int kAdNaN = 1 << 20;
__device__ __forceinline__ double ad_unit(int k) {
  return k == kAdNaN ? CUDART_NAN : d_from((uint32_t)(k + 1023) << 20, 0u);
}
// (0 below the floats' normal range)
__device__ __forceinline__ float ad_unit_f(int k) {
  return k > 127 ? CUDART_NAN_F : k < -126 ? 0.0f : f_from_bits((uint32_t)(k + 127) << 23);
}

// Inverse: the threads' modes z give, per particle q,
//   u[iy][ix] = sum over all modes z exp(+i phi (mx ix + my iy))
// (Hermitian in mx), delivered per grid point to `out(q, i, V, k)`, u = V 2^k, V an
// integer of at most 63 bits, always by the same thread.  top: 2 PB words, zero on
// entry: the largest high words of the particles' modes, then of their column sums.
// Returns with a barrier.  |z| < 2^e at scale 2^(57 - e); the columns' sums, at most nt
// sqrt(2) 2^e < 2^(e + 6), are below 2^61.5 in units of four, and are shifted to
// below 2^57 by their own largest, so that their rounding is 2^-57 of it; then |u|, at most
// nt sqrt(2) of that, is below 2^62 in units of two.
template <class V, int U, class Out>
__device__ void ad_inverse(const AdLayout& L, double* sm, unsigned* top, const Modes<V, U>& z, Out out) {
  const int nt = L.nt, H = L.H, T = blockDim.x, tid = threadIdx.x, units = H * H;
  const int items = L.PB * units;
  const Fx* tw = reinterpret_cast<const Fx*>(sm + L.twx);
  const int own = ad_own(tid, units, L.PB);
  unsigned* colmax = top + L.PB;
  unsigned most = 0;
#pragma unroll
  for (int j = 0; j < U; ++j)
    if (tid + j * T < items)
      most = max(most, max(fx_top(z.re[j][0], z.im[j][0]), fx_top(z.re[j][1], z.im[j][1])));
  atomicMax(top + own, most);
  __syncthreads();
  const auto key = fx_key(z.re[0][0], fx_scale(top[own]));
#pragma unroll
  for (int j = 0; j < U; ++j) {
    const int t = tid + j * T;
    if (t < items) {
      const int q = t / units, v = t - q * units;
      double* R = sm + L.base + q * L.per;
      Fx* ps = reinterpret_cast<Fx*>(R + L.ps);
      Fx* pd = reinterpret_cast<Fx*>(R + L.pd);
      const long long ar = fx_of<57>(z.re[j][0], key), ai = fx_of<57>(z.im[j][0], key);
      if (v < H) {  // p = 0: the unpaired my = 0
        ps[2 * v] = fx_split(ar);
        ps[2 * v + 1] = fx_split(ai);
      } else {
        const long long br = fx_of<57>(z.re[j][1], key), bi = fx_of<57>(z.im[j][1], key);
        ps[2 * v] = fx_split(ar + br);
        ps[2 * v + 1] = fx_split(ai + bi);
        pd[2 * v] = fx_split(ar - br);
        pd[2 * v + 1] = fx_split(ai - bi);
      }
    }
  }
  __syncthreads();
  // columns: Y(iy) = Z0 + sum_{m=1}^{H-1} [s_m cos(phi m iy) + i d_m sin(phi m iy)]
  // for iy = py, and the conjugate sine part for iy = nt - py
  long long yr[U][2], yi[U][2];
#pragma unroll
  for (int j = 0; j < U; ++j) {
    const int t = tid + j * T;
    yr[j][0] = yi[j][0] = yr[j][1] = yi[j][1] = 0;
    if (t < items) {
      const int q = t / units, v = t - q * units;
      const double* R = sm + L.base + q * L.per;
      const Fx* ps = reinterpret_cast<const Fx*>(R + L.ps);
      const Fx* pd = reinterpret_cast<const Fx*>(R + L.pd);
      const int py = v / H, mx = v - py * H;
      FxSum cr = fx_start(ps[2 * mx]), ci = fx_start(ps[2 * mx + 1]), dr{0, 0}, di{0, 0};
      int k = py;
      for (int m = 1; m < H; ++m) {
        const int o = 2 * (m * H + mx);
        const Fx cs = tw[k], sn = tw[nt + k];
        accumulate(cr, ps[o], cs);
        accumulate(ci, ps[o + 1], cs);
        accumulate(dr, pd[o], sn);
        accumulate(di, pd[o + 1], sn);
        k += py;
        if (k >= nt) k -= nt;
      }
      const long long a = fx_round(cr), b = fx_round(ci), c = fx_round(dr), d = fx_round(di);
      yr[j][0] = a - d;
      yi[j][0] = b + c;
      if (py > 0) {
        yr[j][1] = a + d;
        yi[j][1] = b - c;
      }
      // (x ^ x >> 63 is |x| to the last bit)
      long long w = 0;
#pragma unroll
      for (int i = 0; i < 2; ++i) w |= (yr[j][i] ^ (yr[j][i] >> 63)) | (yi[j][i] ^ (yi[j][i] >> 63));
      atomicMax(colmax + q, (unsigned)(w >> 32));
    }
  }
  __syncthreads();
  // the shift that leaves 57 bits
  const int own_shift = max(0, 7 - __clz((int)colmax[own]));
#pragma unroll
  for (int j = 0; j < U; ++j) {
    const int t = tid + j * T;
    if (t < items) {
      const int q = t / units, v = t - q * units;
      Fx* cy = reinterpret_cast<Fx*>(sm + L.base + q * L.per + L.cy);
      const int py = v / H, mx = v - py * H;
      const long long half = (1ll << own_shift) >> 1;
      cy[2 * (py * H + mx)] = fx_split((yr[j][0] + half) >> own_shift);
      cy[2 * (py * H + mx) + 1] = fx_split((yi[j][0] + half) >> own_shift);
      if (py > 0) {
        cy[2 * ((nt - py) * H + mx)] = fx_split((yr[j][1] + half) >> own_shift);
        cy[2 * ((nt - py) * H + mx) + 1] = fx_split((yi[j][1] + half) >> own_shift);
      }
    }
  }
  __syncthreads();
  // rows (Hermitian in mx): u[px] = Re Y0 + 2 (A - B), u[nt - px] = Re Y0 + 2 (A + B),
  // A = sum_{mx>=1} Re Y cos(phi mx px), B = sum_{mx>=1} Im Y sin(phi mx px)
  const int rows = nt * H;
  for (int t = tid; t < L.PB * rows; t += T) {
    const int q = t / rows, v = t - q * rows;
    const Fx* cy = reinterpret_cast<const Fx*>(sm + L.base + q * L.per + L.cy);
    const int iy = v / H, px = v - iy * H;
    const Fx* y = cy + 2 * iy * H;
    FxSum a{0, 0}, b{0, 0};
    int k = px;
    for (int mx = 1; mx < H; ++mx) {
      accumulate(a, y[2 * mx], tw[k]);
      accumulate(b, y[2 * mx + 1], tw[nt + k]);
      k += px;
      if (k >= nt) k -= nt;
    }
    const long long A = fx_round2(a), B = fx_round2(b), m = ((fx_join(y[0]) + 1) >> 1) + 2 * A;
    // z in units of 2^(e - 57), the columns in four times that and shifted, this
    // in two of theirs (the products' units of four, halved by fx_round2)
    const int k2 = top[q] >= 0x7ff00000u ? kAdNaN : fx_scale(top[q]) - 54 + max(0, 7 - __clz((int)colmax[q]));
    out(q, iy * nt + px, m - 2 * B, k2);
    if (px > 0) out(q, iy * nt + nt - px, m + 2 * B, k2);
  }
  __syncthreads();
}

__device__ __forceinline__ double ad_loglik(const FilterDev& fd, const EpochParams* __restrict__ ep,
                                            const double* X) {
  double s = 0.0;
  for (int i = 0; i < fd.m; ++i) {
    const double z = (ep->y[i] - X[fd.obs[i]]) * ep->inv_sigma[i];
    s = fma(z, z, s);
  }
  return -0.5 * s;
}

// The twiddle tables and the AdCoef table (the step table is loaded).
__device__ __forceinline__ void ad_tables(const AdLayout& L, double* sm, int S) {
  double* tw = sm + L.tw;
  Fx* twx = reinterpret_cast<Fx*>(sm + L.twx);
  for (int k = threadIdx.x; k < L.nt; k += blockDim.x) {
    double sn, cs;
    sincospi(2.0 * (double)k / (double)L.nt, &sn, &cs);
    tw[k] = cs;
    tw[L.nt + k] = sn;
    twx[k] = fx_split(__double2ll_rn(cs * 0x1.0p54));
    twx[L.nt + k] = fx_split(__double2ll_rn(sn * 0x1.0p54));
  }
  const StepCoef* sc = reinterpret_cast<const StepCoef*>(sm + L.sc);
  AdCoef* ac = reinterpret_cast<AdCoef*>(sm + L.ac);
  for (int i = threadIdx.x; i < S; i += blockDim.x) {
    const StepCoef& c = sc[i];
    const StepCoef& r = sc[c.ref];
    AdCoef a;
    a.kappa = c.rho2 / c.rho1;
    a.dgamma = (float)(c.gamma - r.gamma);
    a.drho = (float)((c.rho1 - r.rho1) / r.rho1);
    a.pa = ff_from(-(c.pi1 + c.pi2));
    a.pb = ff_from(-c.pi2);
    a.mu = ff_from(c.mu / (double)L.d);
    ac[i] = a;
  }
}

// complex a * b
__device__ __forceinline__ void cmul(double ar, double ai, double br, double bi, double& r, double& i) {
  r = fma(ar, br, -ai * bi);
  i = fma(ar, bi, ai * br);
}
__device__ __forceinline__ double value_of(ff a) { return d_from_f(a.h) + d_from_f(a.l); }
// a pair of floats in a double's registers
__device__ __forceinline__ double ff_bits(ff a) { return d_from(f_bits(a.h), f_bits(a.l)); }
__device__ __forceinline__ ff bits_ff(double a) { return ff{f_from_bits(d_hi(a)), f_from_bits(d_lo(a))}; }

// One block advances PB particles (PB > 1 fills the warps on small grids) on at
// most MAXT threads; U = 2 serves grids of more than 512 units (nt = 45).  The
// second bound holds the registers to what lets two to four blocks share an SM:
// the phases of a block alternate between the FP64 and the integer pipe, so
// other blocks' phases fill the waits (72 registers and some spills against 128:
// n = 20, N = 5000 stage 2 0.95 against 1.70 ms, n = 40, N = 1000 1.11 against
// 1.40 ms, the state's transform then still in integers).
// Measured (GB300), against FP64 transforms and mode steps throughout: n = 20,
// N = 5000 stage 1 0.82 -> 0.41 ms, stage 2 2.26 -> 0.97 ms (1.05 with a cold cache); n = 40,
// N = 1000 0.93 -> 0.43, 2.89 -> 1.14 ms; the FP64 pipe is 85 and 68 % busy at n = 20, 79 and
// 51 % at 40.
template <int STAGE, int U, int PB, int MAXT>
__global__ void __launch_bounds__(MAXT, MAXT == 512 ? 1 : MAXT == 416 || U == 2 ? 2 : 3) k_adstage(const __grid_constant__ FilterDev fd,
                                                                   const EpochParams* __restrict__ ep) {
  extern __shared__ double s_dyn[];
  __shared__ double s_red[32];
  __shared__ double s_th[PB][kPMax];
  __shared__ unsigned s_top[3][2 * PB];  // scales of the fields, then of successive inverses
  __shared__ unsigned s_state[PB];    // the largest high word of the state's modes
  // Scale 2^s_err of the estimates squared and summed in ff: 2^40 over the size 2^e of
  // the state's modes, so that it follows the state's units.  An estimate up to 2^(e +
  // 18) squares and sums within the floats; one that may be above (V 2^k, |V| < 2^62: k +
  // 62 > e + 18) is summed in FP64.
  __shared__ int s_err[PB];
  __shared__ int s_flag;
  const Ctrl* ctrl = fd.ctrl;
  if (ctrl->status != PF_OK) return;
  const int S = ep->S;
  const AdLayout L = ad_layout(fd.d, S, PB);
  double* sm = s_dyn;
  load_steps(reinterpret_cast<StepCoef*>(sm + L.sc), ep, S);  // ends with a barrier
  const StepCoef* sc = reinterpret_cast<const StepCoef*>(sm + L.sc);
  const AdCoef* ac = reinterpret_cast<const AdCoef*>(sm + L.ac);
  const int cur = ctrl->cur;
  const Ensemble src = committed(fd, cur);
  const Ensemble dst = pending(fd, cur);
  const int64_t N = fd.N;
  const int64_t n0 = (int64_t)blockIdx.x * PB;  // the block's first particle
  const uint32_t epoch = ep->epoch;
  const int d = L.d, nt = L.nt, H = L.H, T = blockDim.x, tid = threadIdx.x, units = H * H;
  const double inv_d = 1.0 / (double)d;
  // particle q of the block is n0 + q, gathered from slot l (stage 2: the
  // resampled parent); slots past N repeat the last particle and write nothing, so
  // that they have no say in when the block's estimates leave FP64
  auto particle = [&](int q) -> int64_t { return n0 + q < N ? n0 + q : N - 1; };
  auto slot_of = [&](int q) -> int64_t { return STAGE == 2 ? (int64_t)fd.idx[particle(q)] : particle(q); };
  if (tid < PB) {
    const int q = tid;
    const int64_t n = particle(q);
    double ph[5];
    const int64_t l = slot_of(q);
    if (STAGE == 1) {
      // Step 2: phibar^n = a phi^n + (1 - a) phibar
      for (int i = 0; i < 5; ++i) ph[i] = fd.a * src.phi[i * N + n] + (1.0 - fd.a) * ctrl->phibar[i];
    } else {
      // Step 4a: phi_{j+1}^n = phibar^l + s L z
      double z[6];
      for (int b = 0; b < 3; ++b) {
        const U4 w = draw_block(fd, kRngTheta, (uint32_t)n, epoch, (uint32_t)b);
        normal_pair(w, z[2 * b], z[2 * b + 1]);
      }
      for (int i = 0; i < 5; ++i) {
        double lz = 0.0;
        for (int k = 0; k <= i; ++k) lz = fma(ctrl->L[i * kPMax + k], z[k], lz);
        const double shr = fd.a * src.phi[i * N + l] + (1.0 - fd.a) * ctrl->phibar[i];
        ph[i] = fma(fd.s, lz, shr);
        if (n0 + q < N) dst.phi[i * N + n] = ph[i];
      }
    }
    for (int i = 0; i < 5; ++i) s_th[q][i] = (fd.transform == PF_TRANSFORM_LOG) ? pfm::exp_fixed(ph[i]) : ph[i];
  }
  ad_tables(L, sm, S);
  if (tid < 6 * PB) s_top[tid / (2 * PB)][tid % (2 * PB)] = 0u;
  if (tid < PB) s_state[tid] = 0u;
  __syncthreads();
  // scales of D1 and D2 (the error predictor's, stage 2)
  for (int t = tid; t < PB * d; t += T) {
    const int q = t / d;
    const int64_t o = (int64_t)(t - q * d) * N + slot_of(q);
    const double x = src.x[o], h1 = src.h1[o];
    atomicMax(&s_top[1][q], hi_abs(x - h1));
    if (STAGE == 2) atomicMax(&s_top[2][q], hi_abs(h1 - src.h2[o]));
  }
  __syncthreads();
  // the folded fields
  for (int t = tid; t < PB * units; t += T) {
    const int q = t / units, v = t - q * units;
    const int py = v / H, px = v - py * H;
    double* R = sm + L.base + q * L.per;
    const int my = py ? nt - py : 0, mxx = px ? nt - px : 0;
    const int at[4] = {py * nt + px, py * nt + mxx, my * nt + px, my * nt + mxx};
    double x[4], e[4], f[4];
    const int64_t l = slot_of(q);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int64_t o = (int64_t)at[i] * N + l;
      x[i] = src.x[o];
      const double h1 = src.h1[o];
      e[i] = x[i] - h1;
      if (STAGE == 2) f[i] = h1 - src.h2[o];
    }
    const bool y0 = py == 0, x0 = px == 0;
    ad_fold(R + L.F[0], units, v, y0, x0, x[0], x[1], x[2], x[3]);
    ad_fold(reinterpret_cast<Fx*>(R + L.F[1]), units, v, y0, x0, fx_scale(s_top[1][q]), e[0], e[1], e[2], e[3]);
    if (STAGE == 2)
      ad_fold(reinterpret_cast<Fx*>(R + L.F[2]), units, v, y0, x0, fx_scale(s_top[2][q]), f[0], f[1], f[2], f[3]);
  }
  __syncthreads();
  const double* tw = sm + L.tw;
  const int own = ad_own(tid, units, PB);

  // the history in the Fourier basis, each thread holding its own mode pairs:
  // X_n, X_{n-1} and, while the estimate is formed in FP64 (`wide`), X_{n-2};
  // afterwards fa = X_n - X_{n-1} and, in X_{n-2}'s registers, fb = X_{n-1} - X_{n-2} in ff
  Modes<double, U> x0, x1, xb;
  Modes<ff, U> fa;
  auto each = [&](auto f) {
#pragma unroll
    for (int j = 0; j < U; ++j)
#pragma unroll
      for (int b = 0; b < 2; ++b) f(j, b);
  };
  ad_forward<InFp64>(L, sm, L.F[0], L.tw, 1.0, x0);
  ad_forward<InFx>(L, sm, L.F[1], L.twx, fx_unit(s_top[1][own], -51), x1);
  if (STAGE == 2) ad_forward<InFx>(L, sm, L.F[2], L.twx, fx_unit(s_top[2][own], -51), xb);
  each([&](int j, int b) {
    x1.re[j][b] = x0.re[j][b] - x1.re[j][b];
    x1.im[j][b] = x0.im[j][b] - x1.im[j][b];
    if (STAGE == 2) {
      xb.re[j][b] = x1.re[j][b] - xb.re[j][b];
      xb.im[j][b] = x1.im[j][b] - xb.im[j][b];
    }
  });
  if (tid < 6 * PB) s_top[tid / (2 * PB)][tid % (2 * PB)] = 0u;
  if (STAGE == 2) {
    unsigned top = 0;
    each([&](int j, int b) { top = max(top, fx_top(x0.re[j][b], x0.im[j][b])); });
    if (tid < PB * units) atomicMax(s_state + own, top);
    // the error sums take the fields' place
    for (int t = tid; t < PB * d; t += T) {
      const int q = t / d, i = t - q * d;
      double* R = sm + L.base + q * L.per;
      R[L.F[1] + i] = 0.0;
      R[L.F[2] + i] = 0.0;  // (also the ff zero)
    }
  }
  __syncthreads();
  if (STAGE == 2 && tid < PB) s_err[tid] = 40 - fx_scale(s_state[tid]);  // (read after the first inverse's barriers)
  double lr[U][2], li[U][2];
#pragma unroll
  for (int j = 0; j < U; ++j) {
    const int t = tid + j * T;
    lr[j][0] = li[j][0] = lr[j][1] = li[j][1] = 0.0;
    if (t < PB * units) {
      const int q = t / units, v = t - q * units;
      const int p = v / H, mxm = v - p * H;
      const AdOp op = ad_op(s_th[q]);
      ad_lambda(L, op, tw, p, mxm, lr[j][0], li[j][0]);
      if (p > 0) ad_lambda(L, op, tw, nt - p, mxm, lr[j][1], li[j][1]);
    }
  }

  // Psi over the S substeps (Steps 2 and 4b/4d), mode by mode
  double wr[U][2], wi[U][2];  // W = rho1/(1 - gamma lambda) of substep `ref`
  float gr[U][2], gi[U][2];   // lambda/(1 - gamma lambda) of it
  int ref = -1;
  bool wide = STAGE == 2;
  int inv = 0;  // inverses so far: s_top's slots take turns
  auto next_top = [&]() -> unsigned* {
    // the slot after this one is cleared for the next inverse, two barriers ahead of it
    unsigned* now = s_top[inv % 3];
    if (tid < 2 * PB) s_top[(inv + 1) % 3][tid] = 0u;
    ++inv;
    return now;
  };
#pragma unroll 1
  for (int s = 0; s < S; ++s) {
    const StepCoef c = sc[s];
    const AdCoef a = ac[s];
    if (c.ref != ref) {
      ref = c.ref;
      const double gamma = sc[ref].gamma, rho1 = sc[ref].rho1;
      each([&](int j, int b) {
        const double p = fma(-gamma, lr[j][b], 1.0), q = -gamma * li[j][b];
        const double inv2 = 1.0 / fma(p, p, q * q);
        const double ur = p * inv2, ui = -q * inv2;
        wr[j][b] = rho1 * ur;
        wi[j][b] = rho1 * ui;
        double vr, vi;
        cmul(ur, ui, lr[j][b], li[j][b], vr, vi);
        gr[j][b] = f_from(vr);
        gi[j][b] = f_from(vi);
      });
    }
    const bool cold = c.kind != 2;
    Modes<ff, U> e;
    Modes<double, U> ed;
    each([&](int j, int b) {
      const double xr = x0.re[j][b], xi = x0.im[j][b];
      const double pr = x1.re[j][b], pi = x1.im[j][b];
      // (BDF1: rho1 = 1, kappa = 0)
      const double rr = fma(a.kappa, pr, xr), ri = fma(a.kappa, pi, xi);
      double yr, yi;
      cmul(rr, ri, wr[j][b], wi[j][b], yr, yi);
      // the substep's own gamma and rho1: y (1 + drho + dgamma lambda w)
      const float fr = f_from(yr), fi = f_from(yi);
      const float er = f_fma(a.dgamma, gr[j][b], a.drho), ei = f_mul(a.dgamma, gi[j][b]);
      yr += d_from_f(f_fma(fr, er, -f_mul(fi, ei)));
      yi += d_from_f(f_fma(fr, ei, f_mul(fi, er)));
      if (STAGE == 2) {
        if (wide) {
          double qr, qi;
          if (cold) {
            // the explicit-Euler predictor x_n + h L x_n
            double hr, hi;
            cmul(c.h * lr[j][b], c.h * li[j][b], xr, xi, hr, hi);
            qr = xr + hr;
            qi = xi + hi;
          } else {
            qr = fma(c.pi2, xb.re[j][b], fma(c.pi1, pr, c.pi0 * xr));
            qi = fma(c.pi2, xb.im[j][b], fma(c.pi1, pi, c.pi0 * xi));
          }
          const double f = c.mu * inv_d;
          ed.re[j][b] = f * (yr - qr);
          ed.im[j][b] = f * (yi - qi);
          xb.re[j][b] = pr;
          xb.im[j][b] = pi;
        } else {
          const ff Dr = ff_from(yr - xr), Di = ff_from(yi - xi);
          const ff br = bits_ff(xb.re[j][b]), bi = bits_ff(xb.im[j][b]);
          const ff qr = ff_fma(a.pb, br, ff_mul_raw(a.pa, fa.re[j][b]));
          const ff qi = ff_fma(a.pb, bi, ff_mul_raw(a.pa, fa.im[j][b]));
          e.re[j][b] = ff_mul(a.mu, ff_sub(Dr, qr));
          e.im[j][b] = ff_mul(a.mu, ff_sub(Di, qi));
          xb.re[j][b] = ff_bits(fa.re[j][b]);
          xb.im[j][b] = ff_bits(fa.im[j][b]);
          fa.re[j][b] = Dr;
          fa.im[j][b] = Di;
        }
      }
      x1.re[j][b] = xr;
      x1.im[j][b] = xi;
      x0.re[j][b] = yr;
      x0.im[j][b] = yi;
    });
    if (STAGE == 2) {
      unsigned* top = next_top();
      if (wide) {
        ad_inverse(L, sm, top, ed, [&](int q, int i, long long V, int k) {
          double* EE = sm + L.base + q * L.per + L.F[1];
          const double v = (double)V * ad_unit(k);
          EE[i] = fma(v, v, EE[i]);
        });
        // Small beside the state -- 2^-9 by the largest modes (the estimate's
        // carry 1/d), at most 2^-9 sqrt(d) by the norm -- the next estimates may be
        // formed in ff, to 2^-48 of themselves.
        bool small = !cold && s + 1 < S && sc[s + 1].kind == 2;
        for (int q = 0; q < PB; ++q)
          small = small && top[q] + ((unsigned)(9 + 32 - __clz(d - 1)) << 20) <= s_state[q] && s_state[q] < (1023u + 60u) << 20 &&
                  s_state[q] > (1023u - 40u) << 20;
        if (small) {
          wide = false;
          each([&](int j, int b) {
            fa.re[j][b] = ff_from(x0.re[j][b] - x1.re[j][b]);
            fa.im[j][b] = ff_from(x0.im[j][b] - x1.im[j][b]);
            xb.re[j][b] = ff_bits(ff_from(x1.re[j][b] - xb.re[j][b]));
            xb.im[j][b] = ff_bits(ff_from(x1.im[j][b] - xb.im[j][b]));
          });
        }
      } else {
        ad_inverse(L, sm, top, e, [&](int q, int i, long long V, int k) {
          double* R = sm + L.base + q * L.per;
          const int ku = k + s_err[q];
          if (ku <= -4) {
            ff* EE = reinterpret_cast<ff*>(R + L.F[2]);
            ff v = ff_from((double)V);
            const float u = ad_unit_f(ku);
            v = ff{f_mul(v.h, u), f_mul(v.l, u)};
            EE[i] = ff_fma(v, v, EE[i]);
          } else {  // (also one that is not finite)
            const double v = (double)V * ad_unit(k);
            R[L.F[1] + i] = fma(v, v, R[L.F[1] + i]);
          }
        });
      }
    }
  }

  // back to physical space (scaled by 1/d)
  if (STAGE == 1) {
    ad_inverse(L, sm, next_top(), x0, [&](int q, int i, long long V, int k) {
      sm[L.base + q * L.per + L.F[0] + i] = (double)V * (ad_unit(k) * inv_d);
    });
    double lg = -CUDART_INF;
    if (tid < PB && n0 + tid < N) {
      const int64_t n = n0 + tid;
      const double ll = ad_loglik(fd, ep, sm + L.base + tid * L.per + L.F[0]);
      fd.ll1[n] = ll;
      lg = (src.lw[n] - ctrl->logW) + ll;
      if (!finite_bits(lg)) lg = -CUDART_INF;
      fd.lg[n] = lg;
    }
    stage1_tail(fd, epoch, lg, (int)blockIdx.x, (int)gridDim.x, s_red, &s_flag);
  } else {
    // Steps 4c, 4d: the innovation v = sqrt(kappa E) z' takes the ff sums' place
    const int halves = (d + 1) / 2;
    for (int t = tid; t < PB * halves; t += T) {
      const int q = t / halves, b = t - q * halves;
      const int64_t n = n0 + q;
      double* R = sm + L.base + q * L.per;
      const U4 w = draw_block(fd, kRngInnov, (uint32_t)n, epoch, (uint32_t)b);
      double z0, z1;
      normal_pair(w, z0, z1);
      for (int h = 0; h < 2; ++h) {
        const int i = 2 * b + h;
        if (i >= d) break;
        const double u = ad_unit(-s_err[q]);
        const double E = fma(value_of(reinterpret_cast<ff*>(R + L.F[2])[i]) * u, u, R[L.F[1] + i]);
        R[L.F[2] + i] = pfm::sqrt_fixed(fd.kappa * E) * (h == 0 ? z0 : z1);
      }
    }
    __syncthreads();
    // x, then x_{n-1} and x_{n-2} below it by the differences; F[0] keeps x + v
    // for the log-likelihood, F[1] the running state
    ad_inverse(L, sm, next_top(), x0, [&](int q, int i, long long V, int k) {
      double* R = sm + L.base + q * L.per;
      const double x = (double)V * (ad_unit(k) * inv_d), xv = x + R[L.F[2] + i];
      R[L.F[1] + i] = x;
      R[L.F[0] + i] = xv;
      if (n0 + q < N) dst.x[(int64_t)i * N + n0 + q] = xv;
    });
    auto below = [&](Modes<double, U>& D, double* row) {
      ad_inverse(L, sm, next_top(), D, [&](int q, int i, long long V, int k) {
        double* R = sm + L.base + q * L.per;
        const double x = fma(-(double)V, ad_unit(k) * inv_d, R[L.F[1] + i]);
        R[L.F[1] + i] = x;
        if (n0 + q < N) row[(int64_t)i * N + n0 + q] = x + R[L.F[2] + i];
      });
    };
    each([&](int j, int b) {
      x0.re[j][b] -= x1.re[j][b];
      x0.im[j][b] -= x1.im[j][b];
      xb.re[j][b] = wide ? x1.re[j][b] - xb.re[j][b] : value_of(bits_ff(xb.re[j][b]));
      xb.im[j][b] = wide ? x1.im[j][b] - xb.im[j][b] : value_of(bits_ff(xb.im[j][b]));
    });
    below(x0, dst.h1);
    below(xb, dst.h2);
    double lwn = -CUDART_INF;
    bool bad = false;
    if (tid < PB && n0 + tid < N) {
      // Step 5: new log weight
      const int64_t n = n0 + tid;
      lwn = ad_loglik(fd, ep, sm + L.base + tid * L.per + L.F[0]) - fd.ll1[slot_of(tid)];
      if (!finite_bits(lwn)) {
        lwn = -CUDART_INF;
        bad = true;
      }
      dst.lw[n] = lwn;
    }
    stage2_tail(fd, epoch, lwn, bad, (int)blockIdx.x, (int)gridDim.x, s_red, &s_flag);
  }
}

// Launch shape for a grid side: particles per block PB and units (mode pairs)
// per thread U, and threads per block, a multiple of 32 covering PB H^2 units.
// PB (1, 2 or 4) wastes the fewest lanes in the unit and row passes with at most
// 288 threads; U = 2 only where one particle's units exceed 512.
static void ad_shape(int nt, int* threads, int* upt, int* pb) {
  const int H = (nt + 1) / 2, units = H * H;
  int u = 1;
  while (u < kAdMaxUnitsPerThread && (units + u - 1) / u > 512) u *= 2;
  int best_pb = 1, best_T = 0;
  double best_eff = -1.0;
  for (int p = 1; p <= 4; p *= 2) {
    if (u > 1 && p > 1) break;
    const int need = (p * units + u - 1) / u;
    const int T = ((need > 64 ? need : 64) + 31) / 32 * 32;
    if (p > 1 && T > 288) break;
    // lane efficiency of the unit passes and of the row passes
    const double e_units = (double)(p * units) / (double)(((p * units + T - 1) / T) * T);
    const double e_rows = (double)(p * nt * H) / (double)(((p * nt * H + T - 1) / T) * T);
    const double eff = 0.7 * e_units + 0.3 * e_rows;
    if (eff > best_eff + 0.02) {
      best_eff = eff;
      best_pb = p;
      best_T = T;
    }
  }
  *upt = u;
  *pb = best_pb;
  *threads = best_T;
}

struct AdKernel {
  int upt, pb, max_threads;
  void (*k[2])(const FilterDev, const EpochParams*);
};
static const AdKernel kAdKernels[] = {{1, 1, 416, {k_adstage<1, 1, 1, 416>, k_adstage<2, 1, 1, 416>}},
                                      {1, 1, 512, {k_adstage<1, 1, 1, 512>, k_adstage<2, 1, 1, 512>}},
                                      {1, 2, 288, {k_adstage<1, 1, 2, 288>, k_adstage<2, 1, 2, 288>}},
                                      {1, 4, 288, {k_adstage<1, 1, 4, 288>, k_adstage<2, 1, 4, 288>}},
                                      {2, 1, 288, {k_adstage<1, 2, 1, 288>, k_adstage<2, 2, 1, 288>}}};
static const AdKernel* ad_variant(int T, int upt, int pb) {
  for (const AdKernel& v : kAdKernels)
    if (v.upt == upt && v.pb == pb && T <= v.max_threads) return &v;
  return nullptr;
}

cudaError_t launch_ad_stage(int stage, const FilterDev& fd, const EpochParams* ep, int S,
                            cudaStream_t st) {
  const int nt = ad_side(fd.d);
  if (nt == 0) return cudaErrorInvalidValue;
  int T, upt, pb;
  ad_shape(nt, &T, &upt, &pb);
  const size_t smem = sizeof(double) * (size_t)ad_layout(fd.d, S, pb).total;
  const int H = (nt + 1) / 2;
  const AdKernel* v = ad_variant(T, upt, pb);
  if (T * upt < pb * H * H || !v) return cudaErrorInvalidValue;
  const auto k = v->k[stage == 1 ? 0 : 1];
  cudaError_t e = cudaFuncSetAttribute((const void*)k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  const unsigned blocks = (unsigned)((fd.N + pb - 1) / pb);
  k<<<blocks, T, smem, st>>>(fd, ep);
  return cudaGetLastError();
}

cudaError_t preload_ad_kernels() {
  for (const AdKernel& v : kAdKernels)
    for (const auto k : v.k) {
      cudaFuncAttributes a;
      const cudaError_t e = cudaFuncGetAttributes(&a, (const void*)k);
      if (e != cudaSuccess) return e;
    }
  return cudaSuccess;
}

}  // namespace pfg
