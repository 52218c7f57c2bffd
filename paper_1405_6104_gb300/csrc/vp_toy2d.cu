// vp_toy2d.cu -- batched trials of the two-dimensional toy model of the
// variational pathway scheme (SM, "Illustrative Application in a Toy Model"):
// one particle on U(x, y) under underdamped Langevin dynamics (Eq. Lang,
// BAOAB), with the ratchet-and-pawl bias of Eq. VR, a steered harmonic pull,
// or no bias on z = sqrt(x^2 + y^2), and the functional of Eq. VMDcondition
// accumulated up to the first passage into the product (z <= z_product).
//
// A thread, or a pair of lanes (one per coordinate), owns one trial and keeps
// its state in registers; the only memory traffic is the trial's inputs, its
// outputs, (optionally) its recorded path and the noise.  Arithmetic is FP64
// without contraction (this file is compiled with -fmad=false), in the
// operation order of the equations, so that a trial follows its FP64 definition
// step for step; the white noise is Philox4x32-10 (counter = (0, step, 0 |
// stream)) turned into normals by Box-Muller in FP64.
//
// Bound by this part's FP64 unit: a warp issues one FP64 instruction (a compare
// too) per 64 cycles however many of its lanes are active and however
// independent its instructions are; an SM takes one per 16 to 19 cycles, so
// four warps.  The 2000 trials per bias strength of the model's protocol are a
// warp or two per SM, so a step costs 64 cycles times its FP64 instructions
// per warp.  Hence:
//  - quotients and square roots are formed from an approximate (inverse square)
//    root, one Halley step and Markstein's correction of the rounded result (P.
//    Markstein, IBM J. Res. Dev. 34 (1990) 111): the operators' values but for
//    results next to the midpoint of two numbers (see quotient()), with the
//    reciprocal shared where several quotients have one divisor, in fewer
//    instructions;
//  - comparisons of positive numbers, halving and range checks are integer
//    operations; multiplication by a mass or friction of one is left out;
//  - the noise does not depend on the trial's state, so other warps prepare it:
//    the normals of the next steps by a kernel that fills the GPU, or, in long
//    runs, sqrt(-2 log u) and (cos, sin)(2 pi u) for all 2^23 values a uniform
//    takes, in tables read one step ahead (the very functions, so the same
//    bits);
//  - while trials are few, two lanes share one: each does its own coordinate,
//    and the three well terms and the root, one after another otherwise, go two
//    at a time (55 FP64 instructions per step, one lane per trial 93, the
//    operators and functions in the step 230);
//  - trials that have reached the product leave: the run goes in launches, each
//    over the trials still on their way.
// 8000 rMD trials of 30 000 steps: 211 ms with the operators and functions in
// the step, 118 with one lane per trial and the tables, 76 now (5300 cycles per
// step: 55 FP64 instructions and the exchanges between them); 24 000 trials 292
// and 134 ms.  With every trial running all its steps: 78.4 ms, 82.7 with a mass
// of 2.5, a friction of 0.3 and a third well off the axis, whose multiplications
// and quotient the defaults leave out (210.6 and 211.5 before).
#include <algorithm>
#include <cmath>
#include <cstring>
#include <string>

#include "../../include/vpath.h"
#include "vp_internal.cuh"

namespace vp {
namespace {

struct ToyConst {
  double w4, N1, N2, N3;   // 4 w^2, 4 A s^p of the three terms
  double ss1, ss2, ss3;    // s^2
  double xm, ym, x0, y0;
  double gm, inv_gm;       // gamma m and its reciprocal
  double im, h, dt;        // 1/m, dt/2, dt
  double c1, c2sd;         // exp(-gamma dt), sqrt(1 - c1^2) sqrt(kT/m)
  double sd;               // sqrt(kT/m)
  double zp;               // product threshold
  long long zp_bits;       // the threshold as an integer (positive doubles order as their bits), -1 if not positive
  int bias;
  int plain;               // gamma m and the numerators N are moderate (or N = 0): see quotient()
  int unit_mass, unit_gm;  // 1/m = 1, gamma m = 1
};

// the uniform of a 23-bit word, and the two halves of a Box-Muller draw
__device__ __forceinline__ double uniform_d(uint32_t m) { return ((double)m + 0.5) * (1.0 / 8388608.0); }
__device__ __forceinline__ double normal_radius(double u) { return sqrt(-2.0 * log(u)); }
__device__ __forceinline__ double2 normal_angle(double u) {
  const double two_pi = 6.283185307179586476925286766559;
  double sn, cs;
  sincos(two_pi * u, &sn, &cs);
  return make_double2(cs, sn);
}
// two standard normals from Philox (key = seed) at (atom 0, step, stream)
__device__ __forceinline__ double2 normal2_d(uint32_t k0, uint32_t k1, unsigned long long step, uint32_t stream) {
  const uint4 x = philox4x32_10(make_uint4(0u, (uint32_t)step, (uint32_t)(step >> 32), stream), k0, k1);
  const double r = normal_radius(uniform_d(x.x >> 9));
  const double2 a = normal_angle(uniform_d(x.y >> 9));
  return make_double2(r * a.x, r * a.y);
}

// ---------------------------------------------------------------------------
// quotients and roots
// ---------------------------------------------------------------------------
__device__ __forceinline__ double rcp_approx(double b) {  // relative error below 2^-20
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(b));
  return y;
}
__device__ __forceinline__ double rsqrt_approx(double b) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(b));
  return y;
}
// 1/b within about an ulp: e = 1 - b y0, y = y0 (1 + e + e^2)
__device__ __forceinline__ double reciprocal(double b) {
  const double y = rcp_approx(b), e = fma(-b, y, 1.0);
  return fma(y, fma(e, e, e), y);
}
// 1/sqrt(b) within about an ulp: e = 1 - b y0^2, y = y0 (1 + e/2 + 3 e^2/8)
__device__ __forceinline__ double inv_sqrt(double b) {
  const double y = rsqrt_approx(b), e = fma(-(b * y), y, 1.0);
  return fma(e * y, fma(0.375, e, 0.5), y);
}
// a/b, y = 1/b within half an ulp and 2^-7 (e^3): a y is within two ulps of a/b, so
// what the last step adds is within 2^-51 ulps of what it should be, and the result
// within 1/2 + 2^-51 ulps of a/b.  That is the correctly rounded one unless a/b lies
// within 2^-51 ulps of the midpoint of two numbers, as for a few of the 2^53
// dividends of a divisor; then the wrong neighbour is taken now and then (by 1 of
// the 10 295 such quotients in the tests).  Markstein's proof for these needs a
// correctly rounded reciprocal, two more FP64 instructions, and a second step.
__device__ __forceinline__ double quotient(double a, double b, double y) {
  const double q = a * y;
  return fma(fma(-b, q, a), y, q);
}
// sqrt(b) within 1/2 + 2^-51 ulps likewise, y = 1/sqrt(b) within an ulp
__device__ __forceinline__ double root(double b, double y) {
  const double g = b * y;
  return fma(fma(-g, g, b), 0.5 * y, g);
}
// b in [2^-300, 2^300): far from where the steps above could over- or underflow
__device__ __forceinline__ bool moderate(double b) {
  return (unsigned)(__double2hiint(b) - ((1023 - 300) << 20)) < (600u << 20);
}

__device__ __forceinline__ double half_of(double v) {  // of a number far from the denormals
  return __hiloint2double(__double2hiint(v) - (1 << 20), __double2loint(v));
}
__device__ __forceinline__ bool is_zero(double v) { return ((__double2hiint(v) << 1) | __double2loint(v)) == 0; }
__device__ __forceinline__ bool below(double a, double b) {  // of positive numbers
  return __double_as_longlong(a) < __double_as_longlong(b);
}

// what a step needs at a position: force of the potential, z and grad z
struct ToyPoint {
  double fx, fy, z, ux, uy;
};

// With the operators themselves: wherever a divisor is out of the moderate range
// (grad z = 0 at z = 0)
__device__ __noinline__ ToyPoint toy_point_any(const ToyConst &c, double x, double y) {
  const double r2 = x * x + y * y;
  double gx = c.w4 * r2 * x, gy = c.w4 * r2 * y;
  const double D1 = r2 + c.ss1, q1 = c.N1 / (D1 * D1 * D1);
  gx += q1 * x;
  gy += q1 * y;
  const double D2 = r2 + c.ss2, q2 = c.N2 / (D2 * D2 * D2);
  gx -= q2 * x;
  gy -= q2 * y;
  const double dx = x - c.xm, dy = y - c.ym;
  const double D3 = dx * dx + dy * dy + c.ss3, q3 = c.N3 / (D3 * D3 * D3);
  gx += q3 * dx;
  gy += q3 * dy;
  const double z = sqrt(r2);
  return ToyPoint{-gx, -gy, z, z == 0.0 ? 0.0 : x / z, z == 0.0 ? 0.0 : y / z};
}

// -grad U (the force of the potential; U itself is not needed on the path), z
// and grad z = (x, y)/z; *fast: z is positive and finite
__device__ __forceinline__ ToyPoint toy_point(const ToyConst &c, double x, double y, bool &fast) {
  const double yy = y * y, r2 = x * x + yy;
  const double D1 = r2 + c.ss1, D2 = r2 + c.ss2;
  const double dx = x - c.xm;
  double dy = y, dyy = yy;
  if (!is_zero(c.ym)) {
    dy = y - c.ym;
    dyy = dy * dy;
  }
  const double D3 = dx * dx + dyy + c.ss3;
  const double E1 = D1 * D1 * D1, E2 = D2 * D2 * D2, E3 = D3 * D3 * D3;
  fast = c.plain && moderate(r2) && moderate(E1) && moderate(E2) && moderate(E3);
  if (!fast) return toy_point_any(c, x, y);
  const double q1 = quotient(c.N1, E1, reciprocal(E1)), q2 = quotient(c.N2, E2, reciprocal(E2)),
               q3 = quotient(c.N3, E3, reciprocal(E3));
  const double wr = c.w4 * r2;
  double gx = wr * x, gy = wr * y;
  gx += q1 * x;
  gy += q1 * y;
  gx -= q2 * x;
  gy -= q2 * y;
  gx += q3 * dx;
  gy += q3 * dy;
  const double iz = inv_sqrt(r2), z = root(r2, iz);
  ToyPoint p{-gx, -gy, z, 0.0, 0.0};
  if (c.bias != TOY2D_NONE) {
    p.ux = quotient(x, z, iz);
    p.uy = quotient(y, z, iz);
  }
  return p;
}

// amplitude s of the bias force s grad z: the ratchet (Eq. VR) against the
// running minimum zm, or the steered pull -k z
__device__ __forceinline__ double toy_amplitude(const ToyConst &c, double k, double z, double zm, bool fast) {
  if (!fast && z == 0.0) return 0.0;
  if (c.bias == TOY2D_RATCHET) {
    const bool above = fast ? below(zm, z) : z > zm;
    const double a = above ? z - zm : 0.0;
    return -0.5 * k * a;
  }
  return -k * z;
}

// Phi's share of a step from dt |F_bias|^2
__device__ __forceinline__ double toy_share(const ToyConst &c, double num) {
  if (c.unit_gm) return num;
  return c.plain && (moderate(num) || is_zero(num)) ? quotient(num, c.gm, c.inv_gm) : num / c.gm;
}

// the normals' tables: radius[m] = sqrt(-2 log u), angle[m] = (cos, sin)(2 pi u), u = (m + 1/2) 2^-23
constexpr int TABLE_BITS = 23;
__global__ void __launch_bounds__(256) k_toy_tables(double *radius, double2 *angle) {
  const uint32_t m = blockIdx.x * 256u + threadIdx.x;
  const double u = uniform_d(m);
  radius[m] = normal_radius(u);
  angle[m] = normal_angle(u);
}

// the normals of steps s0 + 1 .. s0 + steps of the listed trials: out[step][trial]
__global__ void __launch_bounds__(256) k_toy_noise(int n, const int *__restrict__ list,
                                                   const unsigned long long *__restrict__ seeds, long long s0,
                                                   long long steps, double2 *out) {
  const long long i = (long long)blockIdx.x * 256 + threadIdx.x;
  if (i >= steps * n) return;
  const long long s = i / n;
  const int q = (int)(i - s * n);
  const unsigned long long seed = seeds[list ? list[q] : q];
  out[i] = normal2_d((uint32_t)seed, (uint32_t)(seed >> 32), (unsigned long long)(s0 + 1 + s), 0u);
}

// per-trial state between launches
struct ToyState {
  double *xv;       // [4 n] x, y, vx, vy
  double *aux;      // [3 n] running minimum of z, force (bias included)
  double *phi;      // [n]
  long long *passage;  // [n]
};

// a launch's trials and noise: the normals themselves ([step][trial]), or the tables
struct ToyLaunch {
  int n;
  const int *list;   // nullptr: trial q is q
  const double *k;
  const unsigned long long *seeds;
  long long s0, s1;  // steps s0 + 1 .. s1; s0 = 0 starts the trials
  const double2 *noise;
  const double *radius;
  const double2 *angle;
  double *path;
  int every;
  long long n_rec;
};

// One lane per trial.
template <bool TABLE>
__global__ void __launch_bounds__(32) k_toy2d(ToyConst c, ToyLaunch l, ToyState st) {
  const int q = blockIdx.x * 32 + threadIdx.x;
  if (q >= l.n) return;
  const int t = l.list ? l.list[q] : q;
  const double k = l.k[t];
  const unsigned long long seed = l.seeds[t];
  const uint32_t k0 = (uint32_t)seed, k1 = (uint32_t)(seed >> 32);
  double *rec = l.path ? l.path + (size_t)t * (size_t)l.n_rec * 2 : nullptr;
  double x, y, vx, vy, zm, fx, fy, Phi;
  bool fast;
  if (l.s0 == 0) {
    x = c.x0;
    y = c.y0;
    const double2 g0 = normal2_d(k0, k1, 0ull, 1u);  // Maxwell-Boltzmann start: stream 1, step 0
    vx = c.sd * g0.x;
    vy = c.sd * g0.y;
    const ToyPoint p = toy_point(c, x, y, fast);
    zm = p.z;
    fx = p.fx;
    fy = p.fy;
    if (c.bias != TOY2D_NONE) {
      const double s = toy_amplitude(c, k, p.z, zm, fast);
      fx += s * p.ux;
      fy += s * p.uy;
    }
    Phi = 0.0;
    if (rec) { rec[0] = x; rec[1] = y; }
  } else {
    if (st.passage[t] >= 0) return;
    x = st.xv[4 * t]; y = st.xv[4 * t + 1]; vx = st.xv[4 * t + 2]; vy = st.xv[4 * t + 3];
    zm = st.aux[3 * t]; fx = st.aux[3 * t + 1]; fy = st.aux[3 * t + 2];
    Phi = st.phi[t];
  }
  long long passage = -1;
  long long r = rec ? l.s0 / l.every + 1 : 0;
  long long due = rec ? r * l.every : 0;  // the step of the next recorded position
  // half kicks: the closing one of a step and the opening one of the next are equal
  auto kick = [&](double f) {
    const double v = c.h * f;
    return c.unit_mass ? v : v * c.im;
  };
  double kx = kick(fx), ky = kick(fy);
  // the noise of the step ahead: its loads are in flight during a step
  double rad = 0.0;
  double2 ang = make_double2(0.0, 0.0);
  auto fetch = [&](long long s) {
    if (TABLE) {
      const uint4 w = philox4x32_10(make_uint4(0u, (uint32_t)s, (uint32_t)((unsigned long long)s >> 32), 0u), k0, k1);
      rad = l.radius[w.x >> (32 - TABLE_BITS)];
      ang = l.angle[w.y >> (32 - TABLE_BITS)];
    } else {
      ang = l.noise[(size_t)(min(s, l.s1) - l.s0 - 1) * (size_t)l.n + q];
    }
  };
  if (l.s1 > l.s0) fetch(l.s0 + 1);
  for (long long s = l.s0 + 1; s <= l.s1; ++s) {
    const double nx = TABLE ? rad * ang.x : ang.x, ny = TABLE ? rad * ang.y : ang.y;
    fetch(s + 1);
    vx += kx;
    vy += ky;
    x += c.h * vx;
    y += c.h * vy;
    vx = c.c1 * vx + c.c2sd * nx;
    vy = c.c1 * vy + c.c2sd * ny;
    x += c.h * vx;
    y += c.h * vy;
    const ToyPoint p = toy_point(c, x, y, fast);
    fx = p.fx;
    fy = p.fy;
    if (c.bias != TOY2D_NONE) {
      const double b = toy_amplitude(c, k, p.z, zm, fast), bx = b * p.ux, by = b * p.uy;
      Phi += toy_share(c, c.dt * (bx * bx + by * by));
      fx += bx;
      fy += by;
    } else if (!c.plain) {
      Phi += toy_share(c, 0.0);
    }
    if (fast ? below(p.z, zm) : p.z < zm) zm = p.z;
    kx = kick(fx);
    ky = kick(fy);
    vx += kx;
    vy += ky;
    if (rec && s == due && r < l.n_rec) { rec[2 * r] = x; rec[2 * r + 1] = y; ++r; due += l.every; }
    if (fast ? __double_as_longlong(p.z) <= c.zp_bits : p.z <= c.zp) { passage = s; break; }
  }
  if (rec && passage >= 0)
    for (; r < l.n_rec; ++r) { rec[2 * r] = nan(""); rec[2 * r + 1] = nan(""); }
  st.xv[4 * t] = x; st.xv[4 * t + 1] = y; st.xv[4 * t + 2] = vx; st.xv[4 * t + 3] = vy;
  st.aux[3 * t] = zm; st.aux[3 * t + 1] = fx; st.aux[3 * t + 2] = fy;
  st.phi[t] = Phi;
  st.passage[t] = passage;
}

// One lane per coordinate: lanes 2q (x) and 2q + 1 (y) of a warp share trial
// q.  Of a pair, the even lane forms the first well term and then the third,
// the odd one the second and then the root; sums of two coordinates' terms
// commute, so both lanes hold the same bits.  A pair that is done runs on
// without effect until its warp is (the exchanges need every lane).
template <bool TABLE>
__global__ void __launch_bounds__(32) k_toy2d_pair(ToyConst c, ToyLaunch l, ToyState st) {
  const unsigned full = 0xffffffffu;
  const bool odd = threadIdx.x & 1;
  const int q0 = blockIdx.x * 16 + (threadIdx.x >> 1), q = min(q0, l.n - 1);
  bool done = q0 >= l.n;
  const int t = l.list ? l.list[q] : q;
  const double k = l.k[t];
  const unsigned long long seed = l.seeds[t];
  const uint32_t k0 = (uint32_t)seed, k1 = (uint32_t)(seed >> 32);
  double *rec = l.path ? l.path + (size_t)t * (size_t)l.n_rec * 2 + odd : nullptr;
  const double off = odd ? c.ym : c.xm, ss = odd ? c.ss2 : c.ss1, N = odd ? c.N2 : c.N1;
  auto other = [&](double v) { return __shfl_xor_sync(full, v, 1); };
  // force of the potential along this lane's coordinate x, z and grad z
  struct Point {
    double f, z, u;
    bool fast;
  };
  auto point = [&](double x) {
    const double xx = x * x, r2 = xx + other(xx);
    const double d = x - off, dd = d * d, D3 = dd + other(dd) + c.ss3;
    const double D = r2 + ss, E = D * D * D, E3 = D3 * D3 * D3;
    Point p;
    p.fast = c.plain && moderate(r2) && moderate(E) && moderate(E3);
    p.fast = __shfl_xor_sync(full, (int)p.fast, 1) && p.fast;
    // the first term (even) and the second (odd)
    const double qa = quotient(N, E, reciprocal(E)), qb = other(qa);
    // the third term (even) and the root (odd), by the same instructions
    const double y0 = odd ? rsqrt_approx(r2) : rcp_approx(E3);
    const double b0 = r2 * y0;
    const double e = fma(-(odd ? b0 : E3), y0, 1.0);
    const double w = e * y0;
    const double y = fma(w, fma(odd ? 0.375 : 1.0, e, odd ? 0.5 : 1.0), y0);
    const double num = odd ? r2 : c.N3;
    const double g = num * y;
    const double v = fma(fma(-(odd ? g : E3), g, num), odd ? half_of(y) : y, g);
    const double vo = other(v), yo = other(y);
    const double q3 = odd ? vo : v, iz = odd ? y : yo;
    p.z = odd ? v : vo;
    double gr = c.w4 * r2 * x;
    gr += (odd ? qb : qa) * x;
    gr -= (odd ? qa : qb) * x;
    gr += q3 * d;
    p.f = -gr;
    p.u = c.bias != TOY2D_NONE ? quotient(x, p.z, iz) : 0.0;
    const double xo = other(x);
    if (!p.fast) {
      const ToyPoint a = toy_point_any(c, odd ? xo : x, odd ? x : xo);
      p.f = odd ? a.fy : a.fx;
      p.z = a.z;
      p.u = odd ? a.uy : a.ux;
    }
    return p;
  };
  double x, v, zm, f, Phi;
  if (l.s0 == 0) {
    x = odd ? c.y0 : c.x0;
    const double2 g0 = normal2_d(k0, k1, 0ull, 1u);  // Maxwell-Boltzmann start: stream 1, step 0
    v = c.sd * (odd ? g0.y : g0.x);
    const Point p = point(x);
    zm = p.z;
    f = p.f;
    if (c.bias != TOY2D_NONE) f += toy_amplitude(c, k, p.z, zm, p.fast) * p.u;
    Phi = 0.0;
    if (rec && !done) rec[0] = x;
  } else {
    done |= st.passage[t] >= 0;
    x = st.xv[4 * t + odd]; v = st.xv[4 * t + 2 + odd];
    zm = st.aux[3 * t]; f = st.aux[3 * t + 1 + odd];
    Phi = st.phi[t];
  }
  long long r = rec ? l.s0 / l.every + 1 : 0;
  long long due = rec ? r * l.every : 0;  // the step of the next recorded position
  auto kick = [&](double a) {
    const double b = c.h * a;
    return c.unit_mass ? b : b * c.im;
  };
  double kk = kick(f);
  double rad = 0.0, ang = 0.0;  // the noise of the step ahead
  auto fetch = [&](long long s) {
    if (TABLE) {
      const uint4 w = philox4x32_10(make_uint4(0u, (uint32_t)s, (uint32_t)((unsigned long long)s >> 32), 0u), k0, k1);
      rad = l.radius[w.x >> (32 - TABLE_BITS)];
      ang = reinterpret_cast<const double *>(l.angle)[2 * (size_t)(w.y >> (32 - TABLE_BITS)) + odd];
    } else {
      ang = reinterpret_cast<const double *>(l.noise)[2 * ((size_t)(min(s, l.s1) - l.s0 - 1) * (size_t)l.n + q) + odd];
    }
  };
  auto leave = [&](long long passage) {
    if (rec && passage >= 0)
      for (; r < l.n_rec; ++r) rec[2 * r] = nan("");
    st.xv[4 * t + odd] = x; st.xv[4 * t + 2 + odd] = v;
    st.aux[3 * t + 1 + odd] = f;
    if (!odd) {
      st.aux[3 * t] = zm;
      st.phi[t] = Phi;
      st.passage[t] = passage;
    }
  };
  if (l.s1 > l.s0) fetch(l.s0 + 1);
  for (long long s = l.s0 + 1; s <= l.s1 && !__all_sync(full, done); ++s) {
    const double n = TABLE ? rad * ang : ang;
    fetch(s + 1);
    v += kk;
    x += c.h * v;
    v = c.c1 * v + c.c2sd * n;
    x += c.h * v;
    const Point p = point(x);
    f = p.f;
    if (c.bias != TOY2D_NONE) {
      const double b = toy_amplitude(c, k, p.z, zm, p.fast) * p.u, bb = b * b;
      Phi += toy_share(c, c.dt * (bb + other(bb)));
      f += b;
    } else if (!c.plain) {
      Phi += toy_share(c, 0.0);
    }
    if (p.fast ? below(p.z, zm) : p.z < zm) zm = p.z;
    kk = kick(f);
    v += kk;
    if (!done) {
      if (rec && s == due && r < l.n_rec) { rec[2 * r] = x; ++r; due += l.every; }
      if (p.fast ? __double_as_longlong(p.z) <= c.zp_bits : p.z <= c.zp) {
        leave(s);
        done = true;
      }
    }
  }
  if (!done) leave(-1);
}

// the trials still on their way (ascending within a block's share) and their
// number (*count = 0 before)
__global__ void __launch_bounds__(256) k_toy_active(const long long *passage, int n, int *list, int *count) {
  __shared__ int part[8], base;
  const int t = blockIdx.x * 256 + threadIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const bool on = t < n && passage[t] < 0;
  const unsigned bal = __ballot_sync(0xffffffffu, on);
  if (lane == 0) part[warp] = __popc(bal);
  __syncthreads();
  int before = 0, all = 0;
  for (int w = 0; w < 8; ++w) {
    before += w < warp ? part[w] : 0;
    all += part[w];
  }
  if (threadIdx.x == 0) base = atomicAdd(count, all);
  __syncthreads();
  if (on) list[base + before + __popc(bal & ((1u << lane) - 1u))] = t;
}

constexpr long long TOY_DRAWS = 1ll << 22;  // draws prepared for a launch at most (64 MB)
constexpr long long TOY_CHUNK = 8192;       // steps of a launch that reads the tables
constexpr long long TOY_COMPACT = 128;      // steps after which the trials that are done are sorted out

int set_err(char *errbuf, int32_t errlen, int code, const std::string &msg) {
  if (errbuf && errlen > 0) {
    std::strncpy(errbuf, msg.c_str(), (size_t)errlen - 1);
    errbuf[errlen - 1] = '\0';
  }
  return code;
}

}  // namespace
}  // namespace vp

using namespace vp;

extern "C" __attribute__((visibility("default"))) int toy2d_run(const toy2d_params *p, int32_t n_trials,
                                                                const double *k, const uint64_t *seeds,
                                                                int64_t n_steps, double *state, double *phi,
                                                                int64_t *passage, double *path, int32_t path_every,
                                                                void *cuda_stream, char *errbuf, int32_t errlen) {
  if (!p || n_trials < 0 || n_steps < 0 || (n_trials > 0 && (!k || !seeds || !phi || !passage)))
    return set_err(errbuf, errlen, SIM_EINVAL, "toy2d_run: null argument or negative size");
  if (path && path_every < 1) return set_err(errbuf, errlen, SIM_EINVAL, "toy2d_run: path_every must be >= 1");
  if (p->bias != TOY2D_NONE && p->bias != TOY2D_RATCHET && p->bias != TOY2D_STEERED)
    return set_err(errbuf, errlen, SIM_EINVAL, "toy2d_run: unknown bias");
  if (p->s_power != 2 && p->s_power != 4) return set_err(errbuf, errlen, SIM_EINVAL, "toy2d_run: s_power must be 2 or 4");
  if (!(p->mass > 0.0) || !(p->gamma >= 0.0) || !(p->kT >= 0.0) || !(p->dt > 0.0))
    return set_err(errbuf, errlen, SIM_EINVAL, "toy2d_run: mass and dt must be > 0, gamma and kT >= 0");
  if (p->bias != TOY2D_NONE && !(p->gamma > 0.0))
    return set_err(errbuf, errlen, SIM_EINVAL, "toy2d_run: the functional needs gamma > 0");
  if (n_trials == 0) return SIM_OK;
  ToyConst c{};
  auto spow = [&](double s) { return p->s_power == 4 ? (s * s) * (s * s) : s * s; };
  c.w4 = 4.0 * p->w * p->w;
  c.N1 = 4.0 * p->A1 * spow(p->s1);
  c.N2 = 4.0 * p->A2 * spow(p->s2);
  c.N3 = 4.0 * p->A3 * spow(p->s3);
  c.ss1 = p->s1 * p->s1;
  c.ss2 = p->s2 * p->s2;
  c.ss3 = p->s3 * p->s3;
  c.xm = p->xm; c.ym = p->ym; c.x0 = p->x0; c.y0 = p->y0;
  c.gm = p->gamma * p->mass;
  c.inv_gm = 1.0 / c.gm;
  c.im = 1.0 / p->mass;
  c.h = 0.5 * p->dt;
  c.dt = p->dt;
  c.c1 = std::exp(-p->gamma * p->dt);
  c.sd = std::sqrt(p->kT / p->mass);
  c.c2sd = std::sqrt(1.0 - c.c1 * c.c1) * c.sd;
  c.zp = p->z_product;
  c.zp_bits = -1;
  if (c.zp > 0.0) std::memcpy(&c.zp_bits, &c.zp, sizeof(c.zp));
  c.bias = p->bias;
  c.unit_mass = c.im == 1.0;
  c.unit_gm = c.gm == 1.0;
  auto sane = [](double v) { return std::fabs(v) > 1e-80 && std::fabs(v) < 1e80; };
  c.plain = sane(c.gm) && (c.N1 == 0.0 || sane(c.N1)) && (c.N2 == 0.0 || sane(c.N2)) && (c.N3 == 0.0 || sane(c.N3));
  const long long n_rec = path ? n_steps / path_every + 1 : 0;
  cudaStream_t st = (cudaStream_t)cuda_stream;
  const size_t n = (size_t)n_trials;
  std::string err;
  auto ck = [&](cudaError_t e, const char *what) {
    if (e != cudaSuccess && err.empty()) err = std::string(what) + ": " + cudaGetErrorString(e);
    return e == cudaSuccess;
  };
  int dev = 0, n_sm = 1;
  if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
  // the trials (k, seed, state, list) and the noise of a launch; the path; the tables
  // (an eighth of all draws at a time, between 1 and 64 MB, but 16 steps at least)
  const double total = (double)n * (double)n_steps;
  const long long want = (long long)std::min<double>(TOY_DRAWS, std::max<double>(1 << 16, total / 8.0));
  long long draws =
      (long long)n * std::max<long long>(1, std::min<long long>(n_steps, std::max<long long>(16, want / (long long)n)));
  double *buf = nullptr, *dpath = nullptr, *tables = nullptr;
  bool ok = !path || ck(cudaMalloc(&dpath, (size_t)n_rec * 2 * n * sizeof(double)), "cudaMalloc");
  // with little memory left the draws of fewer steps at a time, down to one
  for (; ok && cudaMalloc(&buf, (2 * (size_t)draws + n * 12 + 1) * sizeof(double)) != cudaSuccess;) {
    const cudaError_t e = cudaGetLastError();
    if (e != cudaErrorMemoryAllocation || draws == (long long)n) ok = ck(e, "cudaMalloc");
    draws = std::max<long long>(n, draws / 4);
  }
  double2 *dnoise = (double2 *)buf;
  double *dk = buf + 2 * draws;
  unsigned long long *dseed = (unsigned long long *)(dk + n);
  ToyState ts{dk + 2 * n, dk + 6 * n, dk + 9 * n, (long long *)(dk + 10 * n)};
  int *dlist = (int *)(dk + 11 * n), *dcount = (int *)(dk + 12 * n);
  ok = ok && ck(cudaMemcpyAsync(dk, k, n * sizeof(double), cudaMemcpyHostToDevice, st), "cudaMemcpyAsync") &&
       ck(cudaMemcpyAsync(dseed, seeds, n * sizeof(uint64_t), cudaMemcpyHostToDevice, st), "cudaMemcpyAsync");
  int active = n_trials;
  const int *list = nullptr;
  long long since = 0;  // steps since the finished trials were sorted out
  for (long long s0 = 0; ok && active > 0;) {
    // The tables (2^23 draws to fill, as many as a launch prepares twice) once
    // four times as many draws are left; not before the first launch, in which
    // most trials of a strong bias end, unless filling them is a matter of 64
    // steps.
    if (!tables && (s0 > 0 || n >= (size_t)1 << (TABLE_BITS - 6)) &&
        (double)(n_steps - s0) * active > (double)(4ll << TABLE_BITS)) {
      if (cudaMalloc(&tables, (size_t)3 * sizeof(double) << TABLE_BITS) == cudaSuccess) {
        k_toy_tables<<<(1u << TABLE_BITS) / 256, 256, 0, st>>>(tables + ((size_t)2 << TABLE_BITS), (double2 *)tables);
      } else {  // without the memory for them the run goes on as it is
        cudaGetLastError();
        tables = nullptr;
      }
    }
    const long long left = n_steps - s0;
    long long len = std::min(left, tables ? TOY_CHUNK : draws / active);
    if (s0 == 0) len = std::min<long long>(len, std::max<long long>(64, (1 << 16) / active));  // some end at once
    ToyLaunch l{active, list, dk, dseed, s0, s0 + len, dnoise, nullptr, nullptr, dpath, path_every,
                n_rec};
    if (tables) {
      l.radius = tables + ((size_t)2 << TABLE_BITS);
      l.angle = (const double2 *)tables;
    } else if (len > 0) {
      k_toy_noise<<<(unsigned)((len * active + 255) / 256), 256, 0, st>>>(active, l.list, dseed, s0, len, dnoise);
    }
    // one warp per block: the trials spread evenly over the SMs.  Two lanes per
    // trial up to about five warps per SM (8000 trials on 152 SMs: 3.3): beyond,
    // the SM's FP64 unit is full and fewer instructions in all win.  Parameters out
    // of the quotients' range take one lane, whose step goes to the operators at
    // once (8000 trials of 2000 steps with a friction of 1e-85: 15.6 ms in pairs).
    const bool pair = c.plain && (long long)active <= 76ll * n_sm;
    const unsigned blocks = (unsigned)((active + (pair ? 15 : 31)) / (pair ? 16 : 32));
    if (pair) {
      if (tables) k_toy2d_pair<true><<<blocks, 32, 0, st>>>(c, l, ts);
      else k_toy2d_pair<false><<<blocks, 32, 0, st>>>(c, l, ts);
    } else {
      if (tables) k_toy2d<true><<<blocks, 32, 0, st>>>(c, l, ts);
      else k_toy2d<false><<<blocks, 32, 0, st>>>(c, l, ts);
    }
    ok = ck(cudaGetLastError(), "k_toy2d launch");
    s0 += len;
    if (!ok || s0 >= n_steps) break;
    since += len;
    if (since < TOY_COMPACT) continue;
    since = 0;
    list = dlist;
    ok = ck(cudaMemsetAsync(dcount, 0, sizeof(int), st), "cudaMemsetAsync");
    if (!ok) break;
    k_toy_active<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(ts.passage, n_trials, dlist, dcount);
    ok = ck(cudaGetLastError(), "k_toy_active launch") &&
         ck(cudaMemcpyAsync(&active, dcount, sizeof(int), cudaMemcpyDeviceToHost, st), "cudaMemcpyAsync") &&
         ck(cudaStreamSynchronize(st), "cudaStreamSynchronize");
  }
  ok = ok && ck(cudaMemcpyAsync(phi, ts.phi, n * sizeof(double), cudaMemcpyDeviceToHost, st), "cudaMemcpyAsync") &&
       ck(cudaMemcpyAsync(passage, ts.passage, n * sizeof(int64_t), cudaMemcpyDeviceToHost, st), "cudaMemcpyAsync") &&
       (!state || ck(cudaMemcpyAsync(state, ts.xv, 4 * n * sizeof(double), cudaMemcpyDeviceToHost, st),
                     "cudaMemcpyAsync")) &&
       (!path || ck(cudaMemcpyAsync(path, dpath, (size_t)n_rec * 2 * n * sizeof(double), cudaMemcpyDeviceToHost, st),
                    "cudaMemcpyAsync"));
  ck(cudaStreamSynchronize(st), "cudaStreamSynchronize");
  cudaFree(buf);
  if (dpath) cudaFree(dpath);
  if (tables) cudaFree(tables);
  if (!err.empty()) return set_err(errbuf, errlen, SIM_ECUDA, "toy2d_run: " + err);
  return SIM_OK;
}
