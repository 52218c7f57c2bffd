// vp_cv_dev.cuh -- device functions of the reaction coordinate (one warp's
// tile of the contact-pair triangle, one trial's finaliser), shared by the
// separate kernels and the one-kernel step.
#pragma once
#include "vp_cvpair.cuh"
#include "vp_dev.cuh"

namespace vp {

// one tile of the contact-pair triangle of one configuration
struct CvTile {
  int n_cv, bi, bj, min_sep;
  float L, iL, rc2_far;
  float near2;              // set by cv_tile_far
  const float2 *cn;         // the tile's C~_nat
  long long *gx, *gy, *gz;  // the configuration's gradient sums (atom 0)
  double *z_part;           // the tile's partial sum of z
};

// a contribution too large for the tile's accumulators (the sum is the same)
__device__ __forceinline__ void cv_add_large(const CvTile &t, float fx, float fy, float fz, int il, int jc) {
  const long long v[3] = {fx_from(fx), fx_from(fy), fx_from(fz)};
  long long *const gp[3] = {t.gx, t.gy, t.gz};
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    red_add(gp[c] + t.bi * CV_T + il, (long long)(0ull - (unsigned long long)v[c]));
    red_add(gp[c] + t.bj * CV_T + jc, v[c]);
  }
}

// The two pairs' contributions f (per 1/2^32 after rounding, as fx_from rounds
// them) into the tile's accumulators, or straight to memory when one is too
// large for the split; pair 1 only when v1.  |f| < 512: f 2^(32 - CV_SPLIT) +
// 1.5 2^23 is rounded to the high part, what is left of f 2^32 is exact and
// rounds to the low one -- no 64-bit conversion, which the FP64 pipe does.
// SKIP_NAN: a pair whose three components are not numbers adds nothing.
template <bool SKIP_NAN = false, class SH>
__device__ __forceinline__ void cv_accumulate(SH &sh, const CvTile &t, const float2 (&f)[3], int il0, int jc0, int il1,
                                              int jc1, bool v0, bool v1) {
  const float big0 = fmaxf(fmaxf(fabsf(f[0].x), fabsf(f[1].x)), fabsf(f[2].x));
  const float big1 = fmaxf(fmaxf(fabsf(f[0].y), fabsf(f[1].y)), fabsf(f[2].y));
  if (v0 && !(big0 < 512.0f)) {
    if (!SKIP_NAN || big0 == big0) cv_add_large(t, f[0].x, f[1].x, f[2].x, il0, jc0);
    v0 = false;
  }
  if (v1 && !(big1 < 512.0f)) {
    if (!SKIP_NAN || big1 == big1) cv_add_large(t, f[0].y, f[1].y, f[2].y, il1, jc1);
    v1 = false;
  }
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    const float2 m = f2_all(12582912.0f);
    const float2 th = __ffma2_rn(f[q], f2_all(4294967296.0f / (1 << CV_SPLIT)), m);
    const float2 tl = __fadd2_rn(__ffma2_rn(f2_sub(th, m), f2_all(-(float)(1 << CV_SPLIT)), __fmul2_rn(f[q], f2_all(4294967296.0f))), m);
    if (v0) {
      const int hi = __float_as_int(th.x) - 0x4b400000, lo = __float_as_int(tl.x) - 0x4b400000;
      atomicAdd(&sh.s_ghi[il0][q], hi);
      atomicAdd(&sh.s_glo[il0][q], lo);
      atomicAdd(&sh.s_ghi[CV_T + jc0][q], hi);
      atomicAdd(&sh.s_glo[CV_T + jc0][q], lo);
    }
    if (v1) {
      const int hi = __float_as_int(th.y) - 0x4b400000, lo = __float_as_int(tl.y) - 0x4b400000;
      atomicAdd(&sh.s_ghi[il1][q], hi);
      atomicAdd(&sh.s_glo[il1][q], lo);
      atomicAdd(&sh.s_ghi[CV_T + jc1][q], hi);
      atomicAdd(&sh.s_glo[CV_T + jc1][q], lo);
    }
  }
}

// The near pairs e0 and (when v1) e1 of a tile, entries il | jc << 5: their z
// terms, and their gradient contributions into the tile's accumulators.  One
// definition for the warp and the block form of a tile, so both give the same
// bits.
template <class SH>
__device__ __forceinline__ ff2 cv_near_pairs(SH &sh, const CvConst &k, const CvTile &t, unsigned e0, unsigned e1, bool v1) {
  const int il0 = e0 & 31, jc0 = e0 >> 5, il1 = e1 & 31, jc1 = e1 >> 5;
  ff2 dx, dy, dz;
  cv_delta2(sh.s_x[il0], sh.s_x[il1], sh.s_x[CV_T + jc0], sh.s_x[CV_T + jc1], t.L, t.iL, dx, dy, dz);
  const float2 n0 = t.cn[((jc0 - il0) & (CV_T - 1)) * CV_T + il0], n1 = t.cn[((jc1 - il1) & (CV_T - 1)) * CV_T + il1];
  const ff2 cnat = {make_float2(n0.x, n1.x), make_float2(n0.y, n1.y)};
  const ff2 r2 = ff2_add(ff2_add(ff2_sqr(dx), ff2_sqr(dy)), ff2_sqr(dz));
  const CvPair2 cp = cv_contact2<false>(r2, k);
  const float2 h = ff2_sub(cp.Ct, cnat).hi;
  // dz/dx_i = -w d, dz/dx_j = +w d with d = x_j - x_i, w = 2 h C~'(r)/r
  const float2 w = f2_div(__fmul2_rn(__fadd2_rn(h, h), cp.dCt), cp.r, f2_rcp(cp.r));
  const float2 g[3] = {__fmul2_rn(w, dx.hi), __fmul2_rn(w, dy.hi), __fmul2_rn(w, dz.hi)};
  // coincident atoms (w not a number) pull nowhere
  cv_accumulate(sh, t, g, il0, jc0, il1, jc1, w.x == w.x, v1 && w.y == w.y);
  // z term: C~ (C~ - 2 C~_nat) = (C~ - C~_nat)^2 - C~_nat^2
  return ff2_mul(cp.Ct, ff2_sub(cp.Ct, ff2{__fadd2_rn(cnat.hi, cnat.hi), __fadd2_rn(cnat.lo, cnat.lo)}));
}

// whether the pairs of atom xi with xj0 and with xj1 are closer than the contact
// cut-off (FP32; a position that is not a number is near nothing)
__device__ __forceinline__ void cv_are_near(float4 xi, float4 xj0, float4 xj1, float L, float iL, float near2, bool &n0,
                                            bool &n1) {
  const float2 m = f2_all(12582912.0f), il = f2_all(iL), l = f2_all(-L);  // see cv_delta2
  float2 dx = __fadd2_rn(make_float2(xj0.x, xj1.x), f2_all(-xi.x)), dy = __fadd2_rn(make_float2(xj0.y, xj1.y), f2_all(-xi.y)),
         dz = __fadd2_rn(make_float2(xj0.z, xj1.z), f2_all(-xi.z));
  dx = __ffma2_rn(l, f2_sub(__fadd2_rn(__fmul2_rn(dx, il), m), m), dx);
  dy = __ffma2_rn(l, f2_sub(__fadd2_rn(__fmul2_rn(dy, il), m), m), dy);
  dz = __ffma2_rn(l, f2_sub(__fadd2_rn(__fmul2_rn(dz, il), m), m), dz);
  const float2 r2 = __ffma2_rn(dz, dz, __ffma2_rn(dx, dx, __fmul2_rn(dy, dy)));
  n0 = r2.x < near2;
  n1 = r2.y < near2;
}

// the accumulated gradient of atom a (0..63) of the tile, into the sums at gx, gy, gz
template <class SH>
__device__ __forceinline__ void cv_flush_atom(SH &sh, int a, long long *gx, long long *gy, long long *gz) {
  long long g[3];
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    g[q] = (long long)sh.s_ghi[a][q] * (1ll << CV_SPLIT) + (long long)sh.s_glo[a][q];
    if (a < CV_T) g[q] = -g[q];
  }
  if (g[0] | g[1] | g[2]) { red_add(gx, g[0]); red_add(gy, g[1]); red_add(gz, g[2]); }
}

// Whether no pair of the tile can be closer than the contact cut-off: the
// periodic gap of the two 32-atom blocks' bounding boxes (lane l holds atom l
// of either block).  Some 60 instructions that spare a far tile the 800 of its
// distance tests.  Otherwise t.near2 is what those take as near.
__device__ __forceinline__ bool cv_tile_far(CvTile &t, bool iv, bool jv, float3 xi, float3 xj) {
  const float3 ai = iv ? xi : make_float3(0.f, 0.f, 0.f), aj = jv ? xj : make_float3(0.f, 0.f, 0.f);
  const float m = warp_max(fmaxf(fmaxf(fmaxf(fabsf(ai.x), fabsf(ai.y)), fabsf(ai.z)),
                                 fmaxf(fmaxf(fabsf(aj.x), fabsf(aj.y)), fabsf(aj.z))));
  float g2 = 0.f;
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    const float a = q == 0 ? xi.x : q == 1 ? xi.y : xi.z, b = q == 0 ? xj.x : q == 1 ? xj.y : xj.z;
    const float al = warp_min(iv ? a : 3e38f), ah = warp_max(iv ? a : -3e38f);
    const float bl = warp_min(jv ? b : 3e38f), bh = warp_max(jv ? b : -3e38f);
    float dc = 0.5f * (bl + bh) - 0.5f * (al + ah);
    dc = fabsf(dc - t.L * rintf(dc * t.iL)) - 0.5f * ((ah - al) + (bh - bl));
    dc = fmaxf(dc, 0.f);
    g2 += dc * dc;
  }
  const float m2 = m * m;
  t.near2 = cv_near2(t.rc2_far, 4.0f * m2);
  // a gap is off by 1e-6 m at most: with e = sqrt(3) 1e-6 m, (r + e)^2 is below
  // 1.0005 r^2 + 2001 e^2
  return g2 > fmaf(6e-9f, m2, 1.001f * t.rc2_far);
}

// The near pairs of the tile by one warp, in rotation-major order, into
// s_near; returns their number.  s_x: the atoms of both blocks (not a number
// beyond the last).  KEEP: the ballots of the 32 rotations go to kept.
template <bool KEEP>
__device__ __forceinline__ int cv_near_list(const CvTile &t, unsigned short *s_near, const float4 *s_x, unsigned *kept) {
  const int lane = threadIdx.x & 31, sep = t.min_sep - (t.bj - t.bi) * CV_T + lane;
  const float4 xi = s_x[lane];
  const unsigned below = (1u << lane) - 1u;
  int n_near = 0;
#pragma unroll 2
  for (int k = 0; k < CV_T; k += 2) {
    const int j0 = (lane + k) & (CV_T - 1), j1 = (lane + k + 1) & (CV_T - 1);
    bool n0, n1;
    cv_are_near(xi, s_x[CV_T + j0], s_x[CV_T + j1], t.L, t.iL, t.near2, n0, n1);
    n0 = n0 && j0 > sep;
    n1 = n1 && j1 > sep;
    const unsigned b0 = __ballot_sync(0xffffffffu, n0), b1 = __ballot_sync(0xffffffffu, n1);
    if (n0) s_near[n_near + __popc(b0 & below)] = (unsigned short)(lane | (j0 << 5));
    n_near += __popc(b0);
    if (n1) s_near[n_near + __popc(b1 & below)] = (unsigned short)(lane | (j1 << 5));
    n_near += __popc(b1);
    if (KEEP && lane == 0) *reinterpret_cast<uint2 *>(kept + k) = make_uint2(b0, b1);
  }
  return n_near;
}

// The same from kept ballots (in no particular order).
__device__ __forceinline__ int cv_near_list_kept(unsigned short *s_near, const unsigned *kept) {
  const int lane = threadIdx.x & 31;
  unsigned m = kept[lane];  // lane k: rotation k
  int incl = __popc(m);
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const int v = __shfl_up_sync(0xffffffffu, incl, off);
    if (lane >= off) incl += v;
  }
  for (int p = incl - __popc(m); m; m &= m - 1u) {
    const int i = __ffs(m) - 1;
    s_near[p++] = (unsigned short)(i | (((i + lane) & (CV_T - 1)) << 5));
  }
  return __shfl_sync(0xffffffffu, incl, 31);
}

// The same by a block of NW warps, the 32 rotations dealt out over them: the
// ballots into s_bal ...
template <int NW>
__device__ __forceinline__ void cv_ballots_block(const CvTile &t, unsigned *s_bal, const float4 *s_x) {
  constexpr int KW = CV_T / NW;  // rotations per warp
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, sep = t.min_sep - (t.bj - t.bi) * CV_T + lane;
  const float4 xi = s_x[lane];
#pragma unroll
  for (int q = 0; q < KW; q += 2) {
    const int k = warp * KW + q, j0 = (lane + k) & (CV_T - 1), j1 = (lane + k + 1) & (CV_T - 1);
    bool n0, n1;
    cv_are_near(xi, s_x[CV_T + j0], s_x[CV_T + j1], t.L, t.iL, t.near2, n0, n1);
    const unsigned b0 = __ballot_sync(0xffffffffu, n0 && j0 > sep), b1 = __ballot_sync(0xffffffffu, n1 && j1 > sep);
    if (lane == 0) {
      s_bal[k] = b0;
      s_bal[k + 1] = b1;
    }
  }
}
// ... and the list from them (every thread of the block calls, after a barrier)
template <int NW>
__device__ __forceinline__ int cv_near_list_block(unsigned short *s_near, const unsigned *s_bal) {
  constexpr int KW = CV_T / NW;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int incl = __popc(s_bal[lane]);
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const int v = __shfl_up_sync(0xffffffffu, incl, off);
    if (lane >= off) incl += v;
  }
#pragma unroll
  for (int q = 0; q < KW; ++q) {
    const unsigned bal = s_bal[warp * KW + q];
    const int end = __shfl_sync(0xffffffffu, incl, warp * KW + q);
    if ((bal >> lane) & 1u)
      s_near[end - __popc(bal) + __popc(bal & ((1u << lane) - 1u))] =
          (unsigned short)(lane | (((lane + warp * KW + q) & (CV_T - 1)) << 5));
  }
  __syncthreads();
  return __shfl_sync(0xffffffffu, incl, 31);
}

// an atom of a tile; one beyond the last is not a number, and so near nothing
__device__ __forceinline__ float4 cv_atom(bool valid, float3 x) {
  return valid ? make_float4(x.x, x.y, x.z, 0.f) : make_float4(NAN, NAN, NAN, 0.f);
}

// One warp's tile: z partial sum and gradient.  pos(a): position of
// reaction-coordinate atom a.
// KEEP: the number of near pairs and the ballots that list them are left at
// n_kept and kept, for a later pass over the same pairs.
template <bool KEEP = false, class POS>
__device__ __forceinline__ void cv_tile(CvTile t, const CvConst &k, CvWarpShared &sh, POS pos,
                                        int *n_kept = nullptr, unsigned *kept = nullptr) {
  const int lane = threadIdx.x & 31;
  const int i = t.bi * CV_T + lane, j = t.bj * CV_T + lane;
  const bool iv = i < t.n_cv, jv = j < t.n_cv;
  float3 xi = make_float3(0.f, 0.f, 0.f), xj = xi;
  if (iv) xi = pos(i);
  if (jv) xj = pos(j);
  if (cv_tile_far(t, iv, jv, xi, xj)) {
    if (lane == 0) *t.z_part = 0.0;
    if (KEEP && lane == 0) *n_kept = 0;
    return;
  }
  sh.s_x[lane] = cv_atom(iv, xi);
  sh.s_x[CV_T + lane] = cv_atom(jv, xj);
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    sh.s_ghi[lane][q] = 0; sh.s_ghi[CV_T + lane][q] = 0;
    sh.s_glo[lane][q] = 0; sh.s_glo[CV_T + lane][q] = 0;
  }
  __syncwarp();
  const int n_near = cv_near_list<KEEP>(t, sh.s_near, sh.s_x, kept);
  if (KEEP && lane == 0) *n_kept = n_near;
  __syncwarp();
  // the near pairs, densely
  ff zacc = {0.f, 0.f};
  for (int p = lane; p < n_near; p += 64) {
    const bool two = p + 32 < n_near;
    const ff2 v = cv_near_pairs(sh, k, t, sh.s_near[p], sh.s_near[two ? p + 32 : p], two);
    zacc = ff_add(zacc, ff{v.hi.x, v.lo.x});
    if (two) zacc = ff_add(zacc, ff{v.hi.y, v.lo.y});
  }
  __syncwarp();
  if (n_near > 0) {
    if (iv) cv_flush_atom(sh, lane, t.gx + i, t.gy + i, t.gz + i);
    if (jv) cv_flush_atom(sh, CV_T + lane, t.gx + j, t.gy + j, t.gz + j);
  }
  double zl = ff_to_d(zacc);
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) zl += __shfl_xor_sync(0xffffffffu, zl, off);
  if (lane == 0) *t.z_part = zl;
}

// The same tile by a block of NW warps: the rotations of the distance tests
// and the chunks of 32 near pairs are dealt out over the warps.  The near
// pairs keep the order the one-warp form lists them in, and the z terms go
// through shared memory so that each lane of the first warp adds them in that
// order too: z and the gradient are the same bit for bit.
struct CvBlockShared {
  unsigned short s_near[CV_T * CV_T];
  float4 s_x[2 * CV_T];
  int s_ghi[2 * CV_T][3];
  int s_glo[2 * CV_T][3];
  unsigned s_bal[CV_T];
  float2 s_term[CV_T * CV_T];
};

// positions of the tile's 64 atoms into s_x, its gradient sums cleared;
// returns (in every thread) whether the tile is far
template <int NW, class SH, class POS>
__device__ __forceinline__ bool cv_block_begin(CvTile &t, SH &sh, POS pos) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (threadIdx.x < 2 * CV_T) {
    const int a = (warp == 0 ? t.bi : t.bj) * CV_T + lane;
    float3 q = make_float3(0.f, 0.f, 0.f);
    if (a < t.n_cv) q = pos(a);
    sh.s_x[threadIdx.x] = cv_atom(a < t.n_cv, q);
  }
  for (int q = threadIdx.x; q < 2 * CV_T * 3; q += NW * 32) {
    (&sh.s_ghi[0][0])[q] = 0;
    (&sh.s_glo[0][0])[q] = 0;
  }
  __syncthreads();
  return cv_tile_far(t, t.bi * CV_T + lane < t.n_cv, t.bj * CV_T + lane < t.n_cv,
                     make_float3(sh.s_x[lane].x, sh.s_x[lane].y, sh.s_x[lane].z),
                     make_float3(sh.s_x[CV_T + lane].x, sh.s_x[CV_T + lane].y, sh.s_x[CV_T + lane].z));
}

template <int NW, bool KEEP = false, class POS>
__device__ __forceinline__ void cv_tile_block(CvTile t, const CvConst &k, CvBlockShared &sh, POS pos,
                                              int *n_kept = nullptr, unsigned *kept = nullptr) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (cv_block_begin<NW>(t, sh, pos)) {
    if (threadIdx.x == 0) *t.z_part = 0.0;
    if (KEEP && threadIdx.x == 0) *n_kept = 0;
    return;
  }
  cv_ballots_block<NW>(t, sh.s_bal, sh.s_x);
  __syncthreads();
  const int n_near = cv_near_list_block<NW>(sh.s_near, sh.s_bal);
  if (KEEP && warp == NW - 1) {
    kept[lane] = sh.s_bal[lane];
    if (lane == 0) *n_kept = n_near;
  }
  // 64 pairs per warp at a time: warps without any leave their issue slots to the others
  for (int p = 64 * warp + lane; p < n_near; p += 64 * NW) {
    const int p1 = p + 32;
    const bool two = p1 < n_near;
    const ff2 v = cv_near_pairs(sh, k, t, sh.s_near[p], sh.s_near[two ? p1 : p], two);
    sh.s_term[p] = make_float2(v.hi.x, v.lo.x);
    if (two) sh.s_term[p1] = make_float2(v.hi.y, v.lo.y);
  }
  __syncthreads();
  if (warp == 0) {
    ff zacc = {0.f, 0.f};
    for (int p = lane; p < n_near; p += 32) zacc = ff_add(zacc, ff{sh.s_term[p].x, sh.s_term[p].y});
    double zl = ff_to_d(zacc);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) zl += __shfl_xor_sync(0xffffffffu, zl, off);
    if (lane == 0) *t.z_part = zl;
  } else if (warp <= 2 && n_near > 0) {
    const int a = (warp == 1 ? t.bi : t.bj) * CV_T + lane;
    if (a < t.n_cv) cv_flush_atom(sh, (warp - 1) * CV_T + lane, t.gx + a, t.gy + a, t.gz + a);
  }
}

// the tile of work item W (the partial sum of z goes to the item's slot)
__device__ __forceinline__ CvTile cv_item_tile(const Dev &d, const SimConst &c, const CvItem &W) {
  return CvTile{W.n_cv, W.bi, W.bj, c.cv_min_sep, W.box, W.inv_box, c.cv_rc2_far, 0.f,
                d.cnat_ff + (size_t)W.tile * CV_T * CV_T, d.gx + W.cv0, d.gy + W.cv0, d.gz + W.cv0, d.z_part + W.w};
}

// positions of a trial's reaction-coordinate atoms (caller order)
struct CvSlotPos {
  const Dev &d;
  int atom0;
  __device__ __forceinline__ float3 operator()(int a) const {
    const float4 q = d.pos[d.slot_of[atom0 + a]];
    return make_float3(q.x, q.y, q.z);
  }
};


// The finaliser of trial t by one block of any size: the reduction runs over
// CVFIN_THREADS virtual threads in a fixed tree, so z is the same bit for bit
// whatever block runs it.  Returns true in the block that finished the last
// trial of the step (FIN_STEP: the step counter and the kick then advance).
template <int MODE>
__device__ bool cvfin_trial(const Dev &d, const SimConst &c, CvfinShared &sh, int t) {
  double *rz = sh.rz, *rq = sh.rq;
  const TrialInfo T = d.tinfo[t];
  const long long step_now = *d.step;
  for (int v = threadIdx.x; v < CVFIN_THREADS; v += blockDim.x) {
    double zs = 0.0, q = 0.0;
    for (int k = v; k < T.n_work; k += CVFIN_THREADS) zs += d.z_part[T.work0 + k];
    for (int i = v; i < T.n_cv; i += CVFIN_THREADS) {
      double gx = (double)d.gx[T.cv0 + i] * 2.3283064365386963e-10;
      double gy = (double)d.gy[T.cv0 + i] * 2.3283064365386963e-10;
      double gz = (double)d.gz[T.cv0 + i] * 2.3283064365386963e-10;
      q += (gx * gx + gy * gy + gz * gz) * d.inv_gm[T.sysatom0 + i];  // FP64 division is slow on this part
    }
    rz[v] = zs;
    rq[v] = q;
  }
  __syncthreads();
  for (int off = CVFIN_THREADS / 2; off > 0; off >>= 1) {
    for (int v = threadIdx.x; v < off; v += blockDim.x) { rz[v] += rz[v + off]; rq[v] += rq[v + off]; }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    TrialState &S = d.tstate[t];
    const double z = S.zconst + rz[0];
    const double Q = rq[0];
    double a = 0.0, phi = 0.0;
    if (MODE == FIN_INIT) {
      S.zm = z;
    } else {
      a = z > S.zm ? z - S.zm : 0.0;
      if (MODE == FIN_STEP) {
        phi = c.kR_half_d * c.kR_half_d * a * a * Q;
        S.Phi += c.dt_d * phi;
      }
      if (z < S.zm) S.zm = z;
    }
    S.z = z;
    S.a = a;
    S.phi = phi;
    if (!isfinite(z)) atomicOr(d.err, ERR_NONFINITE);
    if (c.rec_cap > 0 && MODE != FIN_KEEP) {
      long long n = MODE == FIN_STEP ? step_now + 1 : step_now;
      double *r = d.rec + ((size_t)t * c.rec_cap + (size_t)(n % c.rec_cap)) * 5;
      r[0] = z; r[1] = S.zm; r[2] = a; r[3] = phi; r[4] = Q;
    }
    if (MODE == FIN_STEP) {
      __threadfence();
      unsigned ticket = atomicAdd(d.done, 1u);
      sh.last = ticket == (unsigned)(d.n_trials - 1);
    } else {
      sh.last = false;
    }
  }
  __syncthreads();
  const bool last = sh.last;
  if (MODE == FIN_STEP && last && threadIdx.x == 0) {
    *d.step = step_now + 1;
    *d.kick = 1.0f;
    *d.done = 0u;
  }
  __syncthreads();  // the shared arrays may be reused by the caller
  return last;
}

}  // namespace vp
