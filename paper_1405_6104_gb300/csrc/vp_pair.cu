// vp_pair.cu -- nonbonded (LJ + reaction field) and bonded forces.
//
// One warp per 8-atom i-cluster.  Lane l takes list entry e0 + l, one j-atom
// (the list holds only j-atoms with at least one pair in it); it loops over
// the 8 i-atoms, so the force on its j-atom is complete after the loop and
// goes to memory with one 64-bit fixed-point reduction per component.  i-forces stay in registers over the whole list
// and are reduced across the warp at the end.  FP32 pair arithmetic,
// order-independent int64 accumulation (2^32 units per kJ/mol/nm), so the
// forces are bit-reproducible.  Bonded forces come from k_bonded; the bonded
// energies (each atom its own share of every bond and angle it is part of)
// from k_bonded_energy, or from the general energy kernel k_pair itself.
#include <algorithm>
#include <type_traits>

#include "vp_dev.cuh"
#include "vp_pair_dev.cuh"

namespace vp {


// a.b, rounded as written (two kernels form it: the same bits in both)
__device__ __forceinline__ float dot3(float3 a, float3 b) {
  return __fmaf_rn(a.z, b.z, __fmaf_rn(a.x, b.x, __fmul_rn(a.y, b.y)));
}

// one atom's share of its bonded energies (bonds: V = k/2 (r - r0)^2, angles
// V = k/2 (theta - theta0)^2), into eb and ea
__device__ __forceinline__ void bonded_energy(const Dev &d, const TrialInfo &T, int o, float4 self, float &eb,
                                              float &ea) {
  const int sa = T.sysatom0 + o;
  const int b0 = d.bt_start[sa], b1 = d.bt_start[sa + 1];
  const float L = T.box, iL = T.inv_box;
  auto image = [&](float x, float x0) {  // of x nearest to x0
    return __fmaf_rn(-L, rintf(__fmul_rn(__fsub_rn(x, x0), iL)), x);
  };
  for (int k = b0; k < b1; ++k) {
    const BTerm bt = d.bterm[k];
    const float4 p1 = d.pos[d.slot_of[T.atom0 + bt.p1]];
    const float3 q1 = make_float3(image(p1.x, self.x), image(p1.y, self.y), image(p1.z, self.z));
    if (bt.kind == 0) {
      // stiff springs: the stretch r - r0 in float-float (exact coordinate
      // differences), so that k (r - r0) keeps FP32 relative accuracy
      const ff dx = ff_diff(q1.x, self.x), dy = ff_diff(q1.y, self.y), dz = ff_diff(q1.z, self.z);
      const ff r = ff_sqrt(ff_add(ff_add(ff_sqr(dx), ff_sqr(dy)), ff_sqr(dz)));
      const float dr = ff_add_f(r, -bt.x0).hi;
      eb = __fmaf_rn(__fmul_rn(__fmul_rn(0.25f, bt.k), dr), dr, eb);
    } else {
      const float4 p2 = d.pos[d.slot_of[T.atom0 + bt.p2]];
      const float3 d1 = make_float3(__fsub_rn(q1.x, self.x), __fsub_rn(q1.y, self.y), __fsub_rn(q1.z, self.z));
      const float3 d2 = make_float3(__fsub_rn(image(p2.x, self.x), self.x), __fsub_rn(image(p2.y, self.y), self.y),
                                    __fsub_rn(image(p2.z, self.z), self.z));
      float3 u = d1, v = d2;  // self is the vertex; p1, p2 the ends
      if (bt.kind == 1) {     // self is an end; p1 vertex, p2 other end
        u = make_float3(-d1.x, -d1.y, -d1.z);
        v = make_float3(__fsub_rn(d2.x, d1.x), __fsub_rn(d2.y, d1.y), __fsub_rn(d2.z, d1.z));
      }
      float cs = __fmul_rn(dot3(u, v), rsqrtf(__fmul_rn(dot3(u, u), dot3(v, v))));
      cs = fminf(1.0f, fmaxf(-1.0f, cs));
      const float dth = acosf(cs) - bt.x0;
      ea = __fmaf_rn(__fmul_rn(__fmul_rn(0.5f / 3.0f, bt.k), dth), dth, ea);
    }
  }
}

// the energies of the 8 pairs of one lane: j-atom (xj, yj, zj, qj, type row tj)
// against the warp's 8 i-atoms, distances rounded as the force kernels round them
template <bool EXACT>
__device__ __forceinline__ void pair_energies(const float (&xi)[CL], const float (&yi)[CL], const float (&zi)[CL],
                                              const float (&qi)[CL], const int (&tio)[CL], float xj, float yj,
                                              float zj, float qj, int tj, unsigned mb, float L, float iL,
                                              const SimConst &c, const float2 *tab, const float *tshift, float &elj,
                                              float &erf) {
#pragma unroll
  for (int a = 0; a < CL; ++a) {
    float dx = __fsub_rn(xj, xi[a]), dy = __fsub_rn(yj, yi[a]), dz = __fsub_rn(zj, zi[a]);
    if (EXACT) {
      dx = __fmaf_rn(-L, rintf(__fmul_rn(dx, iL)), dx);
      dy = __fmaf_rn(-L, rintf(__fmul_rn(dy, iL)), dy);
      dz = __fmaf_rn(-L, rintf(__fmul_rn(dz, iL)), dz);
    }
    const float r2 = __fmaf_rn(dz, dz, __fmaf_rn(dy, dy, __fmul_rn(dx, dx)));
    const bool in = ((mb >> a) & 1u) && (r2 < c.rc2);
    const float rinv = rsqrtf(r2);
    const float rinv2 = __fmul_rn(rinv, rinv);
    const float rinv6 = __fmul_rn(__fmul_rn(rinv2, rinv2), rinv2);
    const float2 cc = tab[tio[a] + tj];
    const float qq = __fmul_rn(qi[a], qj);
    if (in) {
      elj += rinv6 * (cc.y * (1.0f / 12.0f) * rinv6 - cc.x * (1.0f / 6.0f)) - tshift[tio[a] + tj];
      erf += qq * (rinv + c.krf * r2 - c.crf);
    }
  }
}

// Energies (nonbonded and bonded) of one trial, or of all, any number of types:
// one warp per i-cluster.
__global__ void __launch_bounds__(128, 4) k_pair(Dev d, SimConst c, int only_trial) {
  extern __shared__ float2 smem_tab[];
  float2 *tab = smem_tab;
  float *tshift = reinterpret_cast<float *>(smem_tab + c.n_types * c.n_types);
  const int nt2 = c.n_types * c.n_types;
  for (int k = threadIdx.x; k < nt2; k += blockDim.x) {
    tab[k] = d.ljtab[k];
    tshift[k] = d.ljshift[k];
  }
  __syncthreads();
  const int I = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (I >= d.total_clus) return;
  const int t = d.clus_trial[I];
  if (only_trial >= 0 && t != only_trial) return;
  const TrialInfo T = d.tinfo[t];
  if (I - T.clus0 >= d.tstate[t].n_clus) return;
  const float L = T.box, iL = T.inv_box;

  float xi[CL], yi[CL], zi[CL], qi[CL];
  int tio[CL];
#pragma unroll
  for (int a = 0; a < CL; ++a) {
    float4 p = d.pos[I * CL + a];
    xi[a] = p.x; yi[a] = p.y; zi[a] = p.z; qi[a] = p.w;
    tio[a] = d.type[I * CL + a] * c.n_types;
  }
  float elj = 0.0f, erf = 0.0f;

  const int n = d.list_n[I];
  const uint32_t *seg = d.list + (size_t)I * c.list_cap;
  const uint8_t *segm = d.list_m + (size_t)I * c.list_cap;
  // one j-atom entry per lane; software pipeline: the entry two groups ahead
  // and the j-atom of the next group are in flight while the current group is
  // evaluated; idle lanes get an empty mask
  uint32_t ent = lane < n ? seg[lane] : d.idle_entry;
  uint32_t ent_n = 32 + lane < n ? seg[32 + lane] : d.idle_entry;
  float4 pj = d.pos[(int)(ent & J_MASK)];
  int tj = d.type[(int)(ent & J_MASK)];
  for (int e0 = 0; e0 < n; e0 += 32) {
    const uint32_t ent_nn = e0 + 64 + lane < n ? seg[e0 + 64 + lane] : d.idle_entry;
    const int sj_n = (int)(ent_n & J_MASK);
    const float4 pj_n = d.pos[sj_n];
    const int tj_n = d.type[sj_n];
    const unsigned sh = ent >> J_BITS;
    const float xj = pj.x - L * (float)((int)(sh & 3u) - 1);
    const float yj = pj.y - L * (float)((int)((sh >> 2) & 3u) - 1);
    const float zj = pj.z - L * (float)((int)((sh >> 4) & 3u) - 1);
    const unsigned mb = e0 + lane < n ? segm[e0 + lane] : 0u;
    if (ent & E_EXACT)
      pair_energies<true>(xi, yi, zi, qi, tio, xj, yj, zj, pj.w, tj, mb, L, iL, c, tab, tshift, elj, erf);
    else
      pair_energies<false>(xi, yi, zi, qi, tio, xj, yj, zj, pj.w, tj, mb, L, iL, c, tab, tshift, elj, erf);
    ent = ent_n;
    ent_n = ent_nn;
    pj = pj_n;
    tj = tj_n;
  }

  // bonded terms of the 8 i-atoms (lanes 0..7)
  float eb = 0.f, ea = 0.f;
  if (lane < CL) {
    const int o = d.orig[I * CL + lane];
    if (o >= 0) {
      float4 self = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int a = 0; a < CL; ++a)
        if (a == lane) self = make_float4(xi[a], yi[a], zi[a], 0.f);
      bonded_energy(d, T, o, self, eb, ea);
    }
  }

  double e4[4] = {(double)elj, (double)erf, (double)eb, (double)ea};
#pragma unroll
  for (int k = 0; k < 4; ++k)
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) e4[k] += __shfl_xor_sync(0xffffffffu, e4[k], off);
  if (lane == 0)
#pragma unroll
    for (int k = 0; k < 4; ++k) red_add(d.energy + (size_t)t * 5 + k, __double2ll_rn(e4[k] * E_SCALE));
}


// Force-only kernel for any number of LJ types (up to MAX_TYPES; the packed
// kernels' tables hold SMALL_TYPES).  Per warp, shared memory holds the LJ
// coefficients of its 8 i-atoms against every type (row a at a fixed stride,
// so the pair loop addresses them with immediate offsets) and the 27 image
// shifts of its box, registers the i-atoms; the list mask enters the squared
// distance as a penalty (0 or 1e30), so a masked pair falls outside the
// cut-off without any per-pair bit test.  Arithmetic per pair: 3 FADD, 6 FMUL,
// 12 FFMA, 1 RSQ, 1 LDS, 1 FSETP + FSEL.
template <int MINB>
__global__ void __launch_bounds__(PF_WARPS * 32, MINB) k_pair_f(Dev d, SimConst c, const int *clist, int n_items) {
  constexpr int TS = MAX_TYPES;
  __shared__ float2 s_cij[PF_WARPS][CL][TS];
  __shared__ float4 s_sh[PF_WARPS][64];
  __shared__ float s_red[PF_WARPS][3 * CL * 33];
  const int wib = threadIdx.x >> 5;
  const int item = blockIdx.x * PF_WARPS + wib;
  const int lane = threadIdx.x & 31;
  if (item >= n_items) return;
  const int I = clist ? clist[item] : item;
  const int t = d.clus_trial[I];
  const TrialInfo T = d.tinfo[t];
  if (I - T.clus0 >= d.tstate[t].n_clus) return;
  const float L = T.box, iL = T.inv_box;
  const int NT = c.n_types;

  float xi[CL], yi[CL], zi[CL], qi[CL];
  int ti[CL];
#pragma unroll
  for (int a = 0; a < CL; ++a) {
    const float4 p = d.pos[I * CL + a];
    xi[a] = p.x; yi[a] = p.y; zi[a] = p.z; qi[a] = p.w;
    ti[a] = d.type[I * CL + a];
  }
  // per-warp tables: LJ rows of the i-atoms, image shifts (code = (nx+1) | (ny+1)<<2 | (nz+1)<<4)
  for (int k = lane; k < CL * NT; k += 32) {
    const int a = k / NT, tj = k - a * NT;
    int tia = ti[0];
#pragma unroll
    for (int q = 1; q < CL; ++q)
      if (q == a) tia = ti[q];
    s_cij[wib][a][tj] = d.ljtab[tia * NT + tj];
  }
  for (int k = lane; k < 64; k += 32) {
    const int nx = (k & 3) - 1, ny = ((k >> 2) & 3) - 1, nz = ((k >> 4) & 3) - 1;
    s_sh[wib][k] = make_float4(L * nx, L * ny, L * nz, 0.f);
  }
  __syncwarp();
  float fi[CL][3];
#pragma unroll
  for (int a = 0; a < CL; ++a) fi[a][0] = fi[a][1] = fi[a][2] = 0.0f;

  const int n = d.list_n[I], nm = d.list_nm[I];
  const uint32_t *seg = d.list + (size_t)I * c.list_cap;
  const uint8_t *segm = d.list_m + (size_t)I * c.list_cap;
  uint32_t ent = lane < n ? seg[lane] : d.idle_entry;
  uint32_t ent_n = 32 + lane < n ? seg[32 + lane] : d.idle_entry;
  float4 pj = d.pos[(int)(ent & J_MASK)];
  int tj = d.type[(int)(ent & J_MASK)];
  for (int e0 = 0; e0 < n; e0 += 32) {
    const uint32_t ent_nn = e0 + 64 + lane < n ? seg[e0 + 64 + lane] : d.idle_entry;
    const int sj_n = (int)(ent_n & J_MASK);
    const float4 pj_n = d.pos[sj_n];
    const int tj_n = d.type[sj_n];
    const int sj = (int)(ent & J_MASK);
    const float4 shv = s_sh[wib][(ent >> J_BITS) & 63u];
    const float xj = pj.x - shv.x, yj = pj.y - shv.y, zj = pj.z - shv.z, qj = pj.w;
    const bool masked = e0 < nm;
    const unsigned mb = masked && e0 + lane < n ? segm[e0 + lane] : 0u;
    const bool exact = (ent & E_EXACT) != 0u;
    const float2 *row = &s_cij[wib][0][tj];
    // j-force: even and odd i-atoms in two partial sums (the packed variant's order)
    float fjx[2] = {0.f, 0.f}, fjy[2] = {0.f, 0.f}, fjz[2] = {0.f, 0.f};
    // one image per entry; MASKED: the pair masks apply (a group with
    // exclusions or the cluster itself); else the cut-off alone decides, which
    // gives the same forces: a listed pair that failed the list rule is still
    // beyond the cut-off (lists are rebuilt before any atom has moved skin/2)
    auto one_image = [&](auto mtag) {
      constexpr bool MASKED = decltype(mtag)::value;
#pragma unroll
      for (int a = 0; a < CL; ++a) {
        const float4 ia = make_float4(xi[a], yi[a], zi[a], qi[a]);
        const float pen = MASKED ? ((mb & (1u << a)) ? 0.0f : MASK_PEN) : 0.0f;
        const float dx = __fsub_rn(xj, ia.x), dy = __fsub_rn(yj, ia.y), dz = __fsub_rn(zj, ia.z);
        const float r2 = __fmaf_rn(dz, dz, __fmaf_rn(dy, dy, __fmaf_rn(dx, dx, pen)));
        const float rinv = rsqrtf(r2);
        const float rinv2 = __fmul_rn(rinv, rinv);
        const float rinv6 = __fmul_rn(__fmul_rn(rinv2, rinv2), rinv2);
        const float2 cc = row[a * TS];
        const float qq = __fmul_rn(ia.w, qj);
        float tt = __fmaf_rn(cc.y, rinv6, -cc.x);
        tt = __fmul_rn(tt, rinv6);
        tt = __fmaf_rn(qq, rinv, tt);
        tt = __fmul_rn(tt, rinv2);
        float f = __fmaf_rn(-qq, c.two_krf, tt);
        f = r2 < c.rc2 ? f : 0.0f;
        fi[a][0] = __fmaf_rn(-f, dx, fi[a][0]);
        fi[a][1] = __fmaf_rn(-f, dy, fi[a][1]);
        fi[a][2] = __fmaf_rn(-f, dz, fi[a][2]);
        fjx[a & 1] = __fmaf_rn(f, dx, fjx[a & 1]);
        fjy[a & 1] = __fmaf_rn(f, dy, fjy[a & 1]);
        fjz[a & 1] = __fmaf_rn(f, dz, fjz[a & 1]);
      }
    };
    if (!masked) {
      one_image(std::false_type{});
    } else if (!__any_sync(0xffffffffu, exact)) {
      one_image(std::true_type{});
    } else {
      // some entry of this group needs pair-by-pair minimum images
#pragma unroll
      for (int a = 0; a < CL; ++a) {
        const float4 ia = make_float4(xi[a], yi[a], zi[a], qi[a]);
        const float pen = (mb & (1u << a)) ? 0.0f : MASK_PEN;
        float dx = __fsub_rn(xj, ia.x), dy = __fsub_rn(yj, ia.y), dz = __fsub_rn(zj, ia.z);
        if (exact) {
          dx = __fmaf_rn(-L, rintf(__fmul_rn(dx, iL)), dx);
          dy = __fmaf_rn(-L, rintf(__fmul_rn(dy, iL)), dy);
          dz = __fmaf_rn(-L, rintf(__fmul_rn(dz, iL)), dz);
        }
        const float r2 = __fmaf_rn(dz, dz, __fmaf_rn(dy, dy, __fmaf_rn(dx, dx, pen)));
        const float rinv = rsqrtf(r2);
        const float rinv2 = __fmul_rn(rinv, rinv);
        const float rinv6 = __fmul_rn(__fmul_rn(rinv2, rinv2), rinv2);
        const float2 cc = row[a * TS];
        const float qq = __fmul_rn(ia.w, qj);
        float tt = __fmaf_rn(cc.y, rinv6, -cc.x);
        tt = __fmul_rn(tt, rinv6);
        tt = __fmaf_rn(qq, rinv, tt);
        tt = __fmul_rn(tt, rinv2);
        float f = __fmaf_rn(-qq, c.two_krf, tt);
        f = r2 < c.rc2 ? f : 0.0f;
        fi[a][0] = __fmaf_rn(-f, dx, fi[a][0]);
        fi[a][1] = __fmaf_rn(-f, dy, fi[a][1]);
        fi[a][2] = __fmaf_rn(-f, dz, fi[a][2]);
        fjx[a & 1] = __fmaf_rn(f, dx, fjx[a & 1]);
        fjy[a & 1] = __fmaf_rn(f, dy, fjy[a & 1]);
        fjz[a & 1] = __fmaf_rn(f, dz, fjz[a & 1]);
      }
    }
    const float sx = fjx[0] + fjx[1], sy = fjy[0] + fjy[1], sz = fjz[0] + fjz[1];
    if (sx != 0.f || sy != 0.f || sz != 0.f) {
      red_add(d.fx + sj, fx_from(sx));
      red_add(d.fy + sj, fx_from(sy));
      red_add(d.fz + sj, fx_from(sz));
    }
    ent = ent_n;
    ent_n = ent_nn;
    pj = pj_n;
    tj = tj_n;
  }

  // i-forces: column sums of the 32 lanes' partials in a fixed order
  float *r = s_red[wib];
#pragma unroll
  for (int a = 0; a < CL; ++a)
#pragma unroll
    for (int k = 0; k < 3; ++k) r[(3 * a + k) * 33 + lane] = fi[a][k];
  __syncwarp();
  if (lane < 3 * CL) {
    float sum = 0.f;
    for (int l = 0; l < 32; ++l) sum += r[lane * 33 + l];
    const int a = lane / 3, comp = lane - 3 * a;
    const long long val = fx_from(sum);
    if (val != 0) red_add((comp == 0 ? d.fx : comp == 1 ? d.fy : d.fz) + I * CL + a, val);
  }
}

// Packed variant: the same pair loop on FP32x2 arithmetic (FADD2, FMUL2,
// FFMA2: one instruction for two pairs) over the i-atom pairs (2p, 2p+1).
// The i-atoms sit in shared memory as {-x, -x', -y, -y'} {-z, -z', q, q'} and the
// LJ row of an i-atom pair is {c12, c12', -c6, -c6'}; per two pairs the loop
// issues 3 FADD2, 6 FMUL2, 7 FFMA2, 2 RSQ, 3 LDS.128 and, per pair, one mask
// test joined with the cut-off test and a select (a masked pair may compute
// inf or NaN on the way; the select discards it).  The i-force partials accumulate +f*d and are negated once
// (exactly the sum of -f*d: round-to-nearest is sign-symmetric); the j-force
// sums even and odd i-atoms in two partials, as the scalar variants do, so
// all variants give bit-identical forces.


template <int MINB, int U>
__global__ void __launch_bounds__(PF_WARPS * 32, MINB) k_pair_f2(Dev d, SimConst c, unsigned *next, const int *clist,
                                                                   int n_items) {
  __shared__ PairF2Shared<PF_WARPS> sh;
  const int lane = threadIdx.x & 31;
  // persistent warps: each takes the next i-cluster from a counter until none
  // is left, so that short and long lists even out across the SMs
  for (;;) {
    __syncwarp();  // the warp's tables of its previous cluster are no longer read
    unsigned got = 0u;
    if (lane == 0) got = atomicAdd(next, 1u);
    const int item = (int)__shfl_sync(0xffffffffu, got, 0);
    if (item >= n_items) return;
    pair_cluster_f2<U>(d, c, sh, clist ? clist[item] : item);
  }
}

// The same with one warp per block and i-cluster, the blocks dealt out by the
// hardware: without the counter's fetch before every cluster, and with lists
// of every length on every SM (they get shorter along the clusters), a batch
// whose clusters are few per SM is done sooner.
template <int U, int MINB>
__global__ void __launch_bounds__(32, MINB) k_pair_w(Dev d, SimConst c, const int *clist, int n_items) {
  __shared__ PairF2Shared<1> sh;
  PDL_WAIT();
  const int item = blockIdx.x;
  pair_cluster_f2<U>(d, c, sh, clist ? clist[item] : item);
}

// Forces and nonbonded energies in one pass over the lists (24 warps per SM: 132
// us for 16 configurations of 11 040 atoms, 162 with the energy terms scalar and
// behind a branch per pair; 16 warps 150, 20: 138, 28: 161).
__global__ void __launch_bounds__(32, 24) k_pair_e(Dev d, SimConst c) {
  __shared__ PairF2Shared<1, true> sh;
  pair_cluster_f2<1, 1, true>(d, c, sh, blockIdx.x);
}

// Bonded energies, one thread per slot (each atom's share of every term it is
// part of); the 8 atoms of a cluster are added in FP64 before the fixed-point
// sum, as the general energy kernel does.
__global__ void __launch_bounds__(256) k_bonded_energy(Dev d) {
  const int slot = blockIdx.x * 256 + threadIdx.x;
  const bool in = slot < d.total_slots;
  const int t = in ? d.slot_trial[slot] : 0;
  const int o = in ? d.orig[slot] : -1;
  float eb = 0.f, ea = 0.f;
  if (o >= 0) bonded_energy(d, d.tinfo[t], o, d.pos[slot], eb, ea);
  double e2[2] = {(double)eb, (double)ea};
#pragma unroll
  for (int k = 0; k < 2; ++k)
#pragma unroll
    for (int off = 4; off > 0; off >>= 1) e2[k] += __shfl_xor_sync(0xffffffffu, e2[k], off);
  if (in && (slot & (CL - 1)) == 0)
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const long long v = __double2ll_rn(e2[k] * E_SCALE);
      if (v != 0) red_add(d.energy + (size_t)t * 5 + 2 + k, v);
    }
}

__global__ void __launch_bounds__(256) k_bonded(Dev d) {
  bonded_group(d, blockIdx.y, blockIdx.x * blockDim.x + threadIdx.x);
}

void launch_bonded(const Dev &d, cudaStream_t s) {
  if (d.max_nbg <= 0) return;
  k_bonded<<<dim3((unsigned)((d.max_nbg + 255) / 256), (unsigned)d.n_trials), 256, 0, s>>>(d);
}

// Forces and nonbonded energies of every trial in one pass over the lists, in
// place of the force kernel and the general energy kernel (130 and 178 us for
// 16 configurations of 11 040 atoms); for types that fit the packed kernel's
// tables.
bool pair_energy_in_one_pass(const SimConst &c) { return c.n_types <= SMALL_TYPES; }
void launch_pair_energy(const Dev &d, const SimConst &c, cudaStream_t s) {
  k_pair_e<<<(unsigned)d.total_clus, 32, 0, s>>>(d, c);
}
void launch_bonded_energy(const Dev &d, cudaStream_t s) {
  k_bonded_energy<<<(unsigned)((d.total_slots + 255) / 256), 256, 0, s>>>(d);
}

// Variants (all do the same arithmetic in the same order: bit-identical
// forces).  0, 1, 2: any number of types, registers capped for 4, 5 or 6
// blocks per SM.  The others need at most SMALL_TYPES types (else variant 0
// runs): 3, 4: one warp per block, two groups of entries at a time, 20 or 16
// warps per SM; 5, 6: persistent blocks, two groups at a time, 4 or 5 blocks;
// 7, 8: persistent blocks, one group at a time, 6 or 7 blocks.
// The variant of a batch that has not been tuned: the packed kernels whenever
// the types fit.  Up to 300 clusters per SM one warp per block is the faster
// form (the MD step of one 11 040-atom trial 43.1 us against 51.2, of 16
// trials 213 against 219, of ten 30 000-atom trials 352.2 against 352.9), in
// larger batches the persistent one (64 trials 695 against 706 us).  Up to 50
// clusters per SM 128 registers pay more than 20 warps: the step of one trial
// of 1320 / 11 040 / 30 000 atoms 29.1 -> 28.4 / 33.0 -> 32.6 / 53.5 -> 52.2
// us, of four of 11 040 68.3 -> 67.7, but of 16 (157 per SM) 171 -> 174.
int default_pair_variant(const Dev &d, const SimConst &c) {
  if (c.n_types > SMALL_TYPES) return 0;
  return d.total_clus <= 50 * d.n_sm ? 4 : d.total_clus <= 300 * d.n_sm ? 3 : 6;
}

void launch_pair(const Dev &d, const SimConst &c, bool energy, int32_t only_trial, cudaStream_t s, int variant,
                 const int *clist, int n_items) {
  long long threads = (long long)d.total_clus * 32;
  unsigned blocks = (unsigned)((threads + 127) / 128);
  const size_t nt2 = (size_t)c.n_types * c.n_types;
  if (energy || only_trial >= 0) {
    k_pair<<<blocks, 128, nt2 * (sizeof(float2) + sizeof(float)), s>>>(d, c, only_trial);
    return;
  }
  if (!clist) n_items = d.total_clus;
  if (n_items <= 0) return;
  const unsigned fb = (unsigned)((n_items + PF_WARPS - 1) / PF_WARPS);
  if (variant >= 3 && c.n_types > SMALL_TYPES) variant = 0;
  switch (variant) {
    case 1: k_pair_f<5><<<fb, PF_WARPS * 32, 0, s>>>(d, c, clist, n_items); break;
    case 2: k_pair_f<6><<<fb, PF_WARPS * 32, 0, s>>>(d, c, clist, n_items); break;
    case 3: launch_pdl(k_pair_w<2, 20>, dim3(n_items), dim3(32), s, d, c, clist, n_items); break;
    case 4: launch_pdl(k_pair_w<2, 16>, dim3(n_items), dim3(32), s, d, c, clist, n_items); break;
    case 5: case 6: case 7: case 8: {
      // persistent grid: as many blocks as can be resident, sized from the SM
      // count; the counter hands out the i-clusters
      const int minb = variant - 1;
      const unsigned pb = std::min(fb, (unsigned)(d.n_sm * minb));
      cudaMemsetAsync(d.pair_next, 0, sizeof(unsigned), s);
      if (variant == 5) k_pair_f2<4, 2><<<pb, PF_WARPS * 32, 0, s>>>(d, c, d.pair_next, clist, n_items);
      else if (variant == 6) k_pair_f2<5, 2><<<pb, PF_WARPS * 32, 0, s>>>(d, c, d.pair_next, clist, n_items);
      else if (variant == 7) k_pair_f2<6, 1><<<pb, PF_WARPS * 32, 0, s>>>(d, c, d.pair_next, clist, n_items);
      else k_pair_f2<7, 1><<<pb, PF_WARPS * 32, 0, s>>>(d, c, d.pair_next, clist, n_items);
      break;
    }
    default: k_pair_f<4><<<fb, PF_WARPS * 32, 0, s>>>(d, c, clist, n_items); break;
  }
}

}  // namespace vp
