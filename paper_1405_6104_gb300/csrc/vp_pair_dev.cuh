// vp_pair_dev.cuh -- device functions of the force kernels (the packed
// nonbonded pair loop of one i-cluster, the bonded terms of one group),
// shared by the separate kernels and the one-kernel step.
#pragma once
#include <type_traits>

#include "vp_dev.cuh"

namespace vp {

// displacement x_p - x_self under the minimum image, with the image shift
// subtracted from x_p first (exact when the two are within a box length)
__device__ __forceinline__ float3 min_disp(float4 self, float4 other, float L, float iL) {
  float nx = rintf((other.x - self.x) * iL), ny = rintf((other.y - self.y) * iL), nz = rintf((other.z - self.z) * iL);
  return make_float3((other.x - L * nx) - self.x, (other.y - L * ny) - self.y, (other.z - L * nz) - self.z);
}

// launch shape of the force-only pair kernels: warps per block, the penalty
// of a masked pair
constexpr int PF_WARPS = 4;
constexpr float MASK_PEN = 1.0e30f;
// row of an i-force component's 32 partial sums: 16-byte loads without bank conflicts
constexpr int RED_STRIDE = 36;

// the energies' tables of a warp: {c12, c12', -c6, -c6'} (over r^12 and r^6) and
// minus the potential at the cut-off per i-atom pair and type
template <int NW, bool ENERGY>
struct PairEnergyTables {
  float4 s_e4[NW][CL / 2][SMALL_TYPES];
  float2 s_ts[NW][CL / 2][SMALL_TYPES];
};
template <int NW>
struct PairEnergyTables<NW, false> {};

// shared memory of the packed pair kernel's warps
template <int NW, bool ENERGY = false>
struct PairF2Shared : PairEnergyTables<NW, ENERGY> {
  float4 s_c4[NW][CL / 2][SMALL_TYPES];
  float4 s_sh[NW][64];
  float4 s_ip[NW][CL / 2][2];
  alignas(16) float s_red[NW][3 * CL * RED_STRIDE];
};

// The forces of one i-cluster I by the calling warp (packed arithmetic): one
// j-atom entry per lane, U groups of 32 entries at a time.  U = 1 keeps the
// registers low (a high block count per SM hides the j-atom's load).  U = 2
// loads the j-atoms of the next two groups while the current two are
// evaluated, interleaves the two groups' arithmetic (two independent chains
// per warp) and reads each i-atom pair from shared memory once for both: 96
// registers, 20 warps per SM, and still faster at every batch size (64 x
// 11 040 atoms 366 us against 419 with U = 1 and 24 warps; one trial 13
// against 20 us; U = 3 and 4, U = 2 without the early loads, or two iterations
// unrolled (456 us: too much code for the instruction cache) are slower).  An
// odd last group is taken by itself (an idle second one and the wider loads of
// the i-force sums were 2.7% of the time, loading the masked groups' j-atoms when
// they are due another 1.3%).
// Every accumulator takes its terms in the order of the groups either way:
// the same forces bit for bit.
// ENERGY (U = 1): the Lennard-Jones and reaction-field energies too, each lane
// adding its pairs' in the order of the entries and i-atoms.
template <int U, int NW, bool ENERGY = false>
__device__ __forceinline__ void pair_cluster_f2(const Dev &d, const SimConst &c, PairF2Shared<NW, ENERGY> &sh, int I) {
  static_assert(U <= 2, "an odd last group is the only remainder taken");
  static_assert(!ENERGY || U == 1, "the energies' sums take one group at a time");
  constexpr int TS = SMALL_TYPES;
  auto &s_c4 = sh.s_c4;
  auto &s_sh = sh.s_sh;
  auto &s_ip = sh.s_ip;
  auto &s_red = sh.s_red;
  const int wib = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const int NT = c.n_types;
  const int t = d.clus_trial[I];
  // the loads that need only I go out before those that need the trial (one
  // memory round trip less before the pair loop): the list's first two
  // groups (taken only below list_n, read within the cluster's segment), the
  // i-atoms and their types
  const int n = d.list_n[I], nm = d.list_nm[I];
  const uint32_t *seg = d.list + (size_t)I * c.list_cap;
  const uint8_t *segm = d.list_m + (size_t)I * c.list_cap;
  // the list words stream through L2 (the batch's lists are larger than L2)
  // with the evict-first hint, so that they do not push out the positions
  // and force accumulators every lane keeps coming back to
  const uint32_t raw0 = lane < c.list_cap ? __ldcs(seg + lane) : d.idle_entry;
  const uint32_t raw1 = 32 + lane < c.list_cap ? __ldcs(seg + 32 + lane) : d.idle_entry;
  float4 a0 = make_float4(0.f, 0.f, 0.f, 0.f), a1 = a0;
  if (lane < CL / 2) {
    a0 = d.pos[I * CL + 2 * lane];
    a1 = d.pos[I * CL + 2 * lane + 1];
  }
  int ty[2][2] = {{0, 0}, {0, 0}};  // the i-atom types of this lane's table rows (at most two per lane)
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    const int k = lane + 32 * r;
    if (k < (CL / 2) * NT) {
      const int p = k / NT;
      ty[r][0] = d.type[I * CL + 2 * p];
      ty[r][1] = d.type[I * CL + 2 * p + 1];
    }
  }
  const TrialInfo T = d.tinfo[t];
  if (I - T.clus0 >= d.tstate[t].n_clus) return;
  const float L = T.box, iL = T.inv_box;

  if (lane < CL / 2) {
    // negated coordinates: d = xj + (-xi) in one FADD2 (a packed operand has no negate modifier)
    s_ip[wib][lane][0] = make_float4(-a0.x, -a1.x, -a0.y, -a1.y);
    s_ip[wib][lane][1] = make_float4(-a0.z, -a1.z, a0.w, a1.w);
  }
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    const int k = lane + 32 * r;
    if (k < (CL / 2) * NT) {
      const int p = k / NT, tj = k - p * NT;
      const float2 c0 = d.ljtab[ty[r][0] * NT + tj], c1 = d.ljtab[ty[r][1] * NT + tj];
      s_c4[wib][p][tj] = make_float4(c0.y, c1.y, -c0.x, -c1.x);
      if constexpr (ENERGY) {
        sh.s_e4[wib][p][tj] = make_float4(__fmul_rn(c0.y, 1.0f / 12.0f), __fmul_rn(c1.y, 1.0f / 12.0f),
                                          -__fmul_rn(c0.x, 1.0f / 6.0f), -__fmul_rn(c1.x, 1.0f / 6.0f));
        sh.s_ts[wib][p][tj] = make_float2(-d.ljshift[ty[r][0] * NT + tj], -d.ljshift[ty[r][1] * NT + tj]);
      }
    }
  }
  for (int k = lane; k < 64; k += 32) {
    const int ix = (k & 3) - 1, iy = ((k >> 2) & 3) - 1, iz = ((k >> 4) & 3) - 1;
    s_sh[wib][k] = make_float4(L * ix, L * iy, L * iz, 0.f);
  }
  __syncwarp();
  float2 fx[CL / 2], fy[CL / 2], fz[CL / 2];
#pragma unroll
  for (int p = 0; p < CL / 2; ++p) fx[p] = fy[p] = fz[p] = make_float2(0.f, 0.f);
  const float2 m2krf = make_float2(-c.two_krf, -c.two_krf);
  const float rc2 = c.rc2;
  float elj = 0.0f, erf = 0.0f;
  // the energies of the pairs inside the cut-off of i-atom pair p, added in the
  // order of the i-atoms (a pair that is left out may be inf or NaN)
  auto add_energies = [&](int tj, int p, float2 rinv, float2 rinv6, float2 r2, float2 qq, bool inx, bool iny) {
    if constexpr (ENERGY) {
      const float4 e = sh.s_e4[wib][p][tj];
      const float2 lj = __ffma2_rn(make_float2(e.x, e.y), rinv6, make_float2(e.z, e.w));
      const float2 el = __ffma2_rn(rinv6, lj, sh.s_ts[wib][p][tj]);
      const float2 rf = __fadd2_rn(__ffma2_rn(make_float2(c.krf, c.krf), r2, rinv), make_float2(-c.crf, -c.crf));
      elj = inx ? __fadd_rn(elj, el.x) : elj;
      erf = inx ? __fmaf_rn(qq.x, rf.x, erf) : erf;
      elj = iny ? __fadd_rn(elj, el.y) : elj;
      erf = iny ? __fmaf_rn(qq.y, rf.y, erf) : erf;
    }
  };

  // one pair of i-atoms (2p, 2p + 1) against this lane's j-atom (image
  // already applied): the i-forces into fx/fy/fz, the j-force into gx/gy/gz
  struct JAtom {
    float2 x, y, z, q;
    const float4 *row;
    int tj;
    float2 gx, gy, gz;
  };
  auto j_atom = [&](float4 pj, int tj, uint32_t ent) {
    const float4 shv = s_sh[wib][(ent >> J_BITS) & 63u];
    const float xj = pj.x - shv.x, yj = pj.y - shv.y, zj = pj.z - shv.z;
    JAtom j;
    j.x = make_float2(xj, xj);
    j.y = make_float2(yj, yj);
    j.z = make_float2(zj, zj);
    j.q = make_float2(pj.w, pj.w);
    j.row = &s_c4[wib][0][tj];
    j.tj = tj;
    j.gx = j.gy = j.gz = make_float2(0.f, 0.f);
    return j;
  };
  // one image per entry; MASKED: the pair masks apply (a group with
  // exclusions or the cluster itself); else the cut-off alone decides, which
  // gives the same forces: a listed pair that failed the list rule is still
  // beyond the cut-off (lists are rebuilt before any atom has moved skin/2)
  auto pair2 = [&](auto mtag, JAtom &j, int p, float4 i0, float4 i1, unsigned mb) {
    constexpr bool MASKED = decltype(mtag)::value;
    const float2 dx = __fadd2_rn(j.x, make_float2(i0.x, i0.y));
    const float2 dy = __fadd2_rn(j.y, make_float2(i0.z, i0.w));
    const float2 dz = __fadd2_rn(j.z, make_float2(i1.x, i1.y));
    // the mask bit joins the cut-off test (the same forces as the penalty form)
    const float2 r2 = __ffma2_rn(dz, dz, __ffma2_rn(dy, dy, __fmul2_rn(dx, dx)));
    const float2 rinv = make_float2(rsqrtf(r2.x), rsqrtf(r2.y));
    const float2 rinv2 = __fmul2_rn(rinv, rinv);
    const float2 rinv6 = __fmul2_rn(__fmul2_rn(rinv2, rinv2), rinv2);
    const float4 cc = j.row[p * TS];
    const float2 qq = __fmul2_rn(make_float2(i1.z, i1.w), j.q);
    float2 tt = __ffma2_rn(make_float2(cc.x, cc.y), rinv6, make_float2(cc.z, cc.w));
    tt = __fmul2_rn(tt, rinv6);
    tt = __ffma2_rn(qq, rinv, tt);
    tt = __fmul2_rn(tt, rinv2);
    float2 f = __ffma2_rn(qq, m2krf, tt);
    const bool inx = (!MASKED || (mb & (1u << (2 * p)))) && r2.x < rc2,
               iny = (!MASKED || (mb & (1u << (2 * p + 1)))) && r2.y < rc2;
    f.x = inx ? f.x : 0.0f;
    f.y = iny ? f.y : 0.0f;
    add_energies(j.tj, p, rinv, rinv6, r2, qq, inx, iny);
    fx[p] = __ffma2_rn(f, dx, fx[p]);
    fy[p] = __ffma2_rn(f, dy, fy[p]);
    fz[p] = __ffma2_rn(f, dz, fz[p]);
    j.gx = __ffma2_rn(f, dx, j.gx);
    j.gy = __ffma2_rn(f, dy, j.gy);
    j.gz = __ffma2_rn(f, dz, j.gz);
  };
  auto add_j = [&](const JAtom &j, int sj) {
    const float fjx = j.gx.x + j.gx.y, fjy = j.gy.x + j.gy.y, fjz = j.gz.x + j.gz.y;
    if (fjx != 0.f || fjy != 0.f || fjz != 0.f) {
      red_add(d.fx + sj, fx_from(fjx));
      red_add(d.fy + sj, fx_from(fjy));
      red_add(d.fz + sj, fx_from(fjz));
    }
  };
  // a group that needs the pair masks: one image per entry, or (some entry
  // of the group) pair-by-pair minimum images
  auto masked_group = [&](float4 pj, int tj, uint32_t ent, unsigned mb) {
    const bool exact = (ent & E_EXACT) != 0u;
    JAtom j = j_atom(pj, tj, ent);
    if (!__any_sync(0xffffffffu, exact)) {
#pragma unroll
      for (int p = 0; p < CL / 2; ++p) pair2(std::true_type{}, j, p, s_ip[wib][p][0], s_ip[wib][p][1], mb);
    } else {
#pragma unroll
      for (int p = 0; p < CL / 2; ++p) {
        const float4 i0 = s_ip[wib][p][0], i1 = s_ip[wib][p][1];
        const float4 cc = j.row[p * TS];
        float2 f2v, dx2, dy2, dz2, rinv_2, rinv6_2, r2_2, qq_2;
#pragma unroll
        for (int hh = 0; hh < 2; ++hh) {
          const float pen = (mb & (1u << (2 * p + hh))) ? 0.0f : MASK_PEN;
          float dx = __fadd_rn(j.x.x, hh ? i0.y : i0.x), dy = __fadd_rn(j.y.x, hh ? i0.w : i0.z),
                dz = __fadd_rn(j.z.x, hh ? i1.y : i1.x);
          if (exact) {
            dx = __fmaf_rn(-L, rintf(__fmul_rn(dx, iL)), dx);
            dy = __fmaf_rn(-L, rintf(__fmul_rn(dy, iL)), dy);
            dz = __fmaf_rn(-L, rintf(__fmul_rn(dz, iL)), dz);
          }
          const float r2 = __fmaf_rn(dz, dz, __fmaf_rn(dy, dy, __fmaf_rn(dx, dx, pen)));
          const float rinv = rsqrtf(r2);
          const float rinv2 = __fmul_rn(rinv, rinv);
          const float rinv6 = __fmul_rn(__fmul_rn(rinv2, rinv2), rinv2);
          const float qq = __fmul_rn(hh ? i1.w : i1.z, j.q.x);
          float tt = __fmaf_rn(hh ? cc.y : cc.x, rinv6, hh ? cc.w : cc.z);
          tt = __fmul_rn(tt, rinv6);
          tt = __fmaf_rn(qq, rinv, tt);
          tt = __fmul_rn(tt, rinv2);
          float f = __fmaf_rn(qq, -c.two_krf, tt);
          f = r2 < rc2 ? f : 0.0f;
          if (hh) { f2v.y = f; dx2.y = dx; dy2.y = dy; dz2.y = dz; rinv_2.y = rinv; rinv6_2.y = rinv6; r2_2.y = r2; qq_2.y = qq; }
          else { f2v.x = f; dx2.x = dx; dy2.x = dy; dz2.x = dz; rinv_2.x = rinv; rinv6_2.x = rinv6; r2_2.x = r2; qq_2.x = qq; }
        }
        add_energies(j.tj, p, rinv_2, rinv6_2, r2_2, qq_2, r2_2.x < rc2, r2_2.y < rc2);
        fx[p] = __ffma2_rn(f2v, dx2, fx[p]);
        fy[p] = __ffma2_rn(f2v, dy2, fy[p]);
        fz[p] = __ffma2_rn(f2v, dz2, fz[p]);
        j.gx = __ffma2_rn(f2v, dx2, j.gx);
        j.gy = __ffma2_rn(f2v, dy2, j.gy);
        j.gz = __ffma2_rn(f2v, dz2, j.gz);
      }
    }
    add_j(j, (int)(ent & J_MASK));
  };

  if constexpr (U == 1) {
    // entries are fetched two groups ahead, the j-atom itself at the top of
    // its iteration (fewer live registers: a higher block count per SM hides
    // that load better than a prefetch does)
    uint32_t ent = lane < n ? raw0 : d.idle_entry;
    uint32_t ent_n = 32 + lane < n ? raw1 : d.idle_entry;
    for (int e0 = 0; e0 < n; e0 += 32) {
      const uint32_t ent_nn = e0 + 64 + lane < n ? __ldcs(seg + e0 + 64 + lane) : d.idle_entry;
      const int sj = (int)(ent & J_MASK);
      const float4 pj = d.pos[sj];
      const int tj = d.type[sj];
      if (e0 < nm) {  // the pair masks, in the groups that need them (the first nm entries)
        masked_group(pj, tj, ent, e0 + lane < n ? segm[e0 + lane] : 0u);
      } else {
        JAtom j = j_atom(pj, tj, ent);
#pragma unroll
        for (int p = 0; p < CL / 2; ++p) pair2(std::false_type{}, j, p, s_ip[wib][p][0], s_ip[wib][p][1], 0u);
        add_j(j, sj);
      }
      ent = ent_n;
      ent_n = ent_nn;
    }
  } else {
    const int e1 = (min(nm, n) + 31) & ~31;  // the groups from here on need no masks
    auto entry = [&](int e) { return e < n ? __ldcs(seg + e) : d.idle_entry; };
    // the masked groups' j-atoms are loaded a group ahead
    uint32_t em_n = 0u;
    float4 pm_n = make_float4(0.f, 0.f, 0.f, 0.f);
    int tm_n = 0;
    unsigned mb_n = 0u;
    auto masked_load = [&](int e0) {
      const uint32_t w = e0 == 0 ? raw0 : e0 == 32 ? raw1 : entry(e0 + lane);
      em_n = e0 + lane < n ? w : d.idle_entry;
      pm_n = d.pos[em_n & J_MASK];
      tm_n = d.type[em_n & J_MASK];
      mb_n = e0 + lane < n ? segm[e0 + lane] : 0u;
    };
    if (e1 > 0) masked_load(0);
    // the first U clean groups' j-atoms and the next ones' entries are in
    // flight while the masked groups are evaluated
    uint32_t ent[U], ent_n[U];
    float4 pj[U];
    int tj[U];
#pragma unroll
    for (int u = 0; u < U; ++u) ent[u] = entry(e1 + 32 * u + lane);
#pragma unroll
    for (int u = 0; u < U; ++u) ent_n[u] = entry(e1 + 32 * (U + u) + lane);
#pragma unroll
    for (int u = 0; u < U; ++u) {
      pj[u] = d.pos[ent[u] & J_MASK];
      tj[u] = d.type[ent[u] & J_MASK];
    }
    for (int e0 = 0; e0 < e1; e0 += 32) {
      const uint32_t em = em_n;
      const float4 pm = pm_n;
      const int tm = tm_n;
      const unsigned mb = mb_n;
      if (e0 + 32 < e1) masked_load(e0 + 32);
      masked_group(pm, tm, em, mb);
    }
    int e0 = e1;
    for (; e0 + 32 < n; e0 += 32 * U) {
      float4 pj_n[U];
      int tj_n[U];
      uint32_t ent_nn[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        pj_n[u] = d.pos[ent_n[u] & J_MASK];
        tj_n[u] = d.type[ent_n[u] & J_MASK];
        ent_nn[u] = entry(e0 + 32 * (2 * U + u) + lane);
      }
      JAtom j[U];
#pragma unroll
      for (int u = 0; u < U; ++u) j[u] = j_atom(pj[u], tj[u], ent[u]);
#pragma unroll
      for (int p = 0; p < CL / 2; ++p) {
        const float4 i0 = s_ip[wib][p][0], i1 = s_ip[wib][p][1];
#pragma unroll
        for (int u = 0; u < U; ++u) pair2(std::false_type{}, j[u], p, i0, i1, 0u);
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        add_j(j[u], (int)(ent[u] & J_MASK));
        ent[u] = ent_n[u];
        ent_n[u] = ent_nn[u];
        pj[u] = pj_n[u];
        tj[u] = tj_n[u];
      }
    }
    if (e0 < n) {  // an odd last group (the second one would hold idle entries only, which add nothing)
      JAtom j = j_atom(pj[0], tj[0], ent[0]);
#pragma unroll
      for (int p = 0; p < CL / 2; ++p) pair2(std::false_type{}, j, p, s_ip[wib][p][0], s_ip[wib][p][1], 0u);
      add_j(j, (int)(ent[0] & J_MASK));
    }
  }

  // the i-forces (minus these sums), added up in the order of the lanes
  float *r = s_red[wib];
#pragma unroll
  for (int p = 0; p < CL / 2; ++p) {
    const float2 f3[3] = {fx[p], fy[p], fz[p]};
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      r[(6 * p + k) * RED_STRIDE + lane] = f3[k].x;
      r[(6 * p + 3 + k) * RED_STRIDE + lane] = f3[k].y;
    }
  }
  __syncwarp();
  if (lane < 3 * CL) {
    float sum = 0.f;
#pragma unroll
    for (int l = 0; l < 32; l += 4) {
      const float4 v = *reinterpret_cast<const float4 *>(r + lane * RED_STRIDE + l);
      sum = __fadd_rn(__fadd_rn(__fadd_rn(__fadd_rn(sum, v.x), v.y), v.z), v.w);
    }
    const int a = lane / 3, comp = lane - 3 * a;
    const long long val = fx_from(-sum);
    if (val != 0) red_add((comp == 0 ? d.fx : comp == 1 ? d.fy : d.fz) + I * CL + a, val);
  }
  if constexpr (ENERGY) {
    double e2[2] = {(double)elj, (double)erf};
#pragma unroll
    for (int k = 0; k < 2; ++k)
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) e2[k] += __shfl_xor_sync(0xffffffffu, e2[k], off);
    if (lane == 0)
#pragma unroll
      for (int k = 0; k < 2; ++k) red_add(d.energy + (size_t)t * 5 + k, __double2ll_rn(e2[k] * E_SCALE));
  }
}


// Bonded forces, one thread per (trial, group of terms over at most 3 atoms;
// a water's angle and bonds form one group): every term's forces are
// converted to fixed point and summed per atom, exactly, so the group issues
// one reduction per atom and component (exact action-reaction: a bond's
// second atom and an angle's vertex take minus the others' forces).  A kernel of
// its own, beside the pair kernel: inside the pair kernel's warps the per-atom
// term loops ran on 8 of 32 lanes behind chains of dependent loads.
__device__ __forceinline__ void add3(long long (&F)[3][3], int m, long long x, long long y, long long z) {
#pragma unroll
  for (int q = 0; q < 3; ++q)
    if (q == m) { F[q][0] += x; F[q][1] += y; F[q][2] += z; }
}

__device__ __forceinline__ float4 pick3(const float4 (&p)[3], int m) { return m == 0 ? p[0] : m == 1 ? p[1] : p[2]; }

// group k of trial t's system
__device__ __forceinline__ void bonded_group(const Dev &d, int t, int k) {
  const TrialInfo T = d.tinfo[t];
  if (k >= d.sys_nbg[T.sys]) return;
  const BGroup G = d.bgrp[d.sys_bg0[T.sys] + k];
  const float L = T.box, iL = T.inv_box;
  int sl[3];
  float4 p[3];
#pragma unroll
  for (int m = 0; m < 3; ++m) {
    sl[m] = G.at[m] >= 0 ? d.slot_of[T.atom0 + G.at[m]] : -1;
    p[m] = sl[m] >= 0 ? d.pos[sl[m]] : make_float4(0.f, 0.f, 0.f, 0.f);
  }
  long long F[3][3] = {{0, 0, 0}, {0, 0, 0}, {0, 0, 0}};
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    if (q >= G.n) break;
    const int code = G.code[q];
    const float4 par = G.par[q];
    const int li = (code >> 1) & 3, lj = (code >> 3) & 3, ll = (code >> 5) & 3;
    const float4 pa = pick3(p, li), pb = pick3(p, lj);
    if ((code & 1) == 0) {
      // bond a-b, V = k/2 (r - r0)^2: the stretch in float-float (exact coordinate differences)
      const float nx = rintf((pb.x - pa.x) * iL), ny = rintf((pb.y - pa.y) * iL), nz = rintf((pb.z - pa.z) * iL);
      const ff dx = ff_diff(pb.x - L * nx, pa.x), dy = ff_diff(pb.y - L * ny, pa.y), dz = ff_diff(pb.z - L * nz, pa.z);
      const ff r = ff_sqrt(ff_add(ff_add(ff_sqr(dx), ff_sqr(dy)), ff_sqr(dz)));
      const float dr = ff_add_f(ff_add_f(r, -par.x), -par.z).hi;  // r - r0 with r0 in float-float
      const float fs = par.y * dr / r.hi;  // force on a = +k dr (b - a)/r
      const long long fx = fx_from(fs * dx.hi), fy = fx_from(fs * dy.hi), fz = fx_from(fs * dz.hi);
      add3(F, li, fx, fy, fz);
      add3(F, lj, -fx, -fy, -fz);
    } else {
      // angle a-b-c (vertex b), V = k/2 (theta - theta0)^2
      const float4 pc = pick3(p, ll);
      const float3 u = min_disp(pb, pa, L, iL), v = min_disp(pb, pc, L, iL);
      const float uu = u.x * u.x + u.y * u.y + u.z * u.z, vv = v.x * v.x + v.y * v.y + v.z * v.z;
      const float iuv = rsqrtf(uu * vv);
      float cs = (u.x * v.x + u.y * v.y + u.z * v.z) * iuv;
      cs = fminf(1.0f, fmaxf(-1.0f, cs));
      const float dth = acosf(cs) - par.x;
      const float sn = fmaxf(sqrtf(fmaxf(0.0f, 1.0f - cs * cs)), 1e-6f);
      const float g = par.y * dth / sn;
      const float iuu = 1.0f / uu, ivv = 1.0f / vv;
      // forces on the ends: g d cos / d u and g d cos / d v
      const long long ax = fx_from(g * (v.x * iuv - cs * u.x * iuu)), ay = fx_from(g * (v.y * iuv - cs * u.y * iuu)),
                      az = fx_from(g * (v.z * iuv - cs * u.z * iuu));
      const long long cx = fx_from(g * (u.x * iuv - cs * v.x * ivv)), cy = fx_from(g * (u.y * iuv - cs * v.y * ivv)),
                      cz = fx_from(g * (u.z * iuv - cs * v.z * ivv));
      add3(F, li, ax, ay, az);
      add3(F, ll, cx, cy, cz);
      add3(F, lj, -(ax + cx), -(ay + cy), -(az + cz));
    }
  }
#pragma unroll
  for (int m = 0; m < 3; ++m)
    if (sl[m] >= 0) {
      red_add(d.fx + sl[m], F[m][0]);
      red_add(d.fy + sl[m], F[m][1]);
      red_add(d.fz + sl[m], F[m][2]);
    }
}

}  // namespace vp
