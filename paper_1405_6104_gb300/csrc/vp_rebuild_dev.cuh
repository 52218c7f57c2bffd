// vp_rebuild_dev.cuh -- device functions of the list rebuild (binning,
// column scan, bucket fill, column sort, cluster-pair list of one i-cluster),
// shared by the separate kernels and the one-kernel step.  The binning stages
// each live atom (wrapped position, velocity, type, index) in the sort
// buffers; the column sort writes the new layout from there into the arrays.
#pragma once
#include <cooperative_groups.h>

#include "vp_dev.cuh"

namespace vp {

// Slot `slot` of trial t, its atom already loaded (live: the slot holds one):
// wrapped into the box and staged in the sort buffers; returns its grid
// column, or -1 for a slot without an atom.
__device__ __forceinline__ int bin_loaded(const Dev &d, const SimConst &c, const TrialInfo &T, float half_skin2,
                                          int strict, int t, int slot, bool live, int o, float4 p, float4 v,
                                          int ty, unsigned long long n) {
  if (!live) return -1;
  // the slot's atom is staged in the sort buffers (the column sort reads it
  // there and writes the new layout straight into the arrays themselves)
  d.vel_b[slot] = v;
  d.type_b[slot] = ty;
  d.orig_b[slot] = o;
  const float L = T.box, iL = T.inv_box;
  if (c.list_fixed && d.rb[d.n_trials + t] != (uint32_t)n) {
    // fixed-interval lists: an atom farther than skin/2 from where the list
    // was built may have left pairs out (the slot is the one it had then;
    // a forced rebuild follows a new state, not a list interval)
    const float4 r = d.ref_slot[slot];
    const float ddx = p.x - r.x, ddy = p.y - r.y, ddz = p.z - r.z;
    if (ddx * ddx + ddy * ddy + ddz * ddz > half_skin2) {
      atomicAdd(reinterpret_cast<unsigned long long *>(d.diag), 1ull);
      if (strict) atomicOr(d.err, ERR_SKIN);
    }
  }
  float x = p.x - L * floorf(p.x * iL), y = p.y - L * floorf(p.y * iL), z = p.z - L * floorf(p.z * iL);
  x = x >= L ? x - L : (x < 0.0f ? x + L : x);
  y = y >= L ? y - L : (y < 0.0f ? y + L : y);
  z = z >= L ? z - L : (z < 0.0f ? z + L : z);
  z += 0.0f;  // no negative zero in the sort key
  // a coordinate that is not finite, or so large that one wrap cannot bring
  // it into the box (a run that has blown up), is an error; the atom is put
  // at the origin so that every index below stays inside the grid
  if (!(isfinite(x) && isfinite(y) && isfinite(z)) || !(x >= 0.0f && x < L && y >= 0.0f && y < L && z >= 0.0f && z < L)) {
    atomicOr(d.err, ERR_NONFINITE);
    x = y = z = 0.0f;
  }
  d.pos_b[slot] = make_float4(x, y, z, p.w);
  int cx = max(0, min((int)(x * T.inv_col_w), T.ncol - 1));
  int cy = max(0, min((int)(y * T.inv_col_w), T.ncol - 1));
  return cx * T.ncol + cy;
}

// slot `local` of the trial, its column recorded in slot_col and counted (global counters)
__device__ __forceinline__ void bin_slot(const Dev &d, const SimConst &c, float half_skin2, int strict, int t,
                                         int local, unsigned long long n) {
  const TrialInfo T = d.tinfo[t];
  if (local >= T.max_clus * CL) return;
  const int slot = T.slot0 + local;
  const int o = d.orig[slot];
  const bool live = local < d.tstate[t].n_clus * CL && o >= 0;
  const float4 none = make_float4(0.f, 0.f, 0.f, 0.f);
  const int col = bin_loaded(d, c, T, half_skin2, strict, t, slot, live, o, live ? d.pos[slot] : none,
                             live ? d.vel[slot] : none, live ? d.type[slot] : 0, n);
  d.slot_col[slot] = col;
  if (col < 0) return;
  // slots are in column order from the last rebuild, so a warp's atoms fall
  // into one or two columns: one atomic per column and warp
  const unsigned peers = __match_any_sync(__activemask(), col);
  if ((threadIdx.x & 31) == __ffs(peers) - 1) atomicAdd(&d.col_count[T.col0 + col], __popc(peers));
}

template <int NT>
__device__ __forceinline__ void colscan_trial(const Dev &d, int (&s_a)[NT], int (&s_c)[NT], int t) {
  const TrialInfo T = d.tinfo[t];
  int nc = T.ncol * T.ncol;
  int per = (nc + NT - 1) / NT;
  int b = threadIdx.x * per, e = min(b + per, nc);
  int sa = 0, sc = 0, bad = 0;
  for (int c = b; c < e; ++c) {
    int n = d.col_count[T.col0 + c];
    bad |= n > COL_CAP;
    sa += n;
    sc += (n + CL - 1) / CL;
  }
  s_a[threadIdx.x] = sa;
  s_c[threadIdx.x] = sc;
  __syncthreads();
  // Hillis-Steele inclusive scan over the thread sums (fixed order)
  for (int off = 1; off < NT; off <<= 1) {
    int va = threadIdx.x >= off ? s_a[threadIdx.x - off] : 0;
    int vc = threadIdx.x >= off ? s_c[threadIdx.x - off] : 0;
    __syncthreads();
    s_a[threadIdx.x] += va;
    s_c[threadIdx.x] += vc;
    __syncthreads();
  }
  int pa = s_a[threadIdx.x] - sa, pc = s_c[threadIdx.x] - sc;
  for (int c = b; c < e; ++c) {
    int n = d.col_count[T.col0 + c];
    d.col_start[T.col0 + c] = pa;
    d.col_cstart[T.col0 + c] = pc;
    d.col_fill[T.col0 + c] = 0;
    pa += n;
    pc += (n + CL - 1) / CL;
  }
  if (bad) atomicOr(d.err, ERR_COL);
  int total = s_c[NT - 1];
  if (total > T.max_clus) {
    if (threadIdx.x == 0) atomicOr(d.err, ERR_CAPACITY);
    total = T.max_clus;
  }
  if (threadIdx.x == NT - 1) {
    d.tstate[t].n_clus = total;
    const uint32_t n32 = (uint32_t)*d.cur_step;
    d.last_rb[t] = n32;
    atomicAdd(reinterpret_cast<unsigned long long *>(d.diag + 1), 1ull);
    if (d.rb[t] == n32) atomicAdd(reinterpret_cast<unsigned long long *>(d.diag + 2), 1ull);
  }
  // slots past the new clusters become empty (their atoms, if any, are
  // staged in the sort buffers already; the column sort fills the others)
  for (int sl = T.slot0 + total * CL + threadIdx.x; sl < T.slot0 + T.max_clus * CL; sl += NT) {
    const float4 pad = pad_pos(sl);
    d.orig[sl] = -1;
    d.pos[sl] = pad;
    d.ref_slot[sl] = pad;
    d.vel[sl] = make_float4(0.f, 0.f, 0.f, 0.f);
    d.type[sl] = 0;
  }
}

__device__ __forceinline__ void colfill_slot(const Dev &d, int t, int local) {
  const TrialInfo &T = d.tinfo[t];
  if (local >= T.max_clus * CL) return;
  const int slot = T.slot0 + local;
  int c = d.slot_col[slot];
  if (c < 0) return;
  int cg = T.col0 + c;
  // one atomic per column and warp; the lanes of a column take consecutive
  // places (the order inside a bucket is irrelevant: the column sort orders it)
  const unsigned act = __activemask();
  const unsigned peers = __match_any_sync(act, cg);
  const int lane = threadIdx.x & 31, leader = __ffs(peers) - 1;
  int base = 0;
  if (lane == leader) base = atomicAdd(&d.col_fill[cg], __popc(peers));
  base = __shfl_sync(act, base, leader);
  const int p = base + __popc(peers & ((1u << lane) - 1u));
  if (p < COL_CAP && d.col_count[cg] <= COL_CAP) d.bucket[T.atom0 + d.col_start[cg] + p] = slot;
}

// The first part of trial t's rebuild by one thread-block cluster of
// FRONT_CLUSTER blocks of FRONT_THREADS threads, in place of three grid-wide
// kernels: binning, the column scans and the bucket fill.  The column counters
// live in the shared memory of the cluster's first block; the others reach
// them through distributed shared memory.  The order inside a column's bucket
// depends on timing, but the column sort orders every column by (z, atom
// index), so the layout is the same.
// A chain of latencies, so: each thread's loads of FRONT_UNROLL slots go out
// together, the counting atomic returns the atom's place in its bucket (no
// second pass of atomics), column and place stay in registers (slot_col holds
// them only for slots beyond the first FRONT_UNROLL of a thread), the scan
// runs on the shared counters with one barrier, and eight blocks of 512 threads
// spread a trial over eight SMs at 64 registers, two blocks per SM.  14 unequal
// trials 27 -> 17 us per step, 64 trials of 11 040 atoms 20 -> 15, 10 trials of
// 30 000 23 -> 16 (4 blocks of 1024 threads, two atomic passes before; 8 x 512
// with four slots per thread 19 / 17, with two 21 / 18; 8 x 256 25 / 18).
constexpr int FRONT_THREADS = 512;
constexpr int FRONT_CLUSTER = 8;
constexpr int FRONT_UNROLL = 3;
constexpr int MAX_COLS = 64 * 64;  // columns per trial (the host caps the grid at 64 x 64)
constexpr int COL_BITS = 12;
static_assert(MAX_COLS <= 1 << COL_BITS && COL_CAP < 1 << (30 - COL_BITS), "column and place share a word");
struct FrontShared {
  int cnt[MAX_COLS];  // atoms per column, then the column's first place, -1 beyond its capacity (the first block's)
  int wa[32], wc[32];
  int n_clus;         // clusters of the new layout (the first block's)
};

__device__ __forceinline__ void front_scan(const Dev &d, FrontShared &sh, const TrialInfo &T, int t) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nc = T.ncol * T.ncol;
  const int per = (nc + FRONT_THREADS - 1) / FRONT_THREADS;
  const int b = min((int)threadIdx.x * per, nc), e = min(b + per, nc);
  int sa = 0, sc = 0;
  for (int k = b; k < e; ++k) {
    const int n = sh.cnt[k];
    sa += n;
    sc += (n + CL - 1) / CL;
  }
  int ia = sa, ic = sc;  // inclusive sums
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const int va = __shfl_up_sync(0xffffffffu, ia, off), vc = __shfl_up_sync(0xffffffffu, ic, off);
    if (lane >= off) { ia += va; ic += vc; }
  }
  if (lane == 31) { sh.wa[warp] = ia; sh.wc[warp] = ic; }
  __syncthreads();
  int wa = 0, wc = 0, total = 0;
  {
    const int xa = lane < FRONT_THREADS / 32 ? sh.wa[lane] : 0, xc = lane < FRONT_THREADS / 32 ? sh.wc[lane] : 0;
    wa = (int)__reduce_add_sync(0xffffffffu, (unsigned)(lane < warp ? xa : 0));
    wc = (int)__reduce_add_sync(0xffffffffu, (unsigned)(lane < warp ? xc : 0));
    total = (int)__reduce_add_sync(0xffffffffu, (unsigned)xc);
  }
  int pa = wa + ia - sa, pc = wc + ic - sc;
  for (int k = b; k < e; ++k) {
    const int n = sh.cnt[k];
    d.col_count[T.col0 + k] = n;
    d.col_start[T.col0 + k] = pa;
    d.col_cstart[T.col0 + k] = pc;
    if (n > COL_CAP) atomicOr(d.err, ERR_COL);
    sh.cnt[k] = n > COL_CAP ? -1 : pa;
    pa += n;
    pc += (n + CL - 1) / CL;
  }
  if (threadIdx.x == 0) {
    if (total > T.max_clus) {
      atomicOr(d.err, ERR_CAPACITY);
      total = T.max_clus;
    }
    sh.n_clus = total;
    d.tstate[t].n_clus = total;
    atomicAdd(reinterpret_cast<unsigned long long *>(d.diag + 1), 1ull);
    if (d.rb[t] == (uint32_t)*d.cur_step) atomicAdd(reinterpret_cast<unsigned long long *>(d.diag + 2), 1ull);
  }
}

__device__ __forceinline__ void front_trial(const Dev &d, const SimConst &c, float half_skin2, int strict,
                                            FrontShared &sh, int t, unsigned long long n) {
  namespace cgr = cooperative_groups;
  cgr::cluster_group cl = cgr::this_cluster();
  const int rank = (int)cl.block_rank(), lane = threadIdx.x & 31;
  int *cnt0 = cl.map_shared_rank(sh.cnt, 0);
  const TrialInfo T = d.tinfo[t];
  const int n_slots = T.max_clus * CL, n_used = d.tstate[t].n_clus * CL;
  constexpr int STRIDE = FRONT_CLUSTER * FRONT_THREADS;
  const int first = rank * FRONT_THREADS + threadIdx.x;
  if (rank == 0)
    for (int k = threadIdx.x; k < T.ncol * T.ncol; k += FRONT_THREADS) sh.cnt[k] = 0;
  cl.sync();
  int word[FRONT_UNROLL];  // column | place in its bucket << COL_BITS, or -1, of the thread's first slots
  for (int base = first; base - lane < n_slots; base += STRIDE * FRONT_UNROLL) {
    int o[FRONT_UNROLL], at[FRONT_UNROLL];
    float4 p[FRONT_UNROLL], v[FRONT_UNROLL];
    int ty[FRONT_UNROLL];
    unsigned peers[FRONT_UNROLL];
#pragma unroll
    for (int u = 0; u < FRONT_UNROLL; ++u) {
      const int local = base + u * STRIDE, slot = T.slot0 + local;
      const bool in = local < n_used;
      o[u] = in ? d.orig[slot] : -1;
      p[u] = in ? d.pos[slot] : make_float4(0.f, 0.f, 0.f, 0.f);
      v[u] = in ? d.vel[slot] : make_float4(0.f, 0.f, 0.f, 0.f);
      ty[u] = in ? d.type[slot] : 0;
    }
    // slots are in column order from the last rebuild, so a warp's atoms fall
    // into one or two columns: one atomic per column and warp, the lanes of a
    // column take consecutive places
    int w[FRONT_UNROLL];
#pragma unroll
    for (int u = 0; u < FRONT_UNROLL; ++u) {
      w[u] = bin_loaded(d, c, T, half_skin2, strict, t, T.slot0 + base + u * STRIDE, o[u] >= 0, o[u], p[u], v[u], ty[u], n);
      peers[u] = __match_any_sync(0xffffffffu, w[u]);
      at[u] = 0;
      if (w[u] >= 0 && lane == __ffs(peers[u]) - 1) at[u] = atomicAdd(cnt0 + w[u], __popc(peers[u]));
    }
#pragma unroll
    for (int u = 0; u < FRONT_UNROLL; ++u) {
      const int place = __shfl_sync(0xffffffffu, at[u], __ffs(peers[u]) - 1) + __popc(peers[u] & ((1u << lane) - 1u));
      if (w[u] >= 0) w[u] |= min(place, COL_CAP) << COL_BITS;
      const int local = base + u * STRIDE;
      if (base == first) word[u] = w[u];
      else if (local < n_slots) d.slot_col[T.slot0 + local] = w[u];
    }
  }
  cl.sync();
  if (rank == 0) front_scan(d, sh, T, t);
  cl.sync();
  const int n_new = *cl.map_shared_rank(&sh.n_clus, 0) * CL;
  for (int base = first; base < n_slots; base += STRIDE * FRONT_UNROLL) {
    if (base != first) {
#pragma unroll
      for (int u = 0; u < FRONT_UNROLL; ++u)
        word[u] = base + u * STRIDE < n_slots ? d.slot_col[T.slot0 + base + u * STRIDE] : -1;
    }
    int start[FRONT_UNROLL];
#pragma unroll
    for (int u = 0; u < FRONT_UNROLL; ++u) start[u] = word[u] >= 0 ? cnt0[word[u] & ((1 << COL_BITS) - 1)] : -1;
#pragma unroll
    for (int u = 0; u < FRONT_UNROLL; ++u) {
      const int place = word[u] >> COL_BITS, local = base + u * STRIDE, sl = T.slot0 + local;
      if (start[u] >= 0 && place < COL_CAP) d.bucket[T.atom0 + start[u] + place] = sl;
      // slots past the new clusters become empty (their atoms, if any, are
      // staged in the sort buffers already; the column sort fills the others)
      if (local >= n_new && local < n_slots) {
        const float4 pad = pad_pos(sl);
        d.orig[sl] = -1;
        d.pos[sl] = pad;
        d.ref_slot[sl] = pad;
        d.vel[sl] = make_float4(0.f, 0.f, 0.f, 0.f);
        d.type[sl] = 0;
      }
    }
  }
  cl.sync();  // the first block's counters stay alive until every block is done with them
}

struct ColsortShared {
  alignas(16) unsigned long long key[COL_CAP + 1];  // (z, atom index) in bucket order
  int s_old[COL_CAP];                               // slots before this rebuild, idem
  float3 s_pos[COL_CAP];                            // positions in the new order
};

// One column: its atoms in the order of (z, atom index), the new layout.  The
// atoms are read from the sort buffers (staged by the binning: the layout
// before this rebuild) and written in the new order into the arrays
// themselves.  STAMP: the block of column 0 records this step as the trial's
// last rebuild.
// Bound by latency (some twelve columns per SM even when all of 16 trials
// rebuild): so an atom's place is its rank, counted over the column's keys
// without a barrier while its position and velocity load (a bitonic sort of
// 100 keys takes 28 barriers), and the boxes are formed from shared memory.
// 64 trials of 11 040 atoms: 37 -> 22 us per step.
template <bool STAMP>
__device__ __forceinline__ void colsort_column(const Dev &d, ColsortShared &sh, int t, int c) {
  const TrialInfo T = d.tinfo[t];
  if (c >= T.ncol * T.ncol) return;
  if (STAMP && c == 0 && threadIdx.x == 0) d.last_rb[t] = (uint32_t)*d.cur_step;
  const int cg = T.col0 + c;
  const int n = d.col_count[cg];
  const int start = d.col_start[cg], cstart = d.col_cstart[cg];
  __syncthreads();
  // the count is consumed: the column starts from zero at the trial's next rebuild
  if (threadIdx.x == 0) d.col_count[cg] = 0;
  if (n > COL_CAP) return;  // flagged by the column scan
  if (cstart + (n + CL - 1) / CL > T.max_clus) return;  // flagged by the column scan
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    const int s = d.bucket[T.atom0 + start + i];
    sh.s_old[i] = s;
    sh.key[i] = ((unsigned long long)__float_as_uint(d.pos_b[s].z) << 32) | (unsigned)d.orig_b[s];
  }
  if (threadIdx.x == 0) sh.key[n] = ~0ull;  // the keys are read two at a time
  __syncthreads();
  const int ncl = (n + CL - 1) / CL;
  const int base = T.slot0 + cstart * CL;
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    const int old = sh.s_old[i];
    const unsigned long long key = sh.key[i];
    const float4 p = d.pos_b[old], v = d.vel_b[old];
    const auto ty = d.type_b[old];
    int r = 0;
#pragma unroll 4
    for (int m = 0; m < n; m += 2) {
      const ulonglong2 k2 = *reinterpret_cast<const ulonglong2 *>(sh.key + m);
      r += (k2.x < key) + (k2.y < key);
    }
    const int o = (int)(key & 0xffffffffu), ns = base + r;
    sh.s_pos[r] = make_float3(p.x, p.y, p.z);
    d.pos[ns] = p;
    d.ref_slot[ns] = p;  // the position the new list is built from
    d.vel[ns] = v;
    d.orig[ns] = o;
    d.type[ns] = ty;
    d.slot_of[T.atom0 + o] = ns;
  }
  for (int r = n + threadIdx.x; r < ncl * CL; r += blockDim.x) {
    const int ns = base + r;
    const float4 pad = pad_pos(ns);
    d.pos[ns] = pad;
    d.ref_slot[ns] = pad;
    d.vel[ns] = make_float4(0.f, 0.f, 0.f, 0.f);
    d.orig[ns] = -1;
    d.type[ns] = 0;
  }
  __syncthreads();
  // bounding boxes of the 4-atom halves of each cluster, as centre and half
  // extent (real atoms only; an all-padding half gets an empty box, half
  // extents -3e38: farther than any cut-off from everything)
  for (int k = threadIdx.x; k < 2 * ncl; k += blockDim.x) {
    float3 lo = make_float3(3e38f, 3e38f, 3e38f), hi = make_float3(-3e38f, -3e38f, -3e38f);
#pragma unroll
    for (int a = 0; a < CJ; ++a) {
      const int r = k * CJ + a;
      if (r < n) {
        const float3 p = sh.s_pos[r];
        lo.x = fminf(lo.x, p.x); lo.y = fminf(lo.y, p.y); lo.z = fminf(lo.z, p.z);
        hi.x = fmaxf(hi.x, p.x); hi.y = fmaxf(hi.y, p.y); hi.z = fmaxf(hi.z, p.z);
      }
    }
    const int hj = 2 * (T.clus0 + cstart) + k;
    d.bb_c[hj] = make_float4(0.5f * lo.x + 0.5f * hi.x, 0.5f * lo.y + 0.5f * hi.y, 0.5f * lo.z + 0.5f * hi.z, 0.f);
    d.bb_h[hj] = make_float4(0.5f * hi.x - 0.5f * lo.x, 0.5f * hi.y - 0.5f * lo.y, 0.5f * hi.z - 0.5f * lo.z, 0.f);
  }
  // z-bin table: the halves are in ascending z (an all-padding half counts as
  // above everything), so the number of halves whose lower z-bound lies below
  // b L / ZBINS is the first half at or above it
  const int nh = (n + CJ - 1) / CJ;
  for (int b = threadIdx.x; b <= ZBINS; b += blockDim.x) {
    const float zt = (float)b * (T.box / ZBINS);
    int lo = 0, hi = nh;
    while (lo < hi) {
      const int mid = (lo + hi) >> 1;
      if (sh.s_pos[mid * CJ].z < zt) lo = mid + 1; else hi = mid;
    }
    d.col_ztab[(size_t)cg * (ZBINS + 1) + b] = lo;
  }
}

// ---------------------------------------------------------------------------
// cluster-pair list
// ---------------------------------------------------------------------------
// the FP32 list rule: n = rint((xj - xi) * invL); d = (xj - L n) - xi (the
// image of x_j first, as the force kernel forms it); r2 = fma(dz, dz,
// fma(dy, dy, dx*dx)); member iff r2 < rl2.  Also returns the image key
// 9 nx + 3 ny + nz of the counts n (x_j image = x_j - L n).
__device__ __forceinline__ bool list_rule(float4 pi, float4 pj, float L, float iL, float rl2, float &key) {
  const float tx = __fsub_rn(pj.x, pi.x), ty = __fsub_rn(pj.y, pi.y), tz = __fsub_rn(pj.z, pi.z);
  const float qx = rintf(__fmul_rn(tx, iL)), qy = rintf(__fmul_rn(ty, iL)), qz = rintf(__fmul_rn(tz, iL));
  const float dx = __fsub_rn(__fsub_rn(pj.x, __fmul_rn(L, qx)), pi.x);
  const float dy = __fsub_rn(__fsub_rn(pj.y, __fmul_rn(L, qy)), pi.y);
  const float dz = __fsub_rn(__fsub_rn(pj.z, __fmul_rn(L, qz)), pi.z);
  const float r2 = __fmaf_rn(dz, dz, __fmaf_rn(dy, dy, __fmul_rn(dx, dx)));
  key = __fmaf_rn(9.0f, qx, __fmaf_rn(3.0f, qy, qz));
  return r2 < rl2;
}

// A candidate whose atom pairs do not all share the image counts (it spans
// half a box length in some dimension): the per-pair rule for all 8 x 4
// pairs, with validity and self-pair tests; kmin/kmax collect the image keys
// of the passing pairs (exclusions are cleared afterwards).
static __device__ __noinline__ unsigned list_mixed_images(const Dev &d, int I, int Il, int J8, int sj0, float L, float iL,
                                                   float rl2, float &kmin, float &kmax) {
  unsigned mask = 0u;
  for (int b = 0; b < CJ; ++b) {
    const float4 pj = d.pos[sj0 + b];
    const int oj = d.orig[sj0 + b];
    for (int a = 0; a < CL; ++a) {
      const float4 pi = d.pos[I * CL + a];
      const int oi = d.orig[I * CL + a];
      float key;
      const bool v = list_rule(pi, pj, L, iL, rl2, key) && oi >= 0 && oj >= 0 && (J8 != Il || sj0 + b > I * CL + a);
      if (v) {
        kmin = fminf(kmin, key);
        kmax = fmaxf(kmax, key);
        mask |= 1u << (b * CL + a);
      }
    }
  }
  return mask;
}

constexpr int LIST_WARPS = 4;
constexpr int CAND_MAX = 1024;  // candidate 4-atom j-clusters per i-cluster (bounding-box pass)
constexpr int ENT_MAX = 512;    // 4-atom j-clusters with a listed pair per i-cluster
// a candidate word: the half index (J_BITS bits, from the trial's first
// half), the six bits of the image code, the shared-image flag
constexpr unsigned CAND_SAME = 1u << 31;
static_assert(J_BITS + 6 == 31, "candidate word: half index, image code and flag in 32 bits");

// j-atoms of an entry with at least one listed pair: the bytes of the mask
// that are not zero
__device__ __forceinline__ int j_columns(unsigned m) {
  return __popc((((m & 0x7f7f7f7fu) + 0x7f7f7f7fu) | m) & 0x80808080u);
}

// One warp per i-cluster.  Phase 1: lanes test columns, then the 4-atom
// halves of the clusters of each passing column, against the i-cluster's
// bounding box and collect the candidates in order (column-major, then z,
// i.e. ascending j-cluster index).  Phase 2: each lane takes one candidate
// and evaluates the FP32 list rule for all 8 x 4 atom pairs itself, giving
// the entry's mask (bit b * 8 + a for j-atom b and i-atom a: a byte per
// j-atom), image code and exact flag; entries are written in candidate order
// (deterministic).  Phase 3: the i-atoms' exclusions clear their bits in the
// entries (found by binary search).  Phase 4: one list entry per j-atom with
// a listed pair is written out.
//
// Bound by issue slots (a GPU full of rebuilding trials) or by the chain of
// loads (one trial).  Hence: boxes as centre and half extent (the periodic gap
// and the image counts of a box pair come from one rounding per dimension),
// columns before the i-cluster's own left out (their clusters have lower
// indices), z-windows in 64 bins, the halves to test written out once per 32
// columns instead of searched per test, the next step's boxes loaded while the
// current ones are tested, the chain of loads that leads to the excluded
// partners' slots begun before the search, byte masks that phase 4 reads off
// directly.  Of 64 trials of 11 040 atoms, 16 rebuilding in the step: 222 us
// before these, 138 with them; a step of one trial, every fourth with a
// rebuild, 12 -> 6 us on average.  Testing every half of the z-windows pair by
// pair without the box test (215 instead of 179 of them) took 168 us.
struct ListShared {
  unsigned s_cand[LIST_WARPS][CAND_MAX];
  float4 s_xp[LIST_WARPS][CL / 2][2];  // i-atom pairs (2p, 2p+1): {-x, -x', -y, -y'} {-z, -z', 0, 0}
  unsigned s_dirty[LIST_WARPS][ENT_MAX / 32];  // entries whose j-atoms need the pair masks
  unsigned s_mask[LIST_WARPS][ENT_MAX];        // halves to test (phase 1), then the entries' masks (their
                                               // first words overwrite s_cand)
  int4 s_part[LIST_WARPS];  // of the parts of a list: halves found, entries, masked and clean j-atoms
};

// PARTS > 1: that many consecutive warps of the block share the list, each
// doing an equal share of the window's columns.  The shares are consecutive in the
// list's order, so a warp only needs to know how many j-atoms the shares before
// its own hold.  Once per block: s_part holds one list's numbers.
template <int PARTS = 1>
__device__ __forceinline__ void list_cluster(const Dev &d, const SimConst &c, float rl2_bbox, ListShared &sh, int t,
                                             int Il) {
  const int wib = threadIdx.x >> 5, part = wib % PARTS;
  const int lane = threadIdx.x & 31;
  auto &s_xp = sh.s_xp[wib];
  auto &s_dirty = sh.s_dirty[wib];
  unsigned *cand = sh.s_cand[wib], *s_mask = sh.s_mask[wib];
  const TrialInfo T = d.tinfo[t];
  if (Il >= T.max_clus) return;
  const int I = T.clus0 + Il;
  const int n_clus_t = d.tstate[t].n_clus;
  if (Il >= n_clus_t) {
    if (lane == 0) d.list_n[I] = 0;
    return;
  }
  // lane = (i-atom lane & 7, four of its excluded partners at a time from lane >> 3)
  const int xo = d.orig[I * CL + (lane & 7)];
  const float4 xi = d.pos[I * CL + (lane & 7)];
  if (lane < CL) {
    float *x = &s_xp[lane >> 1][0].x + (lane & 1);
    x[0] = -xi.x; x[2] = -xi.y; x[4] = -xi.z;
  }
  if (lane < ENT_MAX / 32) s_dirty[lane] = c.list_fixed ? ~0u : 0u;  // fixed-interval lists: masks everywhere
  // the partners themselves (unused places hold -1) and their number
  const int32_t *xrow = d.excl + (size_t)(T.sysatom0 + max(xo, 0)) * MAX_EXCL;
  const int xn = xo >= 0 ? d.excl_n[T.sysatom0 + xo] : 0;
  const int xa = xo >= 0 ? xrow[lane >> 3] : -1;
  const float3 lo = make_float3(warp_min(xo >= 0 ? xi.x : 3e38f), warp_min(xo >= 0 ? xi.y : 3e38f),
                                warp_min(xo >= 0 ? xi.z : 3e38f));
  const float3 hi = make_float3(warp_max(xo >= 0 ? xi.x : -3e38f), warp_max(xo >= 0 ? xi.y : -3e38f),
                                warp_max(xo >= 0 ? xi.z : -3e38f));
  const float L = T.box, iL = T.inv_box, w = T.col_w;
  const int nc2 = T.ncol * T.ncol;
  const float3 ci = make_float3(0.5f * (lo.x + hi.x), 0.5f * (lo.y + hi.y), 0.5f * (lo.z + hi.z));
  const float3 hw = make_float3(0.5f * (hi.x - lo.x), 0.5f * (hi.y - lo.y), 0.5f * (hi.z - lo.z));
  int n_cand = 0;
  // ---- phase 1: candidate 4-atom j-clusters ----
  // Only the grid columns within reach of the i-cluster's bounding box (one
  // column more on each side for the rounding of the binning) are visited,
  // in ascending column index: the window's x and y column indices, wrapped
  // periodically, are enumerated in sorted order (so the candidates, and the
  // entries, ascend in j-cluster index), from the i-cluster's own x index on
  // (the half list keeps clusters of index >= Il).  Lanes take 32 columns; the
  // halves of the passing columns are then tested as one flat range, 32 per
  // step.
  const float reach = sqrtf(rl2_bbox);
  int wx0, wnx, wy0, wny;  // first column (mod ncol) and count of the window in x and in y
  {
    const int ax = (int)floorf((lo.x - reach) * T.inv_col_w) - 1, bx = (int)floorf((hi.x + reach) * T.inv_col_w) + 1;
    const int ay = (int)floorf((lo.y - reach) * T.inv_col_w) - 1, by = (int)floorf((hi.y + reach) * T.inv_col_w) + 1;
    wnx = min(T.ncol, bx - ax + 1);
    wny = min(T.ncol, by - ay + 1);
    wx0 = wnx == T.ncol ? 0 : ((ax % T.ncol) + T.ncol) % T.ncol;
    wy0 = wny == T.ncol ? 0 : ((ay % T.ncol) + T.ncol) % T.ncol;
  }
  // k-th smallest of {a, a + 1, ..., a + m - 1} mod ncol
  auto kth = [&](int a, int m, int k) {
    const int e = a + m - T.ncol;  // the part that wraps to [0, e)
    return e <= 0 ? a + k : (k < e ? k : a + (k - e));
  };
  // rows of the window below the i-cluster's own x index (a rounding below it is only one row more)
  int row0;
  {
    const int own = max(0, (int)floorf((lo.x - 1e-5f) * T.inv_col_w));
    const int e = max(0, wx0 + wnx - T.ncol);
    row0 = min(own, e) + max(0, min(own - wx0, wnx - e));
  }
  const int nwin = (wnx - row0) * wny;
  const float inv_wny = 1.0f / (float)wny;
  const float half_w = 0.5f * w, img_lim = 0.49999f * L;
  int xs = -1;  // slot of this lane's excluded partner
  const int col_lo = nwin * part / PARTS, col_hi = nwin * (part + 1) / PARTS;
  for (int cb = col_lo; cb < col_hi; cb += 32) {
    const int wi = cb + lane;
    // this lane's column: up to two ranges [a1, a1 + n1), [a2, a2 + n2) of
    // half indices (relative to the trial's first half) whose z-extent can
    // reach the i-cluster: the z-window (and its periodic image) comes from
    // the column's xy gap, the ranges from the column's z-bin table, one bin
    // wider on each side than needed (every half in them is still tested)
    int a1 = 0, n1 = 0, a2 = 0, n2 = 0;
    if (wi < col_hi) {
      const int wr = (int)(((float)wi + 0.5f) * inv_wny);  // wi / wny (exact: wi < 2^12)
      const int cx = kth(wx0, wnx, row0 + wr), cy = kth(wy0, wny, wi - wr * wny);
      const int cc = cx * T.ncol + cy;
      // the geometry first, then every load of the column at once (one
      // memory round trip instead of two)
      float gx = ((float)cx * w + half_w) - ci.x, gy = ((float)cy * w + half_w) - ci.y;
      gx = fmaxf(fabsf(gx - L * rintf(gx * iL)) - (half_w + hw.x), 0.0f);
      gy = fmaxf(fabsf(gy - L * rintf(gy * iL)) - (half_w + hw.y), 0.0f);
      const float g2 = gx * gx + gy * gy;
      if (g2 < rl2_bbox) {
        const float rz = sqrtf(rl2_bbox - g2) * 1.001f + 1e-3f;
        const float za = lo.z - rz, zb = hi.z + rz;
        const bool whole = zb - za >= L;
        // z-bins of the halves that may meet [u, v] (0 <= u <= v <= L): one
        // or two intervals (the periodic image)
        const float zs = ZBINS * iL;
        const bool two = za < 0.f || zb > L;
        const float v1 = za < 0.f ? zb : (zb > L ? zb - L : zb);
        const float u1 = two ? 0.f : za;
        const float u2 = za < 0.f ? za + L : za;
        auto bin_lo = [&](float u) { return max(0, min(ZBINS, (int)floorf(u * zs) - 1)); };
        const int bu1 = bin_lo(u1), bv1 = max(0, min(ZBINS, (int)floorf(v1 * zs) + 2)), bu2 = bin_lo(u2);
        const int *tab = d.col_ztab + (size_t)(T.col0 + cc) * (ZBINS + 1);
        const int ccs = d.col_cstart[T.col0 + cc];
        const int cnext = cc + 1 < nc2 ? d.col_cstart[T.col0 + cc + 1] : n_clus_t;
        const int t1a = tab[bu1], t1b = tab[bv1];
        const int t2a = two ? tab[bu2] : 0;
        const int ncl = max(0, cnext - ccs);
        const int jlo = max(ccs, Il);
        if (ccs + ncl > jlo) {
          const int hs = 2 * (jlo - ccs), he = 2 * ncl;  // local half range of the half list
          int r1a = hs, r1b = he, r2a = 0, r2b = 0;
          if (!whole) {
            r1a = max(max(t1a - 1, 0), hs);
            r1b = min(bv1 >= ZBINS ? he : t1b, he);
            // the second interval reaches up to L, the column's end
            r2a = two ? max(max(t2a - 1, hs), r1b) : 0;  // ascending, no half twice
            r2b = two ? he : 0;
          }
          n1 = max(r1b - r1a, 0);
          n2 = max(r2b - r2a, 0);
          a1 = r1a + 2 * ccs;
          a2 = r2a + 2 * ccs;
        }
      }
    }
    if (cb == col_lo && xa >= 0) xs = d.slot_of[T.atom0 + xa];
    const int cntc = n1 + n2;
    // inclusive scan of the per-column counts
    int incl = cntc;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, incl, off);
      if (lane >= off) incl += v;
    }
    const int total = __shfl_sync(0xffffffffu, incl, 31), first = incl - cntc;
    // the halves of these columns, ENT_MAX at a time
    for (int t0 = 0; t0 < total; t0 += ENT_MAX) {
      const int m = min(ENT_MAX, total - t0);
      __syncwarp();
      for (int u = max(0, t0 - first); u < cntc && first + u < t0 + m; ++u)
        s_mask[first + u - t0] = (unsigned)(u < n1 ? a1 + u : a2 + (u - n1));
      __syncwarp();
      // idle lanes of the last step repeat its last half (and are not counted)
      unsigned Jn = s_mask[min(lane, m - 1)];
      float4 cn = d.bb_c[2 * T.clus0 + Jn], hn = d.bb_h[2 * T.clus0 + Jn];
      for (int q = 0; q < m; q += 32) {
        const unsigned J4 = Jn;
        const float4 cj = cn, hj = hn;
        if (q + 32 < m) {  // the next step's boxes
          Jn = s_mask[min(q + 32 + lane, m - 1)];
          cn = d.bb_c[2 * T.clus0 + Jn];
          hn = d.bb_h[2 * T.clus0 + Jn];
        }
        // periodic gap of the boxes, and the image counts of their centres:
        // all atom pairs share them when no pair can come near half a box
        // length (the 1e-5 L margin covers every rounding here and in the rule)
        float dx = cj.x - ci.x, dy = cj.y - ci.y, dz = cj.z - ci.z;
        const float nx = rintf(dx * iL), ny = rintf(dy * iL), nz = rintf(dz * iL);
        dx = fabsf(dx - L * nx); dy = fabsf(dy - L * ny); dz = fabsf(dz - L * nz);
        const float sx = hj.x + hw.x, sy = hj.y + hw.y, sz = hj.z + hw.z;
        const float gx = fmaxf(dx - sx, 0.f), gy = fmaxf(dy - sy, 0.f), gz = fmaxf(dz - sz, 0.f);
        const bool ok = q + lane < m && gx * gx + gy * gy + gz * gz < rl2_bbox;
        const bool same = fmaxf(fmaxf(dx + sx, dy + sy), dz + sz) < img_lim;
        const unsigned code = (unsigned)(int)(nx + 4.0f * ny + 16.0f * nz + (float)NO_SHIFT);
        const unsigned bal = __ballot_sync(0xffffffffu, ok);
        const int pos = n_cand + __popc(bal & ((1u << lane) - 1u));
        if (ok && pos < CAND_MAX) cand[pos] = J4 | (code << J_BITS) | (same ? CAND_SAME : 0u);
        n_cand += __popc(bal);
      }
    }
  }
  int n_found = n_cand;
  n_cand = min(n_cand, CAND_MAX);
  __syncwarp();
  // ---- phase 2: one candidate 4-atom j-cluster per lane ----
  // Image counts: q = rint(fl(d * invL)) for every atom pair of a candidate
  // with shared images is that of the box centres, so the rule reduces to
  // d - fl(L q) with the same rounding as the per-pair form.  Padding atoms
  // sit far outside every box and fail the distance test on that path.
  const float rl2 = c.rl2;
  int cnt = 0;
  for (int k0 = 0; k0 < n_cand; k0 += 32) {
    const int k = k0 + lane;
    unsigned mask = 0u, w0 = 0u;
    bool dirty = false;
    if (k < n_cand) {
      const unsigned cw = cand[k];
      const unsigned J4 = cw & J_MASK, code = (cw >> J_BITS) & 63u;
      const int J8 = (int)(J4 >> 1);
      const int sj0 = T.slot0 + (int)J4 * CJ;
      const unsigned jw = (unsigned)(2 * T.clus0) + J4;
      w0 = jw | (code << J_BITS);
      dirty = J8 == Il;  // the cluster with itself: pairs below the diagonal masked
      if (cw & CAND_SAME) {
        // the j-atoms' images once, then two i-atoms per packed FP32x2
        // operation; every operation rounds on its own exactly as the
        // per-pair rule does (d = (xj - L n) + (-xi) is (xj - L n) - xi)
        const float sx = __fmul_rn(L, (float)((int)(code & 3u) - 1)), sy = __fmul_rn(L, (float)((int)((code >> 2) & 3u) - 1)),
                    sz = __fmul_rn(L, (float)((int)(code >> 4) - 1));
        float ux[CJ], uy[CJ], uz[CJ];
#pragma unroll
        for (int b = 0; b < CJ; ++b) {
          const float4 pj = d.pos[sj0 + b];
          ux[b] = __fsub_rn(pj.x, sx); uy[b] = __fsub_rn(pj.y, sy); uz[b] = __fsub_rn(pj.z, sz);
        }
#pragma unroll
        for (int p = 0; p < CL / 2; ++p) {
          const float4 i0 = s_xp[p][0], i1 = s_xp[p][1];
#pragma unroll
          for (int b = 0; b < CJ; ++b) {
            const float2 dx = __fadd2_rn(make_float2(ux[b], ux[b]), make_float2(i0.x, i0.y));
            const float2 dy = __fadd2_rn(make_float2(uy[b], uy[b]), make_float2(i0.z, i0.w));
            const float2 dz = __fadd2_rn(make_float2(uz[b], uz[b]), make_float2(i1.x, i1.y));
            const float2 r2 = __ffma2_rn(dz, dz, __ffma2_rn(dy, dy, __fmul2_rn(dx, dx)));
            if (r2.x < rl2) mask |= 1u << (b * CL + 2 * p);
            if (r2.y < rl2) mask |= 1u << (b * CL + 2 * p + 1);
          }
        }
        // inside the i-cluster itself: pairs with the j slot above the i slot
        if (J8 == Il) mask &= (J4 & 1u) ? 0x7f3f1f0fu : 0x07030100u;
      } else {
        float kmin = 3e38f, kmax = -3e38f;
        mask = list_mixed_images(d, I, Il, J8, sj0, L, iL, rl2, kmin, kmax);
        // image counts of the entry from the key 9 nx + 3 ny + nz (each in -1..1)
        const int key = mask ? (int)kmin : 0;
        const int kz = ((key % 3) + 4) % 3 - 1;
        const int ky = (((key - kz) / 3) % 3 + 4) % 3 - 1;
        const int kx = (key - kz - 3 * ky) / 9;
        const bool exact = mask && kmin != kmax;  // pairs that take images one by one need the masks
        w0 = jw | ((unsigned)((kx + 1) | ((ky + 1) << 2) | ((kz + 1) << 4)) << J_BITS) | (exact ? E_EXACT : 0u);
        dirty |= exact;
      }
    }
    const unsigned bal = __ballot_sync(0xffffffffu, mask != 0u);
    const int pos = cnt + __popc(bal & ((1u << lane) - 1u));
    __syncwarp();  // every lane has read its candidate before entries overwrite them
    if (mask != 0u && pos < ENT_MAX) {
      // entries are kept in shared memory until the exclusions are cleared:
      // the first word over the consumed candidates, the mask beside
      cand[pos] = w0;
      s_mask[pos] = mask;
      if (dirty) atomicOr(&s_dirty[pos >> 5], 1u << (pos & 31));
    }
    cnt += __popc(bal);
  }
  const int n_ent = min(cnt, ENT_MAX);
  // ---- phase 3: exclusions ----
  // for each atom excluded from i-atom a, the bit of that pair is cleared in
  // the entry of its 4-atom j-cluster, if this list holds the pair (entries
  // ascend in j-cluster index; a pair inside the i-cluster belongs to the
  // entry with the higher slot as j)
  __syncwarp();
  for (int q = 0; q == 0 || __any_sync(0xffffffffu, xn > q); q += 4) {
    if (q > 0) {  // atoms with more than four excluded partners
      const int x = q + (lane >> 3) < xn ? xrow[q + (lane >> 3)] : -1;
      xs = x >= 0 ? d.slot_of[T.atom0 + x] : -1;
    }
    const int a = lane & 7, si = I * CL + a;
    if (xs > si && (xs >> 3) >= I) {  // else listed from the other side, or not at all
      const unsigned j4 = (unsigned)(xs >> 2);
      int lo_e = 0, hi_e = n_ent;  // first entry with j-cluster >= j4
      while (lo_e < hi_e) {
        const int mid = (lo_e + hi_e) >> 1;
        if ((cand[mid] & J_MASK) < j4) lo_e = mid + 1; else hi_e = mid;
      }
      if (lo_e < n_ent && (cand[lo_e] & J_MASK) == j4) {
        atomicAnd(&s_mask[lo_e], ~(1u << ((xs & 3) * CL + a)));
        atomicOr(&s_dirty[lo_e >> 5], 1u << (lo_e & 31));
      }
    }
  }
  __syncwarp();
  // ---- phase 4: one entry per j-atom with a listed pair ----
  // In entry order, j-atoms ascending; the j-atoms of entries that need the
  // masks first, so that they fill as few groups of 32 entries as possible.
  int n_dirty = 0;
  for (int e0 = 0; e0 < n_ent; e0 += 32) {
    const unsigned dw = s_dirty[e0 >> 5];
    const int e = e0 + lane;
    n_dirty += __reduce_add_sync(0xffffffffu, e < n_ent && ((dw >> lane) & 1u) ? j_columns(s_mask[e]) : 0);
  }
  int pd = 0, pc = n_dirty;  // where the next j-atoms of either kind go
  if constexpr (PARTS > 1) {
    int n_clean = 0;
    for (int e = lane; e < n_ent; e += 32) n_clean += j_columns(s_mask[e]);
    n_clean = (int)__reduce_add_sync(0xffffffffu, (unsigned)n_clean) - n_dirty;
    const int w0 = wib - part;
    if (lane == 0) sh.s_part[wib] = make_int4(n_found, cnt, n_dirty, n_clean);
    // (constant barrier numbers: a block that may use all 16 leaves room for two on an SM)
    if (PARTS == LIST_WARPS) __syncthreads();
    else if (w0 == 0) asm volatile("bar.sync 1, %0;" ::"n"(32 * PARTS) : "memory");
    else asm volatile("bar.sync 2, %0;" ::"n"(32 * PARTS) : "memory");
    int before = 0;
    n_found = cnt = n_dirty = 0;
    for (int q = 0; q < PARTS; ++q) {
      const int4 v = sh.s_part[w0 + q];
      n_found += v.x;
      cnt += v.y;
      n_dirty += v.z;
      if (q < part) { pd += v.z; before += v.w; }
    }
    pc = n_dirty + before;
  }
  uint32_t *segw = d.list + (size_t)I * c.list_cap;
  uint8_t *segm = d.list_m + (size_t)I * c.list_cap;
  for (int e0 = 0; e0 < n_ent; e0 += 32) {
    const int e = e0 + lane;
    const unsigned m = e < n_ent ? s_mask[e] : 0u;
    const bool dirty = (s_dirty[e0 >> 5] >> lane) & 1u;
    const int nj = j_columns(m);
    // inclusive scan over the lanes of both counts at once (16 bits each)
    const int own = dirty ? nj : nj << 16;
    int sdc = own;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, sdc, off);
      if (lane >= off) sdc += v;
    }
    const int before = sdc - own;
    int p = dirty ? pd + (before & 0xffff) : pc + (before >> 16);
    if (nj) {
      const unsigned wd = cand[e];
      const unsigned s0 = (wd & J_MASK) * CJ, rest = wd & ~J_MASK;
#pragma unroll
      for (int b = 0; b < CJ; ++b) {
        const unsigned col = (m >> (b * CL)) & 0xffu;
        if (col) {
          if (p < c.list_cap) {
            segw[p] = (s0 + b) | rest;
            segm[p] = (uint8_t)col;
          }
          ++p;
        }
      }
    }
    const int tot = __shfl_sync(0xffffffffu, sdc, 31);
    pd += tot & 0xffff;
    pc += tot >> 16;
  }
  if (lane == 0 && part == PARTS - 1) {
    d.list_n[I] = min(pc, c.list_cap);
    d.list_nm[I] = min(n_dirty, c.list_cap);
    if (cnt > ENT_MAX || pc > c.list_cap || n_found > CAND_MAX) atomicOr(d.err, ERR_LIST);
  }
}


}  // namespace vp
