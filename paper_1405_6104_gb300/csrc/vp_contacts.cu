// vp_contacts.cu -- the order in which native contacts form along each trial
// and the path similarity of two paths (Sec. "Results": the matrix M of
// contact-formation order and s(k, k'), after Camilloni et al. 2011).
//
// A contact (i, j) of reaction-coordinate atoms is formed when its contact
// value C(r) = (1 - (r/r0)^6)/(1 - (r/r0)^10) exceeds 1/2; with s = (r/r0)^2
// that is s^4 + s^3 - s^2 - s - 1 < 0, i.e. s below the polynomial's positive
// root.  The decision is taken in FP64 on the FP32 positions (exact
// differences), as the definition reads; an FP32 distance far from the
// threshold (outside a 1e-4 relative guard band, some 400 times its rounding
// error) decides alone.  The formation time of a native contact is the step
// from which it has stayed formed (-1: not formed at the last check); checks
// run every `every` steps.
//
// The similarity of two paths counts the ordered contact pairs on which
// their order relations agree.  Only the order of the times within a path
// matters, so they are replaced by dense ranks (on the device: on the host this
// took 2.9 of a call's 3.4 ms for 64 paths of 23 160 contacts); with few
// distinct times (formation times are check steps) the count comes from the
// joint histogram of the two rank arrays in O(n_c + K_a K_b), otherwise from
// all n_c^2 ordered pairs.
#include <algorithm>
#include <climits>
#include <cstring>
#include <string>
#include <thread>
#include <vector>

#include "../../include/vpath.h"
#include "vp_contacts.cuh"

namespace vp {

__device__ __forceinline__ bool contact_formed(float4 pi, float4 pj, float L, float iL, double Ld, double r0,
                                               float r2_lo, float r2_hi) {
  float dx = pj.x - pi.x, dy = pj.y - pi.y, dz = pj.z - pi.z;
  dx -= L * rintf(dx * iL);
  dy -= L * rintf(dy * iL);
  dz -= L * rintf(dz * iL);
  const float r2f = dx * dx + dy * dy + dz * dz;
  if (r2f < r2_lo) return true;
  if (r2f > r2_hi) return false;
  // FP64, every operation rounded on its own (no contraction), in the order of the definition
  double ex = __dsub_rn((double)pj.x, (double)pi.x), ey = __dsub_rn((double)pj.y, (double)pi.y),
         ez = __dsub_rn((double)pj.z, (double)pi.z);
  ex = __dsub_rn(ex, __dmul_rn(Ld, rint(__ddiv_rn(ex, Ld))));
  ey = __dsub_rn(ey, __dmul_rn(Ld, rint(__ddiv_rn(ey, Ld))));
  ez = __dsub_rn(ez, __dmul_rn(Ld, rint(__ddiv_rn(ez, Ld))));
  const double r2 = __dadd_rn(__dadd_rn(__dmul_rn(ex, ex), __dmul_rn(ey, ey)), __dmul_rn(ez, ez));
  const double s = __ddiv_rn(r2, __dmul_rn(r0, r0));
  const double p =
      __dsub_rn(__dmul_rn(__dsub_rn(__dmul_rn(__dsub_rn(__dmul_rn(__dadd_rn(s, 1.0), s), 1.0), s), 1.0), s), 1.0);
  return p < 0.0;
}

// grid: (contacts of the largest system / 256, trials); the step counter has
// just been advanced to the step whose positions are current
__global__ void __launch_bounds__(256) k_contacts(Dev d, ContactDev c) {
  const long long n = *d.step;
  if (n % c.every != 0) return;
  const int t = blockIdx.y;
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  const int sys = c.trial_sys[t];
  if (k >= c.sys_n[sys]) return;
  const int2 pr = c.pairs[c.sys_off[sys] + k];
  const TrialInfo &T = d.tinfo[t];
  const float4 pi = d.pos[d.slot_of[T.atom0 + pr.x]], pj = d.pos[d.slot_of[T.atom0 + pr.y]];
  const bool f = contact_formed(pi, pj, T.box, T.inv_box, (double)T.box, c.r0, c.r2_lo, c.r2_hi);
  long long *tt = c.t + c.t_off[t] + k;
  const long long cur = *tt;
  if (f) {
    if (cur < 0) *tt = n;
  } else if (cur >= 0) {
    *tt = -1;
  }
}

void launch_contacts(const Dev &d, const ContactDev &c, cudaStream_t s) {
  if (c.max_nc <= 0) return;
  dim3 grid((unsigned)((c.max_nc + 255) / 256), (unsigned)d.n_trials);
  k_contacts<<<grid, 256, 0, s>>>(d, c);
}

namespace {

// ---------------------------------------------------------------------------
// dense ranks of the formation times within each path (a negative time, not
// formed, ranks after every formed contact).  Formation times are check
// steps, few per path, so a path's distinct times are collected in a hash set
// (k_distinct), sorted (k_sort_distinct) and looked up (k_rank).  A path of
// more than DISTINCT_CAP distinct times is ranked on the host.
// ---------------------------------------------------------------------------
constexpr int DISTINCT_CAP = 4096;      // distinct times per path the device ranks
constexpr int SET_SLOTS = 8192;         // slots of a path's set in memory ...
constexpr int BLOCK_SLOTS = 1024;       // ... and of the set each block keeps of what it has seen
constexpr int PROBES = 16;              // places tried in the block's set before the path's set is asked
constexpr int RANK_CHUNK = 4096;        // values per block
constexpr long long EMPTY = -1;         // no key is negative

__device__ __forceinline__ long long time_key(long long t) { return t < 0 ? LLONG_MAX : t; }
__device__ __forceinline__ unsigned key_hash(long long k) {
  return (unsigned)(((unsigned long long)k * 0x9E3779B97F4A7C15ull) >> 40);
}

// inserts k into the path's set unless it is there; counts it.  More than
// DISTINCT_CAP keys raise the count past it, which later readers see.
__device__ void set_insert(unsigned long long *set, int *count, long long k) {
  unsigned h = key_hash(k) & (SET_SLOTS - 1);
  for (int q = 0; q < SET_SLOTS; ++q, h = (h + 1) & (SET_SLOTS - 1)) {
    if (*(volatile int *)count > DISTINCT_CAP) return;
    const unsigned long long old = atomicCAS(set + h, (unsigned long long)EMPTY, (unsigned long long)k);
    if (old == (unsigned long long)k) return;
    if (old == (unsigned long long)EMPTY) {
      atomicAdd(count, 1);
      return;
    }
  }
  atomicAdd(count, DISTINCT_CAP + 1);  // the set is full
}

// grid (chunks of RANK_CHUNK values, paths).  Each block remembers the keys it
// has met in shared memory, so that the path's set is asked about once per
// block and distinct key, not once per value.
__global__ void __launch_bounds__(256) k_distinct(const long long *__restrict__ times, long long n_c,
                                                  unsigned long long *sets, int *counts) {
  __shared__ unsigned long long seen[BLOCK_SLOTS];
  const int path = blockIdx.y;
  const long long *t = times + (size_t)path * (size_t)n_c;
  unsigned long long *set = sets + (size_t)path * SET_SLOTS;
  for (int q = threadIdx.x; q < BLOCK_SLOTS; q += 256) seen[q] = (unsigned long long)EMPTY;
  __syncthreads();
  const long long i0 = (long long)blockIdx.x * RANK_CHUNK;
  for (long long i = i0 + threadIdx.x; i < min(n_c, i0 + RANK_CHUNK); i += 256) {
    const long long k = time_key(t[i]);
    unsigned h = (key_hash(k) >> 13) & (BLOCK_SLOTS - 1);
    int state = 0;  // 1: met before; 2: met now; 0 after the loop: no room nearby
    for (int q = 0; q < PROBES && state == 0; ++q, h = (h + 1) & (BLOCK_SLOTS - 1)) {
      unsigned long long v = *(volatile unsigned long long *)(seen + h);
      if (v == (unsigned long long)EMPTY) v = atomicCAS(seen + h, (unsigned long long)EMPTY, (unsigned long long)k);
      if (v == (unsigned long long)k) state = 1;
      else if (v == (unsigned long long)EMPTY) state = 2;
    }
    if (state != 1) set_insert(set, counts + path, k);
  }
}

// one block per path: its distinct times in ascending order and their number
// (-1: more than DISTINCT_CAP)
__global__ void __launch_bounds__(1024) k_sort_distinct(const unsigned long long *sets, const int *counts,
                                                        long long *sorted, int *n_distinct) {
  extern __shared__ long long key[];  // [DISTINCT_CAP]
  __shared__ int n;
  const int path = blockIdx.x;
  const int count = counts[path];
  if (count > DISTINCT_CAP) {
    if (threadIdx.x == 0) n_distinct[path] = -1;
    return;
  }
  if (threadIdx.x == 0) n = 0;
  __syncthreads();
  for (int q = threadIdx.x; q < SET_SLOTS; q += blockDim.x) {
    const long long k = (long long)sets[(size_t)path * SET_SLOTS + q];
    if (k != EMPTY) key[atomicAdd(&n, 1)] = k;
  }
  int p2 = 1;
  while (p2 < count) p2 <<= 1;
  __syncthreads();
  for (int q = count + threadIdx.x; q < p2; q += blockDim.x) key[q] = LLONG_MAX;
  __syncthreads();
  for (int k = 2; k <= p2; k <<= 1)
    for (int j = k >> 1; j > 0; j >>= 1) {
      for (int i = threadIdx.x; i < p2; i += blockDim.x) {
        const int x = i ^ j;
        if (x > i) {
          const long long a = key[i], b = key[x];
          if ((a > b) == ((i & k) == 0)) { key[i] = b; key[x] = a; }
        }
      }
      __syncthreads();
    }
  for (int q = threadIdx.x; q < count; q += blockDim.x) sorted[(size_t)path * DISTINCT_CAP + q] = key[q];
  if (threadIdx.x == 0) n_distinct[path] = count;
}

// grid (chunks, paths): ranks by binary search among the path's distinct
// times (at most DISTINCT_CAP: 16 bits)
__global__ void __launch_bounds__(256) k_rank(const long long *__restrict__ times, long long n_c,
                                              const long long *__restrict__ sorted, const int *__restrict__ n_distinct,
                                              unsigned short *r16, long long ld16) {
  extern __shared__ long long key[];  // [DISTINCT_CAP]
  const int path = blockIdx.y, K = n_distinct[path];
  if (K < 0) return;
  for (int q = threadIdx.x; q < K; q += 256) key[q] = sorted[(size_t)path * DISTINCT_CAP + q];
  __syncthreads();
  const size_t base = (size_t)path * (size_t)n_c, base16 = (size_t)path * (size_t)ld16;
  const long long i0 = (long long)blockIdx.x * RANK_CHUNK;
  for (long long i = i0 + threadIdx.x; i < min(n_c, i0 + RANK_CHUNK); i += 256) {
    const long long k = time_key(times[base + i]);
    int lo = 0, hi = K - 1;
    while (lo < hi) {
      const int mid = (lo + hi) >> 1;
      if (key[mid] < k) lo = mid + 1; else hi = mid;
    }
    r16[base16 + i] = (unsigned short)lo;
  }
}

// the ranks as 32 bits, for the all-pairs kernel (rows of host-ranked paths are
// written over afterwards)
__global__ void __launch_bounds__(256) k_widen(const unsigned short *__restrict__ r16, long long ld16, long long n_c,
                                               int *r32) {
  const long long i = (long long)blockIdx.x * 256 + threadIdx.x;
  if (i < n_c)
    r32[(size_t)blockIdx.y * (size_t)n_c + i] = r16[(size_t)blockIdx.y * (size_t)ld16 + i];
}

// ---------------------------------------------------------------------------
// counting
// ---------------------------------------------------------------------------
constexpr int SIM_TILE = 2048;
constexpr int HIST_CELLS = 4096;        // joint histogram (K_a x K_b) of the counting kernel ...
constexpr int HIST_CELLS_LARGE = 53248; // ... and of its large form (208 KB: one block per SM)

// sign of a - b in {-1, 0, 1}
__device__ __forceinline__ int cmp3(int a, int b) { return (a > b) - (a < b); }

// all ordered pairs: one (path pair, block of i) per block counts the pairs
// (i != j) on which the two paths' order relations agree; keys are the
// paths' dense ranks (order-preserving, unformed contacts last)
__global__ void __launch_bounds__(256) k_similarity(const int *__restrict__ rk, long long n_c,
                                                    const int2 *__restrict__ pp, unsigned long long *count) {
  __shared__ int2 sab[SIM_TILE];
  __shared__ unsigned long long red[256];
  const int2 ab = pp[blockIdx.y];
  const int *ta = rk + (size_t)ab.x * (size_t)n_c, *tb = rk + (size_t)ab.y * (size_t)n_c;
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const int ai = i < n_c ? ta[i] : 0, bi = i < n_c ? tb[i] : 0;
  unsigned int cnt = 0;  // per thread: at most n_c < 2^31
  for (long long j0 = 0; j0 < n_c; j0 += SIM_TILE) {
    __syncthreads();
    for (int q = threadIdx.x; q < SIM_TILE; q += blockDim.x) {
      const long long j = j0 + q;
      sab[q] = j < n_c ? make_int2(ta[j], tb[j]) : make_int2(0, 0);
    }
    __syncthreads();
    if (i < n_c) {
      const int m = (int)(n_c - j0 < SIM_TILE ? n_c - j0 : SIM_TILE);
#pragma unroll 4
      for (int q = 0; q < m; ++q) {
        const int2 v = sab[q];
        cnt += cmp3(ai, v.x) == cmp3(bi, v.y) ? 1u : 0u;
      }
    }
  }
  // the diagonal (j = i) always agrees; it is not an ordered pair
  if (i < n_c) cnt -= 1u;
  red[threadIdx.x] = cnt;
  __syncthreads();
  for (int off = blockDim.x / 2; off > 0; off >>= 1) {
    if (threadIdx.x < off) red[threadIdx.x] += red[threadIdx.x + off];
    __syncthreads();
  }
  if (threadIdx.x == 0) atomicAdd(count + blockIdx.y, red[0]);
}

// few distinct times (K_a K_b <= CELLS): one block per path pair counts
// the same agreements from the joint histogram H[x][y] of the two paths'
// ranks.  Two contacts in one cell tie in both paths (M = 1/2 in both:
// c (c - 1) ordered pairs agree); two contacts in cells strictly below-left
// and above-right of each other are concordant (both ordered pairs agree);
// every other pair disagrees.  So the count is sum c (c - 1) + 2 sum c P,
// with P the number of contacts strictly below-left of the cell.
//
// Bound by the shared-memory atomics of the histogram (a path's contacts fall
// into few cells, so the lanes of a warp collide) and the L2 reads of the
// ranks: the histogram is kept in as many copies as fit, up to one per lane
// (each on its own bank), and the ranks are read eight at a time as 16 bits.
// 2016 pairs of 23 160 contacts, 121 cells: 39 us with one copy and 32-bit
// ranks read one at a time, 26 with these.
template <int CELLS>
__global__ void __launch_bounds__(256) k_similarity_hist(const unsigned short *__restrict__ rk, long long n_c,
                                                         long long ld,  // row length, a multiple of 8
                                                         const int2 *__restrict__ pp, const int *__restrict__ kk,
                                                         const int *__restrict__ list,
                                                         unsigned long long *count) {
  extern __shared__ unsigned H[];  // [CELLS]
  __shared__ unsigned long long red[8];
  const int q = list[blockIdx.x];
  const int2 ab = pp[q];
  const int Ka = kk[ab.x], Kb = kk[ab.y], nc = Ka * Kb;
  const unsigned short *ta = rk + (size_t)ab.x * (size_t)ld, *tb = rk + (size_t)ab.y * (size_t)ld;
  int sh = 0;  // copies of the histogram: 2^sh
  while (sh < 5 && (nc << (sh + 1)) <= CELLS) ++sh;
  const int copies = 1 << sh, mine = threadIdx.x & (copies - 1);
  for (int c = threadIdx.x; c < (nc << sh); c += blockDim.x) H[c] = 0u;
  __syncthreads();
  auto add = [&](unsigned a, unsigned b) { atomicAdd(&H[((a * (unsigned)Kb + b) << sh) + mine], 1u); };
  const long long n8 = n_c / 8;  // eight ranks per load (rows start on 16 bytes)
  for (long long i = threadIdx.x; i < n8; i += blockDim.x) {
    const uint4 a = reinterpret_cast<const uint4 *>(ta)[i], b = reinterpret_cast<const uint4 *>(tb)[i];
    const unsigned av[4] = {a.x, a.y, a.z, a.w}, bv[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
    for (int w = 0; w < 4; ++w) {
      add(av[w] & 0xffffu, bv[w] & 0xffffu);
      add(av[w] >> 16, bv[w] >> 16);
    }
  }
  for (long long i = 8 * n8 + threadIdx.x; i < n_c; i += blockDim.x) add(ta[i], tb[i]);
  __syncthreads();
  // the copies' sum into the first nc words: 256 cells' copies are read before
  // any of these cells is written, and later cells' copies lie above them all
  if (sh > 0) {
    for (int c0 = 0; c0 < nc; c0 += 256) {
      const int c = c0 + threadIdx.x;
      unsigned v = 0;
      if (c < nc)
        for (int u = 0; u < copies; ++u) v += H[(c << sh) + ((u + c) & (copies - 1))];
      __syncthreads();
      if (c < nc) H[c] = v;
      __syncthreads();
    }
  }
  // inclusive prefix along each row, one warp per row
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int x = warp; x < Ka; x += 8) {
    unsigned run = 0;
    for (int y0 = 0; y0 < Kb; y0 += 32) {
      const int y = y0 + lane;
      unsigned v = y < Kb ? H[x * Kb + y] : 0u;
#pragma unroll
      for (int off = 1; off < 32; off <<= 1) {
        const unsigned o = __shfl_up_sync(0xffffffffu, v, off);
        if (lane >= off) v += o;
      }
      v += run;
      if (y < Kb) H[x * Kb + y] = v;
      run = __shfl_sync(0xffffffffu, v, 31);
    }
  }
  __syncthreads();
  // down each column: the cell's own count, and what lies strictly below-left
  unsigned long long acc = 0;
  for (int y = threadIdx.x; y < Kb; y += blockDim.x) {
    unsigned long long below = 0;
    for (int x = 0; x < Ka; ++x) {
      const unsigned long long left = y > 0 ? H[x * Kb + y - 1] : 0u, c = H[x * Kb + y] - left;
      if (c) acc += c * (c - 1ull) + 2ull * c * below;
      below += left;
    }
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
  if (lane == 0) red[warp] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 8; ++w) acc += red[w];
    count[q] = acc;
  }
}

// dense ranks of one path on the host
void rank_on_host(const int64_t *t, int64_t n_c, int *rk) {
  std::vector<int64_t> v((size_t)n_c), u;
  for (int64_t i = 0; i < n_c; ++i) v[(size_t)i] = t[i] < 0 ? INT64_MAX : t[i];
  u = v;
  std::sort(u.begin(), u.end());
  u.erase(std::unique(u.begin(), u.end()), u.end());
  for (int64_t i = 0; i < n_c; ++i) rk[i] = (int)(std::lower_bound(u.begin(), u.end(), v[(size_t)i]) - u.begin());
}

int put_err(char *errbuf, int32_t errlen, int code, const std::string &msg) {
  if (errbuf && errlen > 0) {
    std::strncpy(errbuf, msg.c_str(), (size_t)errlen - 1);
    errbuf[errlen - 1] = '\0';
  }
  return code;
}

}  // namespace
}  // namespace vp

using namespace vp;

extern "C" __attribute__((visibility("default"))) int path_similarity(const int64_t *times, int32_t n_paths,
                                                                      int64_t n_c, const int32_t *pairs,
                                                                      int32_t n_pairs, double *s, void *cuda_stream,
                                                                      char *errbuf, int32_t errlen) {
  if (n_paths < 0 || n_c < 0 || n_pairs < 0 || (n_pairs > 0 && (!pairs || !s)) || (n_paths > 0 && n_c > 0 && !times))
    return put_err(errbuf, errlen, SIM_EINVAL, "path_similarity: null argument or negative size");
  for (int32_t q = 0; q < n_pairs; ++q)
    if (pairs[2 * q] < 0 || pairs[2 * q] >= n_paths || pairs[2 * q + 1] < 0 || pairs[2 * q + 1] >= n_paths)
      return put_err(errbuf, errlen, SIM_EINVAL, "path_similarity: path index out of range");
  if (n_pairs == 0) return SIM_OK;
  if (n_c < 2) {  // no ordered pair: identical by definition
    for (int32_t q = 0; q < n_pairs; ++q) s[q] = 1.0;
    return SIM_OK;
  }
  if (n_c > (1ll << 30)) return put_err(errbuf, errlen, SIM_EINVAL, "path_similarity: too many contacts");
  if (n_pairs > 65535) return put_err(errbuf, errlen, SIM_EINVAL, "path_similarity: at most 65535 pairs per call");
  const size_t nt = (size_t)n_paths * (size_t)n_c, np = (size_t)n_pairs;
  cudaStream_t st = (cudaStream_t)cuda_stream;
  std::string err;
  auto ck = [&](cudaError_t e, const char *what) {
    if (e != cudaSuccess && err.empty()) err = std::string(what) + ": " + cudaGetErrorString(e);
    return e == cudaSuccess;
  };
  // one allocation: the 16-bit ranks, and for a group of paths at a time their
  // times, sets and sorted distinct times (smaller groups with little memory left)
  int32_t group = (int32_t)std::max<int64_t>(1, std::min<int64_t>({(int64_t)n_paths, 256, ((int64_t)1 << 27) / n_c}));
  const long long ld16 = ((long long)n_c + 7) & ~7ll;  // row length of the 16-bit ranks: rows start on 16 bytes
  size_t o_times, o_set, o_cnt, o_sorted, o_k, o_r16, o_pp, o_list, o_all, o_count, o_call;
  char *buf = nullptr;
  bool ok = true;
  for (;;) {
    size_t total = 0;
    auto part = [&](size_t bytes) {
      const size_t off = total;
      total += (bytes + 255) & ~(size_t)255;
      return off;
    };
    o_times = part((size_t)group * (size_t)n_c * 8);
    o_set = part((size_t)group * SET_SLOTS * 8);
    o_cnt = part((size_t)group * 4);
    o_sorted = part((size_t)group * DISTINCT_CAP * 8);
    o_k = part((size_t)n_paths * 4);
    o_r16 = part((size_t)n_paths * (size_t)ld16 * 2);
    o_pp = part(np * 8);
    o_list = part(2 * np * 4);
    o_all = part(np * 8);
    o_count = part(np * 8);
    o_call = part(np * 8);
    if (cudaMalloc(&buf, total) == cudaSuccess) break;
    const cudaError_t e = cudaGetLastError();
    if (e != cudaErrorMemoryAllocation || group == 1) {
      ok = ck(e, "cudaMalloc");
      break;
    }
    group /= 2;
  }
  long long *d_times = (long long *)(buf + o_times), *d_sorted = (long long *)(buf + o_sorted);
  unsigned long long *d_sets = (unsigned long long *)(buf + o_set);
  int *d_cnt = (int *)(buf + o_cnt), *d_k = (int *)(buf + o_k), *d_list = (int *)(buf + o_list);
  unsigned short *d_r16 = (unsigned short *)(buf + o_r16);
  int2 *d_pp = (int2 *)(buf + o_pp), *d_all = (int2 *)(buf + o_all);
  unsigned long long *d_count = (unsigned long long *)(buf + o_count), *d_call = (unsigned long long *)(buf + o_call);
  const int rank_smem = DISTINCT_CAP * (int)sizeof(long long);
  const dim3 chunks((unsigned)((n_c + RANK_CHUNK - 1) / RANK_CHUNK), 1);
  for (int32_t p0 = 0; ok && p0 < n_paths; p0 += group) {
    const int32_t m = std::min(group, n_paths - p0);
    const size_t off = (size_t)p0 * (size_t)n_c;
    ok = ck(cudaMemcpyAsync(d_times, times + off, (size_t)m * (size_t)n_c * 8, cudaMemcpyHostToDevice, st), "cudaMemcpyAsync") &&
         ck(cudaMemsetAsync(d_sets, 0xff, (size_t)m * SET_SLOTS * 8, st), "cudaMemsetAsync") &&
         ck(cudaMemsetAsync(d_cnt, 0, (size_t)m * 4, st), "cudaMemsetAsync");
    if (!ok) break;
    const dim3 g(chunks.x, (unsigned)m);
    k_distinct<<<g, 256, 0, st>>>(d_times, (long long)n_c, d_sets, d_cnt);
    k_sort_distinct<<<(unsigned)m, 1024, rank_smem, st>>>(d_sets, d_cnt, d_sorted, d_k + p0);
    k_rank<<<g, 256, rank_smem, st>>>(d_times, (long long)n_c, d_sorted, d_k + p0,
                                       d_r16 + (size_t)p0 * (size_t)ld16, ld16);
    ok = ck(cudaGetLastError(), "ranking launch");
  }
  std::vector<int> K((size_t)n_paths);
  ok = ok && ck(cudaMemcpyAsync(d_pp, pairs, np * 8, cudaMemcpyHostToDevice, st), "cudaMemcpyAsync") &&
       ck(cudaMemcpyAsync(K.data(), d_k, (size_t)n_paths * 4, cudaMemcpyDeviceToHost, st), "cudaMemcpyAsync") &&
       ck(cudaStreamSynchronize(st), "cudaStreamSynchronize");
  // path pairs by the size of their joint histogram: the counting kernel, its
  // large form, or all ordered contact pairs
  std::vector<int> lists[2], all_list;
  std::vector<int2> all_pp;
  for (int32_t q = 0; ok && q < n_pairs; ++q) {
    const int ka = K[(size_t)pairs[2 * q]], kb = K[(size_t)pairs[2 * q + 1]];
    const long long cells = (long long)ka * (long long)kb;
    const bool hist = ka >= 0 && kb >= 0 && cells <= HIST_CELLS_LARGE;  // (a path the device did not rank has -1)
    if (hist) {
      lists[cells <= HIST_CELLS ? 0 : 1].push_back(q);
    } else {
      all_list.push_back(q);
      all_pp.push_back(make_int2(pairs[2 * q], pairs[2 * q + 1]));
    }
  }
  const size_t na = all_list.size();
  for (int f = 0; ok && f < 2; ++f) {
    const size_t n = lists[f].size();
    if (n == 0) continue;
    int *dl = d_list + (size_t)f * np;
    ok = ck(cudaMemcpyAsync(dl, lists[f].data(), n * 4, cudaMemcpyHostToDevice, st), "cudaMemcpyAsync");
    if (!ok) break;
    if (f == 0) {
      k_similarity_hist<HIST_CELLS><<<(unsigned)n, 256, HIST_CELLS * 4, st>>>(d_r16, (long long)n_c, ld16, d_pp, d_k, dl, d_count);
    } else {
      ok = ck(cudaFuncSetAttribute(k_similarity_hist<HIST_CELLS_LARGE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   HIST_CELLS_LARGE * 4), "cudaFuncSetAttribute");
      if (ok)
        k_similarity_hist<HIST_CELLS_LARGE><<<(unsigned)n, 256, HIST_CELLS_LARGE * 4, st>>>(d_r16, (long long)n_c, ld16, d_pp,
                                                                                            d_k, dl, d_count);
    }
    ok = ok && ck(cudaGetLastError(), "k_similarity_hist launch");
  }
  // all ordered pairs need 32-bit ranks; those of paths of more distinct times
  // than the device ranks come from up to 16 host threads (their number is not
  // needed: only that it exceeds DISTINCT_CAP)
  // They take the place of the times, which are ranked, where they fit (up to 512
  // paths; an allocation and its free take some 100 us).
  int *d_r32 = nt * 4 <= (size_t)group * (size_t)n_c * 8 ? (int *)d_times : nullptr, *r32_own = nullptr;
  std::vector<int> rk;
  if (ok && na > 0) {
    if (!d_r32) {
      ok = ck(cudaMalloc(&r32_own, nt * 4), "cudaMalloc");
      d_r32 = r32_own;
    }
    for (int32_t p0 = 0; ok && p0 < n_paths; p0 += 65535) {
      const int32_t m = std::min(n_paths - p0, 65535);
      k_widen<<<dim3((unsigned)((n_c + 255) / 256), (unsigned)m), 256, 0, st>>>(
          d_r16 + (size_t)p0 * (size_t)ld16, ld16, (long long)n_c, d_r32 + (size_t)p0 * (size_t)n_c);
      ok = ck(cudaGetLastError(), "k_widen launch");
    }
    std::vector<int32_t> many;
    for (int32_t p = 0; p < n_paths; ++p)
      if (K[(size_t)p] < 0) many.push_back(p);
    if (ok && !many.empty()) {
      rk.resize(many.size() * (size_t)n_c);
      auto work = [&](size_t a, size_t b) {
        for (size_t q = a; q < b; ++q)
          rank_on_host(times + (size_t)many[q] * (size_t)n_c, n_c, rk.data() + q * (size_t)n_c);
      };
      const size_t nw =
          std::max<size_t>(1, std::min<size_t>({(size_t)std::thread::hardware_concurrency(), 16, many.size()}));
      std::vector<std::thread> pool;
      for (size_t w = 1; w < nw; ++w) pool.emplace_back(work, many.size() * w / nw, many.size() * (w + 1) / nw);
      work(0, many.size() / nw);
      for (auto &th : pool) th.join();
      for (size_t q = 0; ok && q < many.size(); ++q)
        ok = ck(cudaMemcpyAsync(d_r32 + (size_t)many[q] * (size_t)n_c, rk.data() + q * (size_t)n_c, (size_t)n_c * 4,
                                cudaMemcpyHostToDevice, st), "cudaMemcpyAsync");
    }
  }
  if (ok && na > 0) {
    ok = ck(cudaMemcpyAsync(d_all, all_pp.data(), na * sizeof(int2), cudaMemcpyHostToDevice, st), "cudaMemcpyAsync") &&
         ck(cudaMemsetAsync(d_call, 0, na * sizeof(unsigned long long), st), "cudaMemsetAsync");
    if (ok) {
      dim3 grid((unsigned)((n_c + 255) / 256), (unsigned)na);
      k_similarity<<<grid, 256, 0, st>>>(d_r32, (long long)n_c, d_all, d_call);
      ok = ck(cudaGetLastError(), "k_similarity launch");
    }
  }
  std::vector<unsigned long long> hc(np, 0ull), ha(na, 0ull);
  if (ok && na < np)
    ok = ck(cudaMemcpyAsync(hc.data(), d_count, np * sizeof(unsigned long long), cudaMemcpyDeviceToHost, st),
            "cudaMemcpyAsync");
  if (ok && na > 0)
    ok = ck(cudaMemcpyAsync(ha.data(), d_call, na * sizeof(unsigned long long), cudaMemcpyDeviceToHost, st),
            "cudaMemcpyAsync");
  ck(cudaStreamSynchronize(st), "cudaStreamSynchronize");
  if (ok && err.empty()) {
    for (size_t k = 0; k < na; ++k) hc[(size_t)all_list[k]] = ha[k];
    const double denom = (double)n_c * (double)(n_c - 1);
    for (int32_t q = 0; q < n_pairs; ++q) s[q] = (double)hc[(size_t)q] / denom;
  }
  cudaFree(buf);
  cudaFree(r32_own);
  if (!err.empty()) return put_err(errbuf, errlen, SIM_ECUDA, "path_similarity: " + err);
  return SIM_OK;
}
