// vp_noalloc.cu -- the reaction coordinate z and its gradient for one
// configuration, computed without allocating any device memory.
//
// Some callers cannot call cudaMalloc: a host program whose device memory is
// owned by another allocator (a framework's caching allocator that has
// reserved the memory, or a fixed per-process budget) must not have a library
// take device memory behind its back, and a latency-critical caller cannot
// accept the implicit device-wide synchronisation that cudaMalloc/cudaFree may
// perform.  This entry point serves them: it is a variant of the batched
// reaction-coordinate kernel of vp_cv.cu in which every piece of scratch (the
// per-tile partial sums of z, the fixed-point gradient accumulators and a block
// counter) lives in one file-scope device array of fixed size, and the native
// contact map is evaluated on the fly instead of from a precomputed table.
//
// The array is allocated when the library is loaded and is held by every GPU
// that loads it until the process exits.  Its device address is
// looked up once per device with cudaGetSymbolAddress, with that device
// current, during the first call on that device; that first call should
// therefore come before any stream capture on that device.  All calls share
// the array and it keeps the last call's contents, so each call clears what must
// start at zero, and calls that overlap on the GPU (on different streams) race.
#include <cstring>
#include <mutex>
#include <string>

#include "../../include/vpath.h"
#include "vp_cvpair.cuh"
#include "vp_internal.cuh"

#define VP_API extern "C" __attribute__((visibility("default")))

namespace vp {
namespace noalloc {

constexpr int MAX_CV = 2048;                      // reaction-coordinate atoms per call
constexpr int MAX_NB = MAX_CV / CV_T;             // 64 tile rows
constexpr int MAX_TILES = MAX_NB * MAX_NB;        // tile grid (upper triangle used)
// scratch: 3 gradient components (int64) per atom + one FP64 partial per tile
// (contact and native-map sums) + the block counter: 112 KiB reserved
constexpr size_t SCRATCH_BYTES =
    (size_t)3 * MAX_CV * sizeof(long long) + (size_t)2 * MAX_TILES * sizeof(double);

static __device__ __align__(256) unsigned char g_scratch[SCRATCH_BYTES];

struct Scratch {
  long long *gx, *gy, *gz;
  unsigned *done;   // right after the gradient sums: cleared with them
  double *zpart;
};
constexpr size_t CLEAR_BYTES = (size_t)3 * MAX_CV * sizeof(long long) + 256;

__host__ __device__ inline Scratch carve(unsigned char *base) {
  Scratch s;
  s.gx = reinterpret_cast<long long *>(base);
  s.gy = s.gx + MAX_CV;
  s.gz = s.gy + MAX_CV;
  s.done = reinterpret_cast<unsigned *>(s.gz + MAX_CV);
  s.zpart = reinterpret_cast<double *>(base + CLEAR_BYTES);
  return s;
}
static_assert(CLEAR_BYTES + (size_t)MAX_NB * (MAX_NB + 1) / 2 * sizeof(double) <= SCRATCH_BYTES, "scratch layout");

struct Consts {
  float L, iL;
  float inv_r0sq_hi, inv_r0sq_lo, rs_hi, rs_lo, inv_w_hi, inv_w_lo, rs2, rc2_far;
  double inv_r0sq, rs, inv_w, rc2;
  float rc2_nat;        // a native pair farther than this (FP32 distance squared) is beyond the cut-off
  int n_cv, min_sep;
  int dmin, m, n_tiles; // tiles (bi, bi + dmin + q), q = 0 .. m - 1, the shorter diagonals last
};

// the same rational form of the contact function as the batched kernel
__device__ __forceinline__ ff contact_s(ff s) {
  ff s2 = ff_sqr(s);
  ff s3 = ff_mul(s2, s);
  ff s4 = ff_sqr(s2);
  ff N = ff_add(ff_add_f(s, 1.0f), s2);
  ff D = ff_add(ff_add(N, s3), s4);
  return ff_div(N, D);
}

__device__ __forceinline__ float dcontact(float s) {
  float N = 1.0f + s + s * s;
  float D = N + s * s * s + s * s * s * s;
  float dN = 1.0f + 2.0f * s;
  float dD = dN + 3.0f * s * s + 4.0f * s * s * s;
  return (dN * D - N * dD) / (D * D);
}

// C~ of a native pair at the squared distance d2, in FP64
__device__ __forceinline__ double native_contact(double d2, const Consts &k) {
  if (d2 >= k.rc2) return 0.0;
  const double s = d2 * k.inv_r0sq;
  const double s2 = s * s;
  const double N = 1.0 + s + s2;
  const double C = N / (N + s2 * s + s2 * s2);
  if (d2 <= k.rs * k.rs) return C;
  const double x = (sqrt(d2) - k.rs) * k.inv_w;
  return C * (1.0 - x * x * x * (10.0 - 15.0 * x + 6.0 * x * x));
}

// a contribution too large for the tile's halves (out of line: the kernel is
// short enough for its code to be fetched cold)
static __device__ __noinline__ void add_large(Scratch sc, int i, int j, float gx, float gy, float gz) {
  const long long v[3] = {fx_from(gx), fx_from(gy), fx_from(gz)};
  long long *const sum[3] = {sc.gx, sc.gy, sc.gz};
  for (int c = 0; c < 3; ++c) {
    red_add(sum[c] + i, (long long)(0ull - (unsigned long long)v[c]));
    red_add(sum[c] + j, v[c]);
  }
}

// One kernel: a block of NW warps per 32 x 32 tile of the contact-pair
// triangle lists the pairs that are near in the configuration or in the native
// structure (FP32 distances, a rotation of the tile per warp and step) and
// evaluates them densely; the block that finishes last sums the tiles' shares
// of z in a fixed order and turns the gradient to FP64.
//
// Bound by latency: 136 tiles of 540 atoms, one block per SM, and this part's
// FP64 unit (a warp instruction takes 16 cycles), which the native contact map
// needs.  Hence no square root or division per pair but N / D (and a square
// root in the switching range), none at all for pairs beyond the cut-off in
// the native structure, and eight warps per tile to have their chains of
// float-float operations side by side.  One warp per tile with the full FP64
// contact per pair, and clearing and finishing kernels around it, took 103 us
// (n_cv = 540); this one 24.
constexpr int NW = 8;
struct TileShared {
  unsigned short s_near[CV_T * CV_T];
  float s_x[2 * CV_T][3];
  float s_nf[2 * CV_T][3];
  double s_n[2 * CV_T][3];
  int s_ghi[2 * CV_T][3];   // c >> 24 and the low 24 bits of each contribution c
  unsigned s_glo[2 * CV_T][3];
  unsigned s_bal[CV_T];
  double s_z[NW];
  bool last;
};
constexpr unsigned POS_NEAR = 1u << 10, NAT_NEAR = 1u << 11;

__global__ void __launch_bounds__(NW * 32) k_eval(const float *__restrict__ pos, const double *__restrict__ native,
                                                  Consts k, Scratch sc, double *z_out, double *grad_out) {
  __shared__ TileShared sh;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  double zl = 0.0;
  if ((int)blockIdx.x < k.n_tiles) {
    // diagonal q holds m - q tiles: q (2 m + 1 - q) / 2 of them come before it
    int q = 0, t = blockIdx.x;
    {
      const float h = (float)k.m + 0.5f;
      q = min(k.m - 1, max(0, (int)(h - sqrtf(fmaxf(h * h - 2.0f * (float)t, 0.0f)))));
      while (q > 0 && q * (2 * k.m + 1 - q) / 2 > t) --q;
      while ((q + 1) * (2 * k.m - q) / 2 <= t) ++q;
      t -= q * (2 * k.m + 1 - q) / 2;
    }
    const int bi = t, bj = t + k.dmin + q;
    if (threadIdx.x < 2 * CV_T) {
      const int a = (warp == 0 ? bi : bj) * CV_T + lane;
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        sh.s_x[threadIdx.x][c] = a < k.n_cv ? pos[3 * a + c] : 0.f;
        const double v = a < k.n_cv ? native[3 * a + c] : 0.0;
        sh.s_n[threadIdx.x][c] = v;
        // relative to the tile's first atom: FP32 distances wherever the structure lies
        sh.s_nf[threadIdx.x][c] = (float)(v - native[3 * bi * CV_T + c]);
      }
    }
    for (int e = threadIdx.x; e < 2 * CV_T * 3; e += NW * 32) {
      (&sh.s_ghi[0][0])[e] = 0;
      (&sh.s_glo[0][0])[e] = 0u;
    }
    __syncthreads();
    const int i = bi * CV_T + lane;
    constexpr int KW = CV_T / NW;
    unsigned bal[KW], flags[KW];
#pragma unroll
    for (int u = 0; u < KW; ++u) {
      const int jc = (lane + warp * KW + u) & (CV_T - 1);
      const int j = bj * CV_T + jc;
      flags[u] = 0u;
      if (i < k.n_cv && j < k.n_cv && j - i > k.min_sep) {
        const float *a = sh.s_x[lane], *b = sh.s_x[CV_T + jc];
        float dx = b[0] - a[0], dy = b[1] - a[1], dz = b[2] - a[2];
        const float near2 = cv_near2(k.rc2_far, fmaxf(fmaxf(dx * dx, dy * dy), dz * dz));
        dx -= k.L * rintf(dx * k.iL);
        dy -= k.L * rintf(dy * k.iL);
        dz -= k.L * rintf(dz * k.iL);
        if (dx * dx + dy * dy + dz * dz < near2) flags[u] |= POS_NEAR;
        a = sh.s_nf[lane];
        b = sh.s_nf[CV_T + jc];
        dx = b[0] - a[0]; dy = b[1] - a[1]; dz = b[2] - a[2];
        // (not greater: a native distance that is not a number stays in)
        if (!(dx * dx + dy * dy + dz * dz > k.rc2_nat)) flags[u] |= NAT_NEAR;
      }
      bal[u] = __ballot_sync(0xffffffffu, flags[u] != 0u);
      if (lane == 0) sh.s_bal[warp * KW + u] = bal[u];
    }
    __syncthreads();
    int incl = __popc(sh.s_bal[lane]);
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, incl, off);
      if (lane >= off) incl += v;
    }
    const int n_near = __shfl_sync(0xffffffffu, incl, 31);
#pragma unroll
    for (int u = 0; u < KW; ++u) {
      const int end = __shfl_sync(0xffffffffu, incl, warp * KW + u);
      if (flags[u])
        sh.s_near[end - __popc(bal[u]) + __popc(bal[u] & ((1u << lane) - 1u))] =
            (unsigned short)(lane | (((lane + warp * KW + u) & (CV_T - 1)) << 5) | flags[u]);
    }
    __syncthreads();
    const ff inv_r0sq = {k.inv_r0sq_hi, k.inv_r0sq_lo};
    ff zacc = {0.f, 0.f};
    double z0 = 0.0;
    for (int p = threadIdx.x; p < n_near; p += NW * 32) {
      const unsigned e = sh.s_near[p];
      const int il = e & 31, jc = (e >> 5) & 31;
      double cnat_d = 0.0;
      if (e & NAT_NEAR) {
        const double *a = sh.s_n[il], *b = sh.s_n[CV_T + jc];
        const double dx = b[0] - a[0], dy = b[1] - a[1], dz = b[2] - a[2];
        cnat_d = native_contact(dx * dx + dy * dy + dz * dz, k);
        z0 += cnat_d * cnat_d;
      }
      if (!(e & POS_NEAR)) continue;
      const float *a = sh.s_x[il], *b = sh.s_x[CV_T + jc];
      ff dx = ff_diff(b[0], a[0]), dy = ff_diff(b[1], a[1]), dz = ff_diff(b[2], a[2]);
      const float nx = rintf(dx.hi * k.iL), ny = rintf(dy.hi * k.iL), nz = rintf(dz.hi * k.iL);
      if (nx != 0.f) dx = ff_add_f(dx, -k.L * nx);
      if (ny != 0.f) dy = ff_add_f(dy, -k.L * ny);
      if (nz != 0.f) dz = ff_add_f(dz, -k.L * nz);
      const ff cnat = ff_from_d(cnat_d);
      const ff r2 = ff_add(ff_add(ff_sqr(dx), ff_sqr(dy)), ff_sqr(dz));
      const ff sv = ff_mul(r2, inv_r0sq);
      ff Ct = contact_s(sv);
      const float rf = sqrtf(r2.hi);
      float dCt = dcontact(sv.hi) * 2.0f * rf * inv_r0sq.hi;
      if (r2.hi > k.rs2) {
        const ff r = ff_sqrt(r2);
        const ff x = ff_mul(ff_add(r, ff{-k.rs_hi, -k.rs_lo}), ff{k.inv_w_hi, k.inv_w_lo});
        if (x.hi >= 1.0f) {
          Ct = {0.f, 0.f};
          dCt = 0.f;
        } else {
          ff p2 = ff_add_f(ff_mul_f(x, 6.0f), -15.0f);
          p2 = ff_add_f(ff_mul(p2, x), 10.0f);
          const ff x3 = ff_mul(ff_sqr(x), x);
          const ff S = ff_add_f(ff_neg(ff_mul(x3, p2)), 1.0f);
          const float xf = x.hi;
          const float dS = -30.0f * xf * xf * (1.0f - xf) * (1.0f - xf) * k.inv_w_hi;
          dCt = dCt * S.hi + Ct.hi * dS;
          Ct = ff_mul(Ct, S);
        }
      }
      const ff h = ff_add(Ct, ff_neg(cnat));
      zacc = ff_add(zacc, ff_mul(Ct, ff_add(Ct, ff_neg(ff_mul_f(cnat, 2.0f)))));
      const float wgt = 2.0f * h.hi * dCt / rf;
      const float g[3] = {wgt * dx.hi, wgt * dy.hi, wgt * dz.hi};
      // 32 contributions below 2^16 stay within the 32-bit halves; a larger one
      // goes straight to the sums (contacts of a radius or switching range below
      // some 1e-5 nm).  Coincident atoms (wgt not a number) pull nowhere.
      if (!(fmaxf(fmaxf(fabsf(g[0]), fabsf(g[1])), fabsf(g[2])) < 65536.0f)) {
        if (wgt == wgt) add_large(sc, bi * CV_T + il, bj * CV_T + jc, g[0], g[1], g[2]);
        continue;
      }
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const long long v = fx_from(g[c]);
        atomicAdd(&sh.s_ghi[il][c], (int)((-v) >> 24));
        atomicAdd(&sh.s_glo[il][c], (unsigned)((-v) & 0xffffff));
        atomicAdd(&sh.s_ghi[CV_T + jc][c], (int)(v >> 24));
        atomicAdd(&sh.s_glo[CV_T + jc][c], (unsigned)(v & 0xffffff));
      }
    }
    zl = ff_to_d(zacc) + z0;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) zl += __shfl_xor_sync(0xffffffffu, zl, off);
    if (lane == 0) sh.s_z[warp] = zl;
    __syncthreads();
    // the tile's gradient into the sums, its share of z
    for (int e = threadIdx.x; e < 2 * CV_T * 3; e += NW * 32) {
      const int row = e / 3, c = e - 3 * row;
      const int a = (row < CV_T ? bi : bj) * CV_T + (row & (CV_T - 1));
      const long long v = (long long)sh.s_ghi[row][c] * 16777216ll + (long long)sh.s_glo[row][c];
      if (a < k.n_cv && v != 0) red_add((c == 0 ? sc.gx : c == 1 ? sc.gy : sc.gz) + a, v);
    }
    if (threadIdx.x == 0) {
      double s = 0.0;
      for (int u = 0; u < NW; ++u) s += sh.s_z[u];
      sc.zpart[blockIdx.x] = s;
    }
  }
  // the last block to get here finishes
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) sh.last = atomicAdd(sc.done, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!sh.last) return;
  __threadfence();
  zl = 0.0;
  for (int t = threadIdx.x; t < k.n_tiles; t += NW * 32) zl += __ldcg(sc.zpart + t);
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) zl += __shfl_xor_sync(0xffffffffu, zl, off);
  if (lane == 0) sh.s_z[warp] = zl;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int u = 0; u < NW; ++u) s += sh.s_z[u];
    *z_out = s;
  }
  const double s = 2.3283064365386963e-10;
  for (int i = threadIdx.x; i < k.n_cv; i += NW * 32) {
    grad_out[3 * i] = (double)__ldcg(sc.gx + i) * s;
    grad_out[3 * i + 1] = (double)__ldcg(sc.gy + i) * s;
    grad_out[3 * i + 2] = (double)__ldcg(sc.gz + i) * s;
  }
}

// per-device address of the static scratch
constexpr int MAX_DEVICES = 64;
static unsigned char *g_addr[MAX_DEVICES];
static std::mutex g_mutex;

}  // namespace noalloc
}  // namespace vp

using namespace vp;

static void set_msg(char *buf, int32_t len, const char *msg) {
  if (buf && len > 0) {
    std::strncpy(buf, msg, (size_t)len - 1);
    buf[len - 1] = '\0';
  }
}

VP_API int cv_eval_noalloc(const float *d_pos, const double *d_native, int32_t n_cv, double box,
                           const sim_params *params, double *d_z, double *d_grad, void *cuda_stream, char *errbuf,
                           int32_t errlen) {
  using namespace vp::noalloc;
  if (!params || !d_z || (n_cv > 0 && (!d_pos || !d_native || !d_grad))) {
    set_msg(errbuf, errlen, "cv_eval_noalloc: missing argument");
    return SIM_EINVAL;
  }
  if (n_cv < 0 || n_cv > MAX_CV) {
    set_msg(errbuf, errlen, "cv_eval_noalloc: n_cv exceeds the fixed scratch limit of 2048 atoms");
    return SIM_EINVAL;
  }
  if (!(box > 0.0) || !(params->cv_r0 > 0.0) || !(params->cv_r_cut > params->cv_r_switch) ||
      !(params->cv_r_switch > 0.0) || params->cv_min_sep < 0) {
    set_msg(errbuf, errlen, "cv_eval_noalloc: invalid box or contact parameters");
    return SIM_EINVAL;
  }
  // an error left on this thread by earlier work is reported as such, before
  // anything is launched, so that the check after the launches sees only ours
  {
    const cudaError_t pending = cudaGetLastError();
    if (pending != cudaSuccess) {
      set_msg(errbuf, errlen, (std::string("cv_eval_noalloc: an earlier CUDA error is pending: ") +
                               cudaGetErrorString(pending)).c_str());
      return SIM_ECUDA;
    }
  }
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= MAX_DEVICES) {
    set_msg(errbuf, errlen, "cv_eval_noalloc: no usable current device");
    return SIM_ECUDA;
  }
  unsigned char *base = nullptr;
  {
    std::lock_guard<std::mutex> lock(g_mutex);
    if (!g_addr[dev]) {
      void *p = nullptr;
      cudaError_t e = cudaGetSymbolAddress(&p, g_scratch);
      if (e != cudaSuccess) {
        set_msg(errbuf, errlen, cudaGetErrorString(e));
        return SIM_ECUDA;
      }
      g_addr[dev] = static_cast<unsigned char *>(p);
    }
    base = g_addr[dev];
  }
  cudaStream_t st = (cudaStream_t)cuda_stream;
  const Scratch sc = carve(base);
  Consts k{};
  const float Lf = (float)box;
  k.L = Lf;
  k.iL = (float)(1.0 / (double)Lf);
  auto split = [](double v, float &hi, float &lo) {
    hi = (float)v;
    lo = (float)(v - (double)hi);
  };
  split(1.0 / (params->cv_r0 * params->cv_r0), k.inv_r0sq_hi, k.inv_r0sq_lo);
  split(params->cv_r_switch, k.rs_hi, k.rs_lo);
  split(1.0 / (params->cv_r_cut - params->cv_r_switch), k.inv_w_hi, k.inv_w_lo);
  k.rs2 = (float)(params->cv_r_switch * params->cv_r_switch);
  k.rc2_far = (float)(params->cv_r_cut * params->cv_r_cut * (1.0 + 1e-4));
  k.inv_r0sq = 1.0 / (params->cv_r0 * params->cv_r0);
  k.rs = params->cv_r_switch;
  k.inv_w = 1.0 / (params->cv_r_cut - params->cv_r_switch);
  k.rc2 = params->cv_r_cut * params->cv_r_cut;
  k.n_cv = n_cv;
  k.min_sep = params->cv_min_sep;
  // native distances are taken in FP32 first: the margin covers the rounding of
  // coordinates in structures up to 10 000 nm across
  k.rc2_nat = (float)((params->cv_r_cut + 4e-3) * (params->cv_r_cut + 4e-3));
  const int nb = (n_cv + CV_T - 1) / CV_T;
  // the tile diagonals that hold a pair more than min_sep apart
  k.dmin = k.min_sep < CV_T ? (k.min_sep >= CV_T - 1 ? 1 : 0) : (k.min_sep - CV_T + 1) / CV_T + 1;
  k.m = nb > k.dmin ? nb - k.dmin : 0;
  k.n_tiles = k.m * (k.m + 1) / 2;
  cudaError_t e = cudaMemsetAsync(base, 0, CLEAR_BYTES, st);
  if (e != cudaSuccess) {
    set_msg(errbuf, errlen, cudaGetErrorString(e));
    return SIM_ECUDA;
  }
  k_eval<<<(unsigned)(k.n_tiles > 0 ? k.n_tiles : 1), NW * 32, 0, st>>>(d_pos, d_native, k, sc, d_z, d_grad);
  e = cudaGetLastError();
  if (e != cudaSuccess) {
    set_msg(errbuf, errlen, cudaGetErrorString(e));
    return SIM_ECUDA;
  }
  set_msg(errbuf, errlen, "");
  return SIM_OK;
}
