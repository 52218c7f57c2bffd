// vp_adjoint.cu -- gradient of the bias functional with respect to the frames
// of a trial path (the variational condition of Eq. VMDcondition is stated as
// a functional derivative with respect to the path X(tau)).
//
// Along frames X_0 .. X_N (dt apart), with z_n = z(X_n), g_n = grad z(X_n),
// Q_n = sum_i |g_n,i|^2/(gamma_i m_i), m_n = min_{k<=n} z_k (first minimiser)
// and a_n = (z_n - m_{n-1})_+ (Eq. VR):
//   Phi = sum_{n>=1} dt (k_R/2)^2 a_n^2 Q_n
//   dPhi/dX_n = A_n g_n + B_n H_z(X_n) w_n,   w_i = g_i/(gamma_i m_i),
//   A_n = dt (k_R/2)^2 (2 a_n Q_n [n>=1] - R_n),  B_n = 2 dt (k_R/2)^2 a_n^2,
//   R_n = sum over later l whose running minimum sits at frame n of 2 a_l Q_l.
// Kernels: per (frame, 32x32 tile) warp for z and g (float-float pair math as
// in the batched kernel), per frame block for z_n, Q_n and w, one scan for the
// coefficients, per (frame, tile) warp for H_z w (FP32 pair math, int64
// fixed-point accumulation), and a per-atom combination.
#include <cstring>
#include <string>

#include "vp_adjoint.cuh"
#include "vp_cv_dev.cuh"

namespace vp {

struct AdjDev {
  float *frames;        // [nf][3 n_cv]
  int nf, n_cv, min_sep, n_tiles;
  const int2 *tiles;    // the system's tiles
  const float2 *cnat;   // the system's C~_nat in tile-skew order (float-float)
  const double *inv_gm; // 1 / (gamma_i m_i) of the system's atoms
  float L, iL;
  double zconst;
  long long *gx, *gy, *gz;  // [nf][n_cv]
  long long *hx, *hy, *hz;  // [nf][n_cv], after g
  float *w;                 // [nf][3 n_cv]
  double *zpart;            // [nf][n_tiles]
  double *z, *Q;            // [nf]
  double *coef;             // [2 nf]: A_n, B_n
  double *phi;              // [1]
  int *n_near;              // [nf][n_tiles] near pairs of each tile, and the ballots that list them: left by
  unsigned *near;           // [nf][n_tiles][32] k_adj_cv for k_adj_hw (NULL: the lists are formed again)
};

struct AdjFramePos {
  const float *X;
  __device__ __forceinline__ float3 operator()(int a) const { return make_float3(X[3 * a], X[3 * a + 1], X[3 * a + 2]); }
};

__device__ __forceinline__ CvTile adj_tile(const AdjDev &a, const CvConst &k, int f, int t) {
  const int2 bij = a.tiles[t];
  const size_t base = (size_t)f * a.n_cv;
  return CvTile{a.n_cv, bij.x, bij.y, a.min_sep, a.L, a.iL, k.rc2_far, 0.f, a.cnat + (size_t)t * CV_T * CV_T,
                a.gx + base, a.gy + base, a.gz + base, a.zpart + (size_t)f * a.n_tiles + t};
}

// z partial sums and gradients, a warp (NW = 1) or a block of NW warps per
// (frame, tile): the tile routines of the batched kernel, which evaluate the
// near pairs densely and leave a tile of far blocks at once.  One lane per i
// and a loop over j, near or far, took 625 us for 51 frames of 1800 atoms.
//
// Two pairs per lane on the packed FP32 instructions, two warps per block at 64
// registers: bound by issue (64% of the slots) and the FP32 latency of the 10
// warps an SM holds on average, half of all tiles being far and gone at once.
// The distance tests, some 900 instructions per tile, are made once: this pass
// keeps their ballots and H_z w reads them (132 bytes per tile).  51 frames of
// 1800 atoms (84 303 tiles): call 821 -> 689 us, z and grad z 311 -> 277, H_z w
// 340 -> 230 (one pair per lane, four warps per block, tests in both before).
constexpr int ADJ_WARPS = 2;  // tiles per block of the one-warp form
constexpr int adj_threads(int nw) { return 32 * (nw == 1 ? ADJ_WARPS : nw); }
constexpr int adj_blocks(int nw) { return nw == 1 ? 16 : 8; }  // 64 registers
template <int NW, bool KEEP>
__global__ void __launch_bounds__(adj_threads(NW), adj_blocks(NW)) k_adj_cv(AdjDev a, CvConst k) {
  PDL_WAIT();
  if constexpr (NW == 1) {
    __shared__ CvWarpShared sh[ADJ_WARPS];
    const int w = blockIdx.x * ADJ_WARPS + (threadIdx.x >> 5);
    if (w >= a.nf * a.n_tiles) return;
    const int f = w / a.n_tiles, t = w - f * a.n_tiles;
    cv_tile<KEEP>(adj_tile(a, k, f, t), k, sh[threadIdx.x >> 5], AdjFramePos{a.frames + (size_t)f * 3 * a.n_cv},
                  a.n_near + w, a.near + (size_t)w * CV_T);
  } else {
    __shared__ CvBlockShared sh;
    const int w = blockIdx.x, f = w / a.n_tiles, t = w - f * a.n_tiles;
    cv_tile_block<NW, KEEP>(adj_tile(a, k, f, t), k, sh, AdjFramePos{a.frames + (size_t)f * 3 * a.n_cv}, a.n_near + w,
                            a.near + (size_t)w * CV_T);
  }
}

// per frame: z, Q and w = g/(gamma m) (a stored 1/(gamma m): FP64 division is
// slow on this part)
constexpr int FIN_THREADS = 512;
__global__ void __launch_bounds__(FIN_THREADS) k_adj_fin(AdjDev a) {
  PDL_WAIT();
  __shared__ double rz[FIN_THREADS / 32], rq[FIN_THREADS / 32];
  const int f = blockIdx.x;
  double zs = 0.0, q = 0.0;
  for (int t = threadIdx.x; t < a.n_tiles; t += FIN_THREADS) zs += a.zpart[(size_t)f * a.n_tiles + t];
  const double sc = 2.3283064365386963e-10;
  for (int i = threadIdx.x; i < a.n_cv; i += FIN_THREADS) {
    const size_t k = (size_t)f * a.n_cv + i;
    const double gx = (double)a.gx[k] * sc, gy = (double)a.gy[k] * sc, gz = (double)a.gz[k] * sc;
    const double ig = a.inv_gm[i];
    q += (gx * gx + gy * gy + gz * gz) * ig;
    a.w[3 * k] = (float)(gx * ig);
    a.w[3 * k + 1] = (float)(gy * ig);
    a.w[3 * k + 2] = (float)(gz * ig);
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    zs += __shfl_xor_sync(0xffffffffu, zs, off);
    q += __shfl_xor_sync(0xffffffffu, q, off);
  }
  if ((threadIdx.x & 31) == 0) { rz[threadIdx.x >> 5] = zs; rq[threadIdx.x >> 5] = q; }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int k = 1; k < FIN_THREADS / 32; ++k) { zs += rz[k]; q += rq[k]; }
    a.z[f] = a.zconst + zs;
    a.Q[f] = q;
  }
}

// Coefficients A_n, B_n and Phi from z and Q along the path (z_m starts at
// z_0), one block.  Per SCAN frames: one warp forms the running minimum before
// each frame (a scan of 32 at a time) and a = (z - z_m)_+; all threads write
// the coefficients and the terms of the sums; then one warp adds up Phi and a
// thread what the frames pass on to the frame their running minimum sits at
// (those frames are consecutive, so one running sum, put down when the minimum
// moves).  That last sum is the only chain of a dependent operation per frame
// left, on shared memory; one thread doing everything from global memory took
// 294 us for 501 frames.
constexpr int SCAN = 1024;
__global__ void __launch_bounds__(256) k_adj_scan(const double *z, const double *Q, int nf, double c, double *coef,
                                                  double *phi_out) {
  PDL_WAIT();
  __shared__ double s_z[SCAN], s_q[SCAN], s_a[SCAN];
  __shared__ bool s_new[SCAN];
  __shared__ double s_m;
  const double z0 = z[0];
  // a path that starts at NaN never compares below or above its minimum
  const bool dead = isnan(z0);
  double Phi = 0.0, R = 0.0;  // warp 1, thread 64
  int arg = 0;                // thread 64
  if (threadIdx.x == 0) {
    s_m = z0;
    coef[0] = 0.0;
    coef[1] = 0.0;
  }
  __syncthreads();
  for (int f0 = 1; f0 < nf; f0 += SCAN) {
    const int n = min(SCAN, nf - f0);
    for (int k = threadIdx.x; k < n; k += blockDim.x) {
      s_z[k] = z[f0 + k];
      s_q[k] = Q[f0 + k];
    }
    __syncthreads();
    if (threadIdx.x < 32) {
      double m = s_m;
      for (int b = 0; b < n; b += 32) {
        const int k = b + (int)threadIdx.x;
        const double v = k < n && !isnan(s_z[k]) ? s_z[k] : INFINITY;
        double incl = v;  // least of this and the earlier lanes' values
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
          const double o = __shfl_up_sync(0xffffffffu, incl, off);
          if ((int)threadIdx.x >= off && o < incl) incl = o;
        }
        double before = __shfl_up_sync(0xffffffffu, incl, 1);
        before = threadIdx.x == 0 || m < before ? m : before;  // z_m before frame k
        if (k < n) {
          s_a[k] = !dead && s_z[k] > before ? s_z[k] - before : 0.0;
          s_new[k] = !dead && s_z[k] < before;
        }
        const double last = __shfl_sync(0xffffffffu, incl, 31);
        if (last < m) m = last;
      }
      if (threadIdx.x == 0) s_m = m;
    }
    __syncthreads();
    for (int k = threadIdx.x; k < n; k += blockDim.x) {
      const double a = s_a[k], q = s_q[k];
      coef[2 * (f0 + k) + 1] = 2.0 * c * a * a;
      coef[2 * (f0 + k)] = 2.0 * c * a * q;
      s_a[k] = c * a * a * q;               // the frame's share of Phi ...
      s_q[k] = a > 0.0 ? 2.0 * a * q : 0.0;  // ... and what it passes on
    }
    __syncthreads();
    if (threadIdx.x >= 32 && threadIdx.x < 64) {
      for (int k = threadIdx.x - 32; k < n; k += 32) Phi += s_a[k];
    } else if (threadIdx.x == 64) {
      for (int k = 0; k < n; ++k) {
        R += s_q[k];
        if (s_new[k]) {
          coef[2 * arg] = fma(-c, R, coef[2 * arg]);
          arg = f0 + k;
          R = 0.0;
        }
      }
    }
    __syncthreads();  // the shared arrays are taken anew
  }
  if (threadIdx.x == 64) coef[2 * arg] = fma(-c, R, coef[2 * arg]);
  if (threadIdx.x >= 32 && threadIdx.x < 64) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) Phi += __shfl_xor_sync(0xffffffffu, Phi, off);
    if (threadIdx.x == 32 && phi_out) *phi_out = Phi;
  }
}

// shared memory of a tile of H_z w
struct AdjHwShared {
  unsigned short s_near[CV_T * CV_T];
  float4 s_x[2 * CV_T], s_w[2 * CV_T];
  int s_ghi[2 * CV_T][3];
  int s_glo[2 * CV_T][3];
};

// Two near pairs of H_z w (the second only when v1): a pair adds K (w_j - w_i)
// to atom j and subtracts it from atom i, K v = f'' u (u.v) +
// (f'/r)(v - u (u.v)), f = (C~ - C~_nat)^2.
__device__ __forceinline__ void adj_hw_pairs(AdjHwShared &sh, const CvTile &t, const CvConst &k, unsigned e0, unsigned e1,
                                             bool v1) {
  const int il0 = e0 & 31, jc0 = e0 >> 5, il1 = e1 & 31, jc1 = e1 >> 5;
  ff2 dx, dy, dz;
  cv_delta2(sh.s_x[il0], sh.s_x[il1], sh.s_x[CV_T + jc0], sh.s_x[CV_T + jc1], t.L, t.iL, dx, dy, dz);
  const float2 n0 = t.cn[((jc0 - il0) & (CV_T - 1)) * CV_T + il0], n1 = t.cn[((jc1 - il1) & (CV_T - 1)) * CV_T + il1];
  const ff2 r2 = ff2_add(ff2_add(ff2_sqr(dx), ff2_sqr(dy)), ff2_sqr(dz));
  const CvPair2 cp = cv_contact2<true>(r2, k);
  const float2 h = ff2_sub(cp.Ct, ff2{make_float2(n0.x, n1.x), make_float2(n0.y, n1.y)}).hi;
  const float2 f1 = __fmul2_rn(__fadd2_rn(h, h), cp.dCt);
  const float2 fh = __ffma2_rn(cp.dCt, cp.dCt, __fmul2_rn(h, cp.d2Ct)), f2 = __fadd2_rn(fh, fh);
  const float2 ir = f2_rcp(cp.r);
  const float2 ux = __fmul2_rn(dx.hi, ir), uy = __fmul2_rn(dy.hi, ir), uz = __fmul2_rn(dz.hi, ir);
  const float4 wi0 = sh.s_w[il0], wi1 = sh.s_w[il1], wj0 = sh.s_w[CV_T + jc0], wj1 = sh.s_w[CV_T + jc1];
  const float2 vx = f2_sub(make_float2(wj0.x, wj1.x), make_float2(wi0.x, wi1.x)),
               vy = f2_sub(make_float2(wj0.y, wj1.y), make_float2(wi0.y, wi1.y)),
               vz = f2_sub(make_float2(wj0.z, wj1.z), make_float2(wi0.z, wi1.z));
  const float2 uv = __ffma2_rn(uz, vz, __ffma2_rn(ux, vx, __fmul2_rn(uy, vy)));
  const float2 q = __fmul2_rn(f1, ir);
  const float2 g[3] = {__ffma2_rn(q, f2_nma(ux, uv, vx), __fmul2_rn(__fmul2_rn(f2, ux), uv)),
                       __ffma2_rn(q, f2_nma(uy, uv, vy), __fmul2_rn(__fmul2_rn(f2, uy), uv)),
                       __ffma2_rn(q, f2_nma(uz, uv, vz), __fmul2_rn(__fmul2_rn(f2, uz), uv))};
  // r, and with it every component, is not a number where r^2 is below the normal
  // range: atoms that coincide (K = 0, as C' and C'' vanish with r)
  cv_accumulate<true>(sh, t, g, il0, jc0, il1, jc1, true, v1);
}

// H_z w per frame with a bias, a warp (NW = 1) or a block of NW warps per (frame, tile)
template <int NW, bool KEPT>
__global__ void __launch_bounds__(adj_threads(NW), adj_blocks(NW)) k_adj_hw(AdjDev a, CvConst k) {
  PDL_WAIT();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  __shared__ AdjHwShared s_sh[NW == 1 ? ADJ_WARPS : 1];
  __shared__ unsigned s_bal[CV_T];
  const int w = NW == 1 ? blockIdx.x * ADJ_WARPS + warp : blockIdx.x;
  if (w >= a.nf * a.n_tiles) return;
  if (KEPT && a.n_near[w] == 0) return;
  const int f = w / a.n_tiles;
  if (a.coef[2 * f + 1] == 0.0) return;  // no bias at this frame: no Hessian term
  CvTile t = adj_tile(a, k, f, w - f * a.n_tiles);
  const size_t base = (size_t)f * a.n_cv;
  t.gx = a.hx + base; t.gy = a.hy + base; t.gz = a.hz + base;
  const AdjFramePos pos{a.frames + 3 * base}, wof{a.w + 3 * base};
  AdjHwShared &sh = s_sh[NW == 1 ? warp : 0];
  int n_near;
  if constexpr (NW == 1) {
    const int i = t.bi * CV_T + lane, j = t.bj * CV_T + lane;
    const bool iv = i < t.n_cv, jv = j < t.n_cv;
    float3 xi = make_float3(0.f, 0.f, 0.f), xj = xi, wi = xi, wj = xi;
    if (iv) { xi = pos(i); wi = wof(i); }
    if (jv) { xj = pos(j); wj = wof(j); }
    if (!KEPT && cv_tile_far(t, iv, jv, xi, xj)) return;
    sh.s_x[lane] = cv_atom(iv, xi);
    sh.s_x[CV_T + lane] = cv_atom(jv, xj);
    sh.s_w[lane] = make_float4(wi.x, wi.y, wi.z, 0.f);
    sh.s_w[CV_T + lane] = make_float4(wj.x, wj.y, wj.z, 0.f);
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      sh.s_ghi[lane][q] = 0; sh.s_ghi[CV_T + lane][q] = 0;
      sh.s_glo[lane][q] = 0; sh.s_glo[CV_T + lane][q] = 0;
    }
    __syncwarp();
    if (KEPT) n_near = cv_near_list_kept(sh.s_near, a.near + (size_t)w * CV_T);
    else n_near = cv_near_list<false>(t, sh.s_near, sh.s_x, nullptr);
    if (n_near == 0) return;
    __syncwarp();
  } else {
    const bool far = cv_block_begin<NW>(t, sh, pos);
    if (far) return;
    if (threadIdx.x < 2 * CV_T) {
      const int q = (warp == 0 ? t.bi : t.bj) * CV_T + lane;
      const float3 v = q < t.n_cv ? wof(q) : make_float3(0.f, 0.f, 0.f);
      sh.s_w[threadIdx.x] = make_float4(v.x, v.y, v.z, 0.f);
    }
    if (KEPT) {
      if (warp == NW - 1) s_bal[lane] = a.near[(size_t)w * CV_T + lane];
    } else {
      cv_ballots_block<NW>(t, s_bal, sh.s_x);
    }
    __syncthreads();
    n_near = cv_near_list_block<NW>(sh.s_near, s_bal);
  }
  for (int p = (NW == 1 ? 0 : 64 * warp) + lane; p < n_near; p += 64 * NW) {
    const bool two = p + 32 < n_near;
    adj_hw_pairs(sh, t, k, sh.s_near[p], sh.s_near[two ? p + 32 : p], two);
  }
  if constexpr (NW == 1) __syncwarp(); else __syncthreads();
  for (int q = NW == 1 ? lane : (int)threadIdx.x; q < 2 * CV_T; q += NW * 32) {
    const int atom = (q < CV_T ? t.bi : t.bj) * CV_T + (q & (CV_T - 1));
    if (atom < t.n_cv) cv_flush_atom(sh, q, t.gx + atom, t.gy + atom, t.gz + atom);
  }
}

__global__ void k_adj_out(AdjDev a, double *grad) {
  PDL_WAIT();
  const size_t k = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= (size_t)a.nf * a.n_cv) return;
  const int f = (int)(k / a.n_cv);
  const double A = a.coef[2 * f], B = a.coef[2 * f + 1], sc = 2.3283064365386963e-10;
  grad[3 * k] = A * (double)a.gx[k] * sc + B * (double)a.hx[k] * sc;
  grad[3 * k + 1] = A * (double)a.gy[k] * sc + B * (double)a.hy[k] * sc;
  grad[3 * k + 2] = A * (double)a.gz[k] * sc + B * (double)a.hz[k] * sc;
}

// frames in FP32, the precision the functional is evaluated at; the gradient sums cleared
__global__ void k_adj_begin(AdjDev a, const double *x, size_t n) {
  const size_t k = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n) return;
  a.frames[k] = (float)x[k];
  a.gx[k] = 0;  // gx, gy, gz lie one after another: n = 3 nf n_cv entries
}

// y = x - eta g on frames 1 .. nf-2, rounded to FP32 (so that the returned
// path is exactly the one scored); y = x on the end frames, which stay put
__global__ void k_descend(AdjDev a, const double *x, const double *g, double eta, double *y, size_t per_frame, int nf) {
  const size_t k = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= per_frame * (size_t)nf) return;
  const int f = (int)(k / per_frame);
  const double v = (f == 0 || f == nf - 1) ? x[k] : (double)(float)(x[k] - eta * g[k]);
  y[k] = v;
  a.frames[k] = (float)v;
  a.gx[k] = 0;
}

// |g|^2 over frames 1 .. nf-2: fixed-order block sums, then one block
__global__ void k_sq_interior(const double *g, size_t per_frame, int nf, double *part) {
  __shared__ double red[256];
  double acc = 0.0;
  const size_t lo = per_frame, hi = per_frame * (size_t)(nf > 1 ? nf - 1 : 0);
  for (size_t k = lo + (size_t)blockIdx.x * blockDim.x + threadIdx.x; k < hi; k += (size_t)gridDim.x * blockDim.x)
    acc += g[k] * g[k];
  red[threadIdx.x] = acc;
  __syncthreads();
  for (int off = blockDim.x / 2; off > 0; off >>= 1) {
    if (threadIdx.x < off) red[threadIdx.x] += red[threadIdx.x + off];
    __syncthreads();
  }
  if (threadIdx.x == 0) part[blockIdx.x] = red[0];
}

// ---------------------------------------------------------------------------

void AdjWorkspace::release() {
  if (p) cudaFree(p);
  p = nullptr;
  n = 0;
}

void *AdjWorkspace::reserve(size_t bytes) {
  if (bytes > n) {
    release();
    if (cudaMalloc(&p, bytes) != cudaSuccess) {
      p = nullptr;
      return nullptr;
    }
    n = bytes;
  }
  return p;
}

namespace {

// carves the arrays of one call out of the workspace, 256 bytes apart
struct Carve {
  char *base;
  size_t off = 0;
  template <class T>
  T *take(size_t n) {
    T *r = reinterpret_cast<T *>(base + off);
    off += ((n ? n : 1) * sizeof(T) + 255) & ~(size_t)255;
    return r;
  }
};

// Tiles up to which the near pairs are kept between the two passes (132 bytes
// per tile: 66 MB); the block form stays far below.
constexpr size_t KEEP_NEAR = 500000;

// the arrays every evaluation needs (with base = nullptr only their size
// counts); keep: the near pairs' ballots too
AdjDev adj_arrays(const AdjInput &in, Carve &c, bool keep) {
  const size_t na = (size_t)in.n_frames * in.n_cv;
  AdjDev a{};
  a.nf = in.n_frames; a.n_cv = in.n_cv; a.min_sep = in.min_sep; a.n_tiles = in.n_tiles;
  a.tiles = in.tiles; a.cnat = in.cnat; a.inv_gm = in.inv_gm; a.L = in.L; a.iL = in.iL; a.zconst = in.zconst;
  a.frames = c.take<float>(3 * na);
  a.gx = c.take<long long>(3 * na);
  a.gy = a.gx + na; a.gz = a.gy + na;
  a.hx = c.take<long long>(3 * na);
  a.hy = a.hx + na; a.hz = a.hy + na;
  a.w = c.take<float>(3 * na);
  a.zpart = c.take<double>((size_t)in.n_frames * in.n_tiles);
  a.z = c.take<double>(in.n_frames);
  a.Q = c.take<double>(in.n_frames);
  a.coef = c.take<double>(2 * (size_t)in.n_frames);
  a.phi = c.take<double>(1);
  const size_t tiles = (size_t)in.n_frames * in.n_tiles;
  if (keep && tiles <= KEEP_NEAR) {
    a.n_near = c.take<int>(tiles);
    a.near = c.take<unsigned>(tiles * CV_T);
  }
  return a;
}

// A block per tile up to 128 tiles per SM: these kernels run alone, so the
// block form pays longer than beside the pair kernel (see launch_cv).  5576
// tiles: z and grad z 62 -> 50 us, H_z w 56 -> 37; 84 303 tiles: 277 -> 332 and
// 230 -> 261.
bool block_form(const AdjInput &in, const AdjDev &a) {
  return a.near && (long long)in.n_frames * in.n_tiles <= 128ll * in.n_sm;
}

// The arrays of a call and (extra[k] doubles each) others of its own out of the
// workspace, without the ballots when there is no memory for them (the near
// pairs are then listed again).  False: no memory.
template <int N>
bool adj_reserve(const AdjInput &in, AdjWorkspace &ws, AdjDev &a, const size_t (&extra)[N], double *(&out)[N]) {
  for (int keep = 1; keep >= 0; --keep) {
    Carve size{nullptr};
    adj_arrays(in, size, keep);
    for (size_t n : extra) size.take<double>(n);
    Carve c{(char *)ws.reserve(size.off)};
    if (!c.base) {
      cudaGetLastError();
      continue;
    }
    a = adj_arrays(in, c, keep);
    for (int k = 0; k < N; ++k) out[k] = c.take<double>(extra[k]);
    return true;
  }
  return false;
}

// The kernels of a call are dependent launches (each starts with PDL_WAIT): a
// descent of 41 frames, 22 evaluations of five short kernels, 2567 -> 2280 us.
// Letting the successor start early as well (PDL_TRIGGER): 2410, its blocks
// take places from the tile kernels.
void launch_adj_cv(const AdjInput &in, const AdjDev &a, cudaStream_t st) {
  const long long tiles = (long long)a.nf * a.n_tiles;
  const unsigned grid = (unsigned)((tiles + ADJ_WARPS - 1) / ADJ_WARPS);
  if (tiles > 0) {
    if (block_form(in, a)) launch_pdl(k_adj_cv<CV_BLOCK_WARPS, true>, dim3((unsigned)tiles), dim3(32 * CV_BLOCK_WARPS), st, a, in.k);
    else launch_pdl(a.near ? k_adj_cv<1, true> : k_adj_cv<1, false>, dim3(grid), dim3(32 * ADJ_WARPS), st, a, in.k);
  }
  launch_pdl(k_adj_fin, dim3(a.nf), dim3(FIN_THREADS), st, a);
}

void launch_adj_grad(const AdjInput &in, const AdjDev &a, double *grad, cudaStream_t st) {
  const long long tiles = (long long)a.nf * a.n_tiles;
  const size_t na = (size_t)a.nf * a.n_cv;
  if (na == 0) return;
  cudaMemsetAsync(a.hx, 0, sizeof(long long) * 3 * na, st);
  const unsigned grid = (unsigned)((tiles + ADJ_WARPS - 1) / ADJ_WARPS);
  if (tiles > 0) {
    if (block_form(in, a)) launch_pdl(k_adj_hw<CV_BLOCK_WARPS, true>, dim3((unsigned)tiles), dim3(32 * CV_BLOCK_WARPS), st, a, in.k);
    else launch_pdl(a.near ? k_adj_hw<1, true> : k_adj_hw<1, false>, dim3(grid), dim3(32 * ADJ_WARPS), st, a, in.k);
  }
  launch_pdl(k_adj_out, dim3((unsigned)((na + 255) / 256)), dim3(256), st, a, grad);
}

}  // namespace

int adjoint_frames(const AdjInput &in, AdjWorkspace &ws, cudaStream_t st, std::string &err) {
  const int nf = in.n_frames;
  const size_t nx = 3 * (size_t)nf * in.n_cv;
  AdjDev a;
  double *own[1];
  if (!adj_reserve(in, ws, a, {nx}, own)) { err = "cudaMalloc failed"; return SIM_ECUDA; }
  double *dx = own[0], *dgrad = dx;  // the frames are read once, at the start
  cudaError_t e = cudaMemcpyAsync(dx, in.frames, sizeof(double) * nx, cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess && in.coef)
    e = cudaMemcpyAsync(a.coef, in.coef, sizeof(double) * 2 * nf, cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) {
    if (nx > 0) k_adj_begin<<<(unsigned)((nx + 255) / 256), 256, 0, st>>>(a, dx, nx);
    launch_adj_cv(in, a, st);
    if (!in.coef) launch_pdl(k_adj_scan, dim3(1), dim3(256), st, a.z, a.Q, nf, in.c, a.coef, a.phi);
    launch_adj_grad(in, a, dgrad, st);
    e = cudaGetLastError();
  }
  // The copy back is several times slower into memory that no one has touched
  // yet (a fresh array of 2 MB: 1.1 ms a call against 0.35): its pages are
  // touched here, while the kernels run.  Every byte keeps its value: grad may be
  // frames itself, whose copy to the device, from page-locked memory, may not have
  // read it yet.
  if (e == cudaSuccess && in.grad) {
    volatile char *g = reinterpret_cast<volatile char *>(in.grad);
    for (size_t k = 0; k < nx * sizeof(double); k += 4096) g[k] = g[k];
  }
  if (e == cudaSuccess && in.grad) e = cudaMemcpyAsync(in.grad, dgrad, sizeof(double) * nx, cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess && in.z_out) e = cudaMemcpyAsync(in.z_out, a.z, sizeof(double) * nf, cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess && in.Q_out) e = cudaMemcpyAsync(in.Q_out, a.Q, sizeof(double) * nf, cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess && in.phi && !in.coef) e = cudaMemcpyAsync(in.phi, a.phi, sizeof(double), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  ws.trim();
  if (e != cudaSuccess) { err = cudaGetErrorString(e); return SIM_ECUDA; }
  return SIM_OK;
}

// ---------------------------------------------------------------------------
// refinement of a path by descent on the functional (frames as variables)
// ---------------------------------------------------------------------------
int refine_frames(const AdjInput &in, double *frames, int n_iter, double step, double *phi_hist, int *n_accepted,
                  AdjWorkspace &ws, cudaStream_t st, std::string &err) {
  const int nf = in.n_frames, ncv = in.n_cv;
  const size_t nx = 3 * (size_t)nf * ncv;
  constexpr int SQ_BLOCKS = 64;
  AdjDev a;
  double *own[4];
  if (!adj_reserve(in, ws, a, {nx, nx, nx, (size_t)SQ_BLOCKS}, own)) { err = "cudaMalloc failed"; return SIM_ECUDA; }
  double *X = own[0], *Y = own[1], *G = own[2], *part = own[3];
  const unsigned gx_blocks = (unsigned)((nx + 255) / 256);
  // Phi at the frames now in a.frames (their z and grad z stay for grad())
  auto eval = [&](double &phi) -> cudaError_t {
    launch_adj_cv(in, a, st);
    launch_pdl(k_adj_scan, dim3(1), dim3(256), st, a.z, a.Q, nf, in.c, a.coef, a.phi);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaMemcpyAsync(&phi, a.phi, sizeof(double), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    return e;
  };
  // dPhi/dX into G and its square over the free frames, at the frames just evaluated
  auto grad = [&](double &v) -> cudaError_t {
    launch_adj_grad(in, a, G, st);
    k_sq_interior<<<SQ_BLOCKS, 256, 0, st>>>(G, 3 * (size_t)ncv, nf, part);
    double h[SQ_BLOCKS];
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaMemcpyAsync(h, part, sizeof(h), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    v = 0.0;
    for (int b = 0; e == cudaSuccess && b < SQ_BLOCKS; ++b) v += h[b];
    return e;
  };
  cudaError_t e = cudaMemcpyAsync(X, frames, sizeof(double) * nx, cudaMemcpyHostToDevice, st);
  double phi = 0.0, gg = 0.0;
  if (e == cudaSuccess && nx > 0) k_adj_begin<<<gx_blocks, 256, 0, st>>>(a, X, nx);
  if (e == cudaSuccess) e = eval(phi);
  if (e == cudaSuccess) e = grad(gg);
  if (phi_hist) phi_hist[0] = phi;
  int accepted = 0;
  double eta = step;
  for (int it = 0; it < n_iter && e == cudaSuccess; ++it) {
    bool ok = false;
    // backtracking (Armijo): accept the first step that lowers Phi by at least 1e-4 eta |g|^2
    for (int bt = 0; bt < 40 && e == cudaSuccess && gg > 0.0; ++bt) {
      k_descend<<<gx_blocks, 256, 0, st>>>(a, X, G, eta, Y, 3 * (size_t)ncv, nf);
      double phi_y = 0.0;
      e = eval(phi_y);
      if (e != cudaSuccess) break;
      if (phi_y <= phi - 1e-4 * eta * gg) {
        std::swap(X, Y);
        phi = phi_y;
        ok = true;
        break;
      }
      eta *= 0.5;
    }
    if (e == cudaSuccess && ok) {
      // the accepted path is the one evaluated last: its z, grad z and
      // coefficients are in place
      e = grad(gg);
      ++accepted;
      eta *= 2.0;
    }
    if (phi_hist) phi_hist[it + 1] = phi;
    if (!ok) {  // no step lowers Phi any more: keep the value for the remaining entries
      for (int k = it + 2; phi_hist && k <= n_iter; ++k) phi_hist[k] = phi;
      break;
    }
  }
  if (e == cudaSuccess) e = cudaMemcpyAsync(frames, X, sizeof(double) * nx, cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  ws.trim();
  if (n_accepted) *n_accepted = accepted;
  if (e != cudaSuccess) { err = cudaGetErrorString(e); return SIM_ECUDA; }
  return SIM_OK;
}

int adjoint_coefficients(const double *z, const double *Q, int n, double c, double *coef, double *phi,
                         AdjWorkspace &ws, cudaStream_t st, std::string &err) {
  Carve size{nullptr};
  for (int k = 0; k < 4; ++k) size.take<double>(n);
  size.take<double>(1);
  Carve a{(char *)ws.reserve(size.off)};
  if (!a.base) { err = "cudaMalloc failed"; return SIM_ECUDA; }
  double *dz = a.take<double>(n), *dq = a.take<double>(n), *dp = a.take<double>(1), *dc = a.take<double>(2 * (size_t)n);
  cudaError_t e = cudaMemcpyAsync(dz, z, sizeof(double) * n, cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) e = cudaMemcpyAsync(dq, Q, sizeof(double) * n, cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) {
    launch_pdl(k_adj_scan, dim3(1), dim3(256), st, dz, dq, n, c, dc, dp);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaMemcpyAsync(coef, dc, sizeof(double) * 2 * n, cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess && phi) e = cudaMemcpyAsync(phi, dp, sizeof(double), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  ws.trim();
  if (e != cudaSuccess) { err = cudaGetErrorString(e); return SIM_ECUDA; }
  return SIM_OK;
}

}  // namespace vp
