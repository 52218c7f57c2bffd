// vp_adjoint.cuh -- host interface of the functional-adjoint kernels.
#pragma once
#include <string>

#include "../../include/vpath.h"
#include "vp_cvpair.cuh"

namespace vp {

struct AdjInput {
  const double *frames;  // host [n_frames][3 n_cv]
  int n_frames, n_cv, min_sep, n_tiles;
  const int2 *tiles;     // device: the system's CV tiles
  const float2 *cnat;    // device: the system's C~_nat table (float-float)
  const double *inv_gm;  // device: 1 / (gamma_i m_i) of the system's atoms
  float L, iL;
  double zconst;         // sum of C~_nat^2
  CvConst k;
  double c;              // dt (k_R/2)^2
  int n_sm;              // multiprocessors of the device
  const double *coef;    // host [2 n_frames] (A_n, B_n) or NULL: from the frames (z_m starts at frame 0)
  double *phi, *z_out, *Q_out, *grad;  // host outputs (may be NULL)
};

// Device memory of these calls, kept with the handle between them (a call
// allocated and freed up to 14 arrays before, a third of its time): grown on
// demand, given back after a call that needed more than KEEP bytes and when
// the handle is destroyed.
struct AdjWorkspace {
  static constexpr size_t KEEP = (size_t)256 << 20;
  void *p = nullptr;
  size_t n = 0;
  void *reserve(size_t bytes);  // nullptr when the allocation fails
  void release();
  void trim() { if (n > KEEP) release(); }
};

int adjoint_frames(const AdjInput &in, AdjWorkspace &ws, cudaStream_t st, std::string &err);
int adjoint_coefficients(const double *z, const double *Q, int n, double c, double *coef, double *phi,
                         AdjWorkspace &ws, cudaStream_t st, std::string &err);
// descent on Phi over frames 1 .. n_frames-2 (in.frames is ignored; frames is
// read and overwritten), Armijo backtracking; phi_hist[n_iter + 1]
int refine_frames(const AdjInput &in, double *frames, int n_iter, double step, double *phi_hist, int *n_accepted,
                  AdjWorkspace &ws, cudaStream_t st, std::string &err);

}  // namespace vp
