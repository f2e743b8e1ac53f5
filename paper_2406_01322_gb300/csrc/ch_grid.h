// Host-side state of one channel handle (internal to libchflow).
#pragma once

#include <stdint.h>

#include <vector>

#include "../../include/ch_flow.h"
#include "ch_internal.h"

namespace chf {

const int kMaxSmem = 227 * 1024 - 1024;  // opt-in limit less room for static shared memory

struct Tw {
  void* d64 = nullptr;  // double2[n]
  void* d32 = nullptr;  // float2[n]
  void* ddf = nullptr;  // df2[n] (double-float pairs)
};

// fields through the step: 5 backward (u v w phi Dphi) -> 6 y-padded (phi_y added by the y
// pass) -> 9 products (Sxx-Szz Syy-Szz Sxy Sxz Syz phi^3 u phi v phi w phi)
constexpr int kBw = 5, kYa = 6, kNl = 9;

// backward y-pass map of the step: u v w phi (phi -> i ky phi) Dphi
YMap step_ymap();

// header of a ch_get_state buffer (followed by om, w, phi, h_om, h_w, h_phi)
struct StateHeader {
  uint64_t magic;
  int32_t nx, ny, nz, first;
  int64_t nstep;
  double t;
  int32_t fields_set, pad0;
  uint64_t pad[2];
};
static_assert(sizeof(StateHeader) == 64, "header size");
const uint64_t kStateMagic = 0x3130333234303632ULL;

}  // namespace chf

struct ch_grid {
  ch_params p;
  chf::GridDev g;
  int prec;
  cudaStream_t stream;
  ch_alloc_fn af;
  ch_free_fn ff;
  void* actx;
  std::vector<void*> allocs;

  // state and Adams-Bashforth history, (Mx, Ny, Nz) complex float64
  double2 *om, *w, *phi, *hom, *hw, *hphi;
  // step buffers in working precision
  void *nl, *bw, *ya, *yb;
  // auxiliary float64 buffers for set/get/diagnostics/stage entry points
  double2 *auxA, *auxB;
  double* phys7;
  // right-hand sides / solved sums of the three implicit problems (3 fields), operator table
  double2* R;
  double* fac;
  // small tables and diagnostics scratch
  double* tab;  // go1 go2 go3 ccw dzl qint, nz each
  double2* zcs; // cos(pi j / N), sin(pi j / N), j < N
  double* diag_part;
  double* diag_out;

  chf::FftPlan px[3], py[3], pz, pxu, pyu;  // px, py indexed by precision
  std::vector<chf::Tw> tws;

  long long fs;      // elements per (Mx, Ny, Nz) field
  long long fsy;     // elements per (Mx, Py, Nz) field
  long long fsp;     // elements per physical (Nz, Ny, Nx) field
  int first;         // next step starts Adams-Bashforth
  int fields_set;
  long long nstep;
  double t;
  cudaGraphExec_t gexec;
  int graph_ok;
  cudaStream_t cap;  // private non-blocking stream used only to capture the step graph

  // discrete adjoint: per-line objective partial sums and the reduced value (allocated with the
  // grid), the reverse-sweep workspace (one block, ch_adjoint_begin .. ch_adjoint_end)
  double* obj_part = nullptr;
  void* adj_block = nullptr;
  double2 *a_lam = nullptr, *a_L = nullptr, *a_Rb = nullptr, *a_mu = nullptr, *a_mu2 = nullptr;
  double2 *a_nlb = nullptr, *a_x6 = nullptr, *a_bb = nullptr;
  double* a_phys = nullptr;   // nine real padded fields of the tensor-core x line (use_tx), if obtained
  void* seg_block = nullptr;  // y-padded fields of the states of one recomputed segment
  int seg_cap = 0;            // states that seg_block holds
  int nl_stale = 0;  // 1: the state was replaced by a reverse step; products not recomputed

  // Chebyshev transform of the step: CH_CHEB_FFT (inside zrhs / zbwd) or CH_CHEB_TC (tensor
  // cores, two extra launches); z_auto: the tensor cores although no method was selected.  cf: the
  // coefficients between the transforms and zrhs / zbwd (auxA)
  int cheb = 0, z_auto = 0;
  chf::ChebTc tcf, tcb;
  double2* cf = nullptr;
  int* tc_err = nullptr;

  // tensor-core transforms of the unpadded grid for the entry points that take or give physical
  // fields (use_ax) and of the step's float64 x stage (use_tx) and y stages (tx_y: forward, backward); for
  // the reverse sweep,
  // made when it first begins, tx_yf1: the forward y transform without the 1 / (Px Py), tx_xb1: the
  // transposed forward x transform
  int use_ax = 0, use_tx = 0, tx_y[2] = {0, 0};
  chf::Txy tx;
  chf::TxyPlan tx_yf1, tx_xb1;
};

// the step's z kernels work on Chebyshev coefficients, transformed on the tensor cores
inline bool ch_z_coef(const ch_grid* G) { return G->cheb == CH_CHEB_TC || G->z_auto; }
// stage 3 y backward, 4 x line, 5 y forward of the step runs on the tensor cores
inline bool ch_tx_stage(const ch_grid* G, int stage) {
  return stage == 4 ? G->use_tx != 0 : G->tx_y[stage == 3] != 0;
}
// the same for a member of an ensemble, whose other choice is a grouped launch
bool ch_tx_member(const ch_grid* G, int stage);
// launch schedule of one step on stream s (events optional) and the non-linear evaluation
int ch_launch_step(ch_grid* G, int first, cudaStream_t s, cudaEvent_t* ev);
int ch_eval_nonlinear(ch_grid* G);
// synchronises the stream: CH_ERR_TIMEOUT while the flag of the bounded device waits is set (it stays
// set until ch_device_status), else CH_OK
int ch_sync_status(ch_grid* G);
// ch_set_state; status: answering the flag as ch_sync_status does, with one wait for both
int ch_restore(ch_grid* G, const void* state, bool status);
// bw <- the five backward fields u v w phi D phi of the state, as the step itself forms them
cudaError_t ch_launch_fields(ch_grid* G, cudaStream_t s);
// the x/y stages of the step on stream s: 3 y backward (bw -> ya), 4 x line (ya -> yb), 5 y
// forward with the combinations (yb -> nl)
cudaError_t ch_launch_xy(ch_grid* G, int stage, cudaStream_t s);
// float64 y pass of the reverse sweep (identity field map, scale 1) on the padded grid
cudaError_t ch_launch_y_adj(ch_grid* G, int dir, const double2* in, double2* out, int nf,
                            cudaStream_t s);
// transposed x line of the reverse sweep: ya (y-padded fields of the state), yb (product adjoints,
// overwritten) -> out6
cudaError_t ch_launch_x_adj(ch_grid* G, const double2* ya, double2* out6, cudaStream_t s);
int ch_adjoint_plan(ch_grid* G);
// nf fields of z samples (Mx, Ny, Nz) -> physical rows out[f]; tmp: nf fields
int ch_z_to_rows(ch_grid* G, const double2* in, double2* tmp, int nf, double* const* out);
// u v w phi phi_x phi_y phi_z of the state on the unpadded grid into phys7 ((nz, ny, nx) each)
int ch_state_phys7(ch_grid* G);
// frees the reverse-sweep workspace if allocated
void ch_adjoint_release(ch_grid* G);
