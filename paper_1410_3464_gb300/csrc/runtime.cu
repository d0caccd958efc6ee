// Host runtime behind the C ABI of include/pslbm.h: parameter validation,
// device allocation of the state, node lists and the layout of the work, CUDA-graph
// capture of whole steps, field read-out and batches.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <map>
#include <memory>
#include <mutex>
#include <new>
#include <string>
#include <vector>

#include "../../include/pslbm.h"
#include "launch.h"
#include "step.cuh"

using namespace pslbm;

namespace {

std::mutex g_mu;
cudaStream_t g_own_stream = nullptr;
cudaStream_t g_user_stream = nullptr;
bool g_user_set = false;
std::string g_lib_err;

cudaStream_t lib_stream() {
  if (g_user_set) return g_user_stream;
  if (!g_own_stream) cudaStreamCreateWithFlags(&g_own_stream, cudaStreamNonBlocking);
  return g_own_stream;
}

size_t fsize(int prec) { return prec == PSLBM_FP64 ? 8 : 4; }
size_t gsize(int prec) { return prec == PSLBM_FP64 ? 8 : (prec == PSLBM_FP32 ? 4 : 2); }

struct GraphCache {
  std::map<int64_t, cudaGraphExec_t> exec;
  void clear() {
    for (auto& kv : exec) cudaGraphExecDestroy(kv.second);
    exec.clear();
  }
};

constexpr int NSTAGING = 3;

// Fields of at most this many bytes together are read by way of the handle's own buffer
// (pslbm_read_fields).
constexpr size_t STAGE_BYTES = 1 << 20;

// Launch state shared by a single simulation and a batch: the work list of the
// streaming kernels, the caller's tile shape and staging, and the captured
// graphs.
struct Stepper {
  const Launchers* L = nullptr;
  DevInst* d = nullptr;
  int ninst = 0;
  std::vector<std::pair<int, int>> dims;   // (nx, ny) per instance
  std::vector<const DevInst*> inst;        // host descriptors
  std::vector<int> nfluid, nface, nres;    // listed nodes and reservoirs per instance, as last seen
  long long plan_fluid = 0, plan_face = 0; // their sums when the work was laid out
  bool plan_fused = false;                 // VOP and amendment in one launch
  int64_t since = 0;                       // steps since the lists were made
  DevInst host0{};                         // host descriptor of the first instance
  int mode = M_SINGLE;
  bool fp64 = false;
  Work* work = nullptr;                    // a batch's work entries: streaming kernels, then VOP kernel
  int nwork = 0, nstream = 0, nvop = 0;    // their numbers (nwork 0: not made yet)
  int npot = 0;                            // warps of k_pot in the place of nstream (one simulation)
  int fix_shape = -1;                      // caller's choices, -1: none
  int fix_staged = -1;
  bool staged_ok = false;                  // the caller may ask for staging 1 or 2
  GraphCache graphs;
  void drop_work() {
    graphs.clear();
    if (work) cudaFree(work);
    work = nullptr;
    nwork = 0;
  }
  void release() { drop_work(); }
};

}  // namespace

struct pslbm_s {
  pslbm_params p{};
  int prec = 0;
  int ns = 0;
  long long N = 0;
  DevInst h{};                 // host copy of the device descriptor
  DevInst* d = nullptr;        // device descriptor
  Stepper run;
  std::vector<void*> allocs;
  uint64_t bytes = 0;
  double* rb = nullptr;        // read-back scratch
  size_t rb_bytes = 0;
  std::unique_ptr<char[]> stage;   // host side of a small read-back (STAGE_BYTES at most)
  std::string err;
  pslbm_status sticky = PSLBM_OK;
  int in_batch = 0;
  const Launchers* L = nullptr;
};

struct pslbm_batch_s {
  std::vector<pslbm_t> members;
  DevInst* d = nullptr;
  Stepper run;
  const Launchers* L = nullptr;
  std::string err;
  pslbm_status sticky = PSLBM_OK;
  unsigned long long* mon = nullptr;       // device: (step, status) per member, for pslbm_batch_monitor
  std::vector<unsigned long long> mon_h;
};

namespace {

pslbm_status fail(pslbm_t h, pslbm_status s, const std::string& msg) {
  if (h) {
    h->err = msg;
    if (s == PSLBM_ERR_CUDA || s == PSLBM_ERR_NONFINITE || s == PSLBM_ERR_EOS_DOMAIN)
      h->sticky = s;
  } else {
    std::lock_guard<std::mutex> lk(g_mu);
    g_lib_err = msg;
  }
  return s;
}

#define CK(h, call)                                                                                   \
  do {                                                                                                \
    cudaError_t e_ = (call);                                                                          \
    if (e_ != cudaSuccess) return fail(h, PSLBM_ERR_CUDA, std::string(#call) + ": " + cudaGetErrorString(e_)); \
  } while (0)

pslbm_status check_device() {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return PSLBM_ERR_NODEVICE;
  cudaDeviceProp prop;
  if (cudaGetDeviceProperties(&prop, dev) != cudaSuccess) return PSLBM_ERR_NODEVICE;
  if (!(prop.major == 10 && prop.minor == 3)) return PSLBM_ERR_NODEVICE;
  return PSLBM_OK;
}

std::string validate(const pslbm_params* p) {
  char buf[256];
  if (!p) return "params is NULL";
  if (p->struct_size != sizeof(pslbm_params)) {
    snprintf(buf, sizeof buf, "struct_size %u != %zu", p->struct_size, sizeof(pslbm_params));
    return buf;
  }
  if (p->nx < 1 || p->ny < 1 || (long long)p->nx * p->ny > 100000000LL)
    return "lattice size must be 1..100,000,000 nodes";
  if (p->precision < 0 || p->precision > 3) return "bad precision";
  for (int s = 0; s < 2; ++s)
    if (!(p->tau[s] > 0.5) || !std::isfinite(p->tau[s])) return "tau must be > 0.5";
  if (p->n_species < 0 || p->n_species > PSLBM_MAX_SPECIES) return "n_species out of range";
  if (p->precision >= 2 && p->n_species == 0) return "16-bit solute storage needs species";
  const int ns = p->n_species;
  auto okidx = [&](int i, bool allow_derived) {
    return i == PSLBM_IDX_ABSENT || (i >= 0 && i < ns) || (allow_derived && i == PSLBM_IDX_DERIVED);
  };
  if (!okidx(p->idx_A, true) || !okidx(p->idx_B, false) || !okidx(p->idx_E, false) || !okidx(p->idx_F, false))
    return "species index out of range";
  {
    int ids[4] = {p->idx_A, p->idx_B, p->idx_E, p->idx_F};
    for (int i = 0; i < 4; ++i)
      for (int j = i + 1; j < 4; ++j)
        if (ids[i] >= 0 && ids[i] == ids[j]) return "two roles share one species index";
  }
  for (int k = 0; k < ns; ++k) {
    if (!(p->J0[k] >= 0.0 && p->J0[k] < 1.0)) return "J0 must be in [0, 1)";
    if (!(p->tau_g[k] > 0.5)) return "tau_g must be > 0.5";
  }
  if (p->G11 != 0.0 && !(p->eos_b > 0 && p->eos_R > 0 && p->eos_T > 0)) return "bad EOS constants";
  if (!(p->rho10 != 0.0 && p->rho20 != 0.0)) return "rho10, rho20 must be nonzero";
  // reactive link rule needs kappa = k / (2 J_w) < 1
  if (p->idx_B >= 0 && p->k2 != 0.0 && !(p->k2 >= 0.0 && p->k2 < 0.5 * (1.0 - p->J0[p->idx_B])))
    return "k2 must be in [0, (1 - J0_B)/2)";
  if (p->idx_F >= 0 && p->k4 != 0.0 && !(p->k4 >= 0.0 && p->k4 < 0.5 * (1.0 - p->J0[p->idx_F])))
    return "k4 must be in [0, (1 - J0_F)/2)";
  if (!(p->V_split > 1.0)) return "V_split must be > 1";
  if (!(p->r1_surface_factor >= 0.0) || !std::isfinite(p->r1_surface_factor)) return "r1_surface_factor must be >= 0";
  for (int k = 0; k < PSLBM_MAX_SPECIES; ++k)
    if (!(p->conc_scale[k] >= 0.0) || !std::isfinite(p->conc_scale[k])) return "conc_scale must be >= 0 and finite";
  if (p->inlet_axis < 0 || p->inlet_axis > 1 || p->outlet_axis < 0 || p->outlet_axis > 1) return "axes must be 0 or 1";
  if (p->inlet_period_liq < 0 || p->inlet_period_gas < 0 ||
      (p->inlet_period_gas > 0 && p->inlet_period_liq + p->inlet_period_gas <= 0))
    return "bad inlet periods";
  if (p->inlet_ramp < 0 || (p->inlet_period_gas > 0 &&
                            (p->inlet_ramp > p->inlet_period_liq || p->inlet_ramp > p->inlet_period_gas)))
    return "inlet_ramp must be in [0, min(inlet periods)]";
  return "";
}

template <class R>
void fill_r(DevParamsR<R>& q, const DevParams& P) {
  for (int s = 0; s < 2; ++s) {
    q.tau[s] = R(P.tau[s]);
    q.inv_tau[s] = R(P.inv_tau[s]);
    q.w_adh[s] = R(P.w_adh[s]);
    q.shift_f[s] = R(P.shift_f[s]);
    q.shift_fg[s] = R(P.shift_fg[s]);
    q.rho_fill[s] = R(P.rho_fill[s]);
  }
  q.G11 = R(P.G11);
  q.G12 = R(P.G12);
  q.G21 = R(P.G21);
  q.a0 = R(P.a0);
  q.inv_rho10 = R(1.0 / P.rho10);
  q.inv_rho20 = R(1.0 / P.rho20);
  q.eos_a = R(P.eos_a);
  q.eos_b4 = R(P.eos_b / 4.0);
  q.eos_RT = R(P.eos_R * P.eos_T);
  q.six_over_G11 = R(P.G11 != 0.0 ? 6.0 / P.G11 : 0.0);
  q.gx = R(P.gx);
  q.gy = R(P.gy);
  for (int k = 0; k < MAXS; ++k) {
    q.J0[k] = R(P.J0[k]);
    q.Ja[k] = R(P.Ja[k]);
    q.inv_tau_g[k] = R(P.inv_tau_g[k]);
    q.shift_c[k] = R(P.shift_c[k]);
    q.conc_in[k] = R(P.conc_in[k]);
    q.cR1[k] = R(P.cR1[k]);
    q.cR3[k] = R(P.cR3[k]);
    q.gs_mul[k] = R(P.gs_scale[k]);
    q.gs_div[k] = R(1.0 / P.gs_scale[k]);
  }
  q.k1 = R(P.k1);
  q.k1_inv_Keq = R(P.k1 * P.inv_Keq);
  q.k1_s = R(P.k1 * P.r1_surface_factor);
  q.k1_inv_Keq_s = R(P.k1 * P.r1_surface_factor * P.inv_Keq);
  q.k3 = R(P.k3);
  q.k2 = R(P.k2);
  q.k4 = R(P.k4);
  q.C_F_sat = R(P.C_F_sat);
  q.gas_yield = R(P.gas_yield);
  q.inv_M_C = R(P.inv_M_C);
  q.c_total_per_rho1 = R(P.c_total_per_rho1);
  // link rule with kappa = k / (2 J_w), J_w = J_a: back = (out (1 - kappa) + k C_sat) / (1 + kappa),
  // flux q = out - back = out 2 kappa / (1 + kappa) - k C_sat / (1 + kappa) (no cancellation)
  q.vB_qa = q.vB_sh = q.vF_qa = q.vF_qc = q.vF_sh = R(0);
  if (P.iB >= 0) {
    const double kap = P.k2 / (2.0 * P.Ja[P.iB]);
    q.vB_qa = R(2.0 * kap / (1.0 + kap));
    q.vB_sh = R(P.Ja[P.iB] * P.shift_c[P.iB]);
  }
  if (P.iF >= 0) {
    const double kap = P.k4 / (2.0 * P.Ja[P.iF]);
    q.vF_qa = R(2.0 * kap / (1.0 + kap));
    q.vF_qc = R(P.k4 * P.C_F_sat / (1.0 + kap));
    q.vF_sh = R(P.Ja[P.iF] * P.shift_c[P.iF]);
  }
}

// Whether two parameter blocks agree in everything the streaming kernels read
// through Q (all but the sizes, the rates, the reservoirs and the VOP constants).
bool same_hot_params(const DevParams& a, const DevParams& b) {
  DevParams x, y;
  std::memcpy(&x, &a, sizeof x);
  std::memcpy(&y, &b, sizeof y);
  for (DevParams* p : {&x, &y}) {
    p->nx = p->ny = p->px = p->py = p->row_shift = 0;
    p->row_mul = 0;
    p->per_liq = p->per_gas = p->ramp = p->useB = p->useF = 0;
    p->in_dx = p->in_dy = p->out_dx = p->out_dy = 0;
    p->k1 = p->k2 = p->k3 = p->k4 = p->inv_Keq = p->C_F_sat = p->r1_surface_factor = 0.0;
    p->Vbar_D = p->Vbar_F = p->V_split = 0.0;
    p->seed = 0;
    for (int s = 0; s < 2; ++s) p->rho_in_liq[s] = p->rho_in_gas[s] = p->rho_out[s] = p->rho_out_gas[s] = 0.0;
    for (int k = 0; k < MAXS; ++k) p->conc_in[k] = 0.0;
    auto clear = [](auto& q) {
      q.k1 = q.k1_s = q.k1_inv_Keq = q.k1_inv_Keq_s = q.k2 = q.k3 = q.k4 = q.C_F_sat = 0;
      q.vB_qa = q.vB_sh = q.vF_qa = q.vF_qc = q.vF_sh = 0;
      for (int k = 0; k < MAXS; ++k) q.conc_in[k] = 0;
    };
    clear(p->rf);
    clear(p->rd);
  }
  return std::memcmp(&x, &y, sizeof x) == 0;
}

DevParams to_dev(const pslbm_params* p) {
  DevParams P{};
  P.nx = p->nx;
  P.ny = p->ny;
  P.px = p->periodic_x ? 1 : 0;
  P.py = p->periodic_y ? 1 : 0;
  // node / nx for 0 <= node < 2^31 as a product and a shift: with l = ceil(log2 nx)
  // and m = ceil(2^(31+l) / nx), m nx exceeds 2^(31+l) by less than 2^l, so the
  // quotient's error stays below 1 / nx; m fits 32 bits
  {
    int l = 0;
    while ((1LL << l) < p->nx) ++l;
    P.row_shift = 31 + l;
    P.row_mul = (unsigned)(((1ULL << (31 + l)) + (unsigned)p->nx - 1) / (unsigned)p->nx);
  }
  P.ns = p->n_species;
  P.iA = p->idx_A;
  P.iB = p->idx_B;
  P.iE = p->idx_E;
  P.iF = p->idx_F;
  P.in_dx = p->inlet_axis == 1 ? 0 : 1;
  P.in_dy = p->inlet_axis == 1 ? 1 : 0;
  P.out_dx = p->outlet_axis == 1 ? 0 : -1;
  P.out_dy = p->outlet_axis == 1 ? -1 : 0;
  P.per_liq = p->inlet_period_liq;
  P.per_gas = p->inlet_period_gas;
  P.ramp = p->inlet_ramp;
  for (int s = 0; s < 2; ++s) {
    P.tau[s] = p->tau[s];
    P.w_adh[s] = p->w_adh[s];
    P.shift_f[s] = p->precision == PSLBM_FP64 ? 0.0 : p->rho_ref[s];
    P.shift_fg[s] = p->precision == PSLBM_FP64 ? 0.0 : p->rho_ref_gas[s];
    P.rho_fill[s] = p->rho_ref[s];
    P.rho_in_liq[s] = p->rho_in_liq[s];
    P.rho_in_gas[s] = p->rho_in_gas[s];
    P.rho_out[s] = p->rho_out[s];
    P.rho_out_gas[s] = p->rho_out_gas[s];
  }
  P.G11 = p->G11;
  P.G12 = p->G12;
  P.G21 = p->G21;
  P.a0 = p->a0;
  P.rho10 = p->rho10;
  P.rho20 = p->rho20;
  P.eos_a = p->eos_a;
  P.eos_b = p->eos_b;
  P.eos_R = p->eos_R;
  P.eos_T = p->eos_T;
  P.gx = p->body_force[0];
  P.gy = p->body_force[1];
  for (int k = 0; k < MAXS; ++k) {
    P.J0[k] = p->J0[k];
    P.tau_g[k] = k < p->n_species ? p->tau_g[k] : 1.0;
    P.shift_c[k] = p->precision == PSLBM_FP64 ? 0.0 : p->conc_ref[k];
    P.conc_in[k] = p->conc_in[k];
    // nearest power of two of conc_scale (0: 1), for 16-bit storage only
    double sc = 1.0;
    if (p->precision >= PSLBM_FP32_SOLUTE_F16 && p->conc_scale[k] > 0.0) {
      int e = (int)std::lround(std::log2(p->conc_scale[k]));
      e = std::max(-60, std::min(60, e));
      sc = std::ldexp(1.0, e);
    }
    P.gs_scale[k] = sc;
  }
  for (int s = 0; s < 2; ++s) P.inv_tau[s] = 1.0 / p->tau[s];
  for (int k = 0; k < MAXS; ++k) {
    P.Ja[k] = (1.0 - p->J0[k]) / 4.0;
    P.inv_tau_g[k] = 1.0 / P.tau_g[k];
    P.cR1[k] = (k == p->idx_A ? -1.0 : 0.0) + (k == p->idx_B ? 1.0 : 0.0);
    P.cR3[k] = (k == p->idx_B ? -1.0 : 0.0) + (k == p->idx_E ? -1.0 : 0.0) + (k == p->idx_F ? 1.0 : 0.0);
  }
  P.k1 = p->k1;
  P.r1_surface_factor = p->r1_surface_factor > 0.0 ? p->r1_surface_factor : 1.0;
  P.r1_surf = P.r1_surface_factor != 1.0;
  P.inv_Keq = p->inv_Keq;
  P.k3 = p->k3;
  P.k2 = p->k2;
  P.k4 = p->k4;
  P.C_F_sat = p->C_F_sat;
  P.gas_yield = p->gas_yield;
  P.inv_M_C = p->inv_M_C;
  P.c_total_per_rho1 = p->c_total_per_rho1;
  P.Vbar_D = p->Vbar_D;
  P.Vbar_F = p->Vbar_F;
  P.V_split = p->V_split;
  P.seed = p->seed;
  P.has_g = p->body_force[0] != 0.0 || p->body_force[1] != 0.0;
  // exp(-z) < 2^-55 |a0| for z > ln(2^55 / |a0|); one step up in the high word
  // covers its low bits
  P.phi2_cut = 0x7FFFFFFF;
  if (std::isfinite(p->a0) && std::fabs(p->a0) > 1e-290) {
    const double cut = std::max(1.0, std::log(std::ldexp(1.0, 55) / std::fabs(p->a0)));
    int64_t bits;
    std::memcpy(&bits, &cut, sizeof bits);
    P.phi2_cut = (int)(bits >> 32) + 1;
  }
  P.has_w = p->w_adh[0] != 0.0 || p->w_adh[1] != 0.0;
  P.tau_unit = p->tau[0] == 1.0 && p->tau[1] == 1.0;
  P.has_G11 = p->G11 != 0.0;
  P.has_rev = p->inv_Keq != 0.0;
  P.useB = p->idx_B >= 0 && p->k2 != 0.0;
  P.useF = p->idx_F >= 0 && p->k4 != 0.0;
  fill_r(P.rf, P);
  fill_r(P.rd, P);
  return P;
}

// Whether k_move reads populations of this many bytes (both buffers) with an L2
// policy that lets them go first.  They are read for the last time, and while not
// much more than the 129 MB L2 is in use that keeps what the step and the next one
// still want: FP32, per step, 700x700 (129 MB) 45.9 -> 40.5 us, 1024x512 (138 MB)
// 48.6 -> 42.3, 1200x600 (190 MB) 64.4 -> 60.4.  Above, lines go before the chunks
// that share them have read them: 1448x724 (277 MB) 88.1 -> 93.6, 4096x2048 622 ->
// 698.  FP64 does not care.
bool read_once(size_t bytes) { return bytes <= 220000000; }

// Warps for a list of n entries now (of at most N), each taking 32 entries at a
// time in `turns` turns.  Lists grow as nodes dissolve: with one turn a few warps
// more than needed, so that growth does not give some a second one.
int list_warps(long long n, long long N, double turns) {
  const long long room = turns > 1.0 ? n : std::min(N, n + std::max(2048LL, n / 8));
  return (int)std::max(1.0, std::ceil(double(room) / (32.0 * turns)));
}

// Turns a warp of the streaming kernels takes.  Several, because each saves a
// start (descriptor, step count, list) and has the next turn's list entry in
// flight.  One simulation: one wave of 8 warps an SM (FP64: 16), whose warps sweep the
// list together, so that what neighbours share is met in L2: 1024x512 FP32 48.7 us a
// step, against 56.7 with 16 warps, 54.4 with 8 turns in two waves and 66 with one turn
// (before the evict-first loads).  k_pot, with a third of the loads in flight, takes 16
// in either type (8: 2048x1024 177 us, 16: 161).  Long lists: FP32 8 turns from 80 a
// warp on (one wave and 8 turns: 2048x1024 165 and 179 us, 2896x1448, 65 a warp, 314 and
// 324, 3072x2048, 97 a warp, 477 and 474, 8192x4096 2524 and 2456); FP64 2 turns from 5
// a warp on (768x512 208 and 211, 1024x512, 4.1 a warp, 264 and 265, 1200x600, 5.6 a
// warp, 342 and 336, 2048x1024 913 and 891, 4096x2048 3510 and 3426).  A batch, whose
// members' lists do not join up: 8 turns (FP64 2), fewer where that leaves SMs idle (24
// members 384 us, one wave 405 to 450, one turn 428).
double stream_turns(const Stepper& st, bool pot) {
  if (st.fix_shape >= 0) return SHAPE_TX[st.fix_shape] * SHAPE_TY[st.fix_shape] / 64;
  double chunks = 0;
  for (int f : st.nfluid) chunks += (f + 31) / 32;
  const double sms = device_sms();
  const double wave = sms * (st.fp64 || (pot && st.mode == M_SINGLE) ? 16 : 8);
  if (st.mode == M_SINGLE && chunks <= sms * (st.fp64 ? 5 * 16 : 80 * 8)) return std::max(1.0, chunks / wave);
  double turns = st.fp64 ? 2 : 8;
  while (turns > 1 && chunks / turns < wave) turns /= 2;
  return turns;
}

// Whether every list of minerals is short enough for one launch of VOP and amendment
// with a block an instance (k_vop_amend); a plan that has it keeps it for half as much
// more, or a list around the line would have its plan changed over and over.
bool fused(const Stepper& st) {
  return *std::max_element(st.nface.begin(), st.nface.end()) <= (st.plan_fused ? FUSE_FACE + FUSE_FACE / 2 : FUSE_FACE);
}

// Whether the lists, as last seen, ask for another plan than the one there is: an eighth
// longer (list_warps leaves that much room), half as long, or across the line of `fused`.
bool outgrown(const Stepper& st) {
  auto sum = [](const std::vector<int>& v) {
    long long n = 0;
    for (int k : v) n += k;
    return n;
  };
  auto off = [](long long n, long long plan) { return n > plan + std::max(2048LL, plan / 8) || n < plan / 2; };
  return off(sum(st.nfluid), st.plan_fluid) || off(sum(st.nface), st.plan_face) || fused(st) != st.plan_fused;
}

// Work entries of the streaming kernels (parts of the fluid lists, then chunks of
// 32 reservoir nodes) and of the VOP kernel.  A plan that the lists have outgrown is
// made again; without memory for it the one there is goes on.
cudaError_t ensure_work(Stepper& st) {
  if (st.nwork && !outgrown(st)) return cudaSuccess;
  st.plan_fluid = st.plan_face = 0;
  for (int k : st.nfluid) st.plan_fluid += k;
  for (int k : st.nface) st.plan_face += k;
  st.plan_fused = fused(st);
  auto nodes = [&](int i) { return (long long)st.dims[i].first * st.dims[i].second; };
  if (st.mode == M_SINGLE) {
    st.graphs.clear();
    st.npot = list_warps(st.nfluid[0], nodes(0), stream_turns(st, true));
    st.nstream = list_warps(st.nfluid[0], nodes(0), stream_turns(st, false));
    st.nwork = st.nstream + (st.nres[0] + 31) / 32;
    st.nvop = list_warps(st.nface[0], nodes(0), 1);
    return cudaSuccess;
  }
  const double turns = stream_turns(st, false);
  std::vector<Work> all;
  for (int i = 0; i < (int)st.dims.size(); ++i) {
    const int nw = list_warps(st.nfluid[i], nodes(i), turns);
    for (int c = 0; c < nw; ++c) all.push_back(Work{i, c * 32, nw * 32, -1});
    for (int k = 0; k < st.nres[i]; k += 32) all.push_back(Work{i, 0, 0, k});
  }
  const int nwork = (int)all.size();
  for (int i = 0; i < (int)st.dims.size(); ++i) {
    const int nw = list_warps(st.nface[i], nodes(i), 1);
    for (int c = 0; c < nw; ++c) all.push_back(Work{i, c * 32, nw * 32, -1});
  }
  Work* d = nullptr;
  cudaError_t e = cudaMalloc(&d, all.size() * sizeof(Work));
  if (e == cudaErrorMemoryAllocation && st.nwork) {
    cudaGetLastError();
    return cudaSuccess;
  }
  if (e != cudaSuccess) return e;
  e = cudaMemcpyAsync(d, all.data(), all.size() * sizeof(Work), cudaMemcpyHostToDevice, lib_stream());
  if (e == cudaSuccess) e = cudaStreamSynchronize(lib_stream());
  if (e != cudaSuccess) {
    cudaFree(d);
    return e;
  }
  st.drop_work();
  st.work = d;
  st.nwork = nwork;
  st.nvop = (int)all.size() - nwork;
  return cudaSuccess;
}

pslbm_status dalloc(pslbm_t h, void** ptr, size_t bytes) {
  *ptr = nullptr;
  if (bytes == 0) bytes = 16;
  cudaError_t e = cudaMalloc(ptr, bytes);
  if (e != cudaSuccess) {
    cudaGetLastError();
    *ptr = nullptr;
    return fail(h, e == cudaErrorMemoryAllocation ? PSLBM_ERR_OOM : PSLBM_ERR_CUDA,
                std::string("cudaMalloc: ") + cudaGetErrorString(e));
  }
  h->allocs.push_back(*ptr);
  h->bytes += bytes;
  return PSLBM_OK;
}

void free_all(pslbm_t h) {
  h->run.release();
  for (void* p : h->allocs) cudaFree(p);
  h->allocs.clear();
}

// Enqueue the streaming kernels of one step.
void enqueue_stream(cudaStream_t s, const Stepper& st) {
  const int more = st.mode == M_SINGLE ? st.npot - st.nstream : 0;
  st.L->pot(s, st.work, st.nwork + more, st.nstream + more, st.d, st.host0, st.mode);
  st.L->move(s, st.work, st.nwork, st.nstream, st.d, st.host0, st.mode);
}

// Enqueue the kernels of n steps.
void enqueue_steps(cudaStream_t s, const Stepper& st, int64_t n) {
  for (int64_t i = 0; i < n; ++i) {
    enqueue_stream(s, st);
    if (st.plan_fused) {
      st.L->vop_amend(s, st.ninst, st.d);
      continue;
    }
    st.L->vop(s, st.d, st.work ? st.work + st.nwork : nullptr, st.nvop);
    st.L->amend(s, st.ninst, st.d);
  }
}

// n steps without graph capture, each kernel bracketed by CUDA events on the
// library stream: mean ms per step of the streaming, VOP and amendment kernels and
// of the whole step.
pslbm_status profile_steps(Stepper& st, int64_t n, double* kernel_ms, double* total_ms, std::string& err) {
  cudaStream_t s = lib_stream();
  cudaError_t te = ensure_work(st);
  if (te != cudaSuccess) {
    err = std::string("work list: ") + cudaGetErrorString(te);
    return PSLBM_ERR_CUDA;
  }
  cudaEvent_t ev[4] = {};
  for (int i = 0; i < 4; ++i)
    if (cudaEventCreate(&ev[i]) != cudaSuccess) {
      for (int k = 0; k < i; ++k) cudaEventDestroy(ev[k]);
      err = "cudaEventCreate failed";
      return PSLBM_ERR_CUDA;
    }
  double acc[3] = {0, 0, 0}, tot = 0;
  pslbm_status st_ = PSLBM_OK;
  for (int64_t i = 0; i < n; ++i) {
    cudaEventRecord(ev[0], s);
    enqueue_stream(s, st);
    cudaEventRecord(ev[1], s);
    st.L->vop(s, st.d, st.work ? st.work + st.nwork : nullptr, st.nvop);
    cudaEventRecord(ev[2], s);
    st.L->amend(s, st.ninst, st.d);
    cudaEventRecord(ev[3], s);
    cudaError_t e = cudaEventSynchronize(ev[3]);
    if (e != cudaSuccess) {
      err = std::string("profile step: ") + cudaGetErrorString(e);
      st_ = PSLBM_ERR_CUDA;
      break;
    }
    float ms;
    for (int k = 0; k < 3; ++k) {
      cudaEventElapsedTime(&ms, ev[k], ev[k + 1]);
      acc[k] += ms;
    }
    cudaEventElapsedTime(&ms, ev[0], ev[3]);
    tot += ms;
  }
  for (int i = 0; i < 4; ++i) cudaEventDestroy(ev[i]);
  if (st_ != PSLBM_OK) return st_;
  for (int k = 0; k < 3; ++k) kernel_ms[k] = acc[k] / double(n);
  if (total_ms) *total_ms = tot / double(n);
  return PSLBM_OK;
}

// Initial solid volumes from the node types when the caller gives none:
// V_D = 1 at D(s) nodes, V_F = 1 at F(s) nodes, 0 elsewhere.
__global__ void k_vol_from_mask(const uint8_t* __restrict__ mask, double* __restrict__ V, long long N) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < N; i += (long long)gridDim.x * blockDim.x) {
    const int t = mask[i] & 15;
    V[i] = t == PSLBM_SOLID_D ? 1.0 : 0.0;
    V[N + i] = t == PSLBM_SOLID_F ? 1.0 : 0.0;
  }
}

// First step's liquid threshold from the initial maximum of rho_1 over fluid
// nodes (res[0], -inf without fluid): the maximum in the ordered encoding of
// the step's slot, and half of it in both precisions, as the amendment kernel
// leaves them at the end of a step.
__global__ void k_first_threshold(const double* __restrict__ res, unsigned long long* __restrict__ scal) {
  const double m = res[0];
  const unsigned long long enc = m > -INFINITY ? ord_enc(m) : 0ULL;
  const double th = 0.5 * ord_dec(enc);
  scal[S_MAX0] = enc;
  scal[S_THETA] = (unsigned long long)__double_as_longlong(th);
  scal[S_THETAF] = (unsigned long long)(unsigned)__float_as_int(__double2float_rn(th));
}

// Step count and status bits of every member of a batch, gathered into one
// device buffer (out[2 i], out[2 i + 1]) for a single copy to the host.
__global__ void k_batch_monitor(const DevInst* __restrict__ insts, int n, unsigned long long* __restrict__ out) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    out[2 * i] = insts[i].scal[S_STEP];
    out[2 * i + 1] = insts[i].scal[S_STATUS];
  }
}

// Enqueue the kernels that make an instance's lists from its node types (kinds 2: of
// fluid and of minerals, 3: of reservoirs too).  The counts of the tiles, at most 12
// bytes a node, go where the potentials go, which are not needed between steps.
cudaError_t make_lists(cudaStream_t s, const DevInst& I, int kinds) {
  cudaError_t e = cudaMemsetAsync(I.fbits, 0, (size_t)((I.N + 31) / 32) * 2 * sizeof(unsigned), s);
  if (e != cudaSuccess) return e;
  const int tiles = ((I.P.nx + 31) / 32) * ((I.P.ny + 7) / 8);
  const int blocks = (tiles + ST_WARPS - 1) / ST_WARPS;
  int* counts = (int*)I.pot;
  k_list<false><<<blocks, ST_THREADS, 0, s>>>(I, counts, tiles, kinds);
  k_list_scan<<<1, 1024, 0, s>>>(counts, tiles, I.scal, kinds);
  k_list<true><<<blocks, ST_THREADS, 0, s>>>(I, counts, tiles, kinds);
  return cudaGetLastError();
}

// Steps after which the lists are made again.  They only grow: nodes that dissolve join
// the fluid list out of order and stay on the list of minerals, so that a step takes
// ever longer (100x160 FP32, 1,500 of 13,000 minerals dissolved in 17,000 steps: 19.4 us, with
// new lists 15.8).  Making them takes an instance's share of some 10 us, four launches.
int64_t list_life(const Stepper& st) { return 1024LL * std::max(1, st.ninst / 16); }

// Run n steps, replaying captured graphs of up to 32 steps.
pslbm_status run_steps(Stepper& st, int64_t n, std::string& err) {
  cudaStream_t s = lib_stream();
  cudaError_t te = ensure_work(st);
  if (te != cudaSuccess) {
    err = std::string("work list: ") + cudaGetErrorString(te);
    return PSLBM_ERR_CUDA;
  }
  GraphCache& gc = st.graphs;
  const int64_t K = 32;
  while (n > 0) {
    const int64_t k = n >= K ? K : n;
    auto it = gc.exec.find(k);
    if (it == gc.exec.end()) {
      cudaGraph_t g;
      cudaError_t e = cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal);
      if (e != cudaSuccess) {
        err = std::string("cudaStreamBeginCapture: ") + cudaGetErrorString(e);
        return PSLBM_ERR_CUDA;
      }
      enqueue_steps(s, st, k);
      e = cudaStreamEndCapture(s, &g);
      if (e != cudaSuccess) {
        err = std::string("cudaStreamEndCapture: ") + cudaGetErrorString(e);
        return PSLBM_ERR_CUDA;
      }
      cudaGraphExec_t ex;
      e = cudaGraphInstantiate(&ex, g, 0);
      cudaGraphDestroy(g);
      if (e != cudaSuccess) {
        err = std::string("cudaGraphInstantiate: ") + cudaGetErrorString(e);
        return PSLBM_ERR_CUDA;
      }
      it = gc.exec.emplace(k, ex).first;
    }
    cudaError_t e = cudaGraphLaunch(it->second, s);
    if (e != cudaSuccess) {
      err = std::string("cudaGraphLaunch: ") + cudaGetErrorString(e);
      return PSLBM_ERR_CUDA;
    }
    n -= k;
    st.since += k;
    if (st.since < list_life(st)) continue;
    st.since = 0;
    for (size_t i = 0; i < st.inst.size(); ++i) {
      if (!st.nface[i]) continue;       // no mineral that faces fluid: nothing changes
      e = make_lists(s, *st.inst[i], 2);
      if (e != cudaSuccess) {
        err = std::string("node lists: ") + cudaGetErrorString(e);
        return PSLBM_ERR_CUDA;
      }
    }
  }
  return PSLBM_OK;
}

// Fix the tile shape (tx = ty = 0: none).
pslbm_status set_shape(Stepper& st, int tx, int ty) {
  int idx = -2;
  if (tx == 0 && ty == 0) idx = -1;
  for (int sh = 0; sh < NSHAPES; ++sh)
    if (SHAPE_TX[sh] == tx && SHAPE_TY[sh] == ty) idx = sh;
  if (idx == -2) return PSLBM_ERR_PARAM;
  if (idx >= 0 && st.fix_staged == 1 && SHAPE_TX[idx] * SHAPE_TY[idx] > 256) return PSLBM_ERR_PARAM;
  if (idx != st.fix_shape) st.drop_work();
  st.fix_shape = idx;
  return PSLBM_OK;
}

// Fix the staging (-1: none).  The kernels stage no populations: the choice is
// checked and reported, and changes nothing else.
pslbm_status set_staging(Stepper& st, int mode) {
  if (mode < -1 || mode >= NSTAGING || (mode >= 1 && !st.staged_ok)) return PSLBM_ERR_PARAM;
  if (mode == 1 && st.fix_shape >= 0 && SHAPE_TX[st.fix_shape] * SHAPE_TY[st.fix_shape] > 256) return PSLBM_ERR_PARAM;
  st.fix_staged = mode;
  return PSLBM_OK;
}

// Whether a caller may ask for staging 1 or 2: FP32 populations and rows of a
// multiple of 16 bytes.
bool staging_open(const pslbm_params* p) {
  if (p->precision == PSLBM_FP64) return false;
  return p->nx * 4 % 16 == 0 && (p->n_species == 0 || (int64_t)p->nx * (int64_t)gsize(p->precision) % 16 == 0);
}

// Shape and staging as reported: the caller's, or 32x8 and plain loads.
int shown_shape(const Stepper& st) { return st.fix_shape >= 0 ? st.fix_shape : 1; }
int shown_staging(const Stepper& st) { return st.fix_staged >= 0 ? st.fix_staged : 0; }

pslbm_status status_of(pslbm_t h, unsigned long long st) {
  if (st & ST_NONFINITE) return fail(h, PSLBM_ERR_NONFINITE, "non-finite density on the device");
  if (st & ST_EOS) return fail(h, PSLBM_ERR_EOS_DOMAIN, "Eq. 13 square-root argument negative (rho_1 outside the EOS domain)");
  return PSLBM_OK;
}

// Status bits; the lengths of the lists, which a step's plan depends on, come along.
pslbm_status device_status(pslbm_t h) {
  unsigned long long sc[S_NFACE + 1];
  CK(h, cudaMemcpyAsync(sc, h->h.scal, sizeof sc, cudaMemcpyDeviceToHost, lib_stream()));
  CK(h, cudaStreamSynchronize(lib_stream()));
  h->run.nfluid[0] = (int)sc[S_NFLUID];
  h->run.nface[0] = (int)sc[S_NFACE];
  return status_of(h, sc[S_STATUS]);
}

}  // namespace

extern "C" {

void* pslbm_get_stream(void) { return (void*)lib_stream(); }

pslbm_status pslbm_set_stream(void* s) {
  g_user_set = s != nullptr;
  g_user_stream = (cudaStream_t)s;
  return PSLBM_OK;
}

pslbm_status pslbm_create(const uint8_t* mask, const double* rho1, const double* rho2, const double* conc,
                          const double* vol, const pslbm_params* p, pslbm_t* out) {
  if (!out) return fail(nullptr, PSLBM_ERR_PARAM, "out is NULL");
  *out = nullptr;
  if (!mask || !rho1 || !rho2) return fail(nullptr, PSLBM_ERR_PARAM, "mask, rho1 and rho2 are required");
  std::string v = validate(p);
  if (!v.empty()) return fail(nullptr, PSLBM_ERR_PARAM, v);
  if (check_device() != PSLBM_OK) return fail(nullptr, PSLBM_ERR_NODEVICE, "no sm_103 CUDA device");
  const int ns = p->n_species;
  const Launchers* L = launchers(p->precision, ns);
  if (!L) return fail(nullptr, PSLBM_ERR_PARAM, "no kernels for this precision / species count");

  pslbm_t h = new (std::nothrow) pslbm_s();
  if (!h) return fail(nullptr, PSLBM_ERR_OOM, "host allocation failed");
  h->p = *p;
  h->prec = p->precision;
  h->ns = ns;
  h->L = L;
  const long long N = (long long)p->nx * p->ny;
  h->N = N;
  cudaStream_t s = lib_stream();
  DevInst& I = h->h;
  I.P = to_dev(p);
  I.N = N;
  I.evcap = (int)N;
  pslbm_status st = PSLBM_OK;
  {
    // one device allocation holds the instance's whole state, each part on a
    // 256-byte boundary; the initial
    // threshold's budget partial sums are the last part
    const size_t NP = (size_t)(N + CELL - 1) / CELL * CELL;   // whole cells
    const size_t fb = NP * 18 * fsize(p->precision), gb = NP * 5 * ns * gsize(p->precision);
    I.read_once = read_once(2 * (fb + gb)) ? 1 : 0;
    const size_t sizes[] = {fb, fb, gb, gb, (size_t)N, (size_t)N, (size_t)N * 2 * sizeof(double), (size_t)N,
                            (size_t)N * sizeof(int),
                            (size_t)((N + 31) / 32) * 2 * sizeof(unsigned), S_NSCAL * sizeof(unsigned long long),
                            sizeof(DevInst), (size_t)((BUD_BLOCKS + 1) * NBUD + 2) * sizeof(double), (size_t)N * 4 * fsize(p->precision),
                            (size_t)N, (size_t)N * 2 * sizeof(int)};
    constexpr int NPARTS = sizeof(sizes) / sizeof(sizes[0]);
    size_t offs[NPARTS], total = 0;
    for (int i = 0; i < NPARTS; ++i) {
      offs[i] = total;
      total += ((sizes[i] ? sizes[i] : 16) + 255) / 256 * 256;
    }
    void* arena = nullptr;
    st = dalloc(h, &arena, total);
    if (st != PSLBM_OK) goto fail_cleanup;
    char* base = (char*)arena;
    I.f[0] = base + offs[0];
    I.f[1] = base + offs[1];
    I.g[0] = base + offs[2];
    I.g[1] = base + offs[3];
    I.type[0] = (uint8_t*)(base + offs[4]);
    I.type[1] = (uint8_t*)(base + offs[5]);
    I.V = (double*)(base + offs[6]);
    I.evt = (uint8_t*)(base + offs[7]);
    I.claim = (int*)(base + offs[8]);
    I.fbits = (unsigned*)(base + offs[9]);
    I.mbits = I.fbits + (N + 31) / 32;
    I.scal = (unsigned long long*)(base + offs[10]);
    h->d = (DevInst*)(base + offs[11]);
    I.pot = base + offs[13];
    // the potentials are done with before the VOP kernel runs, and its events with the
    // amendment before the next potentials: both in the same bytes
    I.xs = (double*)I.pot;
    I.evlist = (int*)(I.xs + N);
    static_assert(4 * sizeof(float) >= sizeof(double) + 2 * sizeof(int), "room for xs and evlist");
    I.code = (uint8_t*)(base + offs[14]);
    I.flist = (int*)(base + offs[15]);
    I.mlist = I.flist + N;
    double* part = (double*)(base + offs[12]);
    double* res = part + (size_t)BUD_BLOCKS * NBUD;

    // the inputs are staged in the second population buffer (at least 72
    // bytes per node; they need 17 + 8 ns <= 49), which is cleared once the
    // initialisation kernel has read them
    double* dr1 = (double*)I.f[1];
    double* dr2 = dr1 + N;
    double* dc = (conc && ns) ? dr2 + N : nullptr;
    uint8_t* dmask = (uint8_t*)(dr2 + N + (dc ? (size_t)N * ns : 0));
    cudaError_t e = cudaMemcpyAsync(dmask, mask, N, cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(dr1, rho1, N * sizeof(double), cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(dr2, rho2, N * sizeof(double), cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess && dc) e = cudaMemcpyAsync(dc, conc, N * ns * sizeof(double), cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(I.evt, 0, (size_t)N, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(I.claim, 0, (size_t)N * sizeof(int), s);
    if (e == cudaSuccess) e = cudaMemsetAsync(I.scal, 0, S_NSCAL * sizeof(unsigned long long), s);
    if (e == cudaSuccess) e = cudaMemsetAsync(I.scal + S_LIMIT, 0xff, sizeof(unsigned long long), s);
    if (e == cudaSuccess && ns) e = cudaMemsetAsync(I.g[1], 0, gb, s);
    if (e == cudaSuccess) {
      if (vol) {
        e = cudaMemcpyAsync(I.V, vol, (size_t)N * 2 * sizeof(double), cudaMemcpyHostToDevice, s);
      } else {
        k_vol_from_mask<<<(unsigned)std::min<long long>((N + 255) / 256, 65536), 256, 0, s>>>(dmask, I.V, N);
        e = cudaGetLastError();
      }
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(h->d, &I, sizeof(DevInst), cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) {
      L->init(s, h->d, dmask, dr1, dr2, dc, N);
      e = make_lists(s, I, 3);
    }
    // initial liquid threshold: half the maximum initial rho_1 over fluid
    // nodes (the first budget entry), decoded on the device
    if (e == cudaSuccess) {
      L->budget(s, h->d, part, res);
      k_first_threshold<<<1, 1, 0, s>>>(res, I.scal);
      e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemsetAsync(I.f[1], 0, fb, s);
    // the host copy of the descriptor is read by the copy above before the
    // call returns only for pageable memory; synchronise once for it and for
    // the errors of everything above
    unsigned long long counts[3] = {0, 0, 0};
    static_assert(S_NFACE == S_NFLUID + 1 && S_NRES == S_NFACE + 1, "read together");
    if (e == cudaSuccess) e = cudaMemcpyAsync(counts, I.scal + S_NFLUID, sizeof counts, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    h->run.nfluid.assign(1, (int)counts[0]);
    h->run.nface.assign(1, (int)counts[1]);
    h->run.nres.assign(1, (int)counts[2]);
    I.nres = (int)counts[2];
    I.reslist = I.flist + (N - I.nres);
    if (e == cudaSuccess) e = cudaMemcpyAsync(h->d, &I, sizeof(DevInst), cudaMemcpyHostToDevice, s);
    if (e != cudaSuccess) {
      st = fail(nullptr, e == cudaErrorMemoryAllocation ? PSLBM_ERR_OOM : PSLBM_ERR_CUDA,
                std::string("create: ") + cudaGetErrorString(e));
      goto fail_cleanup;
    }
  }
  h->run.L = L;
  h->run.d = h->d;
  h->run.ninst = 1;
  h->run.dims.assign(1, {p->nx, p->ny});
  h->run.host0 = h->h;
  h->run.inst.assign(1, &h->h);
  h->run.fp64 = p->precision == PSLBM_FP64;
  h->run.staged_ok = staging_open(p);
  {
    cudaError_t e = ensure_work(h->run);
    if (e != cudaSuccess) {
      st = fail(nullptr, e == cudaErrorMemoryAllocation ? PSLBM_ERR_OOM : PSLBM_ERR_CUDA,
                std::string("work list: ") + cudaGetErrorString(e));
      goto fail_cleanup;
    }
  }
  *out = h;
  return PSLBM_OK;
fail_cleanup : {
  std::string m = h->err;
  free_all(h);
  delete h;
  if (!m.empty()) {
    std::lock_guard<std::mutex> lk(g_mu);
    g_lib_err = m;
  }
  return st;
}
}

pslbm_status pslbm_step(pslbm_t h, int64_t n) {
  if (!h) return fail(nullptr, PSLBM_ERR_PARAM, "handle is NULL");
  if (h->sticky) return h->sticky;
  if (n < 0) return fail(h, PSLBM_ERR_PARAM, "n < 0");
  if (h->in_batch) return fail(h, PSLBM_ERR_STATE, "handle is a member of a batch; step the batch");
  if (n == 0) return PSLBM_OK;
  std::string err;
  pslbm_status st = run_steps(h->run, n, err);
  if (st != PSLBM_OK) return fail(h, st, err);
  return PSLBM_OK;
}

pslbm_status pslbm_profile_step(pslbm_t h, int64_t n, double* kernel_ms, double* total_ms) {
  if (!h) return fail(nullptr, PSLBM_ERR_PARAM, "handle is NULL");
  if (h->sticky) return h->sticky;
  if (n < 1 || !kernel_ms) return fail(h, PSLBM_ERR_PARAM, "n < 1 or kernel_ms is NULL");
  if (h->in_batch) return fail(h, PSLBM_ERR_STATE, "handle is a member of a batch");
  std::string err;
  pslbm_status st = profile_steps(h->run, n, kernel_ms, total_ms, err);
  if (st != PSLBM_OK) return fail(h, st, err);
  return device_status(h);
}

pslbm_status pslbm_set_step_limit(pslbm_t h, int64_t limit) {
  if (!h) return fail(nullptr, PSLBM_ERR_PARAM, "handle is NULL");
  if (h->sticky) return h->sticky;
  const unsigned long long v = limit < 0 ? ~0ULL : (unsigned long long)limit;
  CK(h, cudaMemcpyAsync(h->h.scal + S_LIMIT, &v, sizeof v, cudaMemcpyHostToDevice, lib_stream()));
  CK(h, cudaStreamSynchronize(lib_stream()));
  return PSLBM_OK;
}

pslbm_status pslbm_estimate_device_bytes(const pslbm_params* p, uint64_t* bytes) {
  if (!bytes) return fail(nullptr, PSLBM_ERR_PARAM, "bytes is NULL");
  std::string v = validate(p);
  if (!v.empty()) return fail(nullptr, PSLBM_ERR_PARAM, v);
  const uint64_t N = (uint64_t)p->nx * (uint64_t)p->ny;
  const uint64_t per = 2 * 18 * fsize(p->precision) + 2 * 5 * (uint64_t)p->n_species * gsize(p->precision) +
                       2 /*types*/ + 4 * fsize(p->precision) + 1 /*potentials, codes*/ + 16 /*V*/ + 1 /*events*/ + 4 /*claims*/ + 8 /*node lists*/;
  const uint64_t bits = ((N + 31) / 32) * 8;
  // whole cells
  const uint64_t cells = (N + CELL - 1) / CELL * CELL;
  const uint64_t pops = 2 * 18 * fsize(p->precision) + 2 * 5 * (uint64_t)p->n_species * gsize(p->precision);
  *bytes = N * per + (cells - N) * pops + bits + sizeof(DevInst) + S_NSCAL * 8 +
           (uint64_t)((BUD_BLOCKS + 1) * NBUD + 2) * sizeof(double) + 16 * 256;
  return PSLBM_OK;
}

pslbm_status pslbm_set_tile_shape(pslbm_t h, int32_t tile_x, int32_t tile_y) {
  if (!h) return fail(nullptr, PSLBM_ERR_PARAM, "handle is NULL");
  if (set_shape(h->run, tile_x, tile_y) != PSLBM_OK)
    return fail(h, PSLBM_ERR_PARAM,
                "unsupported tile shape (0x0, 16x16, 32x8, 16x32 or 32x16; not the last two while staging 1 is asked for)");
  return PSLBM_OK;
}

pslbm_status pslbm_get_tile_shape(pslbm_t h, int32_t* tile_x, int32_t* tile_y, int32_t* tuned) {
  if (!h) return fail(nullptr, PSLBM_ERR_PARAM, "handle is NULL");
  if (tile_x) *tile_x = SHAPE_TX[shown_shape(h->run)];
  if (tile_y) *tile_y = SHAPE_TY[shown_shape(h->run)];
  if (tuned) *tuned = 1;
  return PSLBM_OK;
}

pslbm_status pslbm_set_staging(pslbm_t h, int32_t mode) {
  if (!h) return fail(nullptr, PSLBM_ERR_PARAM, "handle is NULL");
  if (set_staging(h->run, mode) != PSLBM_OK)
    return fail(h, PSLBM_ERR_PARAM, "staging must be -1, 0, 1 or 2 (1, 2 only with FP32 populations and rows of a multiple of 16 bytes)");
  return PSLBM_OK;
}

pslbm_status pslbm_get_staging(pslbm_t h, int32_t* staged, int32_t* available) {
  if (!h) return fail(nullptr, PSLBM_ERR_PARAM, "handle is NULL");
  if (staged) *staged = shown_staging(h->run);
  if (available) *available = h->run.staged_ok ? 1 : 0;
  return PSLBM_OK;
}

pslbm_status pslbm_monitor(pslbm_t h, int64_t* steps, double* max_rho1, uint32_t* status) {
  if (!h) return fail(nullptr, PSLBM_ERR_PARAM, "handle is NULL");
  if (h->sticky) return h->sticky;
  unsigned long long sc[S_STATUS + 1];
  CK(h, cudaMemcpyAsync(sc, h->h.scal, sizeof sc, cudaMemcpyDeviceToHost, lib_stream()));
  CK(h, cudaStreamSynchronize(lib_stream()));
  const unsigned long long n = sc[S_STEP];
  if (steps) *steps = (int64_t)n;
  // the slot the last step filled (the initial maximum before the first step)
  if (max_rho1) *max_rho1 = ord_dec(sc[S_MAX0 + int(n & 1ULL)]);
  if (status) *status = (uint32_t)sc[S_STATUS];
  if (sc[S_STATUS] & ST_NONFINITE) return fail(h, PSLBM_ERR_NONFINITE, "non-finite density on the device");
  if (sc[S_STATUS] & ST_EOS)
    return fail(h, PSLBM_ERR_EOS_DOMAIN, "Eq. 13 square-root argument negative (rho_1 outside the EOS domain)");
  return PSLBM_OK;
}

pslbm_status pslbm_sync(pslbm_t h) {
  if (!h) return fail(nullptr, PSLBM_ERR_PARAM, "handle is NULL");
  if (h->sticky) return h->sticky;
  cudaError_t e = cudaStreamSynchronize(lib_stream());
  if (e != cudaSuccess) return fail(h, PSLBM_ERR_CUDA, std::string("sync: ") + cudaGetErrorString(e));
  return device_status(h);
}

pslbm_status pslbm_info(pslbm_t h, int64_t* steps, int32_t* nx, int32_t* ny, int32_t* n_species) {
  if (!h) return fail(nullptr, PSLBM_ERR_PARAM, "handle is NULL");
  if (steps) {
    unsigned long long t = 0;
    CK(h, cudaMemcpyAsync(&t, h->h.scal + S_STEP, sizeof t, cudaMemcpyDeviceToHost, lib_stream()));
    CK(h, cudaStreamSynchronize(lib_stream()));
    *steps = (int64_t)t;
  }
  if (nx) *nx = h->p.nx;
  if (ny) *ny = h->p.ny;
  if (n_species) *n_species = h->ns;
  return PSLBM_OK;
}

pslbm_status pslbm_device_bytes(pslbm_t h, uint64_t* bytes) {
  if (!h || !bytes) return fail(h, PSLBM_ERR_PARAM, "NULL argument");
  *bytes = h->bytes;
  return PSLBM_OK;
}

pslbm_status pslbm_read_fields(pslbm_t h, uint32_t fields, void* const* out) {
  if (!h) return fail(nullptr, PSLBM_ERR_PARAM, "handle is NULL");
  if (h->sticky) return h->sticky;
  if (fields & ~0xFFu) return fail(h, PSLBM_ERR_PARAM, "unknown field bits");
  if (fields && !out) return fail(h, PSLBM_ERR_PARAM, "out is NULL");
  const long long N = h->N;
  const int ns = h->ns;
  cudaStream_t s = lib_stream();
  // scratch: rho1, rho2, ux, uy (N each), conc (ns N), type (N bytes), budget
  // partials, budget, step count and status
  const size_t at_part = ((size_t)N * (4 + ns) * sizeof(double) + (size_t)N + 15) / 16 * 16;
  const size_t need = at_part + ((BUD_BLOCKS + 1) * NBUD + 2) * sizeof(double);
  if (h->rb_bytes < need) {
    if (h->rb) {
      cudaFree(h->rb);
      h->bytes -= h->rb_bytes;
    }
    h->rb = nullptr;
    h->rb_bytes = 0;
    cudaError_t e = cudaMalloc(&h->rb, need);
    if (e != cudaSuccess) {
      cudaGetLastError();
      return fail(h, PSLBM_ERR_OOM, "read-back scratch allocation failed");
    }
    h->rb_bytes = need;
    h->bytes += need;
  }
  double* r1 = h->rb;
  double* r2 = r1 + N;
  double* ux = r2 + N;
  double* uy = ux + N;
  double* cc = uy + N;
  uint8_t* ty = (uint8_t*)(cc + (size_t)N * ns);
  double* part = (double*)((char*)h->rb + at_part);
  double* bud = part + BUD_BLOCKS * NBUD;
  if (fields & 0x3F) {
    auto want = [&](uint32_t f, auto* p) { return fields & f ? p : nullptr; };
    h->L->fields(s, h->d, N, want(PSLBM_F_RHO1, r1), want(PSLBM_F_RHO2, r2), want(PSLBM_F_UX, ux), want(PSLBM_F_UY, uy),
                 ns ? want(PSLBM_F_CONC, cc) : nullptr, want(PSLBM_F_TYPE, ty));
    CK(h, cudaGetLastError());
  }
  if (fields & PSLBM_F_BUDGET) {
    h->L->budget(s, h->d, part, bud);
    CK(h, cudaGetLastError());
  }
  // The caller's buffers are copied to one by one: two that happen to adjoin may lie in
  // different page-locked ranges, which one copy must not span.  Few bytes come over
  // into a buffer of the handle, parts that adjoin on the device in one copy, and go on
  // from there (all fields of 128x64 FP64, 0.6 MB: 95 us, with a copy a field 101; what
  // is left over 56 us, with one copy into one block of the caller's, is the second pass
  // over bytes that the host has not in its caches).
  struct Part {
    const char* from;
    size_t bytes;
    uint32_t bit;
  };
  const size_t fb = (size_t)N * sizeof(double);
  const Part parts[] = {{(char*)r1, fb, PSLBM_F_RHO1}, {(char*)r2, fb, PSLBM_F_RHO2}, {(char*)ux, fb, PSLBM_F_UX},
                        {(char*)uy, fb, PSLBM_F_UY}, {(char*)cc, fb * ns, PSLBM_F_CONC}, {(char*)ty, (size_t)N, PSLBM_F_TYPE},
                        {(char*)h->h.V, 2 * fb, PSLBM_F_VOL}};
  constexpr int NPARTS = 7, V_PART = NPARTS - 1;    // all but V in the scratch, one behind the other
  size_t total = 0;
  for (const Part& q : parts) total += fields & q.bit ? q.bytes : 0;
  char* stage = nullptr;
  if (total && total <= STAGE_BYTES) {
    if (!h->stage) h->stage.reset(new (std::nothrow) char[std::min(fb * (6 + ns) + (size_t)N, STAGE_BYTES)]);
    stage = h->stage.get();       // null: no memory, straight to the caller's buffers
  }
  int i = 0;
  if (stage) {
    char* to = stage;
    for (int k = 0; k < NPARTS;) {
      size_t run = fields & parts[k].bit ? parts[k].bytes : 0;
      int e = k + 1;
      if (run)
        while (e < V_PART && (fields & parts[e].bit)) run += parts[e++].bytes;
      if (run) CK(h, cudaMemcpyAsync(to, parts[k].from, run, cudaMemcpyDeviceToHost, s));
      to += run;
      k = e;
    }
    CK(h, cudaStreamSynchronize(s));
    const char* at = stage;
    for (const Part& q : parts) {
      if (!(fields & q.bit)) continue;
      if (q.bytes) std::memcpy(out[i], at, q.bytes);
      at += q.bytes;
      ++i;
    }
  } else {
    for (const Part& q : parts) {
      if (!(fields & q.bit)) continue;
      if (q.bytes) CK(h, cudaMemcpyAsync(out[i], q.from, q.bytes, cudaMemcpyDeviceToHost, s));
      ++i;
    }
  }
  if (!(fields & PSLBM_F_BUDGET)) return device_status(h);
  struct {
    double v[NBUD];
    unsigned long long step, status;
  } b;
  CK(h, cudaMemcpyAsync(&b, bud, sizeof b, cudaMemcpyDeviceToHost, s));
  CK(h, cudaStreamSynchronize(s));
  double* o = (double*)out[i++];
  o[0] = b.v[0] > -INFINITY ? b.v[0] : 0.0;
  o[1] = b.v[1];
  o[2] = b.v[2];
  for (int k = 0; k < ns; ++k) o[3 + k] = b.v[3 + k];
  o[3 + ns] = b.v[3 + MAXS];
  o[4 + ns] = b.v[4 + MAXS];
  o[5 + ns] = (double)b.step;
  return status_of(h, b.status);
}

pslbm_status pslbm_destroy(pslbm_t h) {
  if (!h) return PSLBM_OK;
  cudaStreamSynchronize(lib_stream());
  if (h->rb) cudaFree(h->rb);
  free_all(h);
  delete h;
  return PSLBM_OK;
}

const char* pslbm_last_error(pslbm_t h) {
  if (h) return h->err.c_str();
  return g_lib_err.c_str();
}

// ------------------------------------------------------------------ batches

pslbm_status pslbm_batch_create(int32_t n, const pslbm_t* members, int32_t tile_x, int32_t tile_y,
                                pslbm_batch_t* out) {
  if (!out) return fail(nullptr, PSLBM_ERR_PARAM, "out is NULL");
  *out = nullptr;
  if (n < 1 || !members) return fail(nullptr, PSLBM_ERR_PARAM, "empty batch");
  for (int i = 0; i < n; ++i) {
    if (!members[i] || members[i]->sticky) return fail(nullptr, PSLBM_ERR_PARAM, "invalid member");
    if (members[i]->in_batch) return fail(nullptr, PSLBM_ERR_STATE, "member already in a batch");
    if (members[i]->prec != members[0]->prec || members[i]->ns != members[0]->ns)
      return fail(nullptr, PSLBM_ERR_PARAM, "members differ in precision or species count");
    for (int j = 0; j < i; ++j)
      if (members[j] == members[i]) return fail(nullptr, PSLBM_ERR_PARAM, "duplicate member");
  }
  pslbm_batch_t b = new (std::nothrow) pslbm_batch_s();
  if (!b) return fail(nullptr, PSLBM_ERR_OOM, "host allocation failed");
  b->run.staged_ok = true;
  for (int i = 0; i < n; ++i) b->run.staged_ok = b->run.staged_ok && members[i]->run.staged_ok;
  b->L = members[0]->L;
  b->run.L = b->L;
  if (set_shape(b->run, tile_x, tile_y) != PSLBM_OK) {
    delete b;
    return fail(nullptr, PSLBM_ERR_PARAM, "unsupported tile shape (0x0, 16x16, 32x8, 16x32 or 32x16)");
  }
  std::vector<DevInst> di;
  for (int i = 0; i < n; ++i) {
    b->members.push_back(members[i]);
    di.push_back(members[i]->h);
    b->run.dims.push_back({members[i]->p.nx, members[i]->p.ny});
  }
  cudaStream_t s = lib_stream();
  cudaError_t e = cudaMalloc(&b->d, di.size() * sizeof(DevInst));
  if (e == cudaSuccess) e = cudaMemcpyAsync(b->d, di.data(), di.size() * sizeof(DevInst), cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  b->L = members[0]->L;
  b->run.L = b->L;
  b->run.d = b->d;
  b->run.ninst = n;
  b->run.host0 = members[0]->h;
  b->run.fp64 = members[0]->prec == PSLBM_FP64;
  b->run.mode = M_SHARED;
  for (int i = 0; i < n; ++i) {
    b->run.nfluid.push_back(members[i]->run.nfluid[0]);
    b->run.nface.push_back(members[i]->run.nface[0]);
    b->run.nres.push_back(members[i]->run.nres[0]);
    b->run.inst.push_back(&members[i]->h);
    b->run.since = std::max(b->run.since, members[i]->run.since);
    if (!same_hot_params(members[i]->h.P, members[0]->h.P)) b->run.mode = M_MIXED;
  }
  if (e == cudaSuccess) e = ensure_work(b->run);
  if (e != cudaSuccess) {
    b->run.release();
    if (b->d) cudaFree(b->d);
    delete b;
    return fail(nullptr, e == cudaErrorMemoryAllocation ? PSLBM_ERR_OOM : PSLBM_ERR_CUDA,
                std::string("batch create: ") + cudaGetErrorString(e));
  }
  for (int i = 0; i < n; ++i) members[i]->in_batch = 1;
  *out = b;
  return PSLBM_OK;
}

pslbm_status pslbm_batch_step(pslbm_batch_t b, int64_t n) {
  if (!b) return fail(nullptr, PSLBM_ERR_PARAM, "batch is NULL");
  if (b->sticky) return b->sticky;
  if (n < 0) return fail(nullptr, PSLBM_ERR_PARAM, "n < 0");
  if (n == 0) return PSLBM_OK;
  for (size_t i = 0; i < b->members.size(); ++i) {
    b->run.nfluid[i] = b->members[i]->run.nfluid[0];
    b->run.nface[i] = b->members[i]->run.nface[0];
  }
  std::string err;
  pslbm_status st = run_steps(b->run, n, err);
  if (st != PSLBM_OK) {
    b->sticky = st;
    b->err = err;
    return fail(nullptr, st, err);
  }
  return PSLBM_OK;
}

pslbm_status pslbm_batch_get_tile_shape(pslbm_batch_t b, int32_t* tile_x, int32_t* tile_y, int32_t* tuned) {
  if (!b) return fail(nullptr, PSLBM_ERR_PARAM, "batch is NULL");
  if (tile_x) *tile_x = SHAPE_TX[shown_shape(b->run)];
  if (tile_y) *tile_y = SHAPE_TY[shown_shape(b->run)];
  if (tuned) *tuned = 1;
  return PSLBM_OK;
}

pslbm_status pslbm_batch_set_staging(pslbm_batch_t b, int32_t mode) {
  if (!b) return fail(nullptr, PSLBM_ERR_PARAM, "batch is NULL");
  if (set_staging(b->run, mode) != PSLBM_OK)
    return fail(nullptr, PSLBM_ERR_PARAM, "staging must be -1, 0, 1 or 2 (1, 2 only where every member has them)");
  return PSLBM_OK;
}

pslbm_status pslbm_batch_get_staging(pslbm_batch_t b, int32_t* staged, int32_t* available) {
  if (!b) return fail(nullptr, PSLBM_ERR_PARAM, "batch is NULL");
  if (staged) *staged = shown_staging(b->run);
  if (available) *available = b->run.staged_ok ? 1 : 0;
  return PSLBM_OK;
}

pslbm_status pslbm_batch_sync(pslbm_batch_t b) {
  if (!b) return fail(nullptr, PSLBM_ERR_PARAM, "batch is NULL");
  if (b->sticky) return b->sticky;
  cudaError_t e = cudaStreamSynchronize(lib_stream());
  if (e != cudaSuccess) return fail(nullptr, PSLBM_ERR_CUDA, std::string("batch sync: ") + cudaGetErrorString(e));
  for (pslbm_t m : b->members) {
    pslbm_status st = device_status(m);
    if (st != PSLBM_OK) return st;
  }
  return PSLBM_OK;
}

pslbm_status pslbm_batch_profile_step(pslbm_batch_t b, int64_t n, double* kernel_ms, double* total_ms) {
  if (!b) return fail(nullptr, PSLBM_ERR_PARAM, "batch is NULL");
  if (b->sticky) return b->sticky;
  if (n < 1 || !kernel_ms) return fail(nullptr, PSLBM_ERR_PARAM, "n < 1 or kernel_ms is NULL");
  std::string err;
  pslbm_status st = profile_steps(b->run, n, kernel_ms, total_ms, err);
  if (st != PSLBM_OK) {
    b->sticky = st;
    b->err = err;
    return fail(nullptr, st, err);
  }
  return PSLBM_OK;
}

pslbm_status pslbm_batch_monitor(pslbm_batch_t b, int64_t* min_steps, uint32_t* status) {
  if (!b) return fail(nullptr, PSLBM_ERR_PARAM, "batch is NULL");
  if (b->sticky) return b->sticky;
  const int n = (int)b->members.size();
  cudaStream_t s = lib_stream();
  if (!b->mon) {
    cudaError_t e = cudaMalloc(&b->mon, (size_t)n * 2 * sizeof(unsigned long long));
    if (e != cudaSuccess) {
      cudaGetLastError();
      b->mon = nullptr;
      return fail(nullptr, PSLBM_ERR_OOM, "batch monitor buffer");
    }
    b->mon_h.assign((size_t)n * 2, 0ULL);
  }
  k_batch_monitor<<<(n + 255) / 256, 256, 0, s>>>(b->d, n, b->mon);
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(b->mon_h.data(), b->mon, (size_t)n * 2 * sizeof(unsigned long long), cudaMemcpyDeviceToHost,
                        s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return fail(nullptr, PSLBM_ERR_CUDA, std::string("batch monitor: ") + cudaGetErrorString(e));
  unsigned long long lo = ~0ULL, bits = 0;
  for (int i = 0; i < n; ++i) {
    lo = std::min(lo, b->mon_h[2 * i]);
    bits |= b->mon_h[2 * i + 1];
  }
  if (min_steps) *min_steps = (int64_t)lo;
  if (status) *status = (uint32_t)bits;
  return PSLBM_OK;
}

pslbm_status pslbm_batch_destroy(pslbm_batch_t b) {
  if (!b) return PSLBM_OK;
  cudaStreamSynchronize(lib_stream());
  b->run.release();
  if (b->d) cudaFree(b->d);
  if (b->mon) cudaFree(b->mon);
  for (pslbm_t m : b->members) {
    m->in_batch = 0;
    m->run.since = b->run.since;
  }
  delete b;
  return PSLBM_OK;
}

}  // extern "C"

namespace pslbm {

const Launchers* launchers_f64(int ns);
const Launchers* launchers_f32(int ns);
const Launchers* launchers_f32h(int ns);
const Launchers* launchers_f32b(int ns);
const Launchers* launchers(int prec, int ns) {
  if (ns < 0 || ns > MAXS) return nullptr;
  switch (prec) {
    case PSLBM_FP64: return launchers_f64(ns);
    case PSLBM_FP32: return launchers_f32(ns);
    case PSLBM_FP32_SOLUTE_F16: return launchers_f32h(ns);
    case PSLBM_FP32_SOLUTE_BF16: return launchers_f32b(ns);
  }
  return nullptr;
}

}  // namespace pslbm

// Accessors used by the allocation-free budget entry point (noalloc.cu).
namespace pslbm {
const DevInst* handle_device_inst(pslbm_t h) { return h->d; }
long long handle_nodes(pslbm_t h) { return h->N; }
int handle_precision(pslbm_t h) { return h->prec; }
int handle_species(pslbm_t h) { return h->ns; }
pslbm_status handle_sticky(pslbm_t h) { return h->sticky; }
pslbm_status handle_fail(pslbm_t h, pslbm_status s, const std::string& msg) { return fail(h, s, msg); }
cudaStream_t library_stream() { return lib_stream(); }
}  // namespace pslbm
