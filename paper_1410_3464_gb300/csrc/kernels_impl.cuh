// Explicit instantiation of the step kernels for one storage precision.
// Included by one translation unit per precision with KTF (population storage),
// KTG (solute storage), KR (compute type) and KNAME defined.
#include "launch.h"
#include "step.cuh"
#include "interface.cuh"
#include "aux.cuh"

namespace pslbm {
namespace {

// The kernels of a step are launched with programmatic stream serialisation: a
// kernel's blocks may start while the one before it drains, and wait
// (step_begin) for its end and its writes before they read anything.
template <class... A>
void launch_step(cudaStream_t s, int blocks, int threads, void (*kernel)(A...), A... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)blocks);
  cfg.blockDim = dim3((unsigned)threads);
  cfg.stream = s;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &at;
  // two blocks an SM at most: on larger grids the early blocks take room (1.5 % slower)
  cfg.numAttrs = blocks <= 2 * device_sms() ? 1 : 0;
  cudaLaunchKernelEx(&cfg, kernel, args...);
}

// Streaming kernels over nwork warps; Ik: the descriptor of a single simulation
// (mode M_SINGLE), or of a batch's first member (M_SHARED: all members have its
// hot parameters).
template <int NS>
void pot_l(cudaStream_t s, const Work* work, int nwork, int nstream, const DevInst* insts, const DevInst& Ik, int mode) {
  if (nwork <= 0) return;
  const int blocks = (nwork + ST_WARPS - 1) / ST_WARPS;
  auto k = mode == M_SINGLE ? k_pot<KTF, KR, M_SINGLE> : mode == M_SHARED ? k_pot<KTF, KR, M_SHARED> : k_pot<KTF, KR, M_MIXED>;
  launch_step<const Work*, int, int, const DevInst*, DevInst>(s, blocks, ST_THREADS, k, work, nwork, nstream, insts, Ik);
}
template <int NS>
void move_l(cudaStream_t s, const Work* work, int nwork, int nstream, const DevInst* insts, const DevInst& Ik, int mode) {
  if (nwork <= 0) return;
  const int blocks = (nwork + ST_WARPS - 1) / ST_WARPS;
  auto k = mode == M_SINGLE ? k_move<KTF, KTG, KR, NS, M_SINGLE>
           : mode == M_SHARED ? k_move<KTF, KTG, KR, NS, M_SHARED> : k_move<KTF, KTG, KR, NS, M_MIXED>;
  launch_step<const Work*, int, int, const DevInst*, DevInst>(s, blocks, ST_THREADS, k, work, nwork, nstream, insts, Ik);
}
template <int NS>
void vop_l(cudaStream_t s, const DevInst* insts, const Work* work, int nwork) {
  if (nwork <= 0) return;
  launch_step<const DevInst*, const Work*, int>(s, (nwork + NTHREADS / 32 - 1) / (NTHREADS / 32), NTHREADS,
                                                k_vop<KTF, KTG, KR, NS>, insts, work, nwork);
}
template <int NS>
void amend_l(cudaStream_t s, int ninst, const DevInst* insts) {
  if (ninst <= 0) return;
  launch_step<const DevInst*>(s, ninst, NTHREADS, k_amend<KTF, KTG, KR, NS>, insts);
}
template <int NS>
void vop_amend_l(cudaStream_t s, int ninst, const DevInst* insts) {
  if (ninst <= 0) return;
  launch_step<const DevInst*>(s, ninst, NTHREADS, k_vop_amend<KTF, KTG, KR, NS>, insts);
}
template <int NS>
void init_l(cudaStream_t s, DevInst* I, const uint8_t* m, const double* r1, const double* r2, const double* c,
            long long N) {
  long long blocks = (N + 255) / 256;
  if (blocks > 65536) blocks = 65536;
  k_init<KTF, KTG, KR, NS><<<(int)blocks, 256, 0, s>>>(I, m, r1, r2, c);
}
template <int NS>
void fields_l(cudaStream_t s, const DevInst* I, long long N, double* r1, double* r2, double* ux, double* uy,
              double* c, uint8_t* t) {
  long long blocks = (N + FIELD_THREADS - 1) / FIELD_THREADS;
  if (blocks > 65536) blocks = 65536;
  if (ux || uy) k_fields_pot<KTF, KR><<<(int)blocks, FIELD_THREADS, 0, s>>>(I);
  k_fields<KTF, KTG, KR, NS><<<(int)blocks, FIELD_THREADS, 0, s>>>(I, r1, r2, ux, uy, c, t);
}
template <int NS>
void budget_l(cudaStream_t s, const DevInst* I, double* part, double* out) {
  k_budget_partial<KTF, KTG, KR, NS><<<BUD_BLOCKS, BUD_THREADS, 0, s>>>(I, part);
  k_budget_final<<<1, BUD_FINAL_THREADS, 0, s>>>(I, part, BUD_BLOCKS, out);
}

template <int NS>
constexpr Launchers make() {
  Launchers l{};
  l.pot = &pot_l<NS>;
  l.move = &move_l<NS>;
  l.vop = &vop_l<NS>;
  l.amend = &amend_l<NS>;
  l.vop_amend = &vop_amend_l<NS>;
  l.init = &init_l<NS>;
  l.fields = &fields_l<NS>;
  l.budget = &budget_l<NS>;
  return l;
}
const Launchers table[MAXS + 1] = {make<0>(), make<1>(), make<2>(), make<3>(), make<4>()};

}  // namespace

const Launchers* KNAME(int ns) { return (ns >= 0 && ns <= MAXS) ? &table[ns] : nullptr; }

}  // namespace pslbm
