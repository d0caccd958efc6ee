// The two streaming kernels of a time step (Chen, Kang et al., arXiv 1410.3464,
// Sections 3-4, numerical procedure of Section 4.7):
//   k_pot   -- densities (Eq. 9a), liquid/gas marking (Section 4.5) and the
//              potentials psi_1 (Eq. 13), phi_1, phi_2 (Eq. 15) of every node;
//   k_move  -- forces (Eqs. 11, 14, 16), velocities (Eqs. 17-19), concentration
//              amendment at marking changes (Step 2), homogeneous sources
//              (Eqs. 5a, 5c, 27, 28), D2Q9 collision and push (Eq. 6, halfway
//              bounce-back) and D2Q5 collision and push (Eqs. 20-22), bouncing
//              back at every non-liquid neighbour (no-flux links, Eq. 26; the
//              VOP kernel applies Eqs. 29-31 to the links of minerals).
// State between steps is the pre-collision populations; streaming is a push into
// the other buffer of a ping-pong pair.
#pragma once
#include "device.cuh"

namespace pslbm {

template <class R, class TG, int NS>
__device__ __forceinline__ void conc_at(const TG* gin, int node, const DevParams& P, R* C) {
#pragma unroll
  for (int k = 0; k < NS; ++k) {
    const TG* gk = gin + goff<NS>(node) + k * 5 * CELL;
    R s = gld<R>(P, k, gk);
#pragma unroll
    for (int a = 1; a < 5; ++a) s += gld<R>(P, k, gk + a * CELL);
    C[k] = rp<R>(P).shift_c[k] + s;
  }
}

// Per-thread maximum of rho_1 and status bits of the tiles a thread has done
// since the last flush.
template <class R>
struct TileAcc {
  R mx;
  unsigned status;
};

// Warp reduction of the accumulators into the instance's slots: the exact
// maximum (the atomic only when it can raise the slot) and the status bits.
// Called by all lanes of the warp.
template <class R>
__device__ __forceinline__ void flush_acc(TileAcc<R>& acc, unsigned long long* scal, int cur) {
  R m = acc.mx;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = rmax<R>(m, __shfl_xor_sync(0xffffffffu, m, o));
  const unsigned st = __reduce_or_sync(0xffffffffu, acc.status);
  if ((threadIdx.x & 31) == 0) {
    if (m > R(-1.0 / 0.0)) {
      const unsigned long long enc = ord_enc(double(m));
      unsigned long long* slot = &scal[S_MAX0 + (cur ^ 1)];
      if (enc > *(volatile unsigned long long*)slot) atomicMax(slot, enc);
    }
    if (st) atomicOr(&scal[S_STATUS], (unsigned long long)st);
  }
  acc.mx = R(-1.0 / 0.0);
  acc.status = 0;
}

// Code of a node, one byte: what a step needs to know of a neighbour (fluid,
// marked liquid, reservoir, mineral; fluid and not marked, raw type liquid, raw
// type D(s), fluid and marked).
constexpr int C_FLUID = 1, C_MARK = 2, C_RES = 4, C_MIN = 8, C_FGAS = 16, C_OLDLIQ = 32, C_SOLD = 64, C_FLIQ = 128;
constexpr int C_LIVE = C_FLUID | C_RES;     // test with != 0
// ... by type, before marking; a type outside the enumeration is a wall.
__device__ __forceinline__ int type_code(int t) {
  if (t > T_OUTLET) return 0;
  constexpr unsigned lo = unsigned(C_FLUID | C_OLDLIQ) | unsigned(C_FLUID) << 8 | unsigned(C_MIN | C_SOLD) << 16 |
                          unsigned(C_MIN) << 24;
  constexpr unsigned hi = unsigned(C_RES) << 8 | unsigned(C_RES) << 16;
  return int(__funnelshift_r(t < 4 ? lo : hi, 0u, 8 * (t & 3)) & 0xFFu);
}

// Two values side by side: (psi_1, phi_1), the two fluid components, or two species.
template <class R>
struct Pair {
  R a, b;
};
template <class R> __device__ __forceinline__ Pair<R> mk(R a, R b) { return Pair<R>{a, b}; }
template <class R> __device__ __forceinline__ Pair<R> mk(R a) { return Pair<R>{a, a}; }
template <class R> __device__ __forceinline__ Pair<R> operator+(Pair<R> x, Pair<R> y) {
  return Pair<R>{radd<R>(x.a, y.a), radd<R>(x.b, y.b)};
}
template <class R> __device__ __forceinline__ Pair<R> operator-(Pair<R> x, Pair<R> y) {
  return Pair<R>{rsub<R>(x.a, y.a), rsub<R>(x.b, y.b)};
}
template <class R> __device__ __forceinline__ Pair<R> operator*(Pair<R> x, Pair<R> y) {
  return Pair<R>{rmul<R>(x.a, y.a), rmul<R>(x.b, y.b)};
}
template <class R> __device__ __forceinline__ Pair<R> pfma(Pair<R> x, Pair<R> y, Pair<R> z) {
  return Pair<R>{rfma<R>(x.a, y.a, z.a), rfma<R>(x.b, y.b, z.b)};
}
// Potentials of a node, read with one or two vector loads.
template <class R>
struct alignas(16) Pot {
  R ps, p1, p2, pad;
};
__device__ __forceinline__ Pot<float> ld_pot(const Pot<float>* p) {
  const float4 v = *reinterpret_cast<const float4*>(p);
  return Pot<float>{v.x, v.y, v.z, v.w};
}
__device__ __forceinline__ Pot<double> ld_pot(const Pot<double>* p) {
  const double2 v = *reinterpret_cast<const double2*>(p);
  return Pot<double>{v.x, v.y, p->p2, 0.0};
}
// FP64: rho_1 rides along with the potentials (eight additions less in k_move).
__device__ __forceinline__ double pot_rho1(const Pot<double>* p) { return p->pad; }
__device__ __forceinline__ float pot_rho1(const Pot<float>*) { return 0.f; }

// Both kernels run over the instance's list of fluid nodes (in tile order, kept
// up to date by the amendment kernel when nodes dissolve or fill), so that solid
// nodes cost neither lanes nor loads (1024x512 FP32: 62 us a step over all nodes,
// 54 over the list; FP64 430 and 322).  A warp takes a chunk of the list, 32 nodes
// at a time; a few warps take the reservoir nodes instead.
constexpr int ST_WARPS = 4;
constexpr int ST_THREADS = 32 * ST_WARPS;
// Where a launch finds its instances: one simulation, whose descriptor comes as
// a kernel argument (constant bank), or a batch's work list and descriptors; in
// a batch of equal hot parameters those come as an argument too.
enum { M_SINGLE = 0, M_SHARED = 1, M_MIXED = 2 };

// Start of a step's kernel (kernels_impl.cuh, launch_step): the next kernel may
// launch its blocks as this one's leave room; wait until the one before has
// ended.  Every thread of every block calls it before anything else.
__device__ __forceinline__ void step_begin() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// Work of warp w: 32 list entries from `first` on, and the same again every
// `stride` entries as far as the list goes; or reservoir nodes from entry `res`.
__device__ __forceinline__ bool step_work(bool single, const Work* __restrict__ work, int nwork, int nstream, int w, Work& t) {
  if (w >= nwork) return false;
  if (single) t = Work{0, w * 32, nstream * 32, w >= nstream ? (w - nstream) * 32 : -1};
  else t = work[w];
  return true;
}

// The fluid list, the list of minerals with a fluid axis neighbour and, at creation
// (kinds 3), the reservoir nodes, from the node types.  All go through the lattice by tiles of 32 columns and
// 8 rows, row by row within a tile, so that a warp's chunk of the list stays
// together on the lattice (4096x2048 FP32: 612 us a step, 717 to 766 with the tiles
// in the order of an atomic counter): k_list<false> counts a tile's nodes (a warp a tile),
// k_list_scan turns the counts into positions, k_list<true> writes the lists.
template <bool FILL>
static __global__ void __launch_bounds__(ST_THREADS) k_list(const __grid_constant__ DevInst I, int* __restrict__ counts, int ntiles, int kinds) {
  constexpr unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const int nx = I.P.nx, ny = I.P.ny, ncx = (nx + 31) >> 5;
  const int ti = blockIdx.x * ST_WARPS + (threadIdx.x >> 5);
  if (ti >= ntiles) return;
  const int y0 = ti / ncx * 8, x = (ti % ncx) * 32 + lane;
  const uint8_t* type = I.type[int(I.scal[S_STEP] & 1ULL)];
  int bf = FILL ? counts[ti] : 0, bm = FILL ? counts[ntiles + ti] : 0;
  int br = FILL && kinds > 2 ? int(I.N) - int(I.scal[S_NRES]) + counts[2 * ntiles + ti] : 0;
  const unsigned below = (1u << lane) - 1u;
#pragma unroll 4
  for (int r = 0; r < 8; ++r) {
    const int y = y0 + r;
    const int node = y * nx + x;
    const bool in = x < nx && y < ny;
    const int t = in ? type[node] & T_MASK : T_WALL;
    bool face = false;
    if (in && is_mineral(t)) {
#pragma unroll
      for (int a = 1; a < 5; ++a) {
        int xn, yn;
        if (nbr(I.P, x, y, EX(a), EY(a), xn, yn)) face = face || is_fluid(type[yn * nx + xn] & T_MASK);
      }
    }
    const bool fl = in && is_fluid(t);
    const bool res = kinds > 2 && (t == T_INLET || t == T_OUTLET);
    const unsigned mf = __ballot_sync(FULL, fl), mm = __ballot_sync(FULL, face), mr = __ballot_sync(FULL, res);
    if constexpr (FILL) {
      if (fl) {
        I.flist[bf + __popc(mf & below)] = node;
        atomicOr(&I.fbits[node >> 5], 1u << (node & 31));
      }
      if (face) {
        I.mlist[bm + __popc(mm & below)] = node;
        atomicOr(&I.mbits[node >> 5], 1u << (node & 31));
      }
      if (res) I.flist[br + __popc(mr & below)] = node;
    }
    bf += __popc(mf);
    bm += __popc(mm);
    br += __popc(mr);
  }
  if (!FILL && lane == 0) {
    counts[ti] = bf;
    counts[ntiles + ti] = bm;
    if (kinds > 2) counts[2 * ntiles + ti] = br;
  }
}
// One block: exclusive sums of the count arrays in place, totals into scal.
static __global__ void __launch_bounds__(1024) k_list_scan(int* __restrict__ counts, int ntiles, unsigned long long* scal, int kinds) {
  __shared__ int sums[1024];
  const int per = (ntiles + 1023) / 1024;
  for (int k = 0; k < kinds; ++k) {
    int* c = counts + k * ntiles;
    const int lo = min(threadIdx.x * per, ntiles), hi = min(lo + per, ntiles);
    int s = 0;
    for (int i = lo; i < hi; ++i) s += c[i];
    sums[threadIdx.x] = s;
    __syncthreads();
    for (int o = 1; o < 1024; o <<= 1) {
      const int v = threadIdx.x >= o ? sums[threadIdx.x - o] : 0;
      __syncthreads();
      sums[threadIdx.x] += v;
      __syncthreads();
    }
    int at = sums[threadIdx.x] - s;
    for (int i = lo; i < hi; ++i) {
      const int v = c[i];
      c[i] = at;
      at += v;
    }
    if (threadIdx.x == 1023) scal[S_NFLUID + k] = (unsigned long long)sums[1023];
    __syncthreads();
  }
}

// Reservoir nodes i .. i + 31 of an instance: densities of the step, potentials
// and codes.
template <class TF, class R>
__device__ __noinline__ void reservoir_pot(const DevInst* I, int cur, unsigned long long step, int i) {
  i += threadIdx.x & 31;
  if (i >= I->nres) return;
  const DevParams& P = I->P;
  const int node = I->reslist[i];
  const uint8_t* tin = I->type[cur];
  const uint8_t t = tin[node] & T_MASK;
  const R theta = theta_of<R>(I);
  double a, b;
  reservoir_rho(P, t, step, t == T_OUTLET && outlet_up_liquid<R, TF>(P, tin, (const TF*)I->f[cur], node, theta), a, b);
  unsigned status = 0;
  R ps, p1, p2;
  potentials<R>(P, R(a), R(b), ps, p1, p2, status);
  ((Pot<R>*)I->pot)[node] = Pot<R>{ps, p1, p2, R(0)};
  I->code[node] = (uint8_t)(C_RES | (R(a) > theta ? C_MARK : 0));
  if (status) atomicOr(&I->scal[S_STATUS], (unsigned long long)status);
}

// Bound by its reads: 18 populations a node in, 16 bytes (FP64 32), a code and a type
// out; in FP64 by the equation of state and the exponentials.  A kernel of its own
// because one that also collides had to hold or recompute the ring of neighbours:
// 1,522 warp instructions and a block barrier per 32 nodes, 77 us at 1024x512 FP32
// (FP64 460), where k_pot and k_move take 39 (FP64 254) together (between events, on a
// lattice that the step before has left in L2 as far as it fits).
template <class TF, class R, int MODE>
__global__ void __launch_bounds__(ST_THREADS, sizeof(R) == 8 ? 4 : 8)
    k_pot(const Work* __restrict__ work, int nwork, int nstream, const DevInst* __restrict__ insts,
          const __grid_constant__ DevInst Ik) {
  step_begin();
  const int lane = threadIdx.x & 31;
  Work wk;
  if (!step_work(MODE == M_SINGLE, work, nwork, nstream, blockIdx.x * ST_WARPS + (threadIdx.x >> 5), wk)) return;
  const DevInst& I = MODE == M_SINGLE ? Ik : insts[wk.inst];
  const DevParams& P = I.P;
  const DevParams& Q = MODE == M_MIXED ? P : Ik.P;
  unsigned long long* scal = I.scal;
  const int* flist = I.flist;
  const int head = flist[min(wk.first + lane, (int)I.N - 1)];   // in flight beside the counters
  const unsigned long long step = scal[S_STEP];
  const bool live = step < scal[S_LIMIT];   // else a frozen instance
  const int cur = int(step & 1ULL);
  if (wk.res >= 0) {
    if (live) reservoir_pot<TF, R>(insts + wk.inst, cur, step, wk.res);
    return;
  }
  if (!live) return;
  const int n = (int)scal[S_NFLUID];
  const R theta = theta_of<R>(&I);
  const TF* fin = (const TF*)I.f[cur];
  const uint8_t* tin = I.type[cur];
  uint8_t* __restrict__ tout = I.type[cur ^ 1];
  Pot<R>* __restrict__ pot = (Pot<R>*)I.pot;
  uint8_t* __restrict__ code = I.code;
  TileAcc<R> acc{R(-1.0 / 0.0), 0u};
  {
    // the next node's populations are in flight while a lane reduces one
    R q[18];
    int next = wk.first + lane < n ? head : -1;
    uint8_t tnext = 0;
    auto fetch = [&] {
      if (next < 0) return;
      tnext = tin[next] & T_MASK;
      const TF* fi = fin + foff(next);
#pragma unroll
      for (int a = 0; a < 18; ++a) q[a] = ld<R>(fi + a * CELL);
    };
    fetch();
#pragma unroll 1
    for (int i = wk.first + lane; i < n; i += wk.stride) {
      const int node = next;
      const int t = tnext;
      R d1 = q[0], d2 = q[9];
#pragma unroll
      for (int a = 1; a < 9; ++a) {
        d1 += q[a];
        d2 += q[9 + a];
      }
      next = i + wk.stride < n ? flist[i + wk.stride] : -1;
      fetch();
      if (!is_fluid(t)) continue;     // filled since it was listed
      R r1 = d1, r2 = d2;
      if constexpr (sizeof(R) == 4) {      // FP64 stores no shift
        r1 = fshift<R>(Q, 0, t) + d1;
        r2 = fshift<R>(Q, 1, t) + d2;
      }
      const bool nan1 = is_nan<R>(r1);
      if (nan1 || is_nan<R>(r2)) acc.status |= ST_NONFINITE;
      if (!nan1 && above<R>(r1, acc.mx)) acc.mx = r1;
      R ps, p1, p2;
      potentials<R>(Q, r1, r2, ps, p1, p2, acc.status);
      const bool liq = !nan1 && above<R>(r1, theta);
      pot[node] = Pot<R>{ps, p1, p2, r1};
      code[node] = (uint8_t)(type_code(t) | (liq ? (C_MARK | C_FLIQ) : C_FGAS));
      tout[node] = liq ? T_LIQUID : T_GAS;
    }
  }
  __syncwarp();
  flush_acc(acc, scal, cur);
}

// Reservoir node: push its equilibrium
// state, densities r1 and r2, into its fluid neighbours and the solute
// equilibrium into its liquid ones.
template <class R, class TF, class TG, int NS>
__device__ __forceinline__ void reservoir_push_node(const DevParams& P, const uint8_t* tin, const TF* fin, const TG* gin,
                                                 TF* fout, TG* gout, int x, int y, uint8_t t, R r1, R r2,
                                                 unsigned nbits, bool marked) {
  R ux = R(0), uy = R(0);
  int xn, yn;
  const int dx = (t == T_INLET) ? P.in_dx : P.out_dx, dy = (t == T_INLET) ? P.in_dy : P.out_dy;
  if (nbr(P, x, y, dx, dy, xn, yn)) {
    const int nn = yn * P.nx + xn;
    const uint8_t tnn = tin[nn] & T_MASK;
    if (is_fluid(tnn)) {
      R q1[9], q2[9];
      const TF* fi = fin + foff(nn);
#pragma unroll
      for (int a = 0; a < 9; ++a) {
        q1[a] = ld<R>(fi + a * CELL);
        q2[a] = ld<R>(fi + (9 + a) * CELL);
      }
      R e1 = q1[0], e2 = q2[0];
#pragma unroll
      for (int a = 1; a < 9; ++a) { e1 += q1[a]; e2 += q2[a]; }
      const R jx = (q1[1] - q1[3]) + (q1[5] - q1[6]) + (q1[8] - q1[7]) + (q2[1] - q2[3]) + (q2[5] - q2[6]) +
                   (q2[8] - q2[7]);
      const R jy = (q1[2] - q1[4]) + (q1[5] - q1[8]) + (q1[6] - q1[7]) + (q2[2] - q2[4]) + (q2[5] - q2[8]) +
                   (q2[6] - q2[7]);
      const R rt = (fshift<R>(P, 0, tnn) + e1) + (fshift<R>(P, 1, tnn) + e2);
      ux = jx / rt;
      uy = jy / rt;
    }
  }
  const R uu = half_u2<R>(ux, uy);
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    const R rho = s == 0 ? r1 : r2;
    TF* fo = fout + s * 9 * CELL;
#pragma unroll
    for (int a = 1; a < 9; ++a) {
      const unsigned c = nbits >> (4 * (a - 1));
      if (!(c & C_FLUID)) continue;
      // stored relative to the shift of the receiving node's new phase
      const R dr = rho - ((c & C_MARK) ? rp<R>(P).shift_f[s] : rp<R>(P).shift_fg[s]);
      const R eu = R(EX(a)) * ux + R(EY(a)) * uy;   // exact: e has components 0, +-1
      const R feq = feq_shifted<R>(w9<R>(a), dr, rho, eu, uu);
      nbr(P, x, y, EX(a), EY(a), xn, yn);
      st<TF, R>(fo + a * CELL + foff(yn * P.nx + xn), feq);
    }
  }
  if constexpr (NS > 0) {
    if (marked) {
      R Cr[NS];
#pragma unroll
      for (int k = 0; k < NS; ++k) Cr[k] = rp<R>(P).conc_in[k];
      if (t == T_OUTLET) {
        // the upstream node: west (direction 3) or south (direction 4)
        const unsigned cu = nbits >> (4 * ((P.out_dx != 0 ? 3 : 4) - 1));
#pragma unroll
        for (int k = 0; k < NS; ++k) Cr[k] = R(0);
        if ((cu & (C_FLUID | C_MARK)) == (C_FLUID | C_MARK) && nbr(P, x, y, P.out_dx, P.out_dy, xn, yn))
          conc_at<R, TG, NS>(gin, yn * P.nx + xn, P, Cr);
      }
#pragma unroll
      for (int k = 0; k < NS; ++k) {
        const R Ja = rp<R>(P).Ja[k];
#pragma unroll
        for (int a = 1; a < 5; ++a) {
          const unsigned c = nbits >> (4 * (a - 1));
          if ((c & (C_FLUID | C_MARK)) != (C_FLUID | C_MARK)) continue;
          const R eu = R(EX(a)) * ux + R(EY(a)) * uy;   // exact
          const R geq = geq_shifted<R>(Ja, Cr[k], rp<R>(P).shift_c[k], eu);
          nbr(P, x, y, EX(a), EY(a), xn, yn);
          gst<TG, R>(P, k, gout + (k * 5 + a) * CELL + goff<NS>(yn * P.nx + xn), geq);
        }
      }
    }
  }
}

// Reservoir nodes i .. i + 31 of an instance push their state of this step into
// their neighbours.
template <class TF, class TG, class R, int NS>
__device__ __noinline__ void reservoir_push(const DevInst* I, int cur, unsigned long long step, int i) {
  i += threadIdx.x & 31;
  if (i >= I->nres) return;
  const DevParams& P = I->P;
  const int node = I->reslist[i];
  const uint8_t* tin = I->type[cur];
  const TF* fin = (const TF*)I->f[cur];
  const uint8_t t = tin[node] & T_MASK;
  const R theta = theta_of<R>(I);
  const int x = node % P.nx, y = node / P.nx;
  unsigned nbits = 0u;
#pragma unroll
  for (int a = 1; a < 9; ++a) {
    int xn, yn;
    if (nbr(P, x, y, EX(a), EY(a), xn, yn)) nbits |= unsigned(I->code[yn * P.nx + xn] & 0xF) << (4 * (a - 1));
  }
  double r1, r2;
  reservoir_rho(P, t, step, t == T_OUTLET && outlet_up_liquid<R, TF>(P, tin, fin, node, theta), r1, r2);
  reservoir_push_node<R, TF, TG, NS>(P, tin, fin, (const TG*)I->g[cur], (TF*)I->f[cur ^ 1], (TG*)I->g[cur ^ 1], x, y, t,
                                     R(r1), R(r2), nbits, (I->code[node] & C_MARK) != 0);
}

// Bound by memory latency in FP32 (18 + 5 NS populations and nine potentials in, the
// populations out; 128 registers, so 16 warps an SM at most, and more warps at fewer
// registers measured slower), by the FP64 pipe in FP64, where an instruction of a warp
// takes 64 cycles however many lanes are in: hence no BGK difference at tau = 1, the
// density from k_pot, few comparisons, and lists without idle lanes (1024x512 FP64: 322 us
// a step before, 265 now).  Forms with fewer roundings to share out between directions
// were faster (228) and further from 64 bits: FP64 and FP32 keep the order and the
// rounding of the equations.
// Everything that depends on the node alone is loaded before the first use; the loop
// stays within the instruction cache (nothing rare inline but the Step-2 amendment).
template <class TF, class TG, class R, int NS, int MODE>
__global__ void __launch_bounds__(ST_THREADS, sizeof(R) == 8 ? 2 : 4)
    k_move(const Work* __restrict__ work, int nwork, int nstream, const DevInst* __restrict__ insts,
           const __grid_constant__ DevInst Ik) {
  using PR = Pair<R>;
  constexpr unsigned FULL = 0xffffffffu;
  constexpr int NP = (NS + 1) / 2, NPX = NP > 0 ? NP : 1;
  step_begin();
  const int lane = threadIdx.x & 31;
  Work wk;
  if (!step_work(MODE == M_SINGLE, work, nwork, nstream, blockIdx.x * ST_WARPS + (threadIdx.x >> 5), wk)) return;
  const DevInst& I = MODE == M_SINGLE ? Ik : insts[wk.inst];
  const DevParams& P = I.P;
  const DevParams& Q = MODE == M_MIXED ? P : Ik.P;
  const DevParamsR<R>& rates = rp<R>(P);
  auto pr = [](const R& v) { return MODE == M_SINGLE ? v : __ldg(&v); };
  const int* flist = I.flist;
  const int head = flist[min(wk.first + lane, (int)I.N - 1)];   // in flight beside the counters
  const unsigned long long step = I.scal[S_STEP];
  const bool live = step < I.scal[S_LIMIT];   // else a frozen instance
  const int cur = int(step & 1ULL);
  if (wk.res >= 0) {
    if (live) reservoir_push<TF, TG, R, NS>(insts + wk.inst, cur, step, wk.res);
    return;
  }
  if (!live) return;
  const int n = (int)I.scal[S_NFLUID];
  const TF* fin = (const TF*)I.f[cur];
  TF* __restrict__ fout = (TF*)I.f[cur ^ 1];
  const TG* gin = (const TG*)I.g[cur];
  TG* __restrict__ gout = (TG*)I.g[cur ^ 1];
  const Pot<R>* pot = (const Pot<R>*)I.pot;
  const uint8_t* code = I.code;
  const int nx = P.nx, ny = P.ny;
  const bool px = P.px != 0, py = P.py != 0;
  auto spec = [&](const R* v, int k) { return mk<R>(v[2 * k], v[2 * k + 1]); };
  // populations are read for the last time in this step
  const unsigned long long once = MODE == M_SINGLE && Ik.read_once ? l2_evict_first() : l2_evict_normal();

  int next = wk.first + lane < n ? head : -1;
#pragma unroll 1
  for (int b = wk.first; b < n; b += wk.stride) {
  const int node = next < 0 ? 0 : next;
  const bool in_list = next >= 0;
  next = b + wk.stride + lane < n ? flist[b + wk.stride + lane] : -1;
  // all loads that depend on the node alone go out together
  PR F[9];      // populations of the two components
  {
    const TF* fi = fin + foff(node);
#pragma unroll
    for (int a = 0; a < 9; ++a) F[a] = mk<R>(ld_l2<R>(fi + a * CELL, once), ld_l2<R>(fi + (9 + a) * CELL, once));
  }
  const int c0 = code[node];
  const int y = node_row(P, node), x = node - y * nx;
  // ---- neighbours: index offsets (with periodic wrap) and codes (outside a
  // non-periodic edge a wall)
  const bool vl = x > 0 || px, vr = x + 1 < nx || px, vd = y > 0 || py, vu = y + 1 < ny || py;
  const int ol = x > 0 ? -1 : nx - 1, orr = x + 1 < nx ? 1 : 1 - nx;
  const int od = y > 0 ? -nx : (ny - 1) * nx, ou = y + 1 < ny ? nx : -(ny - 1) * nx;
  int dn[9], nc[9];
  dn[0] = 0;
  nc[0] = c0;
#pragma unroll
  for (int a = 1; a < 9; ++a) {
    dn[a] = (EX(a) > 0 ? orr : EX(a) < 0 ? ol : 0) + (EY(a) > 0 ? ou : EY(a) < 0 ? od : 0);
    const bool in = (EX(a) > 0 ? vr : EX(a) < 0 ? vl : true) && (EY(a) > 0 ? vu : EY(a) < 0 ? vd : true);
    nc[a] = in ? (int)code[node + dn[a]] : 0;
  }
  PR gs[NPX][5];   // solute populations, two species a pair (unused at a node that was gas)
  if constexpr (NS > 0) {
    const TG* gi = gin + goff<NS>(node);
#pragma unroll
    for (int k = 0; k < NP; ++k)
#pragma unroll
      for (int a = 0; a < 5; ++a) {
        const R ga = ld_l2<R>(gi + (2 * k * 5 + a) * CELL, once);
        const R gb = 2 * k + 1 < NS ? ld_l2<R>(gi + ((2 * k + 1) * 5 + a) * CELL, once) : R(0);
        gs[k][a] = mk<R>(ga, gb);
        if constexpr (Is16<TG>::value) gs[k][a] = gs[k][a] * spec(rp<R>(Q).gs_div, k);
      }
  }
  const bool on = in_list && (c0 & C_FLUID);      // else past the end, or filled since it was listed
  const unsigned act = __ballot_sync(FULL, on);
  if (!on) continue;
  const bool liq = (c0 & C_MARK) != 0, was = (c0 & C_OLDLIQ) != 0;
  const uint8_t t = was ? T_LIQUID : T_GAS;
  const int axis = nc[1] | nc[2] | nc[3] | nc[4];
  const int orc = axis | nc[5] | nc[6] | nc[7] | nc[8];
  // ---- force stencils (force_stencils): a non-live neighbour's values are read
  // at its mirror image
  PR sx, sy;      // stencil sums of (psi_1, phi_1)
  R s2x, s2y;     // ... of phi_2
  PR s0;
  R p2c;
  {
    const Pot<R>* pc = pot + node;
    int off[9];
#pragma unroll
    for (int a = 1; a < 9; ++a) {
      const bool lv = (nc[a] & C_LIVE) != 0;
      if (a < 5) {
        off[a] = lv ? dn[a] : 0;
      } else {
        const int ah = EX(a) > 0 ? 1 : 3, av = EY(a) > 0 ? 2 : 4;
        // one live axis neighbour: a flat wall (the other one's offset is 0)
        const bool flat = ((nc[ah] & C_LIVE) != 0) != ((nc[av] & C_LIVE) != 0);
        off[a] = lv ? dn[a] : (flat ? off[ah] + off[av] : 0);
      }
    }
    {
      const Pot<R> q = ld_pot(pc);
      s0 = mk<R>(q.ps, q.p1);
      p2c = q.p2;
    }
    PR v[9];
    R w[9];
#pragma unroll
    for (int a = 1; a < 9; ++a) {
      const Pot<R> q = ld_pot(pc + off[a]);
      v[a] = mk<R>(q.ps, q.p1);
      w[a] = q.p2;
    }
    const PR n9 = mk<R>(R(1.0 / 9.0)), n36 = mk<R>(R(1.0 / 36.0));
    const PR d57 = v[5] - v[7], d86 = v[8] - v[6];
    sx = pfma<R>(n9, v[1] - v[3], n36 * (d57 + d86));
    sy = pfma<R>(n9, v[2] - v[4], n36 * (d57 - d86));
    pair_sums<R>(w, s2x, s2y);
  }
  // ---- moments (Eq. 9)
  PR d, jx, jy;
  PR sh, rho;
  if constexpr (sizeof(R) == 4) {
    d = F[0];
#pragma unroll
    for (int a = 1; a < 9; ++a) d = d + F[a];
    jx = ((F[1] - F[3]) + (F[5] - F[6])) + (F[8] - F[7]);
    jy = ((F[2] - F[4]) + (F[5] - F[8])) + (F[6] - F[7]);
    sh = mk<R>(fshift<R>(Q, 0, t), fshift<R>(Q, 1, t));
    rho = sh + d;
  } else {
    // no shift, and as few FP64 instructions as will do
    R d2 = F[0].b;
#pragma unroll
    for (int a = 1; a < 9; ++a) d2 += F[a].b;
    rho = d = mk<R>(pot_rho1(pot + node), d2);
    const PR q = F[5] - F[7], r = F[8] - F[6];
    jx = (F[1] - F[3]) + (q + r);
    jy = (F[2] - F[4]) + (q - r);
    sh = mk<R>(R(0));
  }
  const R rho1 = rho.a, rho2 = rho.b;
  // ---- forces (Eqs. 11, 14a/b, 16 and the body force; force1, force2)
  PR Fx, Fy;
  {
    const PR m = mk<R>(-rmul<R>(rp<R>(Q).G11, s0.a), -rmul<R>(rp<R>(Q).G21, p2c));
    const R m12 = -rmul<R>(rp<R>(Q).G12, s0.b);
    Fx = m * sx;
    Fy = m * sy;
    Fx.a = rfma<R>(m12, s2x, Fx.a);
    Fy.a = rfma<R>(m12, s2y, Fy.a);
    if (Q.has_w) {
      int ix = 0, iy = 0;   // wall-density sums in units of 1/36
#pragma unroll
      for (int a = 1; a < 9; ++a) {
        const int sw = (nc[a] & C_LIVE) != 0 ? 0 : (a < 5 ? 4 : 1);
        ix += EX(a) * sw;
        iy += EY(a) * sw;
      }
      const PR mw = mk<R>(-rmul<R>(rp<R>(Q).w_adh[0], s0.a), -rmul<R>(rp<R>(Q).w_adh[1], rho2));
      Fx = pfma<R>(mw, mk<R>(rmul<R>(R(ix), R(1.0 / 36.0))), Fx);
      Fy = pfma<R>(mw, mk<R>(rmul<R>(R(iy), R(1.0 / 36.0))), Fy);
    }
    if (Q.has_g) {
      Fx = pfma<R>(rho, mk<R>(rp<R>(Q).gx), Fx);
      Fy = pfma<R>(rho, mk<R>(rp<R>(Q).gy), Fy);
    }
  }
  // ---- velocities (Eqs. 17-19)
  const R it1 = rp<R>(Q).inv_tau[0], it2 = rp<R>(Q).inv_tau[1];
  const R rrt = rrcp<R>(radd<R>(rho1, rho2));
  // both relaxation times 1 (the paper's choice): the same sum, the same bits
  const R rden = Q.tau_unit ? rrt : rrcp<R>(rfma<R>(rho1, it1, rmul<R>(rho2, it2)));
  R urx, ury;
  PR ux, uy;
  {
    const R q1 = is_zero<R>(rho1) ? R(0) : rmul<R>(rp<R>(Q).tau[0], rrcp<R>(rho1));
    const R q2 = is_zero<R>(rho2) ? R(0) : rmul<R>(rp<R>(Q).tau[1], rrcp<R>(rho2));
    const PR q = mk<R>(q1, q2);
    R upx, upy;
    if (sizeof(R) == 8 && Q.tau_unit) {
      upx = rmul<R>(radd<R>(jx.a, jx.b), rrt);
      upy = rmul<R>(radd<R>(jy.a, jy.b), rrt);
      const R h = rmul<R>(R(0.5), rrt);
      urx = rfma<R>(h, radd<R>(Fx.a, Fx.b), upx);
      ury = rfma<R>(h, radd<R>(Fy.a, Fy.b), upy);
    } else {
      upx = u_common<R>(jx.a, jx.b, it1, it2, rden);
      upy = u_common<R>(jy.a, jy.b, it1, it2, rden);
      urx = u_phys<R>(jx.a, jx.b, Fx.a, Fx.b, rrt);
      ury = u_phys<R>(jy.a, jy.b, Fy.a, Fy.b, rrt);
    }
    ux = pfma<R>(Fx, q, mk<R>(upx));
    uy = pfma<R>(Fy, q, mk<R>(upy));
  }
  // ---- solutes: concentration with the Step-2 amendment, sources
  PR S = mk<R>(R(0));      // fluid sources
  PR C[NPX], Sk[NPX];
  if constexpr (NS > 0) {
    if (liq) {
      bool vnb = false;
#pragma unroll
      for (int b = 1; b < 5; ++b) vnb |= (nc[b] & (C_OLDLIQ | C_MARK)) == C_OLDLIQ;
      if (!was || vnb) {
        // Section 4.5 amendment (rare): dC receives the solute handed over by
        // vanishing (liquid -> gas) neighbours, each giving C / (number of its
        // liquid neighbours); an appearing (gas -> liquid) node takes the mean C
        // of its surviving liquid neighbours (0 if none)
        R dC[2 * NPX], cb[2 * NPX];
#pragma unroll
        for (int k = 0; k < 2 * NPX; ++k) dC[k] = cb[k] = R(0);
        int nsrc = 0;
#pragma unroll 1
        for (int q = 1; q < 5; ++q) {
          const int cq = q == 1 ? nc[1] : q == 2 ? nc[2] : q == 3 ? nc[3] : nc[4];
          if (!(cq & C_OLDLIQ)) continue;
          const int nn = node + (q == 1 ? dn[1] : q == 2 ? dn[2] : q == 3 ? dn[3] : dn[4]);
          R Cn[NS];
          if (cq & C_MARK) {
            if (was) continue;
            conc_at<R, TG, NS>(gin, nn, P, Cn);
#pragma unroll
            for (int k = 0; k < NS; ++k) cb[k] += Cn[k];
            ++nsrc;
          } else {
            int nrec = 0;
            const int yn = node_row(P, nn), xn = nn - yn * nx;
            if (xn > 0 || px) nrec += (code[nn + (xn > 0 ? -1 : nx - 1)] & C_FLIQ) ? 1 : 0;
            if (xn + 1 < nx || px) nrec += (code[nn + (xn + 1 < nx ? 1 : 1 - nx)] & C_FLIQ) ? 1 : 0;
            if (yn > 0 || py) nrec += (code[nn + (yn > 0 ? -nx : (ny - 1) * nx)] & C_FLIQ) ? 1 : 0;
            if (yn + 1 < ny || py) nrec += (code[nn + (yn + 1 < ny ? nx : -(ny - 1) * nx)] & C_FLIQ) ? 1 : 0;
            conc_at<R, TG, NS>(gin, nn, P, Cn);
#pragma unroll
            for (int k = 0; k < NS; ++k) dC[k] += Cn[k] / R(nrec);
          }
        }
#pragma unroll
        for (int k = 0; k < NS; ++k) cb[k] = nsrc ? cb[k] / R(nsrc) : R(0);
#pragma unroll
        for (int k = 0; k < NP; ++k) {
          const PR J0 = spec(rp<R>(Q).J0, k), Ja = spec(rp<R>(Q).Ja, k), sc = spec(rp<R>(Q).shift_c, k);
          const PR dk = spec(dC, k), ck = spec(cb, k);
#pragma unroll
          for (int a = 0; a < 5; ++a) {
            const PR ja = a == 0 ? J0 : Ja;
            const PR m = ja * sc;
            gs[k][a] = was ? pfma<R>(ja, dk, gs[k][a]) : pfma<R>(ja, ck + dk, mk<R>(-m.a, -m.b));
          }
        }
      }
#pragma unroll
      for (int k = 0; k < NP; ++k) {
        PR s = gs[k][0];
#pragma unroll
        for (int a = 1; a < 5; ++a) s = s + gs[k][a];
        C[k] = sizeof(R) == 8 ? s : spec(rp<R>(Q).shift_c, k) + s;
      }
      // homogeneous reactions (Eqs. 5a, 5c; sources Eqs. 27, 28)
      R CA = R(0), CB = R(0), CE = R(0), tot = R(0);
#pragma unroll
      for (int k = 0; k < NS; ++k) {
        const R ck = (k & 1) ? C[k / 2].b : C[k / 2].a;
        if (k == Q.iA) CA = ck;
        if (k == Q.iB) CB = ck;
        if (k == Q.iE) CE = ck;
        tot += ck;
      }
      if (Q.iA == -2) CA = clamp0<R>(rfma<R>(rp<R>(Q).c_total_per_rho1, rho1, -tot));
      // Section 2: R1 is faster at the surface of D(s) (a liquid node with a
      // D(s) node on an axis link)
      const bool surf = Q.r1_surf && (axis & C_SOLD);
      R R1 = rmul<R>(surf ? pr(rates.k1_s) : pr(rates.k1), CA);
      if (Q.has_rev)
        R1 = rsub<R>(R1, rmul<R>(rmul<R>(surf ? pr(rates.k1_inv_Keq_s) : pr(rates.k1_inv_Keq), CB),
                                 rsqrt_<R>(rmax<R>(rmul<R>(rho2, rp<R>(Q).inv_M_C), R(0)))));
      const R R3 = rmul<R>(rmul<R>(pr(rates.k3), CB), CE);
#pragma unroll
      for (int k = 0; k < NP; ++k)
        Sk[k] = pfma<R>(spec(rp<R>(Q).cR1, k), mk<R>(R1), spec(rp<R>(Q).cR3, k) * mk<R>(R3));
      const R y1 = rmul<R>(rp<R>(Q).gas_yield, R1);
      S = mk<R>(-y1, y1);
    }
  }

  // ---- fluid collision (Eq. 6, Eq. 8 at u_eq) and push streaming: into the
  // fluid neighbour's slot a, or bounced back into slot OPP(a) here.  Nothing is
  // stored into a reservoir, and FP32 populations are stored relative to the
  // receiving node's new phase: both concern few nodes (odd)
  {
    bool odd = (orc & C_RES) != 0;
    if constexpr (sizeof(R) == 4) odd = odd || ((orc | c0) & (was ? C_FGAS : C_FLIQ)) != 0;
    odd = __any_sync(act, odd);
    const int fo0 = foff(node);
    int to[9];
    to[0] = fo0;
#pragma unroll
    for (int a = 1; a < 9; ++a) to[a] = (nc[a] & C_FLUID) ? foff(node + dn[a]) + a * CELL : fo0 + OPP(a) * CELL;
#pragma unroll
    for (int s = 0; s < 2; ++s) {
      const bool c1 = s == 0;
      const R rs = c1 ? rho.a : rho.b, ds = c1 ? d.a : d.b, vx = c1 ? ux.a : ux.b, vy = c1 ? uy.a : uy.b,
              Ss = c1 ? S.a : S.b, it = c1 ? it1 : it2;
      TF* fo = fout + s * 9 * CELL;
      R feq[9];
      feq_pairs<R>(ds, rs, vx, vy, half_u2<R>(vx, vy), feq);
      if (sizeof(R) == 8 && Q.tau_unit) {
        // FP64 at tau = 1: the collision leaves the equilibrium, and a liquid node's
        // source.  Each direction is rounded by itself: with rho (1 - 1.5 u^2) + S
        // formed once for all nine (30 instructions instead of 44, 64 with the BGK
        // difference) the nine errors had one sign, and the beaker's densities were
        // 2.2e-15 off after 200 steps instead of 5.2e-16
        if constexpr (NS > 0) {
          if (liq) {
#pragma unroll
            for (int a = 0; a < 9; ++a) feq[a] = rfma<R>(w9<R>(a), Ss, feq[a]);
          }
        }
      } else {
#pragma unroll
        for (int a = 0; a < 9; ++a) feq[a] = bgk<R>(c1 ? F[a].a : F[a].b, feq[a], it, w9<R>(a), Ss);
      }
      if (!odd) {
#pragma unroll
        for (int a = 0; a < 9; ++a) st<TF, R>(fo + to[a], feq[a]);
      } else {
        const R shs = c1 ? sh.a : sh.b;
        const R dl = shs - rp<R>(Q).shift_f[s], dg = shs - rp<R>(Q).shift_fg[s];
#pragma unroll
        for (int a = 0; a < 9; ++a) {
          const bool to_liq = (a > 0 && (nc[a] & C_FLUID)) ? (nc[a] & C_MARK) != 0 : liq;
          if (a == 0 || !(nc[a] & C_RES))
            st<TF, R>(fo + to[a], sizeof(R) == 8 ? feq[a] : rfma<R>(w9<R>(a), to_liq ? dl : dg, feq[a]));
        }
      }
    }
  }

  // ---- solute collision (Eqs. 20-22 with u_r) and push streaming
  if constexpr (NS > 0) {
    const int go0 = goff<NS>(node);
    auto put = [&](int k, int to, PR v) {
      gst<TG, R>(Q, 2 * k, gout + 2 * k * 5 * CELL + to, v.a);
      if (2 * k + 1 < NS) gst<TG, R>(Q, 2 * k + 1, gout + (2 * k + 1) * 5 * CELL + to, v.b);
    };
    if (liq) {
      // into a liquid neighbour, out into a liquid reservoir (not stored), or
      // bounced back here (no-flux / mineral link)
      int to[5];
      to[0] = go0;
#pragma unroll
      for (int a = 1; a < 5; ++a) to[a] = (nc[a] & C_FLIQ) ? goff<NS>(node + dn[a]) + a * CELL : go0 + OPP(a) * CELL;
      const PR vx = mk<R>(urx), vy = mk<R>(ury);
#pragma unroll
      for (int k = 0; k < NP; ++k) {
        const PR J0 = spec(rp<R>(Q).J0, k), Ja = spec(rp<R>(Q).Ja, k), it = spec(rp<R>(Q).inv_tau_g, k);
        PR go[5];
        // FP64 (no shift) too: as (1 - 1/tau_g) g + J (C / tau_g + S) + ... it took 13
        // instructions a species instead of 24, but the two weights of g and C did not
        // add up to 1 for tau_g > 2, and the largest error of the plain scene was 1.6 times this one's
        const PR cs = sizeof(R) == 8 ? C[k] : C[k] - spec(rp<R>(Q).shift_c, k), hc = mk<R>(R(0.5)) * C[k];
        const PR sa = Ja * cs, ax = hc * vx, ay = hc * vy;
        const PR ge[5] = {J0 * cs, sa + ax, sa + ay, sa - ax, sa - ay};
#pragma unroll
        for (int a = 0; a < 5; ++a) go[a] = pfma<R>(a == 0 ? J0 : Ja, Sk[k], pfma<R>(ge[a] - gs[k][a], it, gs[k][a]));
#pragma unroll
        for (int a = 0; a < 5; ++a)
          if (a == 0 || (nc[a] & (C_RES | C_MARK)) != (C_RES | C_MARK)) put(k, to[a], go[a]);
      }
    } else {
      // gas node: no solute
#pragma unroll
      for (int k = 0; k < NP; ++k)
#pragma unroll
        for (int a = 0; a < 5; ++a) {
          const PR v = spec(a == 0 ? rp<R>(Q).J0 : rp<R>(Q).Ja, k) * spec(rp<R>(Q).shift_c, k);
          put(k, a * CELL + go0, mk<R>(-v.a, -v.b));
        }
    }
  }
  }
}

}  // namespace pslbm
