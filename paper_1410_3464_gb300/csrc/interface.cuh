// Interface kernels of one time step (Chen, Kang et al., arXiv 1410.3464):
//   k_vop   -- heterogeneous reactions at liquid-mineral links (Eqs. 29-31)
//              and the volume-of-pixel update (Eqs. 32-35, Step 4) with the
//              status decisions (dissolution, precipitation overflow);
//   k_amend -- status changes and the amendment of Step 5 (Section 4.5) at
//              flipped nodes, one block per instance; it ends the step.
// Every gather runs in the fixed order E, N, W, S, so the result does not
// depend on thread scheduling.
#pragma once
#include "step.cuh"

namespace pslbm {

// k_move bounces every solute population that leaves a liquid node
// toward a mineral back into the node (halfway bounce-back).  At a reactive
// link this kernel replaces the bounced value by the reactive link rule: with
// the outgoing population `out`, J_w = (1 - J0)/4 and kappa = k / (2 J_w),
// the returning population is (out (1 - kappa) + k C_sat) / (1 + kappa) and the
// link flux q = out - back is the amount consumed (B by R2 at D(s), F by R4 at
// D(s) or F(s)); E gains the B consumed on the same link.  The flux is computed
// directly, q = out 2 kappa / (1 + kappa) - k C_sat / (1 + kappa), since out and
// back differ by a relative 2 kappa only.  Then V_D -= Vbar_D
// sum q_B, V_F += Vbar_F sum q_F, and the node dissolves, overflows or changes
// between D(s) and F(s).
//
// Only minerals with a liquid axis neighbour change.  The kernel runs over the
// instance's list of minerals that face fluid, a lane a mineral, and sees from
// the codes of this step which of the neighbours are liquid.  Bound by the latency
// of its scattered reads (codes, volumes, then the bounced slots): the list costs
// one round trip, where a bitmap that the streaming kernel marked took three and an
// atomic per mineral link (4096x2048 94 -> 61 us, 24 geometries 62 -> 34).
template <class TF, class TG, class R, int NS>
__device__ __forceinline__ void vop_node(const DevInst* Ip, const DevParams& P, int N, int cur,
                                         unsigned long long step, int node) {
  double* __restrict__ V = Ip->V;
  uint8_t* __restrict__ code = Ip->code;
  // independent loads first: own code, volumes, the four neighbour codes
  const int c0 = code[node];
  double VD = V[node], VF = V[N + node];
  const int y = node_row(P, node), x = node - y * P.nx;
  int nbx[4];
#pragma unroll
  for (int b = 1; b < 5; ++b) {
    int xn = x + EX(b), yn = y + EY(b);
    bool in = true;
    if (xn < 0 || xn >= P.nx) {
      in = P.px != 0;
      xn = xn < 0 ? P.nx - 1 : 0;
    }
    if (yn < 0 || yn >= P.ny) {
      in = in && P.py != 0;
      yn = yn < 0 ? P.ny - 1 : 0;
    }
    nbx[b - 1] = in ? yn * P.nx + xn : -1;
  }
  int cn[4];
#pragma unroll
  for (int b = 0; b < 4; ++b) cn[b] = nbx[b] >= 0 ? code[nbx[b]] : 0;
  if (!(c0 & C_MIN)) return;      // dissolved since it was listed
  const uint8_t t = (c0 & C_SOLD) ? T_SOLID_D : T_SOLID_F;
  int nl = 0;
  int dirs[4];
#pragma unroll
  for (int b = 1; b < 5; ++b) {
    if (!(cn[b - 1] & C_FLIQ)) nbx[b - 1] = -1;
    else dirs[nl++] = b;
  }
  if (nl == 0) return;
  R sB = R(0), sF = R(0);
  if constexpr (NS > 0) {
    TG* __restrict__ gout = (TG*)Ip->g[cur ^ 1];
    const bool useB = (t == T_SOLID_D) && P.useB;
    const bool useF = P.useF != 0;
    // the population that left neighbour nn toward this node was bounced into
    // slot b of nn; gather every slot before writing any
    R oB[4], oE[4], oF[4];
#pragma unroll
    for (int b = 1; b < 5; ++b) {
      const int nn = nbx[b - 1];
      oB[b - 1] = oE[b - 1] = oF[b - 1] = R(0);
      if (nn < 0) continue;
      if (useB) {
        oB[b - 1] = gld<R>(P, P.iB, gout + goff<NS>(nn) + (P.iB * 5 + b) * CELL);
        if (P.iE >= 0) oE[b - 1] = gld<R>(P, P.iE, gout + goff<NS>(nn) + (P.iE * 5 + b) * CELL);
      }
      if (useF) oF[b - 1] = gld<R>(P, P.iF, gout + goff<NS>(nn) + (P.iF * 5 + b) * CELL);
    }
#pragma unroll
    for (int b = 1; b < 5; ++b) {
      const int nn = nbx[b - 1];
      if (nn < 0) continue;
      if (useB) {
        const int iB = P.iB;
        const R sh = rp<R>(P).vB_sh;
        const R out = radd<R>(oB[b - 1], sh);
        const R q = rmul<R>(out, rp<R>(P).vB_qa);
        const R bk = rsub<R>(out, q);
        gst<TG, R>(P, iB, gout + goff<NS>(nn) + (iB * 5 + b) * CELL, rsub<R>(bk, sh));
        sB = radd<R>(sB, q);
        if (P.iE >= 0) gst<TG, R>(P, P.iE, gout + goff<NS>(nn) + (P.iE * 5 + b) * CELL, radd<R>(oE[b - 1], q));
      }
      if (useF) {
        const int iF = P.iF;
        const R sh = rp<R>(P).vF_sh;
        const R out = radd<R>(oF[b - 1], sh);
        const R q = rfma<R>(out, rp<R>(P).vF_qa, -rp<R>(P).vF_qc);
        gst<TG, R>(P, iF, gout + goff<NS>(nn) + (iF * 5 + b) * CELL, rsub<R>(rsub<R>(out, q), sh));
        sF = radd<R>(sF, q);
      }
    }
  }
  // volumes accumulate in FP64: per-step increments are far below FP32 resolution of V
  if (t == T_SOLID_D) VD = __fma_rn(-P.Vbar_D, double(sB), VD);   // Eq. 33
  VF = __fma_rn(P.Vbar_F, double(sF), VF);                        // Eq. 35 (precipitation adds volume)
  if (VD < 0.0) VD = 0.0;
  const double total = VD + VF;
  int ev = EV_NONE;
  if (total <= 0.0) {
    VD = 0.0;
    VF = 0.0;
    ev = EV_DISSOLVE;
  } else {
    const bool sd = VD > 0.0;
    if (sd != (t == T_SOLID_D)) {
      // a solid's type and code change here and in the amendment kernel only, in
      // both type buffers
      Ip->type[0][node] = Ip->type[1][node] = sd ? T_SOLID_D : T_SOLID_F;
      code[node] = (uint8_t)(sd ? C_MIN | C_SOLD : C_MIN);
    }
    if (total >= P.V_split) {
      const double excess = total - 1.0;
      VF = VF - excess;
      const unsigned long long key = P.seed ^ (step << 40) ^ (unsigned long long)node;
      const int pick = int(splitmix64(key) % (unsigned long long)nl);
      ev = EV_OVERFLOW | (dirs[pick] << 4);
      Ip->xs[node] = excess;
    }
  }
  V[node] = VD;
  V[N + node] = VF;
  if (ev != EV_NONE) {
    Ip->evt[node] = (uint8_t)ev;
    const unsigned long long slot = atomicAdd(&Ip->scal[S_NEVENT], 1ULL);
    if (slot < (unsigned long long)Ip->evcap)
      Ip->evlist[slot] = node;
    else
      atomicOr(&Ip->scal[S_STATUS], (unsigned long long)ST_EVOVERFLOW);
  }
}

// Blocks per SM the VOP kernel's register budget targets: five in FP32, four in
// FP64 (twice the registers per value).
template <class R>
constexpr int vop_min_blocks() {
  return sizeof(R) == 8 ? 4 : 5;
}

// A warp per work entry: work[w] of a batch, or the w-th 32 entries of the only
// instance's list; both again every `stride` entries as far as the list goes.
template <class TF, class TG, class R, int NS>
__global__ void __launch_bounds__(NTHREADS, vop_min_blocks<R>())
    k_vop(const DevInst* __restrict__ insts, const Work* __restrict__ work, int nwork) {
  step_begin();
  const int lane = threadIdx.x & 31;
  const int w = (blockIdx.x * (int)blockDim.x + threadIdx.x) >> 5;
  if (w >= nwork) return;
  const Work wk = work ? work[w] : Work{0, w * 32, nwork * 32, -1};
  const DevInst* Ip = insts + wk.inst;
  const int N = (int)Ip->N;
  int node = Ip->mlist[min(wk.first + lane, N - 1)];   // in flight beside the counters
  const unsigned long long step = Ip->scal[S_STEP];
  if (step >= Ip->scal[S_LIMIT]) return;   // frozen instance
  const int n = (int)Ip->scal[S_NFACE];
  for (int i = wk.first + lane; i < n; i += wk.stride) {
    vop_node<TF, TG, R, NS>(Ip, Ip->P, N, int(step & 1ULL), step, node);
    if (i + wk.stride < n) node = Ip->mlist[i + wk.stride];
  }
}

// Append a node to a list unless it is listed (bits).
__device__ __forceinline__ void list_node(unsigned* bits, int* list, unsigned long long* count, int node) {
  const unsigned bit = 1u << (node & 31);
  if (atomicOr(&bits[node >> 5], bit) & bit) return;
  list[(int)atomicAdd(count, 1ULL)] = node;
}

__device__ __forceinline__ bool surv_fluid(uint8_t tf) { return (tf & (T_NEW | T_VANISH)) == 0 && is_fluid(tf & T_MASK); }
__device__ __forceinline__ bool surv_liquid(uint8_t tf) { return tf == T_LIQUID; }

// End of a step for one instance: decode the next step's liquid threshold
// (half the maximum k_pot gathered this step) into both precisions,
// free the slot this step read (it receives the maximum two steps later) and
// advance the step counter.  mx: the encoded maximum of this step's slot,
// S_MAX0 + ((step + 1) & 1).
__device__ __forceinline__ void finish_step(const DevInst* Ip, unsigned long long step, unsigned long long mx) {
  const double th = 0.5 * ord_dec(mx);
  Ip->scal[S_THETA] = (unsigned long long)__double_as_longlong(th);
  Ip->scal[S_THETAF] = (unsigned long long)(unsigned)__float_as_int(float(th));
  Ip->scal[S_MAX0 + int(step & 1ULL)] = 0ULL;
  Ip->scal[S_NEVENT] = 0ULL;
  Ip->scal[S_STEP] = step + 1;
}

// Amendment and end of a step for one instance, by one block.
template <class TF, class TG, class R, int NS>
__device__ __forceinline__ void amend(const DevInst* Ip) {
  // the counters, loaded together (one memory round trip)
  const volatile unsigned long long* sc = Ip->scal;
  const unsigned long long step = sc[S_STEP], limit = sc[S_LIMIT], nev_raw = sc[S_NEVENT], m0 = sc[S_MAX0],
                           m1 = sc[S_MAX1];
  if (step >= limit) return;   // frozen instance
  const unsigned long long mx = (step & 1ULL) ? m0 : m1;
  if (nev_raw == 0) {
    if (threadIdx.x == 0) finish_step(Ip, step, mx);
    return;
  }
  const DevParams& P = Ip->P;
  const long long N = Ip->N;
  const int nev = (int)min(nev_raw, (unsigned long long)Ip->evcap);
  // buffer cur is the state k_move just wrote
  const int cur = int(step & 1ULL) ^ 1;
  TF* F = (TF*)Ip->f[cur];
  TG* G = (TG*)Ip->g[cur];
  uint8_t* T = Ip->type[cur];
  int* vlist = Ip->evlist + Ip->evcap;   // second half: vanishing nodes
  __shared__ int s_nv;
  if (threadIdx.x == 0) s_nv = 0;
  __syncthreads();

  // phase 1: new types; each overflow target sums the excess of its choosers
  for (int i = threadIdx.x; i < nev; i += blockDim.x) {
    const int node = Ip->evlist[i];
    const int code = Ip->evt[node];
    const int x = node % P.nx, y = node / P.nx;
    if ((code & 15) == EV_DISSOLVE) {
      T[node] = T_LIQUID | T_NEW;
    } else if ((code & 15) == EV_OVERFLOW) {
      const int d = code >> 4;
      int xt, yt;
      nbr(P, x, y, EX(d), EY(d), xt, yt);
      const int tgt = yt * P.nx + xt;
      if (atomicCAS(&Ip->claim[tgt], 0, 1) == 0) {
        double acc = 0.0;
#pragma unroll
        for (int b = 1; b < 5; ++b) {
          int xz, yz;
          if (!nbr(P, xt, yt, EX(b), EY(b), xz, yz)) continue;
          const int z = yz * P.nx + xz;
          const int cz = Ip->evt[z];
          if ((cz & 15) != EV_OVERFLOW) continue;
          int xc, yc;
          nbr(P, xz, yz, EX(cz >> 4), EY(cz >> 4), xc, yc);
          if (yc * P.nx + xc == tgt) acc += Ip->xs[z];
        }
        Ip->V[tgt] = 0.0;
        Ip->V[N + tgt] = acc;
        T[tgt] = T_SOLID_F | T_VANISH;
        const int k = atomicAdd(&s_nv, 1);
        vlist[k] = tgt;
      }
    }
  }
  __syncthreads();
  const int nv = s_nv;

  // phase 2: refill dissolved nodes at rest with the mean density of their
  // surviving fluid neighbours and the mean concentration of their surviving
  // liquid neighbours (post-streaming values)
  for (int i = threadIdx.x; i < nev; i += blockDim.x) {
    const int node = Ip->evlist[i];
    if ((Ip->evt[node] & 15) != EV_DISSOLVE) continue;
    const int x = node % P.nx, y = node / P.nx;
    R s1 = R(0), s2 = R(0), sc[NS > 0 ? NS : 1];
#pragma unroll
    for (int k = 0; k < NS; ++k) sc[k] = R(0);
    int nf = 0, nl = 0;
#pragma unroll
    for (int b = 1; b < 5; ++b) {
      int xn, yn;
      if (!nbr(P, x, y, EX(b), EY(b), xn, yn)) continue;
      const long long nn = (long long)yn * P.nx + xn;
      const uint8_t tf = T[nn];
      if (surv_fluid(tf)) {
        s1 += fshift<R>(P, 0, tf) + density_shifted<R>(F, 0, (int)nn);
        s2 += fshift<R>(P, 1, tf) + density_shifted<R>(F, 1, (int)nn);
        ++nf;
      }
      if (surv_liquid(tf)) {
#pragma unroll
        for (int k = 0; k < NS; ++k) {
          const TG* gk = G + goff<NS>((int)nn) + k * 5 * CELL;
          R c = gld<R>(P, k, gk);
#pragma unroll
          for (int a = 1; a < 5; ++a) c += gld<R>(P, k, gk + a * CELL);
          sc[k] += rp<R>(P).shift_c[k] + c;
        }
        ++nl;
      }
    }
    const R r1 = nf ? s1 / R(nf) : rp<R>(P).rho_fill[0];
    const R r2 = nf ? s2 / R(nf) : rp<R>(P).rho_fill[1];
#pragma unroll
    for (int a = 0; a < 9; ++a) {
      const R w = w9<R>(a);
      st<TF, R>(F + foff(node) + a * CELL, rfma<R>(w, r1, -rmul<R>(w, rp<R>(P).shift_f[0])));
      st<TF, R>(F + foff(node) + (9 + a) * CELL, rfma<R>(w, r2, -rmul<R>(w, rp<R>(P).shift_f[1])));
    }
#pragma unroll
    for (int k = 0; k < NS; ++k) {
      const R c = nl ? sc[k] / R(nl) : R(0);
      const R J0 = rp<R>(P).J0[k], Ja = (R(1) - J0) / R(4);
#pragma unroll
      for (int a = 0; a < 5; ++a) {
        const R ja = a == 0 ? J0 : Ja;
        gst<TG, R>(P, k, G + goff<NS>(node) + (k * 5 + a) * CELL, rfma<R>(ja, c, -rmul<R>(ja, rp<R>(P).shift_c[k])));
      }
    }
  }
  __syncthreads();

  // phase 3: surviving neighbours of vanished nodes take equal shares of the
  // vanished node's fluid mass (added at rest) and solute
  for (int i = threadIdx.x; i < nv * 4; i += blockDim.x) {
    const int v = vlist[i >> 2];
    const int b0 = (i & 3) + 1;
    int xr, yr;
    if (!nbr(P, v % P.nx, v / P.nx, EX(b0), EY(b0), xr, yr)) continue;
    const int n = yr * P.nx + xr;
    if (!surv_fluid(T[n])) continue;
    if (atomicCAS(&Ip->claim[n], 0, 2) != 0) continue;
    R add1 = R(0), add2 = R(0), addc[NS > 0 ? NS : 1];
#pragma unroll
    for (int k = 0; k < NS; ++k) addc[k] = R(0);
    const bool nliq = surv_liquid(T[n]);
#pragma unroll
    for (int b = 1; b < 5; ++b) {
      int xv, yv;
      if (!nbr(P, xr, yr, EX(b), EY(b), xv, yv)) continue;
      const long long w = (long long)yv * P.nx + xv;
      if (!(T[w] & T_VANISH)) continue;
      int nf = 0, nl = 0;
#pragma unroll
      for (int c = 1; c < 5; ++c) {
        int xz, yz;
        if (!nbr(P, xv, yv, EX(c), EY(c), xz, yz)) continue;
        const uint8_t tz = T[(long long)yz * P.nx + xz];
        nf += surv_fluid(tz) ? 1 : 0;
        nl += surv_liquid(tz) ? 1 : 0;
      }
      add1 += (fshift<R>(P, 0, T[w]) + density_shifted<R>(F, 0, (int)w)) / R(nf);
      add2 += (fshift<R>(P, 1, T[w]) + density_shifted<R>(F, 1, (int)w)) / R(nf);
      if (nliq && nl) {
#pragma unroll
        for (int k = 0; k < NS; ++k) {
          const TG* gk = G + goff<NS>((int)w) + k * 5 * CELL;
          R c = gld<R>(P, k, gk);
#pragma unroll
          for (int a = 1; a < 5; ++a) c += gld<R>(P, k, gk + a * CELL);
          addc[k] += (rp<R>(P).shift_c[k] + c) / R(nl);
        }
      }
    }
#pragma unroll
    for (int a = 0; a < 9; ++a) {
      const R w = w9<R>(a);
      TF* p1 = F + foff(n) + a * CELL;
      TF* p2 = F + foff(n) + (9 + a) * CELL;
      st<TF, R>(p1, rfma<R>(w, add1, ld<R>(p1)));
      st<TF, R>(p2, rfma<R>(w, add2, ld<R>(p2)));
    }
    if (nliq) {
#pragma unroll
      for (int k = 0; k < NS; ++k) {
        const R J0 = rp<R>(P).J0[k], Ja = (R(1) - J0) / R(4);
#pragma unroll
        for (int a = 0; a < 5; ++a) {
          TG* p = G + goff<NS>(n) + (k * 5 + a) * CELL;
          gst<TG, R>(P, k, p, rfma<R>(a == 0 ? J0 : Ja, addc[k], gld<R>(P, k, p)));
        }
      }
    }
  }
  __syncthreads();

  // phase 4: lists, and the solids' types (both buffers) and codes
  for (int i = threadIdx.x; i < nev; i += blockDim.x) {
    const int node = Ip->evlist[i];
    if ((Ip->evt[node] & 15) != EV_DISSOLVE) continue;
    const int x = node % P.nx, y = node / P.nx;
    list_node(Ip->fbits, Ip->flist, Ip->scal + S_NFLUID, node);
#pragma unroll
    for (int b = 1; b < 5; ++b) {
      int xn, yn;
      if (nbr(P, x, y, EX(b), EY(b), xn, yn) && is_mineral(T[yn * P.nx + xn] & T_MASK))
        list_node(Ip->mbits, Ip->mlist, Ip->scal + S_NFACE, yn * P.nx + xn);
    }
  }
  for (int i = threadIdx.x; i < nv; i += blockDim.x) {
    const int v = vlist[i];
    list_node(Ip->mbits, Ip->mlist, Ip->scal + S_NFACE, v);
    Ip->code[v] = (uint8_t)C_MIN;
    Ip->type[cur ^ 1][v] = T_SOLID_F;
  }
  __syncthreads();
  for (int i = threadIdx.x; i < nv; i += blockDim.x) T[vlist[i]] = T_SOLID_F;
  for (int i = threadIdx.x; i < nev; i += blockDim.x) {
    const int node = Ip->evlist[i];
    if ((Ip->evt[node] & 15) == EV_DISSOLVE) T[node] = T_LIQUID;
  }
  __syncthreads();

  // phase 5: clear the scratch state used by this step
  for (int i = threadIdx.x; i < nv * 4; i += blockDim.x) {
    const int v = vlist[i >> 2];
    int xr, yr;
    if (nbr(P, v % P.nx, v / P.nx, EX((i & 3) + 1), EY((i & 3) + 1), xr, yr)) Ip->claim[yr * P.nx + xr] = 0;
  }
  for (int i = threadIdx.x; i < nv; i += blockDim.x) Ip->claim[vlist[i]] = 0;
  __syncthreads();
  for (int i = threadIdx.x; i < nev; i += blockDim.x) Ip->evt[Ip->evlist[i]] = 0;
  if (threadIdx.x == 0) finish_step(Ip, step, mx);
}

template <class TF, class TG, class R, int NS>
__global__ void __launch_bounds__(NTHREADS) k_amend(const DevInst* __restrict__ insts) {
  step_begin();
  amend<TF, TG, R, NS>(insts + blockIdx.x);
}

// k_vop and k_amend of an instance in one block, for lists that one block can take
// at once (FUSE_FACE).  What the block's threads wrote they read back after a block
// barrier; nothing passes between blocks.  Saves a dependent launch and its round
// trip: 131x67 FP32 12.0 -> 11.4 us a step, 100x160 15.3 -> 14.7, 102x90 FP64 24.0 ->
// 23.4, 201x201 FP64 36.0 -> 35.3.
template <class TF, class TG, class R, int NS>
__global__ void __launch_bounds__(NTHREADS) k_vop_amend(const DevInst* __restrict__ insts) {
  step_begin();
  const DevInst* Ip = insts + blockIdx.x;
  const int N = (int)Ip->N;
  const unsigned long long step = Ip->scal[S_STEP];
  if (step >= Ip->scal[S_LIMIT]) return;   // frozen instance
  const int n = (int)Ip->scal[S_NFACE];    // grows as nodes dissolve
  for (int i = threadIdx.x; i < n; i += blockDim.x)
    vop_node<TF, TG, R, NS>(Ip, Ip->P, N, int(step & 1ULL), step, Ip->mlist[i]);
  __syncthreads();
  amend<TF, TG, R, NS>(Ip);
}

}  // namespace pslbm
