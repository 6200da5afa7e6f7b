// adjoint.cu -- reversible-adjoint backward pass (sm_103a), Sec. "Reverse Mode".
//
// With lambda = dL/dpsi* (Wirtinger) = O psi_N, gates are walked from last to
// first.  With psi and lambda the states right after gate k, a gate
// U = exp(-i theta c H) contributes dL/dtheta = 2 c Im<lambda|H|psi> (H includes
// the control projector), and then both states are uncomputed,
// psi <- U^dag psi, lambda <- U^dag lambda (Eq. apply-back); the outer product
// of Eq. outer-product is never formed, only its contraction with H.
//
// Parameterised gates run one fused pass per gate: each thread loads the
// psi and lambda 2^k-tuples, adds Im sum_m conj(l_m) (G x)_m to its FP64
// partial, applies U^dag to both tuples and stores them.  Block partials land
// in scratch memory and one block folds them pairwise into grad[param] in
// stream order.  The uncompute runs in FP64 (complex128 work buffers) whatever
// the forward precision; checkpoints taken during the forward replace psi at
// segment boundaries so that uncompute drift cannot accumulate across segments.
#include <algorithm>
#include <cmath>
#include <cstring>

#include "common.cuh"

namespace qs {

int expect_raw(const void* data, int dtype, int n, int nreg, const qs_observable* o, qs_state* ws_owner,
               double* host_out);
int apply_observable_c128(const double2* psi, double2* lam, int n, const qs_observable* o, cudaStream_t st);
int promote_to_c128(const void* in, int dtype, double2* out, uint64_t dim, cd f, cudaStream_t st);

constexpr int kAdjThreads = 256;
constexpr int kAdjMaxBlocks = 1216;  // 8 per SM on 152 SMs

template <int K>
struct AdjMat {
  double2 g[1 << (2 * K)];   // generator H on the targets
  double2 ud[1 << (2 * K)];  // U^dagger on the targets
  uint64_t off[1 << K];
};

// Where the gradient of a launch goes: grad[param] += scale * (sum of the CTAs'
// contributions).  Each CTA writes its partial; the CTA that arrives last at
// the counter folds them pairwise in index order (the order does not depend on
// which CTA is last), adds the result and resets the counter for the next
// launch on the stream: no separate fold launch per gate.
struct AdjOut {
  double* partials;   // [gridDim.x]
  unsigned* counter;  // 0 between launches
  double* grad;
  int param;
  double scale;
};

__device__ __forceinline__ void adj_finish(double acc, const AdjOut& out) {
  __shared__ double red[kAdjThreads / 32];
  __shared__ bool last;
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double v = 0.0;
    for (int w = 0; w < kAdjThreads / 32; ++w) v += red[w];
    out.partials[blockIdx.x] = v;
    __threadfence();
    last = atomicAdd(out.counter, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  __shared__ double buf[2048];
  static_assert(kAdjMaxBlocks <= 2048, "one fold buffer");
  for (int i = threadIdx.x; i < 2048; i += blockDim.x) buf[i] = i < (int)gridDim.x ? __ldcg(out.partials + i) : 0.0;
  __syncthreads();
  for (int w = 1024; w > 0; w >>= 1) {
    for (int i = threadIdx.x; i < w; i += blockDim.x) buf[i] += buf[i + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    out.grad[out.param] += out.scale * buf[0];
    *out.counter = 0u;
  }
}

template <int K>
__global__ void __launch_bounds__(kAdjThreads)
k_adjoint_param(double2* __restrict__ psi, double2* __restrict__ lam, uint64_t nitems, IdxSpec s,
                const __grid_constant__ AdjMat<K> M, const AdjOut out) {
  constexpr int D = 1 << K;
  double acc = 0.0;
  for (uint64_t it = (uint64_t)blockIdx.x * kAdjThreads + threadIdx.x; it < nitems;
       it += (uint64_t)gridDim.x * kAdjThreads) {
    const uint64_t base = item_index(it, s);
    double2 x[D], l[D];
#pragma unroll
    for (int m = 0; m < D; ++m) {
      x[m] = psi[base + M.off[m]];
      l[m] = lam[base + M.off[m]];
    }
    // Im sum_m conj(l_m) (G x)_m
#pragma unroll
    for (int m = 0; m < D; ++m) {
      double2 gx = make_double2(0.0, 0.0);
#pragma unroll
      for (int j = 0; j < D; ++j) gx = cfma(M.g[m * D + j], x[j], gx);
      acc += l[m].x * gx.y - l[m].y * gx.x;
    }
#pragma unroll
    for (int m = 0; m < D; ++m) {
      double2 px = make_double2(0.0, 0.0), pl = make_double2(0.0, 0.0);
#pragma unroll
      for (int j = 0; j < D; ++j) {
        px = cfma(M.ud[m * D + j], x[j], px);
        pl = cfma(M.ud[m * D + j], l[j], pl);
      }
      psi[base + M.off[m]] = px;
      lam[base + M.off[m]] = pl;
    }
  }
  adj_finish(acc, out);
}

// Single-target parameterised gates in structured forms (FP64 is scarce on
// this part: the dense 2x2 path spends 64 FP64 multiply-adds per pair):
//   ADJ_DIAG: U^dag = diag(u0, u3), H = diag(g0, g3) real (Rz, shift, phase):
//             ~20 per pair;
//   ADJ_RX:   U^dag = [[c, i s], [i s, c]], H = X (Rx): ~24 per pair.
enum { ADJ_DIAG = 0, ADJ_RX = 1 };

struct AdjForm1 {
  double2 u0, u3;   // ADJ_DIAG: the diagonal of U^dag
  double g0, g3;    // ADJ_DIAG: the diagonal of H
  double c, s;      // ADJ_RX: U^dag = [[c, i s], [i s, c]]
  uint64_t off1;    // offset of the target bit
};

template <int FORM>
__global__ void __launch_bounds__(kAdjThreads)
k_adjoint_param1(double2* __restrict__ psi, double2* __restrict__ lam, uint64_t nitems, IdxSpec s,
                 const __grid_constant__ AdjForm1 F, const AdjOut out) {
  double acc = 0.0;
  for (uint64_t it = (uint64_t)blockIdx.x * kAdjThreads + threadIdx.x; it < nitems;
       it += (uint64_t)gridDim.x * kAdjThreads) {
    const uint64_t b0 = item_index(it, s), b1 = b0 + F.off1;
    double2 x0 = psi[b0], x1 = psi[b1], l0 = lam[b0], l1 = lam[b1];
    if (FORM == ADJ_DIAG) {
      // Im conj(l) H x with H diagonal and real
      acc = fma(F.g0, fma(l0.x, x0.y, -l0.y * x0.x), acc);
      acc = fma(F.g3, fma(l1.x, x1.y, -l1.y * x1.x), acc);
      x0 = cmul(F.u0, x0);
      x1 = cmul(F.u3, x1);
      l0 = cmul(F.u0, l0);
      l1 = cmul(F.u3, l1);
    } else {
      // Im (conj(l0) x1 + conj(l1) x0) for H = X
      acc += fma(l0.x, x1.y, -l0.y * x1.x) + fma(l1.x, x0.y, -l1.y * x0.x);
      const double c = F.c, sn = F.s;
      const double2 nx0 = make_double2(fma(c, x0.x, -sn * x1.y), fma(c, x0.y, sn * x1.x));
      const double2 nx1 = make_double2(fma(c, x1.x, -sn * x0.y), fma(c, x1.y, sn * x0.x));
      const double2 nl0 = make_double2(fma(c, l0.x, -sn * l1.y), fma(c, l0.y, sn * l1.x));
      const double2 nl1 = make_double2(fma(c, l1.x, -sn * l0.y), fma(c, l1.y, sn * l0.x));
      x0 = nx0; x1 = nx1; l0 = nl0; l1 = nl1;
    }
    psi[b0] = x0;
    psi[b1] = x1;
    lam[b0] = l0;
    lam[b1] = l1;
  }
  adj_finish(acc, out);
}

// A run of uncontrolled single-qubit gates on one qubit, some with a parameter, as one
// pass, with the controlled X before (pre) or after it that only renames the pair.
// With (a, b) the pair at the end of the run the pass sums Im conj(l_a) x_a,
// Im conj(l_b) x_b, Im<l|X|x> and Im<l|Y|x>; a member's derivative is 2 c times its
// generator carried to the run's end, decomposed over those four (AdjRun::coef).
// The first row of U^dag is divided by its larger entry (its columns traded when that is
// the second): that entry's products, a quarter of all, are gone.  Psi and lambda then carry
// the same complex factor, which the host keeps (AdjWalk::phi): derivatives are divided by
// its square, a checkpoint is multiplied by it, and once it is past 2^100 a run is applied
// in full (FULL) with the factor taken out.
//   bound: the FP64 rate.  12 operations a pair for the sums and 24 for U^dag on psi and
//   lambda, where Rz, Rx, Rz took 64 in three passes and the X a fourth pass.  The pairs
//   are cut into equal contiguous ranges, four CTAs an SM: a grid-stride loop left a
//   sixth of the FP64 units idle in its last round.  Measured in the differentiation
//   workload (n = 20): 49 us a run and its X (53 us with the four sums reduced one by one, 62
//   us with every entry of U^dag multiplied as well), 121 us as four passes.
constexpr int kAdjMembers = 8;
constexpr int kAdjRunBlocks = 608;  // 4 per SM on 152 SMs

struct AdjRun {
  double2 ud[4];             // U^dag of the run
  uint64_t off1;             // offset of its bit
  uint64_t xmask, xval;      // the X's controls and their values (xmask = 0: no X)
  int pre, members;
  int swap;                  // columns of U^dag (and the coefficients) are traded
  int param[kAdjMembers];
  double coef[kAdjMembers][4];
};

template <bool FULL>
__global__ void __launch_bounds__(kAdjThreads, 4)
k_adjoint_run(double2* __restrict__ psi, double2* __restrict__ lam, uint64_t nitems,
              const __grid_constant__ AdjRun F, double* __restrict__ partials, unsigned* __restrict__ counter,
              double* __restrict__ grad) {
  const uint64_t lo = nitems * blockIdx.x / gridDim.x, hi = nitems * (blockIdx.x + 1) / gridDim.x;
  const uint64_t below = F.off1 - 1;
  double va = 0.0, vb = 0.0, vx = 0.0, vy = 0.0;
  for (uint64_t it = lo + threadIdx.x; it < hi; it += kAdjThreads) {
    const uint64_t b0 = it + (it & ~below), b1 = b0 + F.off1;
    const bool on = F.xmask && (b0 & F.xmask) == F.xval;
    const bool in = (on && !F.pre) != (F.swap != 0), out = on && F.pre;
    const uint64_t ia = in ? b1 : b0, ib = in ? b0 : b1;
    const double2 xa = psi[ia], xb = psi[ib], la = lam[ia], lb = lam[ib];
    va = fma(la.x, xa.y, fma(-la.y, xa.x, va));
    vb = fma(lb.x, xb.y, fma(-lb.y, xb.x, vb));
    vx = fma(la.x, xb.y, fma(-la.y, xb.x, vx));
    vy = fma(lb.x, xa.x, fma(lb.y, xa.y, vy));
    vx = fma(lb.x, xa.y, fma(-lb.y, xa.x, vx));
    vy = fma(-la.x, xb.x, fma(-la.y, xb.y, vy));
    const uint64_t oa = out ? b1 : b0, ob = out ? b0 : b1;
    psi[oa] = cfma(F.ud[1], xb, FULL ? cmul(F.ud[0], xa) : xa);
    psi[ob] = cfma(F.ud[3], xb, cmul(F.ud[2], xa));
    lam[oa] = cfma(F.ud[1], lb, FULL ? cmul(F.ud[0], la) : la);
    lam[ob] = cfma(F.ud[3], lb, cmul(F.ud[2], la));
  }
  // CTA sums, then the CTA that arrives last folds all of them (in an order that does not
  // depend on which it is) and adds every member's derivative
  __shared__ double red[4][kAdjThreads / 32];
  __shared__ double tot[4];
  __shared__ bool last;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  // the four sums over a warp in 6 additions a lane (a thread has three or four pairs: 20,
  // each sum by itself, were a seventh of the kernel's FP64 operations): a lane gives away
  // two sums, then one, and keeps the sum that bits 4 and 3 of its number say
  auto cta_sums = [&](const double (&v)[4]) {
    const bool hi = lane & 16, odd = lane & 8;
    const double a = (hi ? v[2] : v[0]) + __shfl_xor_sync(0xffffffffu, hi ? v[0] : v[2], 16);
    const double b = (hi ? v[3] : v[1]) + __shfl_xor_sync(0xffffffffu, hi ? v[1] : v[3], 16);
    double r = (odd ? b : a) + __shfl_xor_sync(0xffffffffu, odd ? a : b, 8);
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
    if ((lane & 7) == 0) red[lane >> 3][warp] = r;
    __syncthreads();
    if (threadIdx.x < 4) {
      static_assert(kAdjThreads / 32 == 8, "CTA tree below is written for 8 warps");
      const double* r = red[threadIdx.x];
      tot[threadIdx.x] = ((r[0] + r[1]) + (r[2] + r[3])) + ((r[4] + r[5]) + (r[6] + r[7]));
    }
    __syncthreads();
  };
  double v[4] = {va, vb, vx, vy};
  cta_sums(v);
  if (threadIdx.x < 4) partials[threadIdx.x * gridDim.x + blockIdx.x] = tot[threadIdx.x];
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(counter, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!last) return;
  __threadfence();
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    v[k] = 0.0;
    for (int i = threadIdx.x; i < (int)gridDim.x; i += kAdjThreads) v[k] += __ldcg(partials + k * gridDim.x + i);
  }
  __syncthreads();
  cta_sums(v);
  if (threadIdx.x == 0) {
    for (int m = 0; m < F.members; ++m) {
      const double* c = F.coef[m];
      grad[F.param[m]] += (c[0] * tot[0] + c[1] * tot[1]) + (c[2] * tot[2] + c[3] * tot[3]);
    }
    *counter = 0u;
  }
}

// the structured form of a single-target gate, or -1
static int adj_form1(const std::vector<cd>& G, const std::vector<cd>& Ud, AdjForm1* F) {
  const cd z(0, 0);
  if (G[1] == z && G[2] == z && G[0].imag() == 0 && G[3].imag() == 0 && Ud[1] == z && Ud[2] == z) {
    F->u0 = make_double2(Ud[0].real(), Ud[0].imag());
    F->u3 = make_double2(Ud[3].real(), Ud[3].imag());
    F->g0 = G[0].real();
    F->g3 = G[3].real();
    return ADJ_DIAG;
  }
  if (G[0] == z && G[3] == z && G[1] == cd(1, 0) && G[2] == cd(1, 0) && Ud[0] == Ud[3] && Ud[0].imag() == 0 &&
      Ud[1] == Ud[2] && Ud[1].real() == 0) {
    F->c = Ud[0].real();
    F->s = Ud[1].imag();
    return ADJ_RX;
  }
  return -1;
}

template <int K>
static int launch_adjoint_param(double2* psi, double2* lam, int n, const qs_gate_desc& g,
                                const std::vector<cd>& G, const std::vector<cd>& Ud, double* partials,
                                unsigned* counter, double* dgrad, double cfac, cudaStream_t st) {
  const AdjOut out{partials, counter, dgrad, g.param, 2.0 * cfac};
  if constexpr (K == 1) {
    AdjForm1 F;
    memset(&F, 0, sizeof(F));
    const int form = adj_form1(G, Ud, &F);
    if (form >= 0) {
      F.off1 = 1ull << g.locs[0];
      IdxSpec s;
      QS_TRY(make_idx(n, F.off1 | g.ctrl_mask, g.ctrl_vals & g.ctrl_mask, &s));
      const uint64_t items = 1ull << s.item_log2;
      const int nblk = (int)std::min<uint64_t>(kAdjMaxBlocks, std::max<uint64_t>(1, (items + kAdjThreads * 4 - 1) / (kAdjThreads * 4)));
      if (form == ADJ_DIAG)
        k_adjoint_param1<ADJ_DIAG><<<nblk, kAdjThreads, 0, st>>>(psi, lam, items, s, F, out);
      else
        k_adjoint_param1<ADJ_RX><<<nblk, kAdjThreads, 0, st>>>(psi, lam, items, s, F, out);
      QS_LAUNCHED();
      return QS_OK;
    }
  }
  AdjMat<K> M;
  memset(&M, 0, sizeof(M));
  constexpr int D = 1 << K;
  uint64_t locmask = 0;
  for (int j = 0; j < K; ++j) locmask |= 1ull << g.locs[j];
  for (int m = 0; m < D; ++m) {
    uint64_t o = 0;
    for (int j = 0; j < K; ++j)
      if ((m >> j) & 1) o |= 1ull << g.locs[j];
    M.off[m] = o;
  }
  for (int i = 0; i < D * D; ++i) {
    M.g[i] = make_double2(G[i].real(), G[i].imag());
    M.ud[i] = make_double2(Ud[i].real(), Ud[i].imag());
  }
  IdxSpec s;
  QS_TRY(make_idx(n, locmask | g.ctrl_mask, g.ctrl_vals & g.ctrl_mask, &s));
  const uint64_t items = 1ull << s.item_log2;
  const int nblk = (int)std::min<uint64_t>(kAdjMaxBlocks, std::max<uint64_t>(1, (items + kAdjThreads * 4 - 1) / (kAdjThreads * 4)));
  k_adjoint_param<K><<<nblk, kAdjThreads, 0, st>>>(psi, lam, items, s, M, out);
  QS_LAUNCHED();
  return QS_OK;
}

// generator H (on the targets) and factor c with U = exp(-i theta c H)
int gate_generator(const qs_gate_desc& g, std::vector<cd>& G, double* cfac) {
  const int D = 1 << g.nlocs;
  G.assign(D * D, cd(0, 0));
  switch (g.kind) {
    case QS_GATE_RX: G[1] = 1; G[2] = 1; *cfac = 0.5; return QS_OK;
    case QS_GATE_RY: G[1] = cd(0, -1); G[2] = cd(0, 1); *cfac = 0.5; return QS_OK;
    case QS_GATE_RZ: G[0] = 1; G[3] = -1; *cfac = 0.5; return QS_OK;
    case QS_GATE_SHIFT: G[3] = 1; *cfac = -1.0; return QS_OK;
    case QS_GATE_PHASE: G[0] = 1; G[3] = 1; *cfac = -1.0; return QS_OK;
    case QS_GATE_ROT:
      pauli_string(g.nlocs, g.paulis, G);
      *cfac = 0.5;
      return QS_OK;
  }
  return fail(QS_EUNSUPPORTED, "gate kind %d has no parameter gradient", g.kind);
}

// One pass of the backward walk: a gate, or a run of gates on one qubit (with the
// controlled X taken along before or after it).
struct AdjStep {
  std::vector<int> gates;
  int x = -1;
  bool pre = false, dead = false;
};

static bool diagonal_gate(const qs_circuit* c, const qs_gate_desc& g) {
  switch (g.kind) {
    case QS_GATE_RX: case QS_GATE_RY: case QS_GATE_X: case QS_GATE_Y: case QS_GATE_H: return false;
    case QS_GATE_ROT: return g.paulis[0] == 3;
    case QS_GATE_MATRIX: return c->mats[g.mat_offset + 1] == cd(0, 0) && c->mats[g.mat_offset + 2] == cd(0, 0);
  }
  return true;
}

// Whether a run is worth its own pass (36 FP64 operations a pair): two gates or more,
// one with a parameter, not all diagonal (those take 20 each).
static bool adj_run(const qs_circuit* c, const AdjStep& u) {
  bool diag = true, param = false;
  for (int k : u.gates) {
    diag = diag && diagonal_gate(c, c->gates[k]);
    param = param || (c->gates[k].param >= 0 && c->gates[k].kind != QS_GATE_MATRIX);
  }
  return u.gates.size() > 1 && param && !diag;
}

// Gates first .. last - 1 as steps, in circuit order: uncontrolled single-qubit gates on
// one qubit collect in a run (at the place of its first gate: nothing in between touches
// the qubit); a controlled X on a run's qubit right after it, or right before it, goes
// along with it (the run moves to the X's place, past gates on other qubits only).
static void adj_steps(const qs_circuit* c, int first, int last, std::vector<AdjStep>& out) {
  out.clear();
  std::vector<int> open(c->nqubits, -1);  // the run on each qubit that takes further gates
  for (int k = first; k < last; ++k) {
    const qs_gate_desc& g = c->gates[k];
    const int t = g.locs[0];
    const bool one = g.nlocs == 1 && g.ctrl_mask == 0;
    const bool cx = g.nlocs == 1 && g.ctrl_mask && g.kind == QS_GATE_X;
    AdjStep* run = g.nlocs == 1 && open[t] >= 0 ? &out[open[t]] : nullptr;
    if (one && run && (int)run->gates.size() < kAdjMembers) {
      run->gates.push_back(k);
      continue;
    }
    AdjStep u;
    if (cx && run && run->x < 0 && adj_run(c, *run)) {
      u = *run;
      run->dead = true;
    }
    if (cx) {
      u.x = k;
      u.pre = u.gates.empty();
    } else {
      u.gates.push_back(k);
    }
    for (int j = 0; j < g.nlocs; ++j) open[g.locs[j]] = -1;
    for (int q = 0; q < c->nqubits; ++q)
      if ((g.ctrl_mask >> q) & 1) open[q] = -1;
    if (one || (cx && u.pre)) open[t] = (int)out.size();
    out.push_back(std::move(u));
  }
}

namespace {

struct AdjWalk {
  qs_state* s;
  const qs_circuit* c;
  const double* params;
  int n;
  double2 *psi, *lam;
  double *dgrad, *partials;
  unsigned* counter;
  std::vector<cd> U, G;
  cd phi = 1;  // psi and lambda hold phi times the states

  int gate(int k) {
    const qs_gate_desc& g = c->gates[k];
    cudaStream_t st = s->stream;
    QS_TRY(gate_matrix(c, g, params, U));
    dagger(U, g.nlocs);
    if (g.param >= 0 && g.kind != QS_GATE_MATRIX) {
      double cfac = 0;
      QS_TRY(gate_generator(g, G, &cfac));
      cfac /= std::norm(phi);
      switch (g.nlocs) {
        case 1: return launch_adjoint_param<1>(psi, lam, n, g, G, U, partials, counter, dgrad, cfac, st);
        case 2: return launch_adjoint_param<2>(psi, lam, n, g, G, U, partials, counter, dgrad, cfac, st);
        case 3: return launch_adjoint_param<3>(psi, lam, n, g, G, U, partials, counter, dgrad, cfac, st);
      }
      return fail(QS_EUNSUPPORTED, "parameterised gate on %d targets", g.nlocs);
    }
    // psi and lambda are adjacent in the work buffer: one launch over both as
    // a batch of two registers
    Plan p;
    QS_TRY(plan_gate(U.data(), g.nlocs, g.locs, g.ctrl_mask, g.ctrl_vals, &p));
    return launch_plan_on(psi, QS_C128, n, 2, 1ll << n, p, s);
  }

  int run(const AdjStep& u) {
    AdjRun F;
    memset(&F, 0, sizeof(F));
    // from the run's end: E is the product of the gates passed; E H E^dag is a gate's
    // generator at the end of the run
    cd E[4] = {1, 0, 0, 1};
    for (size_t q = u.gates.size(); q-- > 0;) {
      const qs_gate_desc& g = c->gates[u.gates[q]];
      if (g.param >= 0 && g.kind != QS_GATE_MATRIX) {
        double cfac = 0;
        QS_TRY(gate_generator(g, G, &cfac));
        cd M[4];
        for (int i = 0; i < 2; ++i)
          for (int j = 0; j < 2; ++j) {
            cd v = 0;
            for (int a = 0; a < 2; ++a)
              for (int b = 0; b < 2; ++b) v += E[2 * i + a] * G[2 * a + b] * std::conj(E[2 * j + b]);
            M[2 * i + j] = v;
          }
        const double f = 2.0 * cfac / std::norm(phi);
        double* co = F.coef[F.members];
        co[0] = f * M[0].real();
        co[1] = f * M[3].real();
        co[2] = f * M[1].real();
        co[3] = -f * M[1].imag();
        F.param[F.members++] = g.param;
      }
      QS_TRY(gate_matrix(c, g, params, U));
      const cd A[4] = {E[0] * U[0] + E[1] * U[2], E[0] * U[1] + E[1] * U[3], E[2] * U[0] + E[3] * U[2],
                       E[2] * U[1] + E[3] * U[3]};
      std::copy(A, A + 4, E);
    }
    cd D[4] = {std::conj(E[0]), std::conj(E[2]), std::conj(E[1]), std::conj(E[3])};
    F.swap = std::norm(D[1]) > std::norm(D[0]);
    if (F.swap) {
      std::swap(D[0], D[1]);
      std::swap(D[2], D[3]);
      for (int m = 0; m < F.members; ++m) {
        std::swap(F.coef[m][0], F.coef[m][1]);
        F.coef[m][3] = -F.coef[m][3];  // Y with its basis states traded
      }
    }
    // a row without a large entry (a matrix that is not unitary) is applied as it is
    const double size = std::abs(phi);
    const bool far = size > 0x1p100 || size < 0x1p-100, full = far || std::norm(D[0]) < 0.25;
    const cd f = far ? 1.0 / phi : full ? cd(1, 0) : 1.0 / D[0];
    phi *= f;
    for (int k = 0; k < 4; ++k) F.ud[k] = make_double2((f * D[k]).real(), (f * D[k]).imag());
    const int t = c->gates[u.gates[0]].locs[0];
    F.off1 = 1ull << t;
    if (u.x >= 0) {
      F.xmask = c->gates[u.x].ctrl_mask;
      F.xval = c->gates[u.x].ctrl_vals & F.xmask;
      F.pre = u.pre ? 1 : 0;
    }
    const uint64_t items = 1ull << (n - 1);
    const int nblk = (int)std::min<uint64_t>(kAdjRunBlocks, std::max<uint64_t>(1, items / kAdjThreads));
    if (full) k_adjoint_run<true><<<nblk, kAdjThreads, 0, s->stream>>>(psi, lam, items, F, partials, counter, dgrad);
    else k_adjoint_run<false><<<nblk, kAdjThreads, 0, s->stream>>>(psi, lam, items, F, partials, counter, dgrad);
    QS_LAUNCHED();
    return QS_OK;
  }

  int step(const AdjStep& u) {
    if (u.dead) return QS_OK;
    if (adj_run(c, u)) return run(u);
    if (u.x >= 0 && !u.pre) QS_TRY(gate(u.x));
    for (size_t q = u.gates.size(); q-- > 0;) QS_TRY(gate(u.gates[q]));
    if (u.x >= 0 && u.pre) QS_TRY(gate(u.x));
    return QS_OK;
  }
};

}  // namespace

int backward(qs_state* s, const qs_circuit* c, const double* params, const qs_observable* o, int ckpt_every,
             const void* ckpts, void* work, double* host_grad, double* host_loss) {
  if (s->nreg != 1) return fail(QS_EUNSUPPORTED, "qs_backward takes a single register");
  const int n = s->nq[0];
  if (n != c->nqubits) return fail(QS_EINVAL, "circuit has %d qubits, state %d", c->nqubits, n);
  if (ckpt_every < 0 || (ckpt_every > 0 && !ckpts)) return fail(QS_EINVAL, "bad checkpoint arguments");
  if (!work) return fail(QS_EINVAL, "work buffer is NULL");
  cudaStream_t st = s->stream;
  const uint64_t dim = 1ull << n;
  double2* psi = (double2*)work;
  double2* lam = psi + dim;
  const int np = std::max(1, c->nparams);
  if (host_loss) QS_TRY(expect_raw(s->data, s->dtype, n, 1, o, s, host_loss));
  // scratch: grad[np] | partials | counter
  constexpr int kPartials = std::max(kAdjMaxBlocks, 4 * kAdjRunBlocks);
  QS_TRY(ensure_ws(s, s->ws, sizeof(double) * (np + kPartials) + 256));
  double* dgrad = (double*)s->ws.ptr;
  double* partials = dgrad + np;
  unsigned* counter = reinterpret_cast<unsigned*>(partials + kPartials);
  QS_CUDA(cudaMemsetAsync(dgrad, 0, sizeof(double) * np, st));
  QS_CUDA(cudaMemsetAsync(counter, 0, sizeof(unsigned), st));
  QS_TRY(promote_to_c128(s->data, s->dtype, psi, dim, 1, st));
  QS_TRY(apply_observable_c128(psi, lam, n, o, st));
  const size_t ab = amp_bytes(s->dtype);
  AdjWalk w{s, c, params, n, psi, lam, dgrad, partials, counter, {}, {}};
  // segments between checkpoints, last first: psi restarts from the checkpoint at a
  // segment's end, so no run spans one
  const int ng = (int)c->gates.size(), every = ckpt_every > 0 ? ckpt_every : std::max(1, ng);
  std::vector<AdjStep> steps;
  for (int seg = ng > 0 ? (ng - 1) / every : -1; seg >= 0; --seg) {
    const int first = seg * every, last = std::min(ng, first + every);
    if (last < ng) QS_TRY(promote_to_c128((const char*)ckpts + ab * dim * seg, s->dtype, psi, dim, w.phi, st));
    adj_steps(c, first, last, steps);
    for (size_t k = steps.size(); k-- > 0;) QS_TRY(w.step(steps[k]));
  }
  QS_CUDA(cudaMemcpyAsync(host_grad, dgrad, sizeof(double) * c->nparams, cudaMemcpyDeviceToHost, st));
  QS_CUDA(cudaStreamSynchronize(st));
  return QS_OK;
}

}  // namespace qs

// ------------------------------------------------------------------ one gate of the adjoint walk
//
// qs_adjoint_step: the per-gate step of the walk above on two caller-held
// complex128 registers, for callers that walk a circuit themselves (the
// qubit-sharded register, whose gates may need data exchanges in between).

namespace qs {

// the matrix pool of a desc: MATRIX gates read 4^k entries at mat_offset
static int desc_matrix(const qs_gate_desc& g, const double* host_mats, const double* params, std::vector<cd>& U) {
  if (g.kind == QS_GATE_MATRIX) {
    if (!host_mats || g.mat_offset < 0) return fail(QS_EINVAL, "MATRIX gate without its matrix");
    const int D = 1 << g.nlocs;
    U.resize(D * D);
    for (int i = 0; i < D * D; ++i)
      U[i] = cd(host_mats[2 * (g.mat_offset + i)], host_mats[2 * (g.mat_offset + i) + 1]);
    return QS_OK;
  }
  qs_circuit tmp;
  tmp.nqubits = QS_MAXQ;
  return gate_matrix(&tmp, g, params, U);
}

static int check_desc(const qs_gate_desc& g, int n, const double* params) {
  int32_t locs[QS_MAXK];
  if (g.nlocs < 1 || g.nlocs > QS_MAXK) return fail(QS_EINVAL, "gate arity %d", g.nlocs);
  for (int j = 0; j < g.nlocs; ++j) locs[j] = g.locs[j];
  QS_TRY(validate_gate(n, g.nlocs, locs, g.ctrl_mask));
  if (g.param >= 0 && !params) return fail(QS_EINVAL, "the gate needs the parameter vector");
  return QS_OK;
}

}  // namespace qs

using namespace qs;

extern "C" {

int qs_gate_desc_matrices(const qs_gate_desc* g, const double* host_mats, const double* host_params, int dagger_u,
                          double* host_U, double* host_G, double* host_cfac) {
  if (!g) return fail(QS_EINVAL, "null gate");
  QS_TRY(check_desc(*g, QS_MAXQ, host_params));
  const int D = 1 << g->nlocs;
  if (host_U) {
    std::vector<cd> U;
    QS_TRY(desc_matrix(*g, host_mats, host_params, U));
    if (dagger_u) dagger(U, g->nlocs);
    for (int i = 0; i < D * D; ++i) { host_U[2 * i] = U[i].real(); host_U[2 * i + 1] = U[i].imag(); }
  }
  if (host_G || host_cfac) {
    if (g->param < 0) return fail(QS_EINVAL, "the gate has no parameter");
    std::vector<cd> G;
    double cf = 0.0;
    QS_TRY(gate_generator(*g, G, &cf));
    if (host_G)
      for (int i = 0; i < D * D; ++i) { host_G[2 * i] = G[i].real(); host_G[2 * i + 1] = G[i].imag(); }
    if (host_cfac) *host_cfac = cf;
  }
  return QS_OK;
}

int qs_adjoint_step(qs_state* psi, qs_state* lam, const qs_gate_desc* g, const double* host_mats,
                    const double* host_params, double* dev_grad) {
  if (!psi || !lam || !g) return fail(QS_EINVAL, "null argument");
  if (psi->dtype != QS_C128 || lam->dtype != QS_C128) return fail(QS_EINVAL, "qs_adjoint_step takes complex128 states");
  if (psi->nreg != 1 || lam->nreg != 1 || psi->nq[0] != lam->nq[0])
    return fail(QS_EINVAL, "psi and lambda must be single registers of one size");
  if (psi->data == lam->data) return fail(QS_EINVAL, "psi and lambda must be distinct");
  const int n = psi->nq[0];
  QS_TRY(check_desc(*g, n, host_params));
  const bool param = g->param >= 0 && g->kind != QS_GATE_MATRIX;
  if (param && !dev_grad) return fail(QS_EINVAL, "dev_grad is NULL");
  cudaStream_t st = psi->stream;
  std::vector<cd> U;
  QS_TRY(desc_matrix(*g, host_mats, host_params, U));
  dagger(U, g->nlocs);
  double2* x = (double2*)psi->data;
  double2* l = (double2*)lam->data;
  if (!param) {
    Plan p;
    QS_TRY(plan_gate(U.data(), g->nlocs, g->locs, g->ctrl_mask, g->ctrl_vals, &p));
    QS_TRY(launch_plan_on(x, QS_C128, n, 1, 1ll << n, p, psi));
    QS_TRY(launch_plan_on(l, QS_C128, n, 1, 1ll << n, p, psi));
    return QS_OK;
  }
  std::vector<cd> G;
  double cfac = 0.0;
  QS_TRY(gate_generator(*g, G, &cfac));
  QS_TRY(ensure_ws(psi, psi->ws, sizeof(double) * kAdjMaxBlocks + 256));
  double* partials = (double*)psi->ws.ptr;
  unsigned* counter = reinterpret_cast<unsigned*>(partials + kAdjMaxBlocks);
  QS_CUDA(cudaMemsetAsync(counter, 0, sizeof(unsigned), st));
  switch (g->nlocs) {
    case 1: return launch_adjoint_param<1>(x, l, n, *g, G, U, partials, counter, dev_grad, cfac, st);
    case 2: return launch_adjoint_param<2>(x, l, n, *g, G, U, partials, counter, dev_grad, cfac, st);
    case 3: return launch_adjoint_param<3>(x, l, n, *g, G, U, partials, counter, dev_grad, cfac, st);
  }
  return fail(QS_EUNSUPPORTED, "parameterised gate on %d targets", g->nlocs);
}

int qs_sample_shards(int nshards, const double* host_weights, int nshots, const double* host_u,
                     int32_t* host_shard, double* host_u_in_shard) {
  if (nshards < 1 || nshots < 0 || !host_weights || (nshots > 0 && (!host_u || !host_shard || !host_u_in_shard)))
    return fail(QS_EINVAL, "bad arguments");
  // the walk of qs_measure's contract over the shard weights: T = left fold of
  // the weights, t = u T, first shard whose running sum exceeds t (else the last
  // positive weight, else the last shard); its exclusive prefix a gives the
  // uniform of the shard's own sampler u' = (t - a) / P_s, kept below 1
  double total = host_weights[0];
  for (int s = 1; s < nshards; ++s) total = total + host_weights[s];
  for (int i = 0; i < nshots; ++i) {
    if (!(host_u[i] >= 0.0 && host_u[i] < 1.0)) return fail(QS_EINVAL, "uniform %d not in [0, 1)", i);
    const double t = host_u[i] * total;
    double a = 0.0, a_last = 0.0;
    int pick = -1, last = -1;
    for (int s = 0; s < nshards; ++s) {
      const double nxt = a + host_weights[s];
      if (nxt > t) { pick = s; break; }
      if (host_weights[s] > 0.0) { last = s; a_last = a; }
      a = nxt;
    }
    if (pick < 0) {
      if (last >= 0) { pick = last; a = a_last; }
      else { pick = nshards - 1; }
    }
    const double w = host_weights[pick];
    double v = w > 0.0 ? (t - a) / w : 0.0;
    if (!(v >= 0.0)) v = 0.0;
    if (v >= 1.0) v = std::nextafter(1.0, 0.0);
    host_shard[i] = pick;
    host_u_in_shard[i] = v;
  }
  return QS_OK;
}

}  // extern "C"

