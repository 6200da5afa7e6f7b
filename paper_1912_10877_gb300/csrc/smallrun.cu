// smallrun.cu -- a whole circuit of single-target gates on a small register (n <= 14) and
// a diagonal expectation in one launch of one thread-block cluster (sm_103a).
//
// One amplitude a thread, in registers; the highest index bits are the CTA's rank in the
// cluster.  Gates are fused on the host: uncontrolled gates on one qubit into one 2x2, a
// controlled X right after (or before) such a run into a renaming of its outputs (or
// inputs), SWAPs into a relabelling.  An op on a lane bit gets the partner by shuffle, on
// a thread bit through shared memory; the rank bits take part only as controls and in
// diagonal gates: when every op left has its target there, one exchange through the
// cluster's shared memory trades them for the qubits whose next use is farthest.
//
// Bound by the FP64 rate of the cluster's SMs (8 operations an amplitude for a dense op)
// and, below, the latency of an op.  12 qubits complex128, 10 layers of Rz Rx Rz and a
// CNOT ladder (120 dense ops) with <sum ZZ>: 94 us, 75 of them the FP64 arithmetic of 16
// SMs; as 25 dense 5-qubit blocks with a grid barrier after each 169 us.
#include <cooperative_groups.h>

#include <algorithm>
#include <cstring>

#include "common.cuh"

namespace qs {

namespace {

namespace cg = cooperative_groups;

constexpr int kRunMaxQubits = 14;  // 16 CTAs of 1024 threads
constexpr int kRunTerms = 64;

enum { RU_DIAG = 0, RU_X, RU_DENSE, RU_EXCH };

// complex64 holds its matrices as the FP64 ones' high parts and corrections (the rounding of a
// matrix is coherent over the state: 120 of them cost more than the state's own rounding)
template <typename R> struct Corr {};
template <> struct Corr<float> { float2 w[4]; };

// masks and positions are physical index bits
template <typename R>
struct RunOp : Corr<R> {
  uint32_t mask, vals;    // controls of the gate
  uint32_t xmask, xvals;  // RU_DENSE: controls of the X taken along (0: none)
  int8_t kind, t, pre, npair;
  int8_t a[4], b[4];      // RU_EXCH: bits that trade places
  c2_t<R> u[4];           // RU_DIAG: u[0], u[3]
};
template <typename R, int CAP>
struct RunOps {
  RunOp<R> op[CAP];
};
struct RunArgs {
  int n, lc, nops, nterm;
  double* out;
  int8_t place[kRunMaxQubits];  // physical bit of each qubit at the end
  uint32_t z[kRunTerms];
  double c[kRunTerms];
};

__device__ __forceinline__ float2 shfl2(float2 v, int m) {
  return make_float2(__shfl_xor_sync(0xffffffffu, v.x, m), __shfl_xor_sync(0xffffffffu, v.y, m));
}
__device__ __forceinline__ double2 shfl2(double2 v, int m) {
  return make_double2(__shfl_xor_sync(0xffffffffu, v.x, m), __shfl_xor_sync(0xffffffffu, v.y, m));
}

// row r of u times (a, b); complex64: the FP64 row, rounded once
__device__ __forceinline__ double2 row_dot(const RunOp<double>& o, bool r, double2 a, double2 b) {
  return cfma(r ? o.u[3] : o.u[1], b, cmul(r ? o.u[2] : o.u[0], a));
}
__device__ __forceinline__ float2 row_dot(const RunOp<float>& o, bool r, float2 a, float2 b) {
  return cf_dot2(a, r ? o.u[2] : o.u[0], r ? o.w[2] : o.w[0], b, r ? o.u[3] : o.u[1], r ? o.w[3] : o.w[1]);
}
__device__ __forceinline__ double2 diag_mul(const RunOp<double>& o, bool r, double2 x) {
  return cmul(x, r ? o.u[3] : o.u[0]);
}
__device__ __forceinline__ float2 diag_mul(const RunOp<float>& o, bool r, float2 x) {
  return cf_mul(x, r ? o.u[3] : o.u[0], r ? o.w[3] : o.w[0]);
}

template <typename R, int CAP>
__global__ void __launch_bounds__(1024)
k_small_run(c2_t<R>* __restrict__ psi, const __grid_constant__ RunArgs A, const __grid_constant__ RunOps<R, CAP> ops) {
  using T = c2_t<R>;
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ double red[32], part[16];
  T* buf = reinterpret_cast<T*>(smraw);  // two areas for the CTA, two for the cluster
  cg::cluster_group cl = cg::this_cluster();
  const unsigned rank = cl.block_rank();
  const int n = A.n, L = n - A.lc;
  const uint32_t area = 1u << L, tid = threadIdx.x;
  const bool act = tid < area;
  const uint32_t i = (rank << L) | tid;
  T x = act ? psi[i] : cmk<T>(0, 0);
  // Every amplitude of the cluster is loaded before any is stored: a circuit with SWAPs ends
  // on other places than it began on, and its ops may need no barrier of their own (lane
  // targets, diagonal gates, none).  It also lets every CTA start before another touches its
  // shared memory.
  cl.sync();
  int turn = 0, rturn = 0;
  for (int o = 0; o < A.nops; ++o) {
    const RunOp<R>& op = ops.op[o];
    const int kind = op.kind, t = op.t;
    if (kind == RU_DIAG) {
      if ((i & op.mask) == op.vals) x = diag_mul(op, (i >> t) & 1u, x);
      continue;
    }
    T y;
    if (kind == RU_EXCH) {
      T* a = buf + (2 + rturn) * area;
      if (act) a[tid] = x;
      cl.sync();  // an area is written again only after the next exchange's barrier
      uint32_t j = i;
      for (int k = 0; k < op.npair; ++k) {
        const uint32_t d = ((i >> op.a[k]) ^ (i >> op.b[k])) & 1u;
        j ^= (d << op.a[k]) | (d << op.b[k]);
      }
      if (act) x = cl.map_shared_rank(a, j >> L)[j & (area - 1)];
      rturn ^= 1;
      continue;
    }
    if (t < 5) {
      y = shfl2(x, 1 << t);
    } else {
      T* a = buf + turn * area;
      if (act) a[tid] = x;
      __syncthreads();
      y = act ? a[tid ^ (1u << t)] : x;
      turn ^= 1;
    }
    if ((i & op.mask) != op.vals) continue;
    if (kind == RU_X) {
      x = y;
      continue;
    }
    const bool one = (i >> t) & 1u, on = op.xmask && (i & op.xmask) == op.xvals;
    const bool row = one ^ (on && !op.pre), in = one ^ (on && op.pre);
    const T a = in ? y : x, b = in ? x : y;
    x = row_dot(op, row, a, b);
  }
  uint32_t out = 0;
  for (int q = 0; q < n; ++q) out |= ((i >> A.place[q]) & 1u) << q;
  if (act) psi[out] = x;
  if (A.out) {
    double e = 0.0;
    if (act) {
      double w = 0.0;
      for (int t = 0; t < A.nterm; ++t) w += (__popc(i & A.z[t]) & 1) ? -A.c[t] : A.c[t];
      e = w * ((double)x.x * (double)x.x + (double)x.y * (double)x.y);
    }
    for (int s = 16; s > 0; s >>= 1) e += __shfl_xor_sync(0xffffffffu, e, s);
    if ((tid & 31) == 0) red[tid >> 5] = e;
    __syncthreads();
    if (tid < 32) {
      e = tid < (blockDim.x >> 5) ? red[tid] : 0.0;
      for (int s = 16; s > 0; s >>= 1) e += __shfl_xor_sync(0xffffffffu, e, s);
      if (tid == 0) *cl.map_shared_rank(part + rank, 0) = e;
    }
    cl.sync();
    if (rank == 0 && tid < 32) {
      e = tid < (1u << A.lc) ? part[tid & 15] : 0.0;
      for (int s = 16; s > 0; s >>= 1) e += __shfl_xor_sync(0xffffffffu, e, s);
      if (tid == 0) *A.out = e;
    }
  }
  cl.sync();  // no CTA leaves while another may read its shared memory
}

// ------------------------------------------------------------------ host: ops

struct LOp {
  int kind, t;
  cd u[4];
  uint32_t mask = 0, vals = 0, xmask = 0, xvals = 0;
  bool pre = false, dead = false;
  uint32_t qubits() const { return (1u << t) | mask | xmask; }
};

// The circuit as fused ops on qubits, then place[q]: the label that qubit q has at the end
// (SWAPs only rename).  false: a gate outside this path.
bool fuse(const qs_circuit* c, const double* params, std::vector<LOp>& ops, std::vector<int>& label, int* rc) {
  const int n = c->nqubits;
  ops.clear();
  label.resize(n);
  for (int q = 0; q < n; ++q) label[q] = q;
  std::vector<int> run(n, -1), lone(n, -1);  // open op per qubit: a run, the X it may go to
  std::vector<cd> U;
  auto diag = [](const cd* u) { return u[1] == cd(0, 0) && u[2] == cd(0, 0); };
  auto close = [&](int q) {  // the run on q takes no more gates
    if (run[q] >= 0) {
      LOp& r = ops[run[q]];
      if (diag(r.u)) r.kind = RU_DIAG;
      else if (lone[q] >= 0) {  // to the place of the X before it
        LOp& x = ops[lone[q]];
        r.xmask = x.mask;
        r.xvals = x.vals;
        r.pre = true;
        x = r;
        r.dead = true;
      }
    }
    run[q] = lone[q] = -1;
  };
  for (const qs_gate_desc& g : c->gates) {
    uint64_t span = g.ctrl_mask;
    for (int j = 0; j < g.nlocs; ++j) span |= 1ull << g.locs[j];
    if (__builtin_popcountll(span) > QS_MAXK) return false;  // wider than a block
    if (g.kind == QS_GATE_SWAP && !g.ctrl_mask) {
      std::swap(label[g.locs[0]], label[g.locs[1]]);
      continue;
    }
    if (g.nlocs != 1) return false;
    *rc = gate_matrix(c, g, params, U);
    if (*rc != QS_OK) return false;
    const int t = label[g.locs[0]];
    if (!g.ctrl_mask) {
      if (run[t] < 0) {
        LOp o;
        o.kind = RU_DENSE;
        o.t = t;
        std::copy(U.begin(), U.end(), o.u);
        run[t] = (int)ops.size();
        ops.push_back(o);
      } else {
        cd* a = ops[run[t]].u;
        const cd m[4] = {U[0] * a[0] + U[1] * a[2], U[0] * a[1] + U[1] * a[3], U[2] * a[0] + U[3] * a[2],
                         U[2] * a[1] + U[3] * a[3]};
        std::copy(m, m + 4, a);
      }
      continue;
    }
    LOp o;
    o.t = t;
    for (int q = 0; q < n; ++q)
      if ((g.ctrl_mask >> q) & 1) {
        close(label[q]);
        o.mask |= 1u << label[q];
        if ((g.ctrl_vals >> q) & 1) o.vals |= 1u << label[q];
      }
    const bool x = g.kind == QS_GATE_X;
    if (x && run[t] >= 0 && lone[t] < 0 && !diag(ops[run[t]].u)) {  // the run moves here with the X
      LOp r = ops[run[t]];
      ops[run[t]].dead = true;
      r.xmask = o.mask;
      r.xvals = o.vals;
      run[t] = -1;
      ops.push_back(r);
      continue;
    }
    close(t);
    std::copy(U.begin(), U.end(), o.u);
    o.kind = x ? RU_X : diag(o.u) ? RU_DIAG : RU_DENSE;
    if (x) lone[t] = (int)ops.size();
    ops.push_back(o);
  }
  for (int q = 0; q < n; ++q) close(q);
  ops.erase(std::remove_if(ops.begin(), ops.end(), [](const LOp& o) { return o.dead; }), ops.end());
  return true;
}

template <typename R>
RunOp<R> phys(const LOp& l, const std::vector<int>& at) {
  RunOp<R> o;
  std::memset((void*)&o, 0, sizeof(o));
  auto map = [&](uint32_t m) {
    uint32_t r = 0;
    for (size_t q = 0; q < at.size(); ++q) r |= ((m >> q) & 1u) << at[q];
    return r;
  };
  o.kind = (int8_t)l.kind;
  o.t = (int8_t)at[l.t];
  o.pre = l.pre;
  o.mask = map(l.mask);
  o.vals = map(l.vals);
  o.xmask = map(l.xmask);
  o.xvals = map(l.xvals);
  for (int k = 0; k < 4; ++k) {
    o.u[k].x = (R)l.u[k].real();
    o.u[k].y = (R)l.u[k].imag();
    if constexpr (sizeof(R) == 4)
      o.w[k] = make_float2((float)(l.u[k].real() - (double)o.u[k].x), (float)(l.u[k].imag() - (double)o.u[k].y));
  }
  return o;
}

// the ops in an order in which targets are not rank bits (the top lc), with exchanges; an
// op moves earlier only past ops on other qubits.  at[q]: physical bit of label q
template <typename R>
void schedule(std::vector<LOp> left, int n, int lc, std::vector<int>& at, std::vector<RunOp<R>>& out) {
  at.resize(n);
  for (int q = 0; q < n; ++q) at[q] = q;
  const int L = n - lc;
  std::vector<LOp> rest;
  for (;;) {
    rest.clear();
    uint32_t blocked = 0;
    for (const LOp& o : left) {
      if ((o.qubits() & blocked) || (o.kind != RU_DIAG && at[o.t] >= L)) {
        blocked |= o.qubits();
        rest.push_back(o);
      } else {
        out.push_back(phys<R>(o, at));
      }
    }
    if (rest.empty()) return;
    left.swap(rest);
    // rank bits for the labels that are targets last
    std::vector<int> next(n, 1 << 30), order(n);
    for (int k = (int)left.size() - 1; k >= 0; --k)
      if (left[k].kind != RU_DIAG) next[left[k].t] = k;
    for (int q = 0; q < n; ++q) order[q] = q;
    std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return next[a] > next[b]; });
    RunOp<R> x;
    std::memset((void*)&x, 0, sizeof(x));
    x.kind = RU_EXCH;
    std::vector<int> in, outl;
    for (int k = 0; k < n; ++k) {
      const int q = order[k];
      if (k < lc && at[q] < L) in.push_back(q);
      if (k >= lc && at[q] >= L) outl.push_back(q);
    }
    for (size_t k = 0; k < in.size(); ++k) {
      x.a[k] = (int8_t)at[in[k]];
      x.b[k] = (int8_t)at[outl[k]];
      std::swap(at[in[k]], at[outl[k]]);
    }
    x.npair = (int8_t)in.size();
    out.push_back(x);
  }
}

// ------------------------------------------------------------------ host: launch

struct RunCache {
  int dtype = -1, device = -1, kmax = 0;
  bool fits = false, asked = false;
  std::vector<double> params;
  std::vector<RunOp<float>> f;
  std::vector<RunOp<double>> d;
  std::vector<int> place;  // physical bit of each qubit at the end
};

// Whether the ops take less here than the circuit's blocks of kmax qubits would in the
// cooperative launch (k_onelaunch, every SM, a grid barrier a block): a block takes the same time
// whatever the number of its gates, an op grows with the amplitudes that a CTA holds (16 CTAs at
// most).  Nanoseconds, fitted to 2200 pairs of times over 3 to 14 qubits, kmax 2, 4 and 5, circuits
// that spread over the register or pile up on two or five qubits (the times of either side within
// a third of the fit; the path taken at most 1.21 of the better one, in 22 cases over 1.03).
// Measured, complex64 / complex128: 300 controlled Rx on five of 10 qubits 98 / 143 us here, 13 / 15
// us as one block; the same over all 14 qubits 182 / 643 us here, 287 / 483 us as blocks for 200 of
// them; 10 layers of Rz Rx Rz and a CNOT ring on 12 qubits 56 / 97 us here, 151 / 194 us as blocks.
// A circuit with parameters pays the host for the block matrices whenever its angles change, and
// a pass with new angles counts as much as one with the same: half of that (18 ns a gate for every
// row of its block's matrix, 110 ns a gate here) goes to the blocks' side.
template <typename R>
bool cluster_pays(const std::vector<RunOp<R>>& ops, const qs_circuit* c, int kmax) {
  const bool f64 = sizeof(R) == 8;
  const int n = c->nqubits;
  const int64_t a = n > 11 ? 1ll << (n - 11) : 1;  // FP64 warps' shares of a CTA's amplitudes
  int64_t here = 0;
  for (const RunOp<R>& o : ops) switch (o.kind) {
      case RU_DIAG: here += f64 ? 120 + 100 * a : 160 + 12 * a; break;
      case RU_X: here += 180; break;
      case RU_DENSE: here += f64 ? 190 + 230 * a : 240 + 45 * a; break;
      default: here += 500 + 200 * a;
    }
  std::vector<int> widths;
  block_widths(c, kmax, widths);
  const int nb = (int)widths.size();
  const int64_t block = f64 ? (n < 10 ? 4600 : 5800) + 400 * (a - 1) : 4000 + 200 * (a - 1);
  int64_t blocks = 2500 + nb * block;
  if (c->nparams > 0 && nb > 0) {
    int64_t rows = 0;
    for (int b = 0; b < nb; ++b) rows += 1ll << widths[b];
    blocks += 4000 + std::max<int64_t>(0, (9 * rows / nb - 55) * (int64_t)c->gates.size());
  }
  return here <= blocks;
}

// CTAs of the cluster: one for every 128 amplitudes (a warp for each FP64 unit of an SM)
int rank_bits(int n) { return std::max(0, std::min(4, n - 7)); }

template <typename R, int CAP>
int launch_cap(c2_t<R>* psi, const RunArgs& a, const RunOp<R>* ops, bool ask, cudaStream_t st) {
  RunOps<R, CAP> list;
  std::memcpy((void*)list.op, ops, sizeof(RunOp<R>) * a.nops);
  cudaLaunchConfig_t cfg;
  std::memset(&cfg, 0, sizeof(cfg));
  cfg.gridDim = dim3(1u << a.lc);
  cfg.blockDim = dim3(std::max(32, 1 << (a.n - a.lc)));
  cfg.dynamicSmemBytes = (sizeof(c2_t<R>) * 4) << (a.n - a.lc);
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = 1u << a.lc;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  QS_CUDA(cudaFuncSetAttribute(k_small_run<R, CAP>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
  if (cfg.dynamicSmemBytes > 32 * 1024)
    QS_CUDA(cudaFuncSetAttribute(k_small_run<R, CAP>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)cfg.dynamicSmemBytes));
  if (ask) {  // whether the device places a cluster of this size
    int clusters = 0;
    if (cudaOccupancyMaxActiveClusters(&clusters, k_small_run<R, CAP>, &cfg) != cudaSuccess || clusters < 1) {
      cudaGetLastError();
      return QS_EUNSUPPORTED;
    }
  }
  QS_CUDA(cudaLaunchKernelEx(&cfg, k_small_run<R, CAP>, psi, a, list));
  return QS_OK;
}

constexpr int kRunCaps[3] = {48, 144, 320};  // ops of a launch: its parameters hold them

template <typename R>
int launch_run(c2_t<R>* psi, const RunArgs& a, const std::vector<RunOp<R>>& ops, bool ask, cudaStream_t st) {
  static_assert(sizeof(RunOp<R>) * kRunCaps[2] + sizeof(RunArgs) + 64 < 32764, "kernel parameters");
  if (a.nops <= kRunCaps[0]) return launch_cap<R, kRunCaps[0]>(psi, a, ops.data(), ask, st);
  if (a.nops <= kRunCaps[1]) return launch_cap<R, kRunCaps[1]>(psi, a, ops.data(), ask, st);
  return launch_cap<R, kRunCaps[2]>(psi, a, ops.data(), ask, st);
}

}  // namespace

void free_smallrun(const qs_circuit* c) {
  delete static_cast<RunCache*>(c->smallrun);
  c->smallrun = nullptr;
}

// Runs circuit c on the single register at `data`, <o> (Z strings) to dev_out if not NULL.
// QS_EUNSUPPORTED, with nothing launched: the circuit is not one of this path's, or takes
// less as blocks of kmax qubits.
int run_small_circuit(void* data, int dtype, const qs_circuit* c, const double* params, int kmax, const qs_observable* o,
                      double* dev_out, cudaStream_t st) {
  const int n = c->nqubits;
  if (n > kRunMaxQubits || (o && o->terms.size() > (size_t)kRunTerms)) return QS_EUNSUPPORTED;
  int dev = 0;
  QS_CUDA(cudaGetDevice(&dev));
  RunCache* k = static_cast<RunCache*>(c->smallrun);
  const int np = c->nparams;
  if (!k || k->dtype != dtype || k->device != dev || k->kmax != kmax || (int)k->params.size() != np ||
      (np && std::memcmp(k->params.data(), params, sizeof(double) * np) != 0)) {
    free_smallrun(c);
    k = new RunCache();
    c->smallrun = k;  // owned by the circuit
    k->dtype = dtype;
    k->device = dev;
    k->kmax = kmax;
    if (np) k->params.assign(params, params + np);
    std::vector<LOp> ops;
    std::vector<int> label, at;
    int rc = QS_OK;
    k->fits = fuse(c, params, ops, label, &rc);
    if (rc != QS_OK) {
      free_smallrun(c);
      return rc;
    }
    if (k->fits) {
      if (dtype == QS_C64) schedule(ops, n, rank_bits(n), at, k->f);
      else schedule(ops, n, rank_bits(n), at, k->d);
      k->place.resize(n);
      for (int q = 0; q < n; ++q) k->place[q] = at[label[q]];
      k->fits = std::max(k->f.size(), k->d.size()) <= (size_t)kRunCaps[2] &&
                (dtype == QS_C64 ? cluster_pays(k->f, c, kmax) : cluster_pays(k->d, c, kmax));
    }
  }
  if (!k->fits) return QS_EUNSUPPORTED;
  RunArgs a;
  std::memset(&a, 0, sizeof(a));
  a.n = n;
  a.lc = rank_bits(n);
  a.nops = (int)std::max(k->f.size(), k->d.size());
  for (int q = 0; q < n; ++q) a.place[q] = (int8_t)k->place[q];
  if (o) {
    a.out = dev_out;
    for (const auto& t : o->terms) {
      for (int q = 0; q < n; ++q) a.z[a.nterm] |= (uint32_t)((t.z_mask >> q) & 1) << k->place[q];
      a.c[a.nterm++] = t.coeff;
    }
  }
  const int rc = dtype == QS_C64 ? launch_run((float2*)data, a, k->f, !k->asked, st)
                                 : launch_run((double2*)data, a, k->d, !k->asked, st);
  k->asked = true;
  if (rc == QS_EUNSUPPORTED) k->fits = false;
  return rc;
}

}  // namespace qs
