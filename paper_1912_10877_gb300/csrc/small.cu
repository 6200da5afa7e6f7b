// small.cu -- the gate-by-gate path of registers that fit a thread-block cluster, many
// gates in one launch (sm_103a): apply! of a chain (Sec. "Representing Quantum
// Circuits") on small registers, where a launch a gate costs more than its arithmetic.
//
// A register's amplitudes live in the registers of one cluster's threads: index bits
// 0..4 are lanes, the next ones threads, then a thread's own amplitudes, the highest
// the CTA's rank in the cluster.  Every thread works out its own amplitudes' new values;
// the partner's value comes by shuffle, through shared memory, from its own registers or
// from another CTA's shared memory.  Diagonal gates need no exchange.  The arithmetic of
// a gate is that of its kernel in gates.cu, operation for operation, so the amplitudes
// are the same bit for bit.
//
// Bound by latency: a gate is a barrier and a chain of at most four dependent FP64
// operations (87 clocks each), a launch was 4 to 6 us.  One CTA holds 128 amplitudes
// (a warp for each of the SM's four FP64 units) before a second CTA is used, up to
// eight.  QFT of 10 qubits complex128, 55 gates: 17.9 us on the GPU and 19 us a call, 320
// us as 55 launches; of 13 qubits with swaps 84 us.
#include <cooperative_groups.h>

#include <cstring>

#include "common.cuh"

namespace qs {

namespace {

namespace cg = cooperative_groups;

constexpr int kSmallThreads = 1024;
constexpr int kSmallMaxQubits = 14;       // 8 CTAs x 1024 threads x 2 amplitudes
// Amplitudes of all registers up to which the path is taken: a dense complex128 gate on
// 2^17 takes 2 us of FP64 arithmetic wherever it runs, half of what its launch takes
// (4.5 us); beyond, launches are hidden by the arithmetic and a kernel that visits only
// the amplitudes a gate touches is the better one.
constexpr uint64_t kSmallAmps = 1 << 17;

enum { SM_DIAG = 0, SM_SWAP, SM_PERM, SM_REAL, SM_RX, SM_DENSE, SM_SWAP2 };

template <typename R>
struct SmallOp {
  uint32_t mask, vals;  // where it acts: controls (SM_DIAG: the touched subspace)
  int16_t kind, t, t2, pad;
  c2_t<R> u[4];         // SM_DIAG: u[0], u[3] by bit t (t < 0: u[0])
};
template <typename R, int CAP>
struct SmallOps {
  SmallOp<R> op[CAP];
};

__device__ __forceinline__ float2 shfl2(float2 v, int m) {
  return make_float2(__shfl_xor_sync(0xffffffffu, v.x, m), __shfl_xor_sync(0xffffffffu, v.y, m));
}
__device__ __forceinline__ double2 shfl2(double2 v, int m) {
  return make_double2(__shfl_xor_sync(0xffffffffu, v.x, m), __shfl_xor_sync(0xffffffffu, v.y, m));
}

// new value of an amplitude x whose bit t is `one`, partner y (pair_op of gates.cu)
template <typename R>
__device__ __forceinline__ c2_t<R> small_out(int kind, const c2_t<R>* u, c2_t<R> x, c2_t<R> y, bool one) {
  using T = c2_t<R>;
  if (kind == SM_SWAP) return y;
  const T v0 = one ? u[2] : u[0], v1 = one ? u[3] : u[1];  // the row of the matrix
  const T a = one ? y : x, b = one ? x : y;
  T r;
  switch (kind) {
    case SM_PERM:
      return cmul(one ? v0 : v1, y);
    case SM_REAL:
      r.x = fma(v1.x, b.x, v0.x * a.x);
      r.y = fma(v1.x, b.y, v0.x * a.y);
      return r;
    case SM_RX:  // a real diagonal, imaginary beside it
      r.x = fma(one ? v1.x : -v1.y, one ? b.x : b.y, (one ? -v0.y : v0.x) * (one ? a.y : a.x));
      r.y = fma(one ? v1.x : v1.y, one ? b.y : b.x, (one ? v0.y : v0.x) * (one ? a.x : a.y));
      return r;
    default:
      return cfma(v1, b, cmul(v0, a));
  }
}

// E (1 or 2) amplitudes a thread; threads and CTAs as the launch has them
template <typename R, int E, int CAP>
__global__ void __launch_bounds__(kSmallThreads)
k_small(c2_t<R>* __restrict__ psi, int n, int nops, const __grid_constant__ SmallOps<R, CAP> ops) {
  using T = c2_t<R>;
  extern __shared__ __align__(16) unsigned char smraw[];
  T* buf = reinterpret_cast<T*>(smraw);  // two exchange areas of the CTA's amplitudes, two for other CTAs to read
  cg::cluster_group cl = cg::this_cluster();
  const unsigned cs = cl.num_blocks(), rank = cl.block_rank();
  const int lc = 31 - __clz((int)cs), L = n - lc;  // bits of a CTA's amplitudes
  const uint32_t nt = 1u << (L - (E - 1));  // threads that hold amplitudes (may be below a warp)
  static_assert(E == 1 || E == 2, "an own partner is the other amplitude");
  const int lt = 31 - __clz((int)nt);
  const uint32_t tid = threadIdx.x, hi = rank << L, area = 1u << L;
  const bool act = tid < nt;
  T* reg = psi + ((uint64_t)(blockIdx.x / cs) << n) + hi;
  T x[E];
#pragma unroll
  for (int e = 0; e < E; ++e) x[e] = act ? reg[e * nt + tid] : cmk<T>(0, 0);
  int turn = 0, rturn = 0;
  for (int o = 0; o < nops; ++o) {
    const SmallOp<R>& op = ops.op[o];
    const int kind = op.kind, t = op.t;
    const uint32_t mask = op.mask, vals = op.vals;
    if (kind == SM_DIAG) {
#pragma unroll
      for (int e = 0; e < E; ++e) {
        const uint32_t i = hi | (e * nt + tid);
        if ((i & mask) == vals) x[e] = cmul(x[e], t >= 0 && ((i >> t) & 1u) ? op.u[3] : op.u[0]);
      }
      continue;
    }
    T y[E];
    if (kind == SM_SWAP2 || t >= L) {
      // the partner may be in any CTA of the cluster.  The areas alternate: a CTA writes one
      // again only after a barrier that follows every read of it
      T* a = buf + (2 + rturn) * area;
      if (act) {
#pragma unroll
        for (int e = 0; e < E; ++e) a[e * nt + tid] = x[e];
      }
      cl.sync();
#pragma unroll
      for (int e = 0; e < E; ++e) {
        const uint32_t i = hi | (e * nt + tid);
        uint32_t j = i ^ (1u << t);
        if (kind == SM_SWAP2) {
          const uint32_t d = ((i >> t) ^ (i >> op.t2)) & 1u;
          j = i ^ ((d << t) | (d << op.t2));
        }
        if (act) y[e] = cl.map_shared_rank(a, j >> L)[j & (area - 1)];
      }
      rturn ^= 1;
    } else if (t >= lt) {
#pragma unroll
      for (int e = 0; e < E; ++e) y[e] = x[e ^ (E - 1)];
    } else if (t < 5) {
#pragma unroll
      for (int e = 0; e < E; ++e) y[e] = shfl2(x[e], 1 << t);
    } else {
      T* a = buf + turn * area;
      if (act) {
#pragma unroll
        for (int e = 0; e < E; ++e) a[e * nt + tid] = x[e];
      }
      __syncthreads();
      if (act) {
#pragma unroll
        for (int e = 0; e < E; ++e) y[e] = a[(e * nt + tid) ^ (1u << t)];
      }
      turn ^= 1;
    }
#pragma unroll
    for (int e = 0; e < E; ++e) {
      const uint32_t i = hi | (e * nt + tid);
      if ((i & mask) == vals) x[e] = kind == SM_SWAP2 ? y[e] : small_out<R>(kind, op.u, x[e], y[e], (i >> t) & 1u);
    }
  }
  if (act) {
#pragma unroll
    for (int e = 0; e < E; ++e) reg[e * nt + tid] = x[e];
  }
  if (cs > 1) cl.sync();  // no CTA leaves while another may read its shared memory
}

template <typename R>
c2_t<R> cast(cd v) {
  c2_t<R> r;
  r.x = (R)v.real();
  r.y = (R)v.imag();
  return r;
}

// the op of a plan; false: not one of this path's
template <typename R>
bool small_op(const Plan& p, SmallOp<R>* o) {
  std::memset(o, 0, sizeof(*o));
  o->t = (int16_t)p.t;
  o->mask = (uint32_t)p.ctrl_mask;
  o->vals = (uint32_t)p.ctrl_vals;
  if (p.precise) return false;
  switch (p.op) {
    case OP_DIAG1:
      o->kind = SM_DIAG;
      o->mask = (uint32_t)p.mask;
      o->vals = (uint32_t)p.vals;
      o->u[0] = cast<R>(p.d0);
      o->u[3] = cast<R>(p.d1);
      return true;
    case OP_PERMK:
      if (p.k != 2 || p.perm[0] != 0 || p.perm[1] != 2 || p.perm[2] != 1) return false;
      for (int m = 0; m < 4; ++m)
        if (p.pv[m] != cd(1, 0)) return false;
      o->kind = SM_SWAP2;
      o->t = (int16_t)p.locs[0];
      o->t2 = (int16_t)p.locs[1];
      return true;
    case OP_SWAP1: o->kind = SM_SWAP; break;
    case OP_PERM1: o->kind = SM_PERM; break;
    case OP_REAL1: case OP_HLIKE1: o->kind = SM_REAL; break;
    case OP_RXLIKE1: o->kind = SM_RX; break;
    case OP_DENSE1: o->kind = SM_DENSE; break;
    default: return false;
  }
  for (int k = 0; k < 4; ++k) o->u[k] = cast<R>(p.u[k]);
  return true;
}

template <typename R, int E, int CAP>
int launch_small(c2_t<R>* psi, int n, int nreg, const SmallOp<R>* ops, int nops, cudaStream_t st) {
  const int lc = std::max(0, std::min(3, n - 7));  // CTAs a register: 128 amplitudes each, up to 8 of them
  const int threads = std::max(32, (1 << (n - lc)) / E);
  SmallOps<R, CAP> list;
  std::memcpy(list.op, ops, sizeof(SmallOp<R>) * nops);
  cudaLaunchConfig_t cfg;
  std::memset(&cfg, 0, sizeof(cfg));
  cfg.gridDim = dim3((unsigned)nreg << lc);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = sizeof(c2_t<R>) * 4 << (n - lc);
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = 1u << lc;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  if (cfg.dynamicSmemBytes > 48 * 1024)
    QS_CUDA(cudaFuncSetAttribute(k_small<R, E, CAP>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)cfg.dynamicSmemBytes));
  QS_CUDA(cudaLaunchKernelEx(&cfg, k_small<R, E, CAP>, psi, n, nops, list));
  return QS_OK;
}

constexpr int kSmallList = 56, kLongList = 360;  // ops of a launch: its parameters hold them (at most 32 KB)

template <typename R>
int run_small(c2_t<R>* psi, int n, int nreg, const std::vector<Plan>& plans, cudaStream_t st) {
  std::vector<SmallOp<R>> ops(plans.size());
  for (size_t i = 0; i < plans.size(); ++i)
    if (!small_op<R>(plans[i], &ops[i])) return fail(QS_EINVAL, "a plan outside the small-register path");
  for (size_t at = 0; at < ops.size();) {
    const int left = (int)(ops.size() - at), k = std::min(left, kLongList);
    const bool two = n > 13;  // 1024 threads a CTA hold 2^13 amplitudes
    if (k <= kSmallList) {
      QS_TRY(two ? (launch_small<R, 2, kSmallList>(psi, n, nreg, ops.data() + at, k, st))
                 : (launch_small<R, 1, kSmallList>(psi, n, nreg, ops.data() + at, k, st)));
    } else {
      QS_TRY(two ? (launch_small<R, 2, kLongList>(psi, n, nreg, ops.data() + at, k, st))
                 : (launch_small<R, 1, kLongList>(psi, n, nreg, ops.data() + at, k, st)));
    }
    at += k;
  }
  return QS_OK;
}

}  // namespace

bool small_register(int n, int nreg) {
  return n <= kSmallMaxQubits && ((uint64_t)nreg << n) <= kSmallAmps;
}

bool small_plan(const Plan& p) {
  SmallOp<float> o;
  return small_op<float>(p, &o);
}

// A lone gate is the cheaper launch of its own kernel (10 qubits: 6.0 us a call against 7.6).
// At 14 qubits complex128 the FP64 arithmetic of a cluster's eight SMs takes about as long as the
// launch it saves: the first launch's 5 us have to come out of what a list's gates gain (tenths of
// a microsecond each).  Measured, here and as launches: a dense 2x2 on every qubit 86.0 and 84.0
// us, H 41 and 57, Rx 57.7 and 57.4; H on two qubits 10.3 and 8.3; two controlled X 6.1 and 7.4, two
// T 8.2 and 12.4; six controlled Rx 20.5 and 24.6; 2, 6 and 20 controlled dense gates 16.0, 36.9 and
// 96 against 12.3, 32.8 and 113.  Registers of a batch have a cluster each, launches more to do
// (eight of them, 60 gates Rx: 61 us here, 86 as launches).
bool small_pays(int dtype, int n, int nreg, const std::vector<Plan>& plans) {
  if (plans.size() < 2) return false;
  if (dtype == QS_C64 || n < kSmallMaxQubits || nreg > 1) return true;
  int gain = 0;
  for (const Plan& p : plans) {
    const bool ctrl = p.ctrl_mask != 0;
    if (p.op == OP_DENSE1) gain += ctrl ? 7 : 0;
    else if (p.op == OP_RXLIKE1) gain += ctrl ? 12 : 3;
    else if (p.op == OP_REAL1 || p.op == OP_HLIKE1) gain += ctrl ? 20 : 15;
    else gain += 26;
    if (gain > 50) return true;
  }
  return false;
}

int apply_small(void* data, int dtype, int n, int nreg, const std::vector<Plan>& plans, cudaStream_t st) {
  if (dtype == QS_C64) return run_small<float>((float2*)data, n, nreg, plans, st);
  return run_small<double>((double2*)data, n, nreg, plans, st);
}

}  // namespace qs
