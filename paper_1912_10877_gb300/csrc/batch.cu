// batch.cu -- batched registers of uneven sizes in one persistent launch
// (Sec. "Batched Quantum Registers"; forward, expectation and reversible
// adjoint of Sec. "Reverse Mode"), complex64.
//
// Every register has its own circuit, parameters and diagonal observable.  The
// host schedules each circuit into fused tile passes (tiles.cuh); a persistent
// grid of 512-thread CTAs takes registers from an atomic counter in
// decreasing-cost order.  A register of n <= 13 qubits lives in shared memory
// for the whole forward, expectation and backward (its lambda too); a larger
// register streams 2^13-amplitude tiles through L2 / HBM once per pass.
// Inside a tile each phase keeps 16 amplitudes per thread in registers.
//
// Backward (Eq. apply-back): the passes and phases run in reverse; for each
// gate, in reverse order, a thread adds Im sum conj(lambda) (G psi) over its
// pairs (for a run of gates on one qubit, the four sums that all their derivatives
// come from) (FP32 over <= 8 pairs, then FP32 warp shuffles, FP64 from the warp
// level up) and uncomputes psi and lambda with U^dagger in FP32, using the
// structured Rx / Ry / diagonal forms of the inverse rotations.  The
// register's gradient lives in shared memory (FP64) and is written once.
#include <algorithm>
#include <cmath>
#include <cstddef>
#include <cstring>
#include <numeric>
#include <unordered_map>

#include "tiles.cuh"

namespace qs {

constexpr int kMaxRegParams = 2048;
constexpr int kMaxPhaseOps = 64;    // gates with a parameter in a phase
constexpr int kMaxPhaseVals = 128;  // sums of its backward ops
constexpr int kMaxRun = 4;          // gates of a fused run
constexpr int kBatchTile = kMaxTileBits;

struct GSpec {           // one circuit gate of one register
  int32_t kind;
  int32_t param;         // global index into params (-1: theta)
  double theta;
  double2 mat[4];        // MATRIX gates (1 target)
};

struct FMem {            // members of a fused op (applied in order)
  int32_t count;
  int32_t g[kMaxRun];    // global GSpec indices
  int32_t rec0;          // backward: first of its GMem records (TK_RUN), else -1
};

struct BReg {
  int32_t n, m, npass, pass0;
  int32_t nparam, nterm, term0, pad;
  int64_t amp_off;       // elements into the batch state
  int64_t work_off;      // elements into psi/lambda work buffers (n > 13), -1 otherwise
  int64_t param_off;     // into params / grad
  double cost;
};

struct BTerm {
  double coeff;
  uint64_t z;
};

struct BArgs {
  float2* state;
  float2* wpsi;          // backward work copies of psi (registers larger than the tile)
  float2* wlam;          // lambda (same)
  float4* wpsif;         // precise path: double-float psi work copies
  float4* wlamf;         // precise path: double-float lambda
  const float2* flo;     // precise path: corrections U - U_hi of the forward ops (4 each)
  const float2* dtlo;    // precise path: corrections of the diagonal tables (16 each)
  const float2* blo;     // precise path: corrections of the backward ops' U^dagger (4 each)
  const BReg* regs;
  const int32_t* order;
  const TPass* passes;
  const TPhase* phases;
  const TOp* fops;
  const TOp* bops;
  const GMem* gmem;
  const float2* dtab;    // TK_DIAG16 factor tables
  const DRun* druns;     // TK_DIAGRUN entries
  const float4* rtab;    // TK_DIAGRUN tables (kRunTab a run)
  const BTerm* terms;
  double* loss;
  double* grad;
  int* counter;
  int nreg;
  int flags;
};

enum { BF_RESET = 1, BF_GRAD = 2 };

// ------------------------------------------------------------------ device: ops on the amplitudes of a phase
//
// A phase of RB register bits (RB = 2..4) keeps 2^RB amplitudes per thread in
// registers.  The complex64 path computes in FP32.  The precise path of the
// batched engine (PREC) applies the forward gates with compensated matrices
// (every FP32 entry U_hi has a correction U_lo = U - U_hi kept beside it, so
// the state sees U to ~2^-48 while it is still stored and multiplied in FP32)
// and runs the reversible uncompute of psi and lambda in double-float
// arithmetic (each real number a pair hi + lo of FP32 values, ~48 bits): the
// uncompute is FP64-class without the FP64 units, which run at 1/64 of the
// FP32 rate on this GPU.

__device__ __forceinline__ float2 cmulf(float2 a, float2 b) {
  return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ float2 cmaf(float2 a, float2 b, float2 c) {  // a*b + c
  c.x = fmaf(a.x, b.x, c.x);
  c.x = fmaf(-a.y, b.y, c.x);
  c.y = fmaf(a.x, b.y, c.y);
  c.y = fmaf(a.y, b.x, c.y);
  return c;
}
__device__ __forceinline__ float imcj(float2 p, float2 q) { return fmaf(p.x, q.y, -p.y * q.x); }  // Im(conj(p) q)
__device__ __forceinline__ float recj(float2 p, float2 q) { return fmaf(p.x, q.x, p.y * q.y); }   // Re(conj(p) q)

// (a, b) <- U (a, b) for the structured kinds; U row-major in u0..u3
// a diagonal whose first entry is exactly 1 (shift, controlled phases): only b changes
constexpr int TK_DIAGB = 16;
// a real 2x2
constexpr int TK_REAL = 17;

template <int KIND>
__device__ __forceinline__ void pair_apply(float2& a, float2& b, float2 u0, float2 u1, float2 u2, float2 u3) {
  if (KIND == TK_SWAP) {
    const float2 t = a; a = b; b = t;
  } else if (KIND == TK_DIAGB) {
    b = cmulf(b, u3);
  } else if (KIND == TK_DIAG) {
    a = cmulf(a, u0);
    b = cmulf(b, u3);
  } else if (KIND == TK_RX) {  // [[c, i s], [i s, c]] (c = u0.x, s = u1.y)
    const float c = u0.x, s = u1.y;
    const float2 na = make_float2(fmaf(c, a.x, -s * b.y), fmaf(c, a.y, s * b.x));
    const float2 nb = make_float2(fmaf(c, b.x, -s * a.y), fmaf(c, b.y, s * a.x));
    a = na; b = nb;
  } else if (KIND == TK_RY) {  // real [[c, u1], [u2, c]]
    const float c = u0.x, p = u1.x, q = u2.x;
    const float2 na = make_float2(fmaf(c, a.x, p * b.x), fmaf(c, a.y, p * b.y));
    const float2 nb = make_float2(fmaf(q, a.x, c * b.x), fmaf(q, a.y, c * b.y));
    a = na; b = nb;
  } else if (KIND == TK_REAL) {
    const float2 na = make_float2(fmaf(u0.x, a.x, u1.x * b.x), fmaf(u0.x, a.y, u1.x * b.y));
    const float2 nb = make_float2(fmaf(u2.x, a.x, u3.x * b.x), fmaf(u2.x, a.y, u3.x * b.y));
    a = na; b = nb;
  } else {
    const float2 na = cmaf(u1, b, cmulf(u0, a));
    const float2 nb = cmaf(u3, b, cmulf(u2, a));
    a = na; b = nb;
  }
}

// compensated forward (cf_mul / cf_dot2: the FP64-exact matrix applied to the
// FP32 amplitudes in double-float, each output rounded to FP32 once)
template <int KIND>
__device__ __forceinline__ void pair_apply_c(float2& a, float2& b, const float2 (&u)[4], const float2 (&w)[4]) {
  if (KIND == TK_SWAP) {
    const float2 t = a; a = b; b = t;
  } else if (KIND == TK_DIAG) {
    a = cf_mul(a, u[0], w[0]);
    b = cf_mul(b, u[3], w[3]);
  } else {
    const float2 na = cf_dot2(a, u[0], w[0], b, u[1], w[1]);
    const float2 nb = cf_dot2(a, u[2], w[2], b, u[3], w[3]);
    a = na; b = nb;
  }
}

template <int RB, int T, int KIND, bool CTRL>
__device__ __forceinline__ void op_fwd(float2 (&x)[1 << RB], const TOp& op) {
  const int cm = op.cmask, cv = op.cval;
  const float2 u0 = op.u[0], u1 = op.u[1], u2 = op.u[2], u3 = op.u[3];
#pragma unroll
  for (int j = 0; j < (1 << RB); ++j) {
    if (j & (1 << T)) continue;
    if (CTRL && (j & cm) != cv) continue;
    pair_apply<KIND>(x[j], x[j | (1 << T)], u0, u1, u2, u3);
  }
}

template <int RB, int T, int KIND, bool CTRL>
__device__ __forceinline__ void op_fwd_c(float2 (&x)[1 << RB], const TOp& op, const float2* lo) {
  const int cm = op.cmask, cv = op.cval;
  const float2 u[4] = {op.u[0], op.u[1], op.u[2], op.u[3]};
  const float2 w[4] = {lo[0], lo[1], lo[2], lo[3]};
#pragma unroll
  for (int j = 0; j < (1 << RB); ++j) {
    if (j & (1 << T)) continue;
    if (CTRL && (j & cm) != cv) continue;
    pair_apply_c<KIND>(x[j], x[j | (1 << T)], u, w);
  }
}

// A run's 2x2 with X on the same bit, before it (PRE) or after, where the X is
// controlled: C >= 0: by phase bit C; else on every pair if `on`.  The X renames the
// inputs or outputs of the pairs it acts on.
template <int RB, int T, int C, bool PRE>
__device__ __forceinline__ void op_fwd_x(float2 (&x)[1 << RB], const TOp& op, bool on) {
  if constexpr (T < RB && C < RB && C != T) {
    const bool sw = C < 0 && on;
    constexpr int P = PRE ? 1 : 2;  // columns or rows trade places
    const float2 u0 = sw ? op.u[P] : op.u[0], u1 = sw ? op.u[P ^ 1] : op.u[1];
    const float2 u2 = sw ? op.u[P ^ 2] : op.u[2], u3 = sw ? op.u[P ^ 3] : op.u[3];
#pragma unroll
    for (int j = 0; j < (1 << RB); ++j) {
      if (j & (1 << T)) continue;
      const bool ren = C >= 0 && ((j >> (C < 0 ? 0 : C)) & 1);
      const int k = j | (1 << T), ja = PRE && ren ? k : j, jb = PRE && ren ? j : k;
      const float2 a = x[ja], b = x[jb];
      const float2 na = cmaf(u1, b, cmulf(u0, a)), nb = cmaf(u3, b, cmulf(u2, a));
      x[!PRE && ren ? k : j] = na;
      x[!PRE && ren ? j : k] = nb;
    }
  }
}
template <int RB, int T, int C, bool PRE>
__device__ __forceinline__ void op_fwd_x_c(float2 (&x)[1 << RB], const TOp& op, const float2* lo, bool on) {
  if constexpr (T < RB && C < RB && C != T) {
    const bool sw = C < 0 && on;
    constexpr int P = PRE ? 1 : 2;
    const float2 u0 = sw ? op.u[P] : op.u[0], u1 = sw ? op.u[P ^ 1] : op.u[1];
    const float2 u2 = sw ? op.u[P ^ 2] : op.u[2], u3 = sw ? op.u[P ^ 3] : op.u[3];
    const float2 w0 = lo[sw ? P : 0], w1 = lo[sw ? P ^ 1 : 1], w2 = lo[sw ? P ^ 2 : 2], w3 = lo[sw ? P ^ 3 : 3];
#pragma unroll
    for (int j = 0; j < (1 << RB); ++j) {
      if (j & (1 << T)) continue;
      const bool ren = C >= 0 && ((j >> (C < 0 ? 0 : C)) & 1);
      const int k = j | (1 << T), ja = PRE && ren ? k : j, jb = PRE && ren ? j : k;
      const float2 na = cf_dot2(x[ja], u0, w0, x[jb], u1, w1), nb = cf_dot2(x[ja], u2, w2, x[jb], u3, w3);
      x[!PRE && ren ? k : j] = na;
      x[!PRE && ren ? j : k] = nb;
    }
  }
}

// x_j *= (bit T of j ? p1 : p0)
template <int RB, int T>
__device__ __forceinline__ void mul_by_bit(float2 (&x)[1 << RB], float2 p0, float2 p1) {
#pragma unroll
  for (int j = 0; j < (1 << RB); ++j) x[j] = cmulf(x[j], ((j >> T) & 1) ? p1 : p0);
}

// x_j *= p1 where bit T of j is 1
template <int RB, int T>
__device__ __forceinline__ void mul_bit1(float2 (&x)[1 << RB], float2 p1) {
#pragma unroll
  for (int j = 0; j < (1 << RB); ++j)
    if ((j >> T) & 1) x[j] = cmulf(x[j], p1);
}

// one entry of a run where its controls hold, by a thread of index bits gb
__device__ __forceinline__ void run_entry(const DRun* e, uint32_t gb, float2& p0, float2& p1) {
  const uint4* w = reinterpret_cast<const uint4*>(e);
  const uint4 a = w[0], b = w[1];  // tmask, tval, gate, tq | u0, u3
  const float2 u0 = make_float2(__uint_as_float(b.x), __uint_as_float(b.y));
  const float2 u3 = make_float2(__uint_as_float(b.z), __uint_as_float(b.w));
  const bool on = (gb & a.x) == a.y;
  float2 f0 = u0, f1 = u3;
  if (a.w != 0xffffffffu) {  // target outside the phase: one factor by its bit
    f0 = ((gb >> (a.w & 31u)) & 1u) ? u3 : u0;
    f1 = f0;
  }
  const float2 q0 = cmulf(p0, f0), q1 = cmulf(p1, f1);
  p0 = on ? q0 : p0;
  p1 = on ? q1 : p1;
}

// What a TK_DIAGRUN op reads besides its record: the pass's entries, its runs' tables
// and, in the tile engine, the products of each run's tile-id entries for this tile.  In
// shared memory, so that the op loops carry one pointer for it.
struct RunCtx {
  const DRun* entries;
  const float4* tab;
  const float4* tile;  // NULL: those entries are applied thread by thread
};

// a TK_DIAGRUN op: the products p0, p1 of its entries' factors, then one pass over the
// amplitudes by phase bit t.  The table look-ups replace up to n - 4 entries tested and
// multiplied by every thread (QFT of 29 qubits, first pass: 20.7 -> 11.0 ms, with the
// phases no longer cut at 64 gates).
template <int RB>
__device__ __forceinline__ void diag_run(float2 (&x)[1 << RB], const TOp& op, const RunCtx& rc, uint32_t gb) {
  const int run = __float_as_int(op.cfac2);
  const float4* tab = rc.tab + run * kRunTab;
  const float4 a = tab[threadIdx.x & 31], b = tab[32 + (threadIdx.x >> 5)];
  float2 p0 = make_float2(1.f, 0.f);
  float2 p1 = cmulf(make_float2(a.z, a.w), make_float2(b.z, b.w));
  const bool one0 = op.gen == 1;
  if (!one0) p0 = cmulf(make_float2(a.x, a.y), make_float2(b.x, b.y));
  uint32_t k = 0;
  if (rc.tile) {
    const float4 t = rc.tile[run];
    if (!one0) p0 = cmulf(p0, make_float2(t.x, t.y));
    p1 = cmulf(p1, make_float2(t.z, t.w));
    k = op.shared;
  }
  const DRun* e = rc.entries + op.param;
  for (; k < op.count; ++k) run_entry(e + k, gb, p0, p1);
  if (one0) {
    switch (op.t) {
      case 0: mul_bit1<RB, 0>(x, p1); break;
      case 1: mul_bit1<RB, 1>(x, p1); break;
      case 2: if constexpr (RB > 2) mul_bit1<RB, 2>(x, p1); break;
      default: if constexpr (RB > 3) mul_bit1<RB, 3>(x, p1); break;
    }
  } else {
    switch (op.t) {
      case 0: mul_by_bit<RB, 0>(x, p0, p1); break;
      case 1: mul_by_bit<RB, 1>(x, p0, p1); break;
      case 2: if constexpr (RB > 2) mul_by_bit<RB, 2>(x, p0, p1); break;
      default: if constexpr (RB > 3) mul_by_bit<RB, 3>(x, p0, p1); break;
    }
  }
}

// A TK_REALRUN op: the layer of one qubit of a QFT (H, then the controlled phases on it) in
// one dispatch.  Bound by instruction issue: H, table and run as ops of their own took 490
// instructions a thread for the 16 amplitudes, two thirds of them record loads, jumps and
// register moves, and multiplied the 8 amplitudes that the table leaves alone as well
// (QFT of 29 qubits: 26.3 -> 20.6 ms; its passes 11.0, 7.3, 6.4 -> 7.5, 5.1, 5.4).
template <int RB, int T>
__device__ __forceinline__ void real_run(float2 (&x)[1 << RB], const TOp& op, const RunCtx& rc, const float2* dtab,
                                         uint32_t gb) {
  if constexpr (T < RB) {
    const int run = __float_as_int(op.cfac2);
    const float4* tab = rc.tab + run * kRunTab;
    const float4 a = tab[threadIdx.x & 31], b = tab[32 + (threadIdx.x >> 5)];
    float2 p = cmulf(make_float2(a.z, a.w), make_float2(b.z, b.w));
    uint32_t k = 0;
    if (rc.tile) {
      const float4 t = rc.tile[run];
      p = cmulf(p, make_float2(t.z, t.w));
      k = op.shared;
    }
    float2 p0 = make_float2(1.f, 0.f);  // stays 1
    for (; k < op.count; ++k) run_entry(rc.entries + op.param + k, gb, p0, p);
    op_fwd<RB, T, TK_REAL, false>(x, op);
    if (op.pad) {
      const float2* d = dtab + 16 * (op.pad - 1);
#pragma unroll
      for (int j = 0; j < (1 << RB); j += 2) {
        if (T > 0 && !((j >> T) & 1)) continue;
        const float4 f = *reinterpret_cast<const float4*>(d + j);
        if (T > 0) x[j] = cmulf(x[j], cmulf(p, make_float2(f.x, f.y)));
        x[j + 1] = cmulf(x[j + 1], cmulf(p, make_float2(f.z, f.w)));
      }
    } else {
      mul_bit1<RB, T>(x, p);
    }
  }
}

// Forward op forms by TOp::var: 0 out-of-phase diagonal, 1 diagonal table,
// 2 + t controlled swap, 6 + t / 10 + t diagonal without / with phase-local
// controls, 14 + t / 18 + t dense without / with them (t: target phase bit),
// 22 a run of diagonal gates (TK_DIAGRUN), 23 + t dense and real without controls (H:
// half the multiply-adds), 27 + 10 t + (0, or 1 + control bit, then the
// same with the X before) TK_DENSEX
enum { FV_DIAGOUT = 0, FV_DIAG16 = 1, FV_SWAP = 2, FV_DIAG = 6, FV_DIAGC = 10, FV_DENSE = 14, FV_DENSEC = 18,
       FV_DIAGRUN = 22, FV_REAL = 23, FV_DENSEX = 27 };

template <int RB, int T, int KIND, bool CTRL, bool COMP>
__device__ __forceinline__ void fwd_form(float2 (&x)[1 << RB], const TOp& op, const float2* lo) {
  if constexpr (T < RB) {
    if constexpr (KIND == TK_SWAP) {
      op_fwd<RB, T, TK_SWAP, true>(x, op);
    } else if constexpr (COMP) {
      op_fwd_c<RB, T, KIND, CTRL>(x, op, lo);
    } else if constexpr (KIND == TK_DIAG) {
      if (op.u[0].x == 1.f && op.u[0].y == 0.f) op_fwd<RB, T, TK_DIAGB, CTRL>(x, op);
      else op_fwd<RB, T, TK_DIAG, CTRL>(x, op);
    } else {
      op_fwd<RB, T, KIND, CTRL>(x, op);
    }
  }
}

template <int RB, bool COMP>
__device__ __forceinline__ void apply_fwd_var(float2 (&x)[1 << RB], const TOp& op, const float2* lo,
                                              const RunCtx& rc, uint32_t gb) {
  switch (op.var) {
    case FV_DIAGRUN:
      if constexpr (!COMP) diag_run<RB>(x, op, rc, gb);
      break;
    case FV_REAL + 0: if constexpr (!COMP) fwd_form<RB, 0, TK_REAL, false, COMP>(x, op, lo); break;
    case FV_REAL + 1: if constexpr (!COMP) fwd_form<RB, 1, TK_REAL, false, COMP>(x, op, lo); break;
    case FV_REAL + 2: if constexpr (!COMP) fwd_form<RB, 2, TK_REAL, false, COMP>(x, op, lo); break;
    case FV_REAL + 3: if constexpr (!COMP) fwd_form<RB, 3, TK_REAL, false, COMP>(x, op, lo); break;
    case FV_SWAP + 0: fwd_form<RB, 0, TK_SWAP, true, COMP>(x, op, lo); break;
    case FV_SWAP + 1: fwd_form<RB, 1, TK_SWAP, true, COMP>(x, op, lo); break;
    case FV_SWAP + 2: fwd_form<RB, 2, TK_SWAP, true, COMP>(x, op, lo); break;
    case FV_SWAP + 3: fwd_form<RB, 3, TK_SWAP, true, COMP>(x, op, lo); break;
    case FV_DIAG + 0: fwd_form<RB, 0, TK_DIAG, false, COMP>(x, op, lo); break;
    case FV_DIAG + 1: fwd_form<RB, 1, TK_DIAG, false, COMP>(x, op, lo); break;
    case FV_DIAG + 2: fwd_form<RB, 2, TK_DIAG, false, COMP>(x, op, lo); break;
    case FV_DIAG + 3: fwd_form<RB, 3, TK_DIAG, false, COMP>(x, op, lo); break;
    case FV_DIAGC + 0: fwd_form<RB, 0, TK_DIAG, true, COMP>(x, op, lo); break;
    case FV_DIAGC + 1: fwd_form<RB, 1, TK_DIAG, true, COMP>(x, op, lo); break;
    case FV_DIAGC + 2: fwd_form<RB, 2, TK_DIAG, true, COMP>(x, op, lo); break;
    case FV_DIAGC + 3: fwd_form<RB, 3, TK_DIAG, true, COMP>(x, op, lo); break;
    case FV_DENSE + 0: fwd_form<RB, 0, TK_DENSE, false, COMP>(x, op, lo); break;
    case FV_DENSE + 1: fwd_form<RB, 1, TK_DENSE, false, COMP>(x, op, lo); break;
    case FV_DENSE + 2: fwd_form<RB, 2, TK_DENSE, false, COMP>(x, op, lo); break;
    case FV_DENSE + 3: fwd_form<RB, 3, TK_DENSE, false, COMP>(x, op, lo); break;
    case FV_DENSEC + 0: fwd_form<RB, 0, TK_DENSE, true, COMP>(x, op, lo); break;
    case FV_DENSEC + 1: fwd_form<RB, 1, TK_DENSE, true, COMP>(x, op, lo); break;
    case FV_DENSEC + 2: fwd_form<RB, 2, TK_DENSE, true, COMP>(x, op, lo); break;
    case FV_DENSEC + 3: fwd_form<RB, 3, TK_DENSE, true, COMP>(x, op, lo); break;
    default: break;
  }
}

// TK_DENSEX ops; on: the controls outside the phase hold
template <int RB, bool COMP>
__device__ __forceinline__ void apply_densex(float2 (&x)[1 << RB], const TOp& op, const float2* lo, bool on) {
  switch (op.var) {
    case FV_DENSEX + 0: if constexpr (COMP) op_fwd_x_c<RB, 0, -1, false>(x, op, lo, on); else op_fwd_x<RB, 0, -1, false>(x, op, on); break;
    case FV_DENSEX + 2: if constexpr (COMP) op_fwd_x_c<RB, 0, 1, false>(x, op, lo, on); else op_fwd_x<RB, 0, 1, false>(x, op, on); break;
    case FV_DENSEX + 3: if constexpr (COMP) op_fwd_x_c<RB, 0, 2, false>(x, op, lo, on); else op_fwd_x<RB, 0, 2, false>(x, op, on); break;
    case FV_DENSEX + 4: if constexpr (COMP) op_fwd_x_c<RB, 0, 3, false>(x, op, lo, on); else op_fwd_x<RB, 0, 3, false>(x, op, on); break;
    case FV_DENSEX + 5: if constexpr (COMP) op_fwd_x_c<RB, 0, -1, true>(x, op, lo, on); else op_fwd_x<RB, 0, -1, true>(x, op, on); break;
    case FV_DENSEX + 7: if constexpr (COMP) op_fwd_x_c<RB, 0, 1, true>(x, op, lo, on); else op_fwd_x<RB, 0, 1, true>(x, op, on); break;
    case FV_DENSEX + 8: if constexpr (COMP) op_fwd_x_c<RB, 0, 2, true>(x, op, lo, on); else op_fwd_x<RB, 0, 2, true>(x, op, on); break;
    case FV_DENSEX + 9: if constexpr (COMP) op_fwd_x_c<RB, 0, 3, true>(x, op, lo, on); else op_fwd_x<RB, 0, 3, true>(x, op, on); break;
    case FV_DENSEX + 10: if constexpr (COMP) op_fwd_x_c<RB, 1, -1, false>(x, op, lo, on); else op_fwd_x<RB, 1, -1, false>(x, op, on); break;
    case FV_DENSEX + 11: if constexpr (COMP) op_fwd_x_c<RB, 1, 0, false>(x, op, lo, on); else op_fwd_x<RB, 1, 0, false>(x, op, on); break;
    case FV_DENSEX + 13: if constexpr (COMP) op_fwd_x_c<RB, 1, 2, false>(x, op, lo, on); else op_fwd_x<RB, 1, 2, false>(x, op, on); break;
    case FV_DENSEX + 14: if constexpr (COMP) op_fwd_x_c<RB, 1, 3, false>(x, op, lo, on); else op_fwd_x<RB, 1, 3, false>(x, op, on); break;
    case FV_DENSEX + 15: if constexpr (COMP) op_fwd_x_c<RB, 1, -1, true>(x, op, lo, on); else op_fwd_x<RB, 1, -1, true>(x, op, on); break;
    case FV_DENSEX + 16: if constexpr (COMP) op_fwd_x_c<RB, 1, 0, true>(x, op, lo, on); else op_fwd_x<RB, 1, 0, true>(x, op, on); break;
    case FV_DENSEX + 18: if constexpr (COMP) op_fwd_x_c<RB, 1, 2, true>(x, op, lo, on); else op_fwd_x<RB, 1, 2, true>(x, op, on); break;
    case FV_DENSEX + 19: if constexpr (COMP) op_fwd_x_c<RB, 1, 3, true>(x, op, lo, on); else op_fwd_x<RB, 1, 3, true>(x, op, on); break;
    case FV_DENSEX + 20: if constexpr (COMP) op_fwd_x_c<RB, 2, -1, false>(x, op, lo, on); else op_fwd_x<RB, 2, -1, false>(x, op, on); break;
    case FV_DENSEX + 21: if constexpr (COMP) op_fwd_x_c<RB, 2, 0, false>(x, op, lo, on); else op_fwd_x<RB, 2, 0, false>(x, op, on); break;
    case FV_DENSEX + 22: if constexpr (COMP) op_fwd_x_c<RB, 2, 1, false>(x, op, lo, on); else op_fwd_x<RB, 2, 1, false>(x, op, on); break;
    case FV_DENSEX + 24: if constexpr (COMP) op_fwd_x_c<RB, 2, 3, false>(x, op, lo, on); else op_fwd_x<RB, 2, 3, false>(x, op, on); break;
    case FV_DENSEX + 25: if constexpr (COMP) op_fwd_x_c<RB, 2, -1, true>(x, op, lo, on); else op_fwd_x<RB, 2, -1, true>(x, op, on); break;
    case FV_DENSEX + 26: if constexpr (COMP) op_fwd_x_c<RB, 2, 0, true>(x, op, lo, on); else op_fwd_x<RB, 2, 0, true>(x, op, on); break;
    case FV_DENSEX + 27: if constexpr (COMP) op_fwd_x_c<RB, 2, 1, true>(x, op, lo, on); else op_fwd_x<RB, 2, 1, true>(x, op, on); break;
    case FV_DENSEX + 29: if constexpr (COMP) op_fwd_x_c<RB, 2, 3, true>(x, op, lo, on); else op_fwd_x<RB, 2, 3, true>(x, op, on); break;
    case FV_DENSEX + 30: if constexpr (COMP) op_fwd_x_c<RB, 3, -1, false>(x, op, lo, on); else op_fwd_x<RB, 3, -1, false>(x, op, on); break;
    case FV_DENSEX + 31: if constexpr (COMP) op_fwd_x_c<RB, 3, 0, false>(x, op, lo, on); else op_fwd_x<RB, 3, 0, false>(x, op, on); break;
    case FV_DENSEX + 32: if constexpr (COMP) op_fwd_x_c<RB, 3, 1, false>(x, op, lo, on); else op_fwd_x<RB, 3, 1, false>(x, op, on); break;
    case FV_DENSEX + 33: if constexpr (COMP) op_fwd_x_c<RB, 3, 2, false>(x, op, lo, on); else op_fwd_x<RB, 3, 2, false>(x, op, on); break;
    case FV_DENSEX + 35: if constexpr (COMP) op_fwd_x_c<RB, 3, -1, true>(x, op, lo, on); else op_fwd_x<RB, 3, -1, true>(x, op, on); break;
    case FV_DENSEX + 36: if constexpr (COMP) op_fwd_x_c<RB, 3, 0, true>(x, op, lo, on); else op_fwd_x<RB, 3, 0, true>(x, op, on); break;
    case FV_DENSEX + 37: if constexpr (COMP) op_fwd_x_c<RB, 3, 1, true>(x, op, lo, on); else op_fwd_x<RB, 3, 1, true>(x, op, on); break;
    case FV_DENSEX + 38: if constexpr (COMP) op_fwd_x_c<RB, 3, 2, true>(x, op, lo, on); else op_fwd_x<RB, 3, 2, true>(x, op, on); break;
    default: break;
  }
}

// Backward op: first this thread's share of Im<lambda|G|psi> over its pairs
// (GK 0: none; 1: diagonal generator diag(g0, g3); 2: X; 3: Y), then
// psi <- U^dag psi and lambda <- U^dag lambda.
template <int RB, int T, int KIND, int GK, bool CTRL>
__device__ __forceinline__ float op_bwd(float2 (&x)[1 << RB], float2 (&l)[1 << RB], const TOp& op, float g0, float g3) {
  const int cm = op.cmask, cv = op.cval;
  const float2 u0 = op.u[0], u1 = op.u[1], u2 = op.u[2], u3 = op.u[3];
  float acc = 0.f;
#pragma unroll
  for (int j = 0; j < (1 << RB); ++j) {
    if (j & (1 << T)) continue;
    if (CTRL && (j & cm) != cv) continue;
    const int k = j | (1 << T);
    if (GK == 1) acc += fmaf(g0, imcj(l[j], x[j]), g3 * imcj(l[k], x[k]));
    if (GK == 2) acc += imcj(l[j], x[k]) + imcj(l[k], x[j]);
    if (GK == 3) acc += recj(l[k], x[j]) - recj(l[j], x[k]);
    pair_apply<KIND>(x[j], x[k], u0, u1, u2, u3);
    pair_apply<KIND>(l[j], l[k], u0, u1, u2, u3);
  }
  return acc;
}

// A TK_RUN op.  With (a, b) the pair at the end of the run (an X after it undone: the
// pair swapped where it acted), the thread's shares of Im conj(l_a) x_a, Im conj(l_b) x_b,
// Im<l|X|x>, Im<l|Y|x> to v; then the run's U^dagger (and an X before it undone: the
// outputs swapped).  22 multiply-adds an amplitude for the whole run, where Rz Rx Rz gate
// by gate took 32, three dispatches and three sums over the warp, and the X a fourth.
template <int RB, int T, int C, bool PRE>
__device__ __forceinline__ void op_bwd_run(float2 (&x)[1 << RB], float2 (&l)[1 << RB], const TOp& op, bool on,
                                           float (&v)[4]) {
  if constexpr (T < RB && C < RB && C != T) {
    const bool sw = C < 0 && on;
    constexpr int P = PRE ? 2 : 1;  // the outputs' rows or the inputs' columns trade places
    const float2 u0 = sw ? op.u[P] : op.u[0], u1 = sw ? op.u[P ^ 1] : op.u[1];
    const float2 u2 = sw ? op.u[P ^ 2] : op.u[2], u3 = sw ? op.u[P ^ 3] : op.u[3];
    float va = 0.f, vb = 0.f, vx = 0.f, vy = 0.f;
#pragma unroll
    for (int j = 0; j < (1 << RB); ++j) {
      if (j & (1 << T)) continue;
      const bool ren = C >= 0 && ((j >> (C < 0 ? 0 : C)) & 1);
      const int k = j | (1 << T), ja = !PRE && ren ? k : j, jb = !PRE && ren ? j : k;
      const float2 xa = x[ja], xb = x[jb], la = l[ja], lb = l[jb];
      va = fmaf(la.x, xa.y, fmaf(-la.y, xa.x, va));
      vb = fmaf(lb.x, xb.y, fmaf(-lb.y, xb.x, vb));
      vx = fmaf(la.x, xb.y, fmaf(-la.y, xb.x, vx));
      vx = fmaf(lb.x, xa.y, fmaf(-lb.y, xa.x, vx));
      vy = fmaf(lb.x, xa.x, fmaf(lb.y, xa.y, vy));
      vy = fmaf(-la.x, xb.x, fmaf(-la.y, xb.y, vy));
      const int oa = PRE && ren ? k : j, ob = PRE && ren ? j : k;
      x[oa] = cmaf(u1, xb, cmulf(u0, xa));
      x[ob] = cmaf(u3, xb, cmulf(u2, xa));
      l[oa] = cmaf(u1, lb, cmulf(u0, la));
      l[ob] = cmaf(u3, lb, cmulf(u2, la));
    }
    const bool neg = !PRE && sw;
    v[0] = neg ? vb : va;
    v[1] = neg ? va : vb;
    v[2] = vx;
    v[3] = neg ? -vy : vy;
  }
}

// backward op forms (TOp::var = 13 t + form): 0 controlled swap, 1 / 2 diagonal /
// dense without a parameter, then X, Y, Z, P1, I generators, each without and
// with phase-local controls
template <int RB, int T, int F>
__device__ __forceinline__ float bwd_form(float2 (&x)[1 << RB], float2 (&l)[1 << RB], const TOp& op) {
  if constexpr (T >= RB) {
    return 0.f;
  } else if constexpr (F == 0) {
    return op_bwd<RB, T, TK_SWAP, 0, true>(x, l, op, 0.f, 0.f);
  } else if constexpr (F == 1) {
    return op_bwd<RB, T, TK_DIAG, 0, true>(x, l, op, 0.f, 0.f);
  } else if constexpr (F == 2) {
    return op_bwd<RB, T, TK_DENSE, 0, true>(x, l, op, 0.f, 0.f);
  } else {
    constexpr bool C = ((F - 3) & 1) != 0;
    constexpr int G = (F - 3) / 2;
    if constexpr (G == 0) return op_bwd<RB, T, TK_RX, 2, C>(x, l, op, 0.f, 0.f);
    else if constexpr (G == 1) return op_bwd<RB, T, TK_RY, 3, C>(x, l, op, 0.f, 0.f);
    else if constexpr (G == 2) return op_bwd<RB, T, TK_DIAG, 1, C>(x, l, op, 1.f, -1.f);
    else if constexpr (G == 3) return op_bwd<RB, T, TK_DIAG, 1, C>(x, l, op, 0.f, 1.f);
    else return op_bwd<RB, T, TK_DIAG, 1, C>(x, l, op, 1.f, 1.f);
  }
}

template <int RB>
__device__ __forceinline__ float apply_bwd_var(float2 (&x)[1 << RB], float2 (&l)[1 << RB], const TOp& op) {
  switch (op.var) {
    case 0: return bwd_form<RB, 0, 0>(x, l, op);
    case 1: return bwd_form<RB, 0, 1>(x, l, op);
    case 2: return bwd_form<RB, 0, 2>(x, l, op);
    case 3: return bwd_form<RB, 0, 3>(x, l, op);
    case 4: return bwd_form<RB, 0, 4>(x, l, op);
    case 5: return bwd_form<RB, 0, 5>(x, l, op);
    case 6: return bwd_form<RB, 0, 6>(x, l, op);
    case 7: return bwd_form<RB, 0, 7>(x, l, op);
    case 8: return bwd_form<RB, 0, 8>(x, l, op);
    case 9: return bwd_form<RB, 0, 9>(x, l, op);
    case 10: return bwd_form<RB, 0, 10>(x, l, op);
    case 11: return bwd_form<RB, 0, 11>(x, l, op);
    case 12: return bwd_form<RB, 0, 12>(x, l, op);
    case 13: return bwd_form<RB, 1, 0>(x, l, op);
    case 14: return bwd_form<RB, 1, 1>(x, l, op);
    case 15: return bwd_form<RB, 1, 2>(x, l, op);
    case 16: return bwd_form<RB, 1, 3>(x, l, op);
    case 17: return bwd_form<RB, 1, 4>(x, l, op);
    case 18: return bwd_form<RB, 1, 5>(x, l, op);
    case 19: return bwd_form<RB, 1, 6>(x, l, op);
    case 20: return bwd_form<RB, 1, 7>(x, l, op);
    case 21: return bwd_form<RB, 1, 8>(x, l, op);
    case 22: return bwd_form<RB, 1, 9>(x, l, op);
    case 23: return bwd_form<RB, 1, 10>(x, l, op);
    case 24: return bwd_form<RB, 1, 11>(x, l, op);
    case 25: return bwd_form<RB, 1, 12>(x, l, op);
    case 26: return bwd_form<RB, 2, 0>(x, l, op);
    case 27: return bwd_form<RB, 2, 1>(x, l, op);
    case 28: return bwd_form<RB, 2, 2>(x, l, op);
    case 29: return bwd_form<RB, 2, 3>(x, l, op);
    case 30: return bwd_form<RB, 2, 4>(x, l, op);
    case 31: return bwd_form<RB, 2, 5>(x, l, op);
    case 32: return bwd_form<RB, 2, 6>(x, l, op);
    case 33: return bwd_form<RB, 2, 7>(x, l, op);
    case 34: return bwd_form<RB, 2, 8>(x, l, op);
    case 35: return bwd_form<RB, 2, 9>(x, l, op);
    case 36: return bwd_form<RB, 2, 10>(x, l, op);
    case 37: return bwd_form<RB, 2, 11>(x, l, op);
    case 38: return bwd_form<RB, 2, 12>(x, l, op);
    case 39: return bwd_form<RB, 3, 0>(x, l, op);
    case 40: return bwd_form<RB, 3, 1>(x, l, op);
    case 41: return bwd_form<RB, 3, 2>(x, l, op);
    case 42: return bwd_form<RB, 3, 3>(x, l, op);
    case 43: return bwd_form<RB, 3, 4>(x, l, op);
    case 44: return bwd_form<RB, 3, 5>(x, l, op);
    case 45: return bwd_form<RB, 3, 6>(x, l, op);
    case 46: return bwd_form<RB, 3, 7>(x, l, op);
    case 47: return bwd_form<RB, 3, 8>(x, l, op);
    case 48: return bwd_form<RB, 3, 9>(x, l, op);
    case 49: return bwd_form<RB, 3, 10>(x, l, op);
    case 50: return bwd_form<RB, 3, 11>(x, l, op);
    case 51: return bwd_form<RB, 3, 12>(x, l, op);
    default: return 0.f;
  }
}

// TK_RUN forms: BV_RUN + 10 t + (0, or 1 + control bit of the X; then the same with the X
// before the run)
constexpr int BV_RUN = 64;

template <int RB>
__device__ __forceinline__ void apply_bwd_run(float2 (&x)[1 << RB], float2 (&l)[1 << RB], const TOp& op, bool on,
                                              float (&v)[4]) {
  switch (op.var) {
    case BV_RUN + 0: op_bwd_run<RB, 0, -1, false>(x, l, op, on, v); break;
    case BV_RUN + 2: op_bwd_run<RB, 0, 1, false>(x, l, op, on, v); break;
    case BV_RUN + 3: op_bwd_run<RB, 0, 2, false>(x, l, op, on, v); break;
    case BV_RUN + 4: op_bwd_run<RB, 0, 3, false>(x, l, op, on, v); break;
    case BV_RUN + 5: op_bwd_run<RB, 0, -1, true>(x, l, op, on, v); break;
    case BV_RUN + 7: op_bwd_run<RB, 0, 1, true>(x, l, op, on, v); break;
    case BV_RUN + 8: op_bwd_run<RB, 0, 2, true>(x, l, op, on, v); break;
    case BV_RUN + 9: op_bwd_run<RB, 0, 3, true>(x, l, op, on, v); break;
    case BV_RUN + 10: op_bwd_run<RB, 1, -1, false>(x, l, op, on, v); break;
    case BV_RUN + 11: op_bwd_run<RB, 1, 0, false>(x, l, op, on, v); break;
    case BV_RUN + 13: op_bwd_run<RB, 1, 2, false>(x, l, op, on, v); break;
    case BV_RUN + 14: op_bwd_run<RB, 1, 3, false>(x, l, op, on, v); break;
    case BV_RUN + 15: op_bwd_run<RB, 1, -1, true>(x, l, op, on, v); break;
    case BV_RUN + 16: op_bwd_run<RB, 1, 0, true>(x, l, op, on, v); break;
    case BV_RUN + 18: op_bwd_run<RB, 1, 2, true>(x, l, op, on, v); break;
    case BV_RUN + 19: op_bwd_run<RB, 1, 3, true>(x, l, op, on, v); break;
    case BV_RUN + 20: op_bwd_run<RB, 2, -1, false>(x, l, op, on, v); break;
    case BV_RUN + 21: op_bwd_run<RB, 2, 0, false>(x, l, op, on, v); break;
    case BV_RUN + 22: op_bwd_run<RB, 2, 1, false>(x, l, op, on, v); break;
    case BV_RUN + 24: op_bwd_run<RB, 2, 3, false>(x, l, op, on, v); break;
    case BV_RUN + 25: op_bwd_run<RB, 2, -1, true>(x, l, op, on, v); break;
    case BV_RUN + 26: op_bwd_run<RB, 2, 0, true>(x, l, op, on, v); break;
    case BV_RUN + 27: op_bwd_run<RB, 2, 1, true>(x, l, op, on, v); break;
    case BV_RUN + 29: op_bwd_run<RB, 2, 3, true>(x, l, op, on, v); break;
    case BV_RUN + 30: op_bwd_run<RB, 3, -1, false>(x, l, op, on, v); break;
    case BV_RUN + 31: op_bwd_run<RB, 3, 0, false>(x, l, op, on, v); break;
    case BV_RUN + 32: op_bwd_run<RB, 3, 1, false>(x, l, op, on, v); break;
    case BV_RUN + 33: op_bwd_run<RB, 3, 2, false>(x, l, op, on, v); break;
    case BV_RUN + 35: op_bwd_run<RB, 3, -1, true>(x, l, op, on, v); break;
    case BV_RUN + 36: op_bwd_run<RB, 3, 0, true>(x, l, op, on, v); break;
    case BV_RUN + 37: op_bwd_run<RB, 3, 1, true>(x, l, op, on, v); break;
    case BV_RUN + 38: op_bwd_run<RB, 3, 2, true>(x, l, op, on, v); break;
    default: break;
  }
}

// ------------------------------------------------------------------ device: double-float arithmetic
//
// A double-float value is an unevaluated sum hi + lo of two FP32 numbers with
// |lo| <= ulp(hi) / 2 (Dekker 1971).  The building blocks are Knuth's
// error-free TwoSum and the FMA form of TwoProduct (the rounding error of
// a * b is fma(a, b, -a * b) exactly); a sum of products accumulates the large
// parts with TwoSum and every small part in a running FP32 correction, and is
// renormalised once at the end (Joldes, Muller and Popescu, ACM TOMS 2017,
// give the error bounds of these double-word operations).  The _rn
// intrinsics keep the compiler from fusing the exact-error steps.

struct ffc {         // complex double-float: (h.x + l.x) + i (h.y + l.y)
  float2 h, l;
};


struct DWAcc {       // running sum s + e of double-float products
  float s, e;
};

// (xh + xl) * (yh + yl) without the xl * yl term (below 2^-48 relative)
__device__ __forceinline__ void dw_first(DWAcc& A, float xh, float xl, float yh, float yl) {
  A.s = __fmul_rn(xh, yh);
  A.e = fmaf(xh, yl, fmaf(xl, yh, fmaf(xh, yh, -A.s)));
}
__device__ __forceinline__ void dw_add(DWAcc& A, float xh, float xl, float yh, float yl) {
  const float p = __fmul_rn(xh, yh);
  const float pe = fmaf(xh, yl, fmaf(xl, yh, fmaf(xh, yh, -p)));
  float s, t;
  two_sum(A.s, p, s, t);
  A.s = s;
  A.e = __fadd_rn(A.e, __fadd_rn(t, pe));
}
__device__ __forceinline__ void dw_out(const DWAcc& A, float& h, float& l) { two_sum(A.s, A.e, h, l); }

// a * u for complex double-floats (u = uh + ul)
__device__ __forceinline__ ffc ff_cmul(const ffc& a, float2 uh, float2 ul) {
  DWAcc re, im;
  dw_first(re, a.h.x, a.l.x, uh.x, ul.x);
  dw_add(re, -a.h.y, -a.l.y, uh.y, ul.y);
  dw_first(im, a.h.x, a.l.x, uh.y, ul.y);
  dw_add(im, a.h.y, a.l.y, uh.x, ul.x);
  ffc r;
  dw_out(re, r.h.x, r.l.x);
  dw_out(im, r.h.y, r.l.y);
  return r;
}

// u0 * a + u1 * b for complex double-floats
__device__ __forceinline__ ffc ff_cdot2(const ffc& a, float2 u0h, float2 u0l, const ffc& b, float2 u1h, float2 u1l) {
  DWAcc re, im;
  dw_first(re, a.h.x, a.l.x, u0h.x, u0l.x);
  dw_add(re, -a.h.y, -a.l.y, u0h.y, u0l.y);
  dw_add(re, b.h.x, b.l.x, u1h.x, u1l.x);
  dw_add(re, -b.h.y, -b.l.y, u1h.y, u1l.y);
  dw_first(im, a.h.x, a.l.x, u0h.y, u0l.y);
  dw_add(im, a.h.y, a.l.y, u0h.x, u0l.x);
  dw_add(im, b.h.x, b.l.x, u1h.y, u1l.y);
  dw_add(im, b.h.y, b.l.y, u1h.x, u1l.x);
  ffc r;
  dw_out(re, r.h.x, r.l.x);
  dw_out(im, r.h.y, r.l.y);
  return r;
}

// (a, b) <- U (a, b) in double-float; U = u + w (hi + lo), row-major
template <int KIND>
__device__ __forceinline__ void pair_apply_ff(ffc& a, ffc& b, const float2 (&u)[4], const float2 (&w)[4]) {
  if (KIND == TK_SWAP) {
    const ffc t = a; a = b; b = t;
  } else if (KIND == TK_DIAG) {
    a = ff_cmul(a, u[0], w[0]);
    b = ff_cmul(b, u[3], w[3]);
  } else if (KIND == TK_RX) {  // [[c, i s], [i s, c]]: a' = c a + i s b
    const float ch = u[0].x, cl = w[0].x, sh = u[1].y, sl = w[1].y;
    DWAcc r0, i0, r1, i1;
    dw_first(r0, a.h.x, a.l.x, ch, cl); dw_add(r0, -b.h.y, -b.l.y, sh, sl);
    dw_first(i0, a.h.y, a.l.y, ch, cl); dw_add(i0, b.h.x, b.l.x, sh, sl);
    dw_first(r1, b.h.x, b.l.x, ch, cl); dw_add(r1, -a.h.y, -a.l.y, sh, sl);
    dw_first(i1, b.h.y, b.l.y, ch, cl); dw_add(i1, a.h.x, a.l.x, sh, sl);
    dw_out(r0, a.h.x, a.l.x); dw_out(i0, a.h.y, a.l.y);
    dw_out(r1, b.h.x, b.l.x); dw_out(i1, b.h.y, b.l.y);
  } else if (KIND == TK_RY) {  // real [[c, p], [q, c]]
    const float ch = u[0].x, cl = w[0].x, ph = u[1].x, pl = w[1].x, qh = u[2].x, ql = w[2].x;
    DWAcc r0, i0, r1, i1;
    dw_first(r0, a.h.x, a.l.x, ch, cl); dw_add(r0, b.h.x, b.l.x, ph, pl);
    dw_first(i0, a.h.y, a.l.y, ch, cl); dw_add(i0, b.h.y, b.l.y, ph, pl);
    dw_first(r1, a.h.x, a.l.x, qh, ql); dw_add(r1, b.h.x, b.l.x, ch, cl);
    dw_first(i1, a.h.y, a.l.y, qh, ql); dw_add(i1, b.h.y, b.l.y, ch, cl);
    dw_out(r0, a.h.x, a.l.x); dw_out(i0, a.h.y, a.l.y);
    dw_out(r1, b.h.x, b.l.x); dw_out(i1, b.h.y, b.l.y);
  } else {
    const ffc na = ff_cdot2(a, u[0], w[0], b, u[1], w[1]);
    const ffc nb = ff_cdot2(a, u[2], w[2], b, u[3], w[3]);
    a = na; b = nb;
  }
}

// the backward op of the precise path: gradient share from the hi parts
// (FP32 products, FP64 above the warp), then the double-float uncompute
template <int RB, int T, int KIND, int GK, bool CTRL>
__device__ __forceinline__ float op_bwd_ff(ffc (&x)[1 << RB], ffc (&l)[1 << RB], const TOp& op, const float2* lo,
                                           float g0, float g3) {
  const int cm = op.cmask, cv = op.cval;
  const float2 u[4] = {op.u[0], op.u[1], op.u[2], op.u[3]};
  const float2 w[4] = {lo[0], lo[1], lo[2], lo[3]};
  float acc = 0.f;
#pragma unroll
  for (int j = 0; j < (1 << RB); ++j) {
    if (j & (1 << T)) continue;
    if (CTRL && (j & cm) != cv) continue;
    const int k = j | (1 << T);
    if (GK == 1) acc += fmaf(g0, imcj(l[j].h, x[j].h), g3 * imcj(l[k].h, x[k].h));
    if (GK == 2) acc += imcj(l[j].h, x[k].h) + imcj(l[k].h, x[j].h);
    if (GK == 3) acc += recj(l[k].h, x[j].h) - recj(l[j].h, x[k].h);
    pair_apply_ff<KIND>(x[j], x[k], u, w);
    pair_apply_ff<KIND>(l[j], l[k], u, w);
  }
  return acc;
}

// op_bwd_run with the double-float uncompute (sums from the hi parts)
template <int RB, int T, int C, bool PRE>
__device__ __forceinline__ void op_bwd_run_ff(ffc (&x)[1 << RB], ffc (&l)[1 << RB], const TOp& op, const float2* lo,
                                              bool on, float (&v)[4]) {
  if constexpr (T < RB && C < RB && C != T) {
    const bool sw = C < 0 && on;
    constexpr int P = PRE ? 2 : 1;
    const float2 u[4] = {sw ? op.u[P] : op.u[0], sw ? op.u[P ^ 1] : op.u[1], sw ? op.u[P ^ 2] : op.u[2],
                         sw ? op.u[P ^ 3] : op.u[3]};
    const float2 w[4] = {lo[sw ? P : 0], lo[sw ? P ^ 1 : 1], lo[sw ? P ^ 2 : 2], lo[sw ? P ^ 3 : 3]};
    float va = 0.f, vb = 0.f, vx = 0.f, vy = 0.f;
#pragma unroll
    for (int j = 0; j < (1 << RB); ++j) {
      if (j & (1 << T)) continue;
      const bool ren = C >= 0 && ((j >> (C < 0 ? 0 : C)) & 1);
      const int k = j | (1 << T), ja = !PRE && ren ? k : j, jb = !PRE && ren ? j : k;
      ffc xa = x[ja], xb = x[jb], la = l[ja], lb = l[jb];
      va = fmaf(la.h.x, xa.h.y, fmaf(-la.h.y, xa.h.x, va));
      vb = fmaf(lb.h.x, xb.h.y, fmaf(-lb.h.y, xb.h.x, vb));
      vx = fmaf(la.h.x, xb.h.y, fmaf(-la.h.y, xb.h.x, vx));
      vx = fmaf(lb.h.x, xa.h.y, fmaf(-lb.h.y, xa.h.x, vx));
      vy = fmaf(lb.h.x, xa.h.x, fmaf(lb.h.y, xa.h.y, vy));
      vy = fmaf(-la.h.x, xb.h.x, fmaf(-la.h.y, xb.h.y, vy));
      pair_apply_ff<TK_DENSE>(xa, xb, u, w);
      pair_apply_ff<TK_DENSE>(la, lb, u, w);
      const int oa = PRE && ren ? k : j, ob = PRE && ren ? j : k;
      x[oa] = xa; x[ob] = xb;
      l[oa] = la; l[ob] = lb;
    }
    const bool neg = !PRE && sw;
    v[0] = neg ? vb : va;
    v[1] = neg ? va : vb;
    v[2] = vx;
    v[3] = neg ? -vy : vy;
  }
}
template <int RB>
__device__ __forceinline__ void apply_bwd_run_ff(ffc (&x)[1 << RB], ffc (&l)[1 << RB], const TOp& op, const float2* lo,
                                                 bool on, float (&v)[4]) {
  switch (op.var) {
    case BV_RUN + 0: op_bwd_run_ff<RB, 0, -1, false>(x, l, op, lo, on, v); break;
    case BV_RUN + 2: op_bwd_run_ff<RB, 0, 1, false>(x, l, op, lo, on, v); break;
    case BV_RUN + 3: op_bwd_run_ff<RB, 0, 2, false>(x, l, op, lo, on, v); break;
    case BV_RUN + 5: op_bwd_run_ff<RB, 0, -1, true>(x, l, op, lo, on, v); break;
    case BV_RUN + 7: op_bwd_run_ff<RB, 0, 1, true>(x, l, op, lo, on, v); break;
    case BV_RUN + 8: op_bwd_run_ff<RB, 0, 2, true>(x, l, op, lo, on, v); break;
    case BV_RUN + 10: op_bwd_run_ff<RB, 1, -1, false>(x, l, op, lo, on, v); break;
    case BV_RUN + 11: op_bwd_run_ff<RB, 1, 0, false>(x, l, op, lo, on, v); break;
    case BV_RUN + 13: op_bwd_run_ff<RB, 1, 2, false>(x, l, op, lo, on, v); break;
    case BV_RUN + 15: op_bwd_run_ff<RB, 1, -1, true>(x, l, op, lo, on, v); break;
    case BV_RUN + 16: op_bwd_run_ff<RB, 1, 0, true>(x, l, op, lo, on, v); break;
    case BV_RUN + 18: op_bwd_run_ff<RB, 1, 2, true>(x, l, op, lo, on, v); break;
    case BV_RUN + 20: op_bwd_run_ff<RB, 2, -1, false>(x, l, op, lo, on, v); break;
    case BV_RUN + 21: op_bwd_run_ff<RB, 2, 0, false>(x, l, op, lo, on, v); break;
    case BV_RUN + 22: op_bwd_run_ff<RB, 2, 1, false>(x, l, op, lo, on, v); break;
    case BV_RUN + 25: op_bwd_run_ff<RB, 2, -1, true>(x, l, op, lo, on, v); break;
    case BV_RUN + 26: op_bwd_run_ff<RB, 2, 0, true>(x, l, op, lo, on, v); break;
    case BV_RUN + 27: op_bwd_run_ff<RB, 2, 1, true>(x, l, op, lo, on, v); break;
    default: break;
  }
}

template <int RB, int T, bool CTRL>
__device__ __forceinline__ float op_bwd_ff_c(ffc (&x)[1 << RB], ffc (&l)[1 << RB], const TOp& op, const float2* lo) {
  switch (op.gen) {
    case GEN_X: return op_bwd_ff<RB, T, TK_RX, 2, CTRL>(x, l, op, lo, 0.f, 0.f);
    case GEN_Y: return op_bwd_ff<RB, T, TK_RY, 3, CTRL>(x, l, op, lo, 0.f, 0.f);
    case GEN_Z: return op_bwd_ff<RB, T, TK_DIAG, 1, CTRL>(x, l, op, lo, 1.f, -1.f);
    case GEN_P1: return op_bwd_ff<RB, T, TK_DIAG, 1, CTRL>(x, l, op, lo, 0.f, 1.f);
    default: return op_bwd_ff<RB, T, TK_DIAG, 1, CTRL>(x, l, op, lo, 1.f, 1.f);  // GEN_I
  }
}

template <int RB, int T>
__device__ __forceinline__ float op_bwd_ff_t(ffc (&x)[1 << RB], ffc (&l)[1 << RB], const TOp& op, const float2* lo) {
  if (op.gen == GEN_NONE) {
    if (op.kind == TK_SWAP) return op_bwd_ff<RB, T, TK_SWAP, 0, true>(x, l, op, lo, 0.f, 0.f);
    if (op.kind == TK_DIAG) return op_bwd_ff<RB, T, TK_DIAG, 0, true>(x, l, op, lo, 0.f, 0.f);
    return op_bwd_ff<RB, T, TK_DENSE, 0, true>(x, l, op, lo, 0.f, 0.f);
  }
  return op.cmask ? op_bwd_ff_c<RB, T, true>(x, l, op, lo) : op_bwd_ff_c<RB, T, false>(x, l, op, lo);
}

template <int RB>
__device__ __forceinline__ float apply_bwd_ff(ffc (&x)[1 << RB], ffc (&l)[1 << RB], const TOp& op, const float2* lo) {
  switch (op.t) {
    case 0: return op_bwd_ff_t<RB, 0>(x, l, op, lo);
    case 1: return op_bwd_ff_t<RB, 1>(x, l, op, lo);
    case 2: if constexpr (RB > 2) return op_bwd_ff_t<RB, 2>(x, l, op, lo); return 0.f;
    default: if constexpr (RB > 3) return op_bwd_ff_t<RB, 3>(x, l, op, lo); return 0.f;
  }
}

// ------------------------------------------------------------------ device: the persistent kernel

constexpr int kWarps = kTileThreads / 32;

// The functions below that are not inlined take shared memory as byte offsets into the
// dynamic array: through a generic pointer every access costs 64-bit address
// arithmetic and a generic load (with the phase index arithmetic below: 8 % fewer
// instructions in a QFT pass, batch of 1024 registers 112 -> 107 ms).
template <typename T>
__device__ __forceinline__ T* sh(uint32_t off) {
  extern __shared__ __align__(16) unsigned char smraw[];
  return reinterpret_cast<T*>(smraw + off);
}

struct BShared {
  double grad[kMaxRegParams];
  alignas(16) float red[kMaxPhaseVals * kWarps];  // in the forward: a pass's TK_DIAGRUN entries
  double lred[kWarps];
  uint32_t rowoff[1 << (kMaxTileBits - kRowBits)];  // register offset of each 32-amplitude tile row (current pass)
  RunCtx rc;
  int reg;
};

// Tile rows: tile-local bits 0..4 are register qubits 0..4 (planner seed), so a
// row of 32 amplitudes is contiguous (256 bytes).  rowoff[] holds the register
// offset of every row of the current pass; tile_base() the offset of a tile.
__device__ void set_rows(uint32_t* rowoff, const TPass& p, int m) {
  for (uint32_t row = threadIdx.x; row < (1u << (m - kRowBits)); row += blockDim.x) {
    uint32_t o = 0;
    for (int k = kRowBits; k < m; ++k) o |= ((row >> (k - kRowBits)) & 1u) << p.tbits[k];
    rowoff[row] = o;
  }
  __syncthreads();
}

__device__ __forceinline__ uint64_t tile_base(uint64_t tile, const TPass& p, int g) {
  uint64_t o = 0;
  for (int k = 0; k < g; ++k) o |= ((tile >> k) & 1ull) << p.gbits[k];
  return o;
}

// Stage one or two tiles (2^m amplitudes each) between global and shared
// memory.  Each thread issues up to 8 16-byte loads per tile before any shared
// store (4096 loads of one tile in flight per CTA).
constexpr int kLdChunk = 8;

template <bool TWO>
__device__ __noinline__ void load_tiles(uint32_t o0, const float2* src0, uint32_t o1, const float2* src1,
                                        uint32_t rows, int m) {
  float2 *sm0 = sh<float2>(o0), *sm1 = sh<float2>(o1);
  const uint32_t* rowoff = sh<uint32_t>(rows);
  const uint32_t nq = 1u << (m - 1);  // float4 per tile
  constexpr int C = TWO ? kLdChunk / 2 : kLdChunk;
  for (uint32_t q0 = 0; q0 < nq; q0 += C * kTileThreads) {
    float4 v0[C], v1[C];
#pragma unroll
    for (int k = 0; k < C; ++k) {
      const uint32_t q = q0 + threadIdx.x + k * kTileThreads;
      if (q < nq) {
        const uint32_t off = rowoff[q >> 4] + 2 * (q & 15);
        v0[k] = *reinterpret_cast<const float4*>(src0 + off);
        if (TWO) v1[k] = *reinterpret_cast<const float4*>(src1 + off);
      }
    }
#pragma unroll
    for (int k = 0; k < C; ++k) {
      const uint32_t q = q0 + threadIdx.x + k * kTileThreads;
      if (q < nq) {
        const uint32_t l = 2 * q;
        sm0[swz(l)] = make_float2(v0[k].x, v0[k].y);
        sm0[swz(l + 1)] = make_float2(v0[k].z, v0[k].w);
        if (TWO) {
          sm1[swz(l)] = make_float2(v1[k].x, v1[k].y);
          sm1[swz(l + 1)] = make_float2(v1[k].z, v1[k].w);
        }
      }
    }
  }
}

template <bool TWO>
__device__ __noinline__ void store_tiles(uint32_t o0, float2* dst0, uint32_t o1, float2* dst1, uint32_t rows, int m) {
  const float2 *sm0 = sh<float2>(o0), *sm1 = sh<float2>(o1);
  const uint32_t* rowoff = sh<uint32_t>(rows);
  const uint32_t nq = 1u << (m - 1);
  for (uint32_t q = threadIdx.x; q < nq; q += kTileThreads) {
    const uint32_t off = rowoff[q >> 4] + 2 * (q & 15);
    const uint32_t l = 2 * q;
    const float2 a = sm0[swz(l)], b = sm0[swz(l + 1)];
    *reinterpret_cast<float4*>(dst0 + off) = make_float4(a.x, a.y, b.x, b.y);
    if (TWO) {
      const float2 c = sm1[swz(l)], d = sm1[swz(l + 1)];
      *reinterpret_cast<float4*>(dst1 + off) = make_float4(c.x, c.y, d.x, d.y);
    }
  }
}

__device__ __forceinline__ void load_tile(uint32_t sm, const float2* src, uint32_t rows, int m) {
  load_tiles<false>(sm, src, 0, nullptr, rows, m);
}
__device__ __forceinline__ void store_tile(uint32_t sm, float2* dst, uint32_t rows, int m) {
  store_tiles<false>(sm, dst, 0, nullptr, rows, m);
}

// double-float tiles of psi and lambda (one float4 = hi.re, hi.im, lo.re, lo.im
// per amplitude, in global and shared memory)
__device__ __noinline__ void load_tiles_ff(uint32_t o0, const float4* src0, uint32_t o1, const float4* src1,
                                           uint32_t rows, int m) {
  float4 *sm0 = sh<float4>(o0), *sm1 = sh<float4>(o1);
  const uint32_t* rowoff = sh<uint32_t>(rows);
  const uint32_t cnt = 1u << m;
  constexpr int C = kLdChunk / 2;
  for (uint32_t q0 = 0; q0 < cnt; q0 += C * kTileThreads) {
    float4 v0[C], v1[C];
#pragma unroll
    for (int k = 0; k < C; ++k) {
      const uint32_t q = q0 + threadIdx.x + k * kTileThreads;
      if (q < cnt) {
        const uint32_t off = rowoff[q >> kRowBits] + (q & 31u);
        v0[k] = src0[off];
        v1[k] = src1[off];
      }
    }
#pragma unroll
    for (int k = 0; k < C; ++k) {
      const uint32_t q = q0 + threadIdx.x + k * kTileThreads;
      if (q < cnt) {
        sm0[swz(q)] = v0[k];
        sm1[swz(q)] = v1[k];
      }
    }
  }
}

__device__ __noinline__ void store_tiles_ff(uint32_t o0, float4* dst0, uint32_t o1, float4* dst1, uint32_t rows, int m) {
  const float4 *sm0 = sh<float4>(o0), *sm1 = sh<float4>(o1);
  const uint32_t* rowoff = sh<uint32_t>(rows);
  const uint32_t cnt = 1u << m;
  for (uint32_t q = threadIdx.x; q < cnt; q += kTileThreads) {
    const uint32_t off = rowoff[q >> kRowBits] + (q & 31u);
    dst0[off] = sm0[swz(q)];
    dst1[off] = sm1[swz(q)];
  }
}

// Tile-local index of a thread's first amplitude: zeros put in at the phase's register
// bits (keep[k]: the bits below the k-th of them; rb steps of two instructions)
template <int RB>
__device__ __forceinline__ uint32_t phase_base(uint32_t tid, const TPhase& ph) {
  uint32_t b = tid;
#pragma unroll
  for (int k = 0; k < RB; ++k) b += b & ~(uint32_t)ph.keep[k];
  return b;
}

// global register index bits of this thread's amplitudes outside the phase: its place
// in the tile's rows (register qubits 0..4 are the tile's bits 0..4)
__device__ __forceinline__ uint32_t thread_global(uint32_t base, const uint32_t* rowoff, uint32_t tbase) {
  return tbase + rowoff[base >> kRowBits] + (base & 31u);
}

// shared-memory slot of amplitude j of a phase: swz is linear over XOR, so
// slot(j) = swz(base) ^ (XOR of swz(offset of bit b) over the set bits b of j);
// the per-bit values stay in registers instead of reloading sroff[j]
struct PhaseSlots {
  uint32_t b, s0, s1, s2, s3;
};
__device__ __forceinline__ PhaseSlots phase_slots(uint32_t sb, const TPhase& ph) {
  return PhaseSlots{sb, ph.sroff[1], ph.sroff[2], ph.sroff[4], ph.sroff[8]};
}
__device__ __forceinline__ uint32_t slot(const PhaseSlots& p, int j) {
  uint32_t o = p.b;
  if (j & 1) o ^= p.s0;
  if (j & 2) o ^= p.s1;
  if (j & 4) o ^= p.s2;
  if (j & 8) o ^= p.s3;
  return o;
}

// An op record in registers from four 16-byte loads issued together: one
// memory latency per op, instead of a chain of dependent field loads behind
// the op's control test and kind branches
__device__ __forceinline__ TOp load_op(const TOp* p) {
  const uint4* s = reinterpret_cast<const uint4*>(p);
  const uint4 a = s[0], b = s[1], c = s[2], d = s[3];
  TOp r;
  r.kind = (uint8_t)(a.x & 0xffu);
  r.t = (uint8_t)((a.x >> 8) & 0xffu);
  r.cmask = (uint8_t)((a.x >> 16) & 0xffu);
  r.cval = (uint8_t)(a.x >> 24);
  r.gen = (uint8_t)(a.y & 0xffu);
  r.shared = (uint8_t)((a.y >> 8) & 0xffu);
  r.var = (uint8_t)((a.y >> 16) & 0xffu);
  r.val = (uint8_t)(a.y >> 24);
  r.param = (int32_t)a.z;
  r.cfac2 = __uint_as_float(a.w);
  r.tmask = b.x;
  r.tval = b.y;
  r.count = b.z;
  r.pad = b.w;
  r.u[0] = make_float2(__uint_as_float(c.x), __uint_as_float(c.y));
  r.u[1] = make_float2(__uint_as_float(c.z), __uint_as_float(c.w));
  r.u[2] = make_float2(__uint_as_float(d.x), __uint_as_float(d.y));
  r.u[3] = make_float2(__uint_as_float(d.z), __uint_as_float(d.w));
  return r;
}

// ---- shared-memory copies of a pass's phase records and ops
//
// Every tile of a pass runs the same phases, so a CTA that streams tiles reads
// each op record once per tile.  Read from global memory, those records are
// evicted from L1 by the tile traffic and every op then waits on L2 before
// its first arithmetic (the records are read by a chain of dependent loads:
// the control test, the kind, the target, the matrix).  The pass's records are
// therefore copied into shared memory once per pass, with the phases' op
// indices rebased to the pass's first op.  A pass larger than the staging
// area keeps reading global memory.
constexpr int kStagePhases = 32;
constexpr int kStageOps = 512;
constexpr int kStageRuns = 256;  // forward: TK_DIAGRUN entries
constexpr int kStageMems = 224;  // backward: GMem records
static_assert(sizeof(TOp) == 64 && sizeof(TOp) % 16 == 0, "TOp is copied as 16-byte words");
static_assert(sizeof(DRun) == 32 && sizeof(GMem) == 32, "records are copied as 16-byte words");
static_assert(sizeof(DRun) * kStageRuns <= sizeof(BShared::red), "a pass's entries in the forward");
constexpr size_t kStagePhaseBytes = (sizeof(TPhase) * kStagePhases + 15) & ~size_t(15);
constexpr size_t kStageBytes = kStagePhaseBytes + sizeof(TOp) * kStageOps;  // then the records
constexpr size_t kStageMemBytes = sizeof(GMem) * kStageMems;
constexpr int kMaxSmem = 227 * 1024;  // of a CTA

struct StagedPass {
  const TPhase* ph;  // the pass's first phase
  const TOp* ops;    // op table the phases index
  int first;         // index of ops[0] in the global op table (0 when not staged)
  const DRun* runs;  // the pass's TK_DIAGRUN entries (forward)
  const GMem* mem;   // GMem records the ops index (backward)
};

// FWD: the forward ops (fop0 / nfop), else the backward ops (bop0 / nbop).
// buf: kStageBytes of shared memory, or nullptr; rec: `room` records of it.  Every thread of
// the CTA calls this (it ends with a barrier when it copies).
template <bool FWD>
__device__ StagedPass stage_pass(const TPass& p, const TPhase* phases, const TOp* ops, unsigned char* buf, void* rec,
                                 int room, const DRun* druns, const GMem* gmem) {
  StagedPass r{phases + p.phase0, ops, 0, FWD ? druns + p.drun0 : nullptr, gmem};
  if (!buf || p.nphase <= 0 || p.nphase > kStagePhases) return r;
  if (FWD && p.ndrun > room) return r;
  const TPhase& f0 = phases[p.phase0];
  const TPhase& fl = phases[p.phase0 + p.nphase - 1];
  const int first = FWD ? f0.fop0 : f0.bop0;
  const int count = FWD ? fl.fop0 + fl.nfop - first : fl.bop0 + fl.nbop - first;
  if (count < 0 || count > kStageOps) return r;
  TPhase* sph = reinterpret_cast<TPhase*>(buf);
  TOp* sop = reinterpret_cast<TOp*>(buf + kStagePhaseBytes);
  constexpr int W = (int)(sizeof(TOp) / 16);
  const uint4* src = reinterpret_cast<const uint4*>(ops + first);
  uint4* dst = reinterpret_cast<uint4*>(sop);
  for (int i = threadIdx.x; i < count * W; i += blockDim.x) dst[i] = src[i];
  if ((int)threadIdx.x < p.nphase) {
    TPhase q = phases[p.phase0 + threadIdx.x];
    if (FWD) q.fop0 -= first;
    else q.bop0 -= first;
    sph[threadIdx.x] = q;
  }
  // a pass with more GMem records than the area holds reads those from global memory
  uint4* rd = reinterpret_cast<uint4*>(rec);
  const bool recs = FWD || p.nmem <= room;
  const uint4* rs = FWD ? reinterpret_cast<const uint4*>(druns + p.drun0) : reinterpret_cast<const uint4*>(gmem + p.mem0);
  for (int i = threadIdx.x; recs && i < (FWD ? p.ndrun : p.nmem) * 2; i += blockDim.x) rd[i] = rs[i];
  __syncthreads();
  if (FWD) return StagedPass{sph, sop, first, reinterpret_cast<const DRun*>(rd), nullptr};
  return StagedPass{sph, sop, first, nullptr, recs ? reinterpret_cast<const GMem*>(rd) - p.mem0 : gmem};
}

// out-of-phase diagonal gate with phase-local controls: x_j *= f where (j & cm) == cv
template <int RB>
__device__ __forceinline__ void diag_masked(float2 (&x)[1 << RB], float2 f, int cm, int cv) {
#pragma unroll
  for (int j = 0; j < (1 << RB); ++j)
    if ((j & cm) == cv) x[j] = cmulf(x[j], f);
}

// COMP: compensated matrices (flo: 4 corrections per forward op, dtlo: 16 per
// diagonal table); out-of-phase diagonal factors are then applied one by one
template <int RB, bool COMP, bool RESLOT>
__device__ __forceinline__ void phase_fwd_body(float2* sm, const TPhase* php, const TOp* fops, const float2* dtab,
                                               const float2* flo, const float2* dtlo, const RunCtx& rc,
                                               const uint32_t* rowoff, int m, uint32_t tbase) {
  constexpr int A = 1 << RB;
  const TPhase& ph = *php;
  const int ntb = m - RB;
  if (threadIdx.x < (1u << ntb)) {
    const uint32_t base = phase_base<RB>(threadIdx.x, ph);
    const PhaseSlots ps = phase_slots(swz(base), ph);
    const uint32_t gb = thread_global(base, rowoff, tbase);
    float2 x[A];
#pragma unroll
    for (int j = 0; j < A; ++j) x[j] = sm[slot(ps, j)];
    // factors of out-of-phase diagonal gates without phase-local controls are
    // scalars for this thread: they commute with the phase and are applied once
    float2 pend = make_float2(1.f, 0.f);
    bool has_pend = false;
    for (int o = 0; o < ph.nfop; ++o) {
      const int oi = ph.fop0 + o;
      const TOp cur = load_op(fops + oi);
      const bool on = (gb & cur.tmask) == cur.tval;
      // The order of the tests shows in the whole loop.  Batches: runs first (their circuits are
      // made of them).  Tile engine: the plain kinds first, behind one test (440 controlled Rx on
      // 24 qubits 3.08 -> 2.84 ms, 300 gates Rx, Ry and controlled Z 2.49 -> 2.41; a QFT's 18.2 ms
      // stay)
      if constexpr (RESLOT) {
        if (cur.kind == TK_DENSEX) {
          apply_densex<RB, COMP>(x, cur, COMP ? flo + 4 * oi : nullptr, on);
          continue;
        }
      } else {
        if (cur.kind <= TK_DIAGRUN) {
          if (on) apply_fwd_var<RB, COMP>(x, cur, COMP ? flo + 4 * oi : nullptr, rc, gb);
          continue;
        }
        if (cur.kind >= TK_DENSEX) {
          if (cur.kind == TK_DENSEX) {
            apply_densex<RB, COMP>(x, cur, COMP ? flo + 4 * oi : nullptr, on);
            continue;
          }
          switch (cur.t) {  // TK_REALRUN
            case 0: real_run<RB, 0>(x, cur, rc, dtab, gb); break;
            case 1: real_run<RB, 1>(x, cur, rc, dtab, gb); break;
            case 2: real_run<RB, 2>(x, cur, rc, dtab, gb); break;
            default: real_run<RB, 3>(x, cur, rc, dtab, gb); break;
          }
          continue;
        }
      }
      if (!on) continue;
      if (cur.kind == TK_DIAGOUT) {
        const bool b1 = (gb >> cur.t) & 1u;
        const float2 f = b1 ? cur.u[3] : cur.u[0];
        if (COMP) {
          const float2 fl = flo[4 * oi + (b1 ? 3 : 0)];
#pragma unroll
          for (int j = 0; j < A; ++j)
            if ((j & cur.cmask) == cur.cval) x[j] = cf_mul(x[j], f, fl);
        } else if (f.x == 1.f && f.y == 0.f) {
          // a factor of exactly 1 (the |0> entry of a shift or controlled phase)
        } else if (cur.cmask == 0) {
          pend = cmulf(pend, f);
          has_pend = true;
        } else {
          diag_masked<RB>(x, f, cur.cmask, cur.cval);
        }
      } else if (cur.kind == TK_DIAG16) {
        const float2* t = dtab + 16 * cur.param;
        if (COMP) {
          const float2* tl = dtlo + 16 * cur.param;
#pragma unroll
          for (int j = 0; j < A; ++j) x[j] = cf_mul(x[j], t[j], tl[j]);
        } else {
#pragma unroll
          for (int j = 0; j < A; ++j) x[j] = cmulf(x[j], t[j]);
        }
      } else if constexpr (RESLOT) {
        apply_fwd_var<RB, COMP>(x, cur, COMP ? flo + 4 * oi : nullptr, rc, gb);
      }
    }
    if (!COMP && has_pend) {
#pragma unroll
      for (int j = 0; j < A; ++j) x[j] = cmulf(x[j], pend);
    }
    // RESLOT: the slot offsets again (from shared memory) rather than live
    // through the op loop (fewer spills in k_batch; slower in the tile engine,
    // whose loop does not spill)
    const PhaseSlots ps2 = RESLOT ? phase_slots(swz(phase_base<RB>(threadIdx.x, ph)), ph) : ps;
#pragma unroll
    for (int j = 0; j < A; ++j) sm[slot(ps2, j)] = x[j];
  }
  __syncthreads();
}

// All phases of a pass on one tile, in order (one call per tile).  SITE gives
// each call site its own copy: ptxas allocates a called function's registers
// per kernel, and one copy shared by the resident and streamed loops of
// k_batch spilled several times as much (ptxas -v) as two copies do; SITE 2
// is the tile engine's pass.
template <int RB, bool COMP, int SITE = 0>
__device__ __noinline__ void run_tile_fwd(uint32_t sm, const TPhase* ph, int nphase, const TOp* fops,
                                          const float2* dtab, const float2* flo, const float2* dtlo, uint32_t rc,
                                          uint32_t rows, int m, uint32_t tbase) {
  for (int f = 0; f < nphase; ++f)
    phase_fwd_body<RB, COMP, SITE != 2>(sh<float2>(sm), ph + f, fops, dtab, flo, dtlo, *sh<RunCtx>(rc),
                                        sh<uint32_t>(rows), m, tbase);
}

// backward of an out-of-phase diagonal gate: the generator is diagonal on the
// target (Z, P1 or 1), whose value is fixed for this thread
__device__ __forceinline__ float diagout_sign(const TOp& op, bool b) {
  switch (op.gen) {
    case GEN_Z: return b ? -1.f : 1.f;
    case GEN_P1: return b ? 1.f : 0.f;
    case GEN_I: return 1.f;
    default: return 0.f;
  }
}

template <int RB>
__device__ __forceinline__ float diagout_bwd(float2 (&x)[1 << RB], float2 (&l)[1 << RB], const TOp& op, uint32_t gb) {
  const bool b = (gb >> op.t) & 1u;
  const float2 d = b ? op.u[3] : op.u[0];
  const int cm = op.cmask, cv = op.cval;
  float acc = 0.f;
#pragma unroll
  for (int j = 0; j < (1 << RB); ++j) {
    if ((j & cm) != cv) continue;
    acc += imcj(l[j], x[j]);
    x[j] = cmulf(x[j], d);
    l[j] = cmulf(l[j], d);
  }
  return diagout_sign(op, b) * acc;
}

template <int RB>
__device__ __forceinline__ float diagout_bwd_ff(ffc (&x)[1 << RB], ffc (&l)[1 << RB], const TOp& op, const float2* lo,
                                                uint32_t gb) {
  const bool b = (gb >> op.t) & 1u;
  const float2 d = b ? op.u[3] : op.u[0];
  const float2 dl = b ? lo[3] : lo[0];
  const int cm = op.cmask, cv = op.cval;
  float acc = 0.f;
#pragma unroll
  for (int j = 0; j < (1 << RB); ++j) {
    if ((j & cm) != cv) continue;
    acc += imcj(l[j].h, x[j].h);
    x[j] = ff_cmul(x[j], d, dl);
    l[j] = ff_cmul(l[j], d, dl);
  }
  return diagout_sign(op, b) * acc;
}

// Warp sums of the gradient ops' lane partials, two ops at a time: the two
// shuffle trees interleave, so a warp waits on one chain of shuffle latencies
// per pair of ops instead of per op.  pend / pend_o hold the first op of a pair
// (pend_o is the same in every lane).
__device__ __forceinline__ void warp_partial(float part, int o, float& pend, int& pend_o, float* red, int lane,
                                             int warp) {
  if (pend_o < 0) {
    pend = part;
    pend_o = o;
    return;
  }
#pragma unroll
  for (int s = 16; s > 0; s >>= 1) {
    pend += __shfl_xor_sync(0xffffffffu, pend, s);
    part += __shfl_xor_sync(0xffffffffu, part, s);
  }
  if (lane == 0) {
    red[pend_o * kWarps + warp] = pend;
    red[o * kWarps + warp] = part;
  }
  pend_o = -1;
}
__device__ __forceinline__ void flush_partial(float pend, int pend_o, float* red, int lane, int warp) {
  if (pend_o < 0) return;
#pragma unroll
  for (int s = 16; s > 0; s >>= 1) pend += __shfl_xor_sync(0xffffffffu, pend, s);
  if (lane == 0) red[pend_o * kWarps + warp] = pend;
}

// warp sums of the four values of a TK_RUN op: each step halves the values a lane still
// carries (6 shuffles, where four trees take 20); lanes 0, 8, 16, 24 hold one each
__device__ __forceinline__ void warp_sums4(const float (&v)[4], float* red, int lane, int warp) {
  const bool h = lane & 16, q = lane & 8;
  float a = h ? v[2] : v[0], b = h ? v[3] : v[1];
  a += __shfl_xor_sync(0xffffffffu, h ? v[0] : v[2], 16);
  b += __shfl_xor_sync(0xffffffffu, h ? v[1] : v[3], 16);
  float c = q ? b : a;
  c += __shfl_xor_sync(0xffffffffu, q ? a : b, 8);
#pragma unroll
  for (int s = 4; s > 0; s >>= 1) c += __shfl_xor_sync(0xffffffffu, c, s);
  if ((lane & 7) == 0) red[(lane >> 3) * kWarps + warp] = c;
}

// fold the warp partials of every parameterised op of a phase: the 16 warp
// partials of a sum are added by 16 lanes in a TwoSum tree (the double-float
// sum s + e of the FP32 partials, exact to ~2^-48), one op per 16 lanes, all
// ops at once; then lane k of the 16 adds the op's k-th record, its combination of
// the op's sums in double-float, to the FP64 accumulator.  Records whose
// parameter another one of the phase shares are added by one thread afterwards.
// (FP64 arithmetic runs at 1/64 of the FP32 rate here: summing in FP64 took
// one warp thousands of cycles per phase while the others waited.)
__device__ __forceinline__ void fold_phase_grad(const TPhase& ph, const TOp* bops, const GMem* gmem, const float* red,
                                                double* gacc) {
  static_assert(kWarps == 16, "one op per 16 lanes");
  const int nbop = ph.nbop, bop0 = ph.bop0;
  for (int base = 0; base < nbop * kWarps; base += blockDim.x) {
    const int t = base + (int)threadIdx.x;
    const int o = t >> 4, w = t & 15;
    const TOp* op = bops + bop0 + (o < nbop ? o : 0);
    const int recs = o < nbop ? (int)op->count : 0;
    const bool run = recs && op->kind == TK_RUN;
    const float* r = red + op->val * kWarps + w;
    float s[4], e[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      s[k] = e[k] = 0.f;
      if (k > 0 && !__any_sync(0xffffffffu, run)) continue;
      if (k == 0 ? recs > 0 : run) s[k] = r[k * kWarps];
#pragma unroll
      for (int d = 8; d > 0; d >>= 1) {
        const float so = __shfl_xor_sync(0xffffffffu, s[k], d), eo = __shfl_xor_sync(0xffffffffu, e[k], d);
        float q, f;
        two_sum(s[k], so, q, f);
        s[k] = q;
        e[k] = __fadd_rn(__fadd_rn(e[k], eo), f);
      }
    }
    if (w < recs) {
      const GMem m = gmem[op->param + w];
      float hs = 0.f, he = 0.f;
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const float p = __fmul_rn(m.c[k], s[k]);
        const float pe = fmaf(m.c[k], e[k], fmaf(m.c[k], s[k], -p));
        float q, f;
        two_sum(hs, p, q, f);
        hs = q;
        he = __fadd_rn(he, __fadd_rn(f, pe));
      }
      if (!m.shared) gacc[m.param] += (double)hs + (double)he;
    }
  }
  __syncthreads();
  if (ph.nshared == 0) return;
  if (threadIdx.x == 0) {
    for (int q = 0; q < nbop; ++q) {
      const TOp& op = bops[bop0 + q];
      for (int k = 0; k < (int)op.count; ++k) {
        const GMem& m = gmem[op.param + k];
        if (!m.shared) continue;
        double g = 0.0;
        for (int i = 0; i < (op.kind == TK_RUN ? 4 : 1); ++i) {
          double v = 0.0;
          for (int w = 0; w < kWarps; ++w) v += (double)red[(op.val + i) * kWarps + w];
          g += (double)m.c[i] * v;
        }
        gacc[m.param] += g;
      }
    }
  }
  __syncthreads();
}

template <int RB>
__device__ __forceinline__ void phase_bwd_body(float2* sx, float2* sl, const TPhase* php, const TOp* bops,
                                               const GMem* gmem, int m, const uint32_t* rowoff, float* red, double* gacc, uint32_t tbase) {
  // the phase record is read where it lies (the pass's shared-memory copy when
  // staged): with 2 x 2^RB live amplitudes per thread there are no registers
  // to spare for a copy of it
  constexpr int A = 1 << RB;
  const TPhase& ph = *php;
  const int ntb = m - RB;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const bool active = threadIdx.x < (1u << ntb);
  const int nbop = ph.nbop, bop0 = ph.bop0;
  float2 x[A], l[A];
  const uint32_t base = active ? phase_base<RB>(threadIdx.x, ph) : 0u;
  const uint32_t gb = thread_global(base, rowoff, tbase);
  const PhaseSlots ps = phase_slots(swz(base), ph);
  if (active) {
#pragma unroll
    for (int j = 0; j < A; ++j) {
      const uint32_t o = slot(ps, j);
      x[j] = sx[o];
      l[j] = sl[o];
    }
  }
  float pend = 0.f;  // warp partial of a gradient op waiting for a partner (pend_o >= 0)
  int pend_o = -1;
  // Runs and other ops each in a loop of their own: as branches of one loop they cost the gates that
  // are no runs 17 instructions an op (80 registers of 15 qubits, 200 Rz: 1.50 ms, 1.37 before the
  // runs came in and now; the batch of 1024 registers 91.4 -> 90.3)
  for (int o = nbop - 1; o >= 0; --o) {
    TOp op = load_op(bops + bop0 + o);
    while (op.kind == TK_RUN) {
      float v[4] = {0.f, 0.f, 0.f, 0.f};
      if (active) apply_bwd_run<RB>(x, l, op, op.cmask && (gb & op.tmask) == op.tval, v);
      warp_sums4(v, red + op.val * kWarps, lane, warp);
      if (--o < 0) break;
      op = load_op(bops + bop0 + o);
    }
    if (o < 0) break;
    float part = 0.f;
    if (active && (gb & op.tmask) == op.tval)
      part = op.kind == TK_DIAGOUT ? diagout_bwd<RB>(x, l, op, gb) : apply_bwd_var<RB>(x, l, op);
    if (op.gen != GEN_NONE) warp_partial(part, op.val, pend, pend_o, red, lane, warp);
  }
  flush_partial(pend, pend_o, red, lane, warp);
  if (active) {
#pragma unroll
    for (int j = 0; j < A; ++j) {
      const uint32_t o = slot(ps, j);
      sx[o] = x[j];
      sl[o] = l[j];
    }
  }
  __syncthreads();
  fold_phase_grad(ph, bops, gmem, red, gacc);
}

// All phases of a pass on one tile, last phase first: one call per tile, so
// that the callers' loop state is saved once per tile rather than per phase
template <int RB>
__device__ __noinline__ void run_tile_bwd(uint32_t sx, uint32_t sl, const TPhase* ph, int nphase, const TOp* bops,
                                          const GMem* gmem, int m, uint32_t rows, uint32_t red, uint32_t gacc, uint32_t tbase) {
  for (int f = nphase - 1; f >= 0; --f)
    phase_bwd_body<RB>(sh<float2>(sx), sh<float2>(sl), ph + f, bops, gmem, m, sh<uint32_t>(rows), sh<float>(red),
                       sh<double>(gacc), tbase);
}

template <int RB>
__device__ __noinline__ void run_phase_bwd_ff(uint32_t ox, uint32_t ol, const TPhase* php, const TOp* bops,
                                              const GMem* gmem, const float2* blo, int m, uint32_t rows, uint32_t ored,
                                              uint32_t ogacc, uint32_t tbase) {
  float4 *sx = sh<float4>(ox), *sl = sh<float4>(ol);
  const uint32_t* rowoff = sh<uint32_t>(rows);
  float* red = sh<float>(ored);
  double* gacc = sh<double>(ogacc);
  constexpr int A = 1 << RB;
  const TPhase& ph = *php;
  const int ntb = m - RB;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const bool active = threadIdx.x < (1u << ntb);
  const int nbop = ph.nbop, bop0 = ph.bop0;
  ffc x[A], l[A];
  const uint32_t base = active ? phase_base<RB>(threadIdx.x, ph) : 0u;
  const uint32_t gb = thread_global(base, rowoff, tbase);
  const PhaseSlots ps = phase_slots(swz(base), ph);
  if (active) {
#pragma unroll
    for (int j = 0; j < A; ++j) {
      const uint32_t o = slot(ps, j);
      const float4 a = sx[o], b = sl[o];
      x[j].h = make_float2(a.x, a.y);
      x[j].l = make_float2(a.z, a.w);
      l[j].h = make_float2(b.x, b.y);
      l[j].l = make_float2(b.z, b.w);
    }
  }
  float pend = 0.f;
  int pend_o = -1;
  // the other ops in a loop of their own, so that what the runs spill does not lie on their way
  // (spill loads 1412 -> 396 bytes; batch of 200 registers 52.4 -> 50.8 ms)
  for (int o = nbop - 1; o >= 0; --o) {
    TOp op = load_op(bops + bop0 + o);
    while (op.kind != TK_RUN) {
      float part = 0.f;
      if (active && (gb & op.tmask) == op.tval)
        part = op.kind == TK_DIAGOUT ? diagout_bwd_ff<RB>(x, l, op, blo + 4 * (bop0 + o), gb)
                                     : apply_bwd_ff<RB>(x, l, op, blo + 4 * (bop0 + o));
      if (op.gen != GEN_NONE) warp_partial(part, op.val, pend, pend_o, red, lane, warp);
      if (--o < 0) break;
      op = load_op(bops + bop0 + o);
    }
    if (o < 0) break;
    float v[4] = {0.f, 0.f, 0.f, 0.f};
    if (active) apply_bwd_run_ff<RB>(x, l, op, blo + 4 * (bop0 + o), op.cmask && (gb & op.tmask) == op.tval, v);
    warp_sums4(v, red + op.val * kWarps, lane, warp);
  }
  flush_partial(pend, pend_o, red, lane, warp);
  if (active) {
#pragma unroll
    for (int j = 0; j < A; ++j) {
      const uint32_t o = slot(ps, j);
      sx[o] = make_float4(x[j].h.x, x[j].h.y, x[j].l.x, x[j].l.y);
      sl[o] = make_float4(l[j].h.x, l[j].h.y, l[j].l.x, l[j].l.y);
    }
  }
  __syncthreads();
  fold_phase_grad(ph, bops, gmem, red, gacc);
}

// the diagonal observable's weight w(i) = sum_t c_t (-1)^popcount(i & z_t)
__device__ __forceinline__ double obs_weight(uint64_t gi, const BTerm* terms, int nterm) {
  double w = 0.0;
  for (int t = 0; t < nterm; ++t) w += (__popcll(gi & terms[t].z) & 1) ? -terms[t].coeff : terms[t].coeff;
  return w;
}

// loss partial and lambda = w psi for the diagonal observable, over a tile in smem
__device__ double expect_tile(float2* sx, float2* sl, uint64_t tbase, const uint32_t* rowoff, int m,
                              const BTerm* terms, int nterm) {
  const uint32_t cnt = 1u << m;
  double acc = 0.0;
  for (uint32_t l = threadIdx.x; l < cnt; l += blockDim.x) {
    const uint64_t gi = tbase + rowoff[l >> kRowBits] + (l & 31u);
    const double w = obs_weight(gi, terms, nterm);
    const float2 a = sx[swz(l)];
    acc += w * ((double)a.x * a.x + (double)a.y * a.y);
    const float wf = (float)w;
    sl[swz(l)] = make_float2(wf * a.x, wf * a.y);
  }
  return acc;
}

// the same from a complex64 tile into double-float psi and lambda tiles
// (w psi formed in FP64 and split into hi + lo)
__device__ double expect_tile_ff(const float2* s2, float4* sxf, float4* slf, uint64_t tbase, const uint32_t* rowoff,
                                 int m, const BTerm* terms, int nterm) {
  const uint32_t cnt = 1u << m;
  double acc = 0.0;
  for (uint32_t l = threadIdx.x; l < cnt; l += blockDim.x) {
    const uint64_t gi = tbase + rowoff[l >> kRowBits] + (l & 31u);
    const double w = obs_weight(gi, terms, nterm);
    const float2 a = s2[swz(l)];
    acc += w * ((double)a.x * a.x + (double)a.y * a.y);
    const double lr = w * (double)a.x, li = w * (double)a.y;
    const float hr = (float)lr, hi = (float)li;
    sxf[swz(l)] = make_float4(a.x, a.y, 0.f, 0.f);
    slf[swz(l)] = make_float4(hr, hi, (float)(lr - (double)hr), (float)(li - (double)hi));
  }
  return acc;
}

__device__ void block_loss(double e, BShared& S, double* out) {
  for (int s = 16; s > 0; s >>= 1) e += __shfl_xor_sync(0xffffffffu, e, s);
  if ((threadIdx.x & 31) == 0) S.lred[threadIdx.x >> 5] = e;
  __syncthreads();
  if (threadIdx.x == 0) {
    static_assert(kWarps == 16, "loss tree below is written for 16 warps");
    const double* v = S.lred;
    *out = (((v[0] + v[1]) + (v[2] + v[3])) + ((v[4] + v[5]) + (v[6] + v[7]))) +
           (((v[8] + v[9]) + (v[10] + v[11])) + ((v[12] + v[13]) + (v[14] + v[15])));
  }
}

// The per-register phase loops of k_batch live in their own (not inlined)
// functions: a phase call then sees only the loop's few live values, and the
// phase functions keep their amplitudes in registers.
template <int RB>
__device__ __noinline__ void batch_bwd_resident(uint32_t sx, uint32_t sl, const TPass* P, int npass, int m,
                                                const TPhase* phases, const TOp* bops, const GMem* gmem, uint32_t rows,
                                                uint32_t red, uint32_t gacc) {
  for (int pi = npass - 1; pi >= 0; --pi)
    run_tile_bwd<RB>(sx, sl, phases + P[pi].phase0, P[pi].nphase, bops, gmem, m, rows, red, gacc, 0u);
}

template <int RB>
__device__ __noinline__ void batch_bwd_resident_ff(uint32_t sx, uint32_t sl, const TPass* P, int npass, int m,
                                                   const TPhase* phases, const TOp* bops, const GMem* gmem,
                                                   const float2* blo, uint32_t rows, uint32_t red, uint32_t gacc) {
  for (int pi = npass - 1; pi >= 0; --pi) {
    const int ph0 = P[pi].phase0;
    for (int f = P[pi].nphase - 1; f >= 0; --f)
      run_phase_bwd_ff<RB>(sx, sl, phases + ph0 + f, bops, gmem, blo, m, rows, red, gacc, 0u);
  }
}

template <int RB>
__device__ __noinline__ void batch_bwd_streamed(uint32_t sx, uint32_t sl, const TPass* P, int npass, int m, int g,
                                                float2* wp, float2* wl, const TPhase* phases, const TOp* bops,
                                                const GMem* gmem, uint32_t rows, uint32_t red, uint32_t gacc, unsigned char* stage) {
  const uint64_t ntile = 1ull << g;
  for (int pi = npass - 1; pi >= 0; --pi) {
    const TPass& p = P[pi];
    set_rows(sh<uint32_t>(rows), p, m);
    const StagedPass sp = stage_pass<false>(p, phases, bops, stage, stage + kStageBytes, kStageMems, nullptr, gmem);
    for (uint64_t t = 0; t < ntile; ++t) {
      const uint64_t tb = tile_base(t, p, g);
      load_tiles<true>(sx, wp + tb, sl, wl + tb, rows, m);
      __syncthreads();
      run_tile_bwd<RB>(sx, sl, sp.ph, p.nphase, sp.ops, sp.mem, m, rows, red, gacc, (uint32_t)tb);
      store_tiles<true>(sx, wp + tb, sl, wl + tb, rows, m);
      __syncthreads();
    }
  }
}

template <int RB>
__device__ __noinline__ void batch_bwd_streamed_ff(uint32_t sx, uint32_t sl, const TPass* P, int npass, int m, int g,
                                                   float4* wp, float4* wl, const TPhase* phases, const TOp* bops,
                                                   const GMem* gmem, const float2* blo, uint32_t rows, uint32_t red, uint32_t gacc,
                                                   unsigned char* stage) {
  const uint64_t ntile = 1ull << g;
  for (int pi = npass - 1; pi >= 0; --pi) {
    const TPass& p = P[pi];
    set_rows(sh<uint32_t>(rows), p, m);
    const StagedPass sp = stage_pass<false>(p, phases, bops, stage, stage + kStageBytes, kStageMems, nullptr, gmem);
    const float2* lo = blo + 4 * (size_t)sp.first;
    for (uint64_t t = 0; t < ntile; ++t) {
      const uint64_t tb = tile_base(t, p, g);
      load_tiles_ff(sx, wp + tb, sl, wl + tb, rows, m);
      __syncthreads();
      for (int f = p.nphase - 1; f >= 0; --f)
        run_phase_bwd_ff<RB>(sx, sl, sp.ph + f, sp.ops, sp.mem, lo, m, rows, red, gacc, (uint32_t)tb);
      store_tiles_ff(sx, wp + tb, sl, wl + tb, rows, m);
      __syncthreads();
    }
  }
}

// cp.async copies (8 bytes each: the swizzled slots of a 16-byte pair may be
// swapped) of the next tile into a second buffer while the current one is computed
__device__ __forceinline__ void cp_async8(void* smem, const void* gmem) {
  const uint32_t d = (uint32_t)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(d), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_prev() { asm volatile("cp.async.wait_group 1;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_group 0;\n" ::: "memory"); }

// issue the copies of one tile (2^m amplitudes) into sm (no wait)
__device__ __forceinline__ void load_tile_async(uint32_t o, const float2* src, uint32_t rows, int m) {
  float2* sm = sh<float2>(o);
  const uint32_t* rowoff = sh<uint32_t>(rows);
  const uint32_t n = 1u << m;
  for (uint32_t l = threadIdx.x; l < n; l += kTileThreads)
    cp_async8(sm + swz(l), src + rowoff[l >> kRowBits] + (l & 31u));
}

template <int RB, bool COMP>
__device__ __noinline__ void batch_fwd_streamed(uint32_t sx, uint32_t sx2, float2* st, const TPass* P, int npass,
                                                int m, int g, const TPhase* phases, const TOp* fops,
                                                const float2* dtab, const float2* flo, const float2* dtlo,
                                                const DRun* druns, const float4* rtab, uint32_t rc, uint32_t rows,
                                                unsigned char* stage) {
  const uint64_t ntile = 1ull << g;
  for (int pi = 0; pi < npass; ++pi) {
    const TPass& p = P[pi];
    set_rows(sh<uint32_t>(rows), p, m);
    const StagedPass sp = stage_pass<true>(p, phases, fops, stage, sh<float>((uint32_t)offsetof(BShared, red)), kStageRuns,
                                           druns, nullptr);
    const float2* lo = COMP ? flo + 4 * (size_t)sp.first : nullptr;
    if (threadIdx.x == 0) *sh<RunCtx>(rc) = RunCtx{sp.runs, rtab + kRunTab * p.run0, nullptr};
    // two tile buffers (sx, sx2): the next tile's copies are in flight while
    // the current one is computed
    load_tile_async(sx, st + tile_base(0, p, g), rows, m);
    cp_async_commit();
    for (uint64_t t = 0; t < ntile; ++t) {
      const uint32_t cur = (t & 1) ? sx2 : sx;
      if (t + 1 < ntile) load_tile_async((t & 1) ? sx : sx2, st + tile_base(t + 1, p, g), rows, m);
      cp_async_commit();
      cp_async_wait_prev();
      __syncthreads();
      const uint64_t tb = tile_base(t, p, g);
      run_tile_fwd<RB, COMP, 1>(cur, sp.ph, p.nphase, sp.ops, dtab, lo, dtlo, rc, rows, m, (uint32_t)tb);
      store_tile(cur, st + tb, rows, m);
      __syncthreads();
    }
    cp_async_wait_all();
  }
}

// CTAs per SM the register budget is sized for (two CTAs of 3-qubit phases, at
// 64 registers a thread, spilled and measured slower: 247 vs 213 ms per batch)
template <int RB, bool PREC>
constexpr int kBatchMinBlocks = 1;

// Shared memory of k_batch after the BShared header: the complex64 path holds
// psi and lambda tiles (2 x 2^13 x 8 bytes); the precise path holds double-float
// psi and lambda tiles (2 x 2^m x 16 bytes) and a complex64 forward tile.
template <int RB, bool PREC>
__global__ void __launch_bounds__(kTileThreads, kBatchMinBlocks<RB, PREC>) k_batch(BArgs a) {
  extern __shared__ __align__(16) unsigned char smraw[];
  BShared& S = *reinterpret_cast<BShared*>(smraw);
  constexpr int MT = kTileThreads == 512 ? 9 + RB : 0;  // largest tile: 512 threads x 2^RB amplitudes
  static_assert(MT >= kRowBits + RB && MT <= kMaxTileBits, "tile size");
  unsigned char* body = smraw + ((sizeof(BShared) + 255) & ~size_t(255));
  float2* sx = reinterpret_cast<float2*>(body);                   // complex64 psi tile (forward, and FP32 backward)
  float2* sl = sx + (1 << MT);                                    // complex64 lambda tile (FP32 backward)
  float4* sxf = reinterpret_cast<float4*>(body + (size_t)8 * (1 << MT));   // double-float psi (precise)
  float4* slf = sxf + (1 << MT);                                           // double-float lambda (precise)
  unsigned char* stage = body + (size_t)(PREC ? 40 : 16) * (1 << MT);      // a pass's records (streamed registers)
  // byte offsets of the above
  const uint32_t ox = (uint32_t)(body - smraw), ol = ox + (uint32_t)sizeof(float2) * (1u << MT);
  const uint32_t oxf = ol, olf = oxf + (uint32_t)sizeof(float4) * (1u << MT);
  const uint32_t orows = (uint32_t)offsetof(BShared, rowoff), ored = (uint32_t)offsetof(BShared, red);
  const uint32_t ograd = (uint32_t)offsetof(BShared, grad), orc = (uint32_t)offsetof(BShared, rc);
  const int tid = threadIdx.x;
  for (;;) {
    if (tid == 0) S.reg = atomicAdd(a.counter, 1);
    __syncthreads();
    const int ri = S.reg;
    __syncthreads();
    if (ri >= a.nreg) break;
    const int reg = a.order[ri];
    const BReg R = a.regs[reg];
    const int n = R.n, m = R.m, g = n - m;
    const bool grad = (a.flags & BF_GRAD) != 0;
    for (int i = tid; i < R.nparam; i += blockDim.x) S.grad[i] = 0.0;
    float2* st = a.state + R.amp_off;
    const uint64_t ntile = 1ull << g;
    const TPass* P = a.passes + R.pass0;
    if (g == 0) {
      // ---- whole register in shared memory
      set_rows(S.rowoff, P[0], m);
      if (a.flags & BF_RESET) {
        for (uint32_t l = tid; l < (1u << m); l += blockDim.x) sx[swz(l)] = make_float2(l == 0 ? 1.f : 0.f, 0.f);
      } else {
        load_tile(ox, st, orows, m);
      }
      __syncthreads();
      for (int pi = 0; pi < R.npass; ++pi) {
        if (!PREC) {
          if (tid == 0) S.rc = RunCtx{a.druns + P[pi].drun0, a.rtab + kRunTab * P[pi].run0, nullptr};
          __syncthreads();
        }
        run_tile_fwd<RB, PREC>(ox, a.phases + P[pi].phase0, P[pi].nphase, a.fops, a.dtab, a.flo, a.dtlo, orc, orows, m, 0u);
      }
      store_tile(ox, st, orows, m);  // psi_N
      if (PREC) {
        block_loss(expect_tile_ff(sx, sxf, slf, 0, S.rowoff, m, a.terms + R.term0, R.nterm), S, a.loss + reg);
        __syncthreads();
        if (grad) batch_bwd_resident_ff<RB>(oxf, olf, P, R.npass, m, a.phases, a.bops, a.gmem, a.blo, orows, ored, ograd);
      } else {
        block_loss(expect_tile(sx, sl, 0, S.rowoff, m, a.terms + R.term0, R.nterm), S, a.loss + reg);
        __syncthreads();
        if (grad) batch_bwd_resident<RB>(ox, ol, P, R.npass, m, a.phases, a.bops, a.gmem, orows, ored, ograd);
      }
    } else {
      // ---- tiles streamed through global memory
      if (a.flags & BF_RESET) {
        for (uint64_t i = tid; i < (1ull << n); i += blockDim.x) st[i] = make_float2(i == 0 ? 1.f : 0.f, 0.f);
        __syncthreads();
      }
      batch_fwd_streamed<RB, PREC>(ox, ol, st, P, R.npass, m, g, a.phases,
                                   a.fops, a.dtab, a.flo, a.dtlo, a.druns, a.rtab, orc, orows, stage);
      // expectation, lambda = O psi, and the work copy of psi for the uncompute
      double e = 0.0;
      const TPass& p0 = P[0];
      set_rows(S.rowoff, p0, m);
      for (uint64_t t = 0; t < ntile; ++t) {
        const uint64_t tb = tile_base(t, p0, g);
        load_tile(ox, st + tb, orows, m);
        __syncthreads();
        if (PREC) {
          e += expect_tile_ff(sx, sxf, slf, tb, S.rowoff, m, a.terms + R.term0, R.nterm);
          __syncthreads();
          if (grad) store_tiles_ff(oxf, a.wpsif + R.work_off + tb, olf, a.wlamf + R.work_off + tb, orows, m);
        } else {
          e += expect_tile(sx, sl, tb, S.rowoff, m, a.terms + R.term0, R.nterm);
          __syncthreads();
          if (grad) store_tiles<true>(ox, a.wpsi + R.work_off + tb, ol, a.wlam + R.work_off + tb, orows, m);
        }
        __syncthreads();
      }
      block_loss(e, S, a.loss + reg);
      __syncthreads();
      if (grad) {
        if (PREC)
          batch_bwd_streamed_ff<RB>(oxf, olf, P, R.npass, m, g, a.wpsif + R.work_off, a.wlamf + R.work_off, a.phases,
                                    a.bops, a.gmem, a.blo, orows, ored, ograd, stage);
        else
          batch_bwd_streamed<RB>(ox, ol, P, R.npass, m, g, a.wpsi + R.work_off, a.wlam + R.work_off, a.phases,
                                 a.bops, a.gmem, orows, ored, ograd, stage);
      }
    }
    __syncthreads();
    if (grad)
      for (int i = tid; i < R.nparam; i += blockDim.x) a.grad[R.param_off + i] = S.grad[i];
    __syncthreads();
  }
}

// bytes of dynamic shared memory of k_batch<RB, PREC>
static constexpr size_t batch_smem(int rb, bool prec) {
  const size_t mt = (size_t)1 << (9 + rb);
  return ((sizeof(BShared) + 255) & ~size_t(255)) + (prec ? (8 + 32) * mt : 16 * mt) + kStageBytes + kStageMemBytes;
}
// 195 KB leave 60 KB of L1, a byte more 28 (the state's tiles stream through it: batch of 1024
// registers 91.4 ms, 93.9 with 2 KB more)
static_assert(batch_smem(kRB, false) <= 195 * 1024 && batch_smem(3, true) <= kMaxSmem, "a register's shared memory");

// the instantiation of k_batch for a phase width and path
static const void* batch_kernel(int rb, bool prec) {
  if (prec) return rb == 2 ? (const void*)k_batch<2, true> : (const void*)k_batch<3, true>;
  switch (rb) {
    case 2: return (const void*)k_batch<2, false>;
    case 3: return (const void*)k_batch<3, false>;
    default: return (const void*)k_batch<4, false>;
  }
}


// ------------------------------------------------------------------ device: fused forward passes of large registers

struct FArgs {
  float2* state;
  const TPass* pass;
  const TPhase* phases;
  const TOp* fops;
  const float2* dtab;
  const DRun* druns;
  const float4* rtab;
  const int2* runs;        // first tile-id entry (in the pass) and their count, a run
  int m, g;
  uint64_t ntile;          // tiles per register
  uint64_t reg_stride;     // amplitudes per register
  int nreg;
};

constexpr int kTileRuns = 48;  // runs of a pass whose tables and tile products shared memory holds
constexpr int kTileTabs = 48;  // TK_DIAG16 tables of a pass that it holds
constexpr uint32_t kTileBytes = sizeof(float2) << kBatchTile;

// k_fused_pass's shared memory: offsets known to the compiler, so that what the op loop
// reads costs no pointer and no generic load.  With the diagonal tables here instead of in
// global memory, and a tile's place found by one OR over the warp instead of a loop over the
// tile-id bits and a 64-bit division: passes of a QFT of 29 qubits 7.5, 5.1, 5.4 -> 6.6,
// 4.5, 4.8 ms (a wait for a global or generic load was the first stall).
constexpr uint32_t kFpBuf = sizeof(uint32_t) << (kMaxTileBits - kRowBits);  // after the rows' offsets: two tiles
constexpr uint32_t kFpStage = kFpBuf + 2 * kTileBytes;                      // phases, ops, runs' entries (stage_pass)
constexpr uint32_t kFpOps = kFpStage + (uint32_t)kStagePhaseBytes;
constexpr uint32_t kFpRuns = kFpOps + (uint32_t)sizeof(TOp) * kStageOps;
constexpr uint32_t kFpTile = kFpRuns + (uint32_t)sizeof(DRun) * kStageRuns;  // the runs' tile products, for two tiles
constexpr uint32_t kFpTab = kFpTile + 2 * sizeof(float4) * kTileRuns;  // the runs' tables
constexpr uint32_t kFpDiag = kFpTab + sizeof(float4) * kTileRuns * kRunTab;
constexpr uint32_t kFpCtx = kFpDiag + sizeof(float2) * 16 * kTileTabs;
constexpr uint32_t kFpBytes = kFpCtx + sizeof(RunCtx);
static_assert(kFpBytes <= kMaxSmem && kFpRuns % 16 == 0 && kFpTile % 16 == 0, "a pass's shared memory");

// run_tile_fwd of a pass whose records and tables all lie in shared memory
__device__ __noinline__ void run_tile_staged(uint32_t sm, int nphase, uint32_t tile, int m, uint32_t tbase) {
  for (int f = 0; f < nphase; ++f) {
    const RunCtx rc{sh<DRun>(kFpRuns), sh<float4>(kFpTab), sh<float4>(tile)};
    phase_fwd_body<kRB, false, false>(sh<float2>(sm), sh<TPhase>(kFpStage) + f, sh<TOp>(kFpOps), sh<float2>(kFpDiag),
                                      nullptr, nullptr, rc, sh<uint32_t>(0), m, tbase);
  }
}

// products of the tile-id entries of the pass's runs for the tile at tb: 16 lanes a run
__device__ __forceinline__ void tile_products(float4* out, const DRun* entries, const int2* runs, int nrun, uint32_t tb) {
  for (int r0 = 0; r0 < nrun; r0 += kTileThreads / 16) {
    const int r = r0 + (int)threadIdx.x / 16;
    float2 p0 = make_float2(1.f, 0.f), p1 = p0;
    if (r < nrun) {
      const int2 e = runs[r];
      for (int k = threadIdx.x & 15; k < e.y; k += 16) run_entry(entries + e.x + k, tb, p0, p1);
    }
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) {
      p0 = cmulf(p0, make_float2(__shfl_xor_sync(0xffffffffu, p0.x, o), __shfl_xor_sync(0xffffffffu, p0.y, o)));
      p1 = cmulf(p1, make_float2(__shfl_xor_sync(0xffffffffu, p1.x, o), __shfl_xor_sync(0xffffffffu, p1.y, o)));
    }
    if (r < nrun && (threadIdx.x & 15) == 0) out[r] = make_float4(p0.x, p0.y, p1.x, p1.y);
  }
}

// One pass over every register of a uniform batch: CTA-strided over tiles,
// each tile staged in shared memory once and run through all phases of the pass.
//
// Two tile buffers: the next tile's amplitudes are copied into one with
// cp.async (8-byte copies into the swizzled slots) while the phases run on the
// other, so the pass does not wait on the state's DRAM latency once per tile.
__global__ void __launch_bounds__(kTileThreads, 1) k_fused_pass(FArgs a) {
  const TPass& p = *a.pass;
  set_rows(sh<uint32_t>(0), p, a.m);
  const StagedPass sp = stage_pass<true>(p, a.phases, a.fops, sh<unsigned char>(kFpStage), sh<DRun>(kFpRuns), kStageRuns,
                                       a.druns, nullptr);
  // the runs' tables, and their tile products for this tile and the one before
  const bool held = p.nrun <= kTileRuns;
  const bool staged = held && p.ndt <= kTileTabs && sp.ph != a.phases + p.phase0;
  float4* rtab = sh<float4>(kFpTab);
  RunCtx* rc = sh<RunCtx>(kFpCtx);
  if (held)
    for (int i = threadIdx.x; i < p.nrun * kRunTab; i += blockDim.x) rtab[i] = a.rtab[kRunTab * p.run0 + i];
  if (staged) {
    const int count = sp.ph[p.nphase - 1].fop0 + sp.ph[p.nphase - 1].nfop;
    for (int i = threadIdx.x; i < 16 * p.ndt; i += blockDim.x) sh<float2>(kFpDiag)[i] = a.dtab[16 * p.dt0 + i];
    TOp* ops = sh<TOp>(kFpOps);
    for (int i = threadIdx.x; i < count; i += blockDim.x) {
      if (ops[i].kind == TK_DIAG16) ops[i].param -= p.dt0;
      if (ops[i].kind == TK_REALRUN && ops[i].pad) ops[i].pad -= (uint32_t)p.dt0;
    }
  }
  const uint64_t total = a.ntile * (uint64_t)a.nreg;
  // a tile's offset in its register: each lane places one bit of the tile's number
  const int lane = threadIdx.x & 31, gbit = lane < a.g ? p.gbits[lane] : 0;
  auto tile_src = [&](uint64_t t, uint32_t& tb) {
    const uint32_t tl = (uint32_t)(t & (a.ntile - 1));
    tb = __reduce_or_sync(0xffffffffu, lane < a.g ? ((tl >> lane) & 1u) << gbit : 0u);
    return a.state + (t >> a.g) * a.reg_stride + tb;
  };
  const int nphase = p.nphase;
  uint32_t tb = 0;
  if (blockIdx.x < total) load_tile_async(kFpBuf, tile_src(blockIdx.x, tb), 0, a.m);
  cp_async_commit();
  int i = 0;
  for (uint64_t t = blockIdx.x; t < total; t += gridDim.x, ++i) {
    const uint32_t sx = kFpBuf + (i & 1) * kTileBytes;
    const uint64_t tn = t + gridDim.x;
    if (tn < total) {
      uint32_t tbn;
      load_tile_async(kFpBuf + ((i + 1) & 1) * kTileBytes, tile_src(tn, tbn), 0, a.m);
    }
    cp_async_commit();
    float2* base = tile_src(t, tb);
    const uint32_t ot = kFpTile + (i & 1) * (uint32_t)sizeof(float4) * kTileRuns;
    float4* rt = held ? sh<float4>(ot) : nullptr;
    if (held) tile_products(rt, sp.runs, a.runs + p.run0, p.nrun, tb);
    if (threadIdx.x == 0 && !staged) *rc = RunCtx{sp.runs, held ? rtab : a.rtab + kRunTab * p.run0, rt};
    cp_async_wait_prev();  // this tile's copies (all groups but the one just issued)
    __syncthreads();
    if (staged) run_tile_staged(sx, nphase, ot, a.m, tb);
    else run_tile_fwd<kRB, false, 2>(sx, sp.ph, nphase, sp.ops, a.dtab, nullptr, nullptr, kFpCtx, 0, a.m, tb);
    store_tile(sx, base, 0, a.m);
    __syncthreads();
  }
  cp_async_wait_all();
}


// One backward pass over a single large register (complex64 psi and lambda
// work copies): CTA-strided over tiles; every CTA accumulates the pass's
// gradient contributions in its own FP64 shared-memory slots and writes them
// to partials[blockIdx.x][param]; k_fold_partials sums the CTAs in order.
struct FBArgs {
  float2* wpsi;
  float2* wlam;
  const TPass* pass;
  const TPhase* phases;
  const TOp* bops;
  const GMem* gmem;
  int vals;              // gradient sums of a phase, at most
  int m, g, nparam;
  int stage;             // GMem records that stage_pass's area after the tiles has room for (-1: no area)
  uint64_t ntile;
  double* partials;      // [gridDim.x][nparam]
};

__global__ void __launch_bounds__(kTileThreads, 1) k_fused_bwd_pass(FBArgs a) {
  extern __shared__ __align__(16) unsigned char smraw[];
  uint32_t* rowoff = reinterpret_cast<uint32_t*>(smraw);
  float* red = reinterpret_cast<float*>(rowoff + (1 << (kMaxTileBits - kRowBits)));
  double* gacc = reinterpret_cast<double*>(red + a.vals * kWarps);
  float2* sx = reinterpret_cast<float2*>(gacc + ((a.nparam + 1) & ~1));
  float2* sl = sx + (1 << a.m);
  unsigned char* stage = a.stage >= 0 ? reinterpret_cast<unsigned char*>(sl + (1 << a.m)) : nullptr;
  const TPass& p = *a.pass;
  for (int i = threadIdx.x; i < a.nparam; i += blockDim.x) gacc[i] = 0.0;
  set_rows(rowoff, p, a.m);
  const StagedPass sp = stage_pass<false>(p, a.phases, a.bops, stage, stage ? stage + kStageBytes : nullptr, a.stage,
                                        nullptr, a.gmem);
  auto at = [&](const void* q) { return (uint32_t)((const unsigned char*)q - smraw); };
  for (uint64_t t = blockIdx.x; t < a.ntile; t += gridDim.x) {
    const uint64_t tb = tile_base(t, p, a.g);
    load_tiles<true>(at(sx), a.wpsi + tb, at(sl), a.wlam + tb, 0, a.m);
    __syncthreads();
    run_tile_bwd<kRB>(at(sx), at(sl), sp.ph, p.nphase, sp.ops, sp.mem, a.m, 0, at(red), at(gacc), (uint32_t)tb);
    store_tiles<true>(at(sx), a.wpsi + tb, at(sl), a.wlam + tb, 0, a.m);
    __syncthreads();
  }
  for (int i = threadIdx.x; i < a.nparam; i += blockDim.x) a.partials[(size_t)blockIdx.x * a.nparam + i] = gacc[i];
}

__global__ void k_fold_partials(const double* __restrict__ partials, int nblk, int nparam, double* __restrict__ grad) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= nparam) return;
  double v = 0.0;
  for (int b = 0; b < nblk; ++b) v += partials[(size_t)b * nparam + i];
  grad[i] += v;
}

// lambda = O psi for complex64 work copies (FP32 arithmetic, FP64 coefficients)
struct ObsC64 {
  int nt;
  uint64_t x[64];
  uint64_t z[64];
  int ny[64];
  float c[64];
};

__global__ void __launch_bounds__(256) k_apply_obs_c64(const float2* __restrict__ psi, float2* __restrict__ lam,
                                                       uint64_t dim, int accumulate, const __grid_constant__ ObsC64 o) {
  const uint64_t i = (uint64_t)blockIdx.x * 256 + threadIdx.x;
  if (i >= dim) return;
  float2 acc = accumulate ? lam[i] : make_float2(0.f, 0.f);
  for (int t = 0; t < o.nt; ++t) {
    const uint64_t j = i ^ o.x[t];
    const float2 v = psi[j];
    const float s = (__popcll(j & o.z[t]) & 1) ? -o.c[t] : o.c[t];
    float re, im;
    switch (o.ny[t] & 3) {
      case 0: re = v.x; im = v.y; break;
      case 1: re = -v.y; im = v.x; break;
      case 2: re = -v.x; im = -v.y; break;
      default: re = v.y; im = -v.x; break;
    }
    acc.x = fmaf(s, re, acc.x);
    acc.y = fmaf(s, im, acc.y);
  }
  lam[i] = acc;
}

// ------------------------------------------------------------------ device: matrices from parameters

// member of a TK_DIAG16 table: a diagonal gate on the phase bits
struct DMem {
  int32_t g;                 // global GSpec index
  uint8_t tb, cm, cv, pad;   // phase-local target bit, control mask and values
};

struct DRef {
  int32_t mem0, count;       // members in dmem[]
};

struct PrepArgs {
  const GSpec* gspec;
  const FMem* fmem;
  const FMem* bmem;
  GMem* gmem;
  float2* flo;             // if not NULL: corrections of the forward matrices (precise path)
  float2* blo;             // backward U^dagger corrections
  float2* dtlo;            // diagonal table corrections
  const DMem* dmem;
  const DRef* dref;
  TOp* fops;
  TOp* bops;
  float2* dtab;
  DRun* druns;
  const DRun* tabent;      // lane and warp entries of the runs: masks over table index bits
  const int4* tabs;        // per run: first of them, lane entries, warp entries
  float4* rtab;
  const double* params;
  int nfop, nbop, ndiag, ndrun, nrun;
};

__device__ void gate_mat(const GSpec& gs, const double* params, double2 (&U)[4]) {
  const double th = gs.param >= 0 ? params[gs.param] : gs.theta;
  double s, c;
  sincos(th * 0.5, &s, &c);
  const double h = 0.70710678118654752440;
  auto set = [&](double a0, double a1, double b0, double b1, double c0, double c1, double d0, double d1) {
    U[0] = make_double2(a0, a1); U[1] = make_double2(b0, b1); U[2] = make_double2(c0, c1); U[3] = make_double2(d0, d1);
  };
  switch (gs.kind) {
    case QS_GATE_X: set(0, 0, 1, 0, 1, 0, 0, 0); break;
    case QS_GATE_Y: set(0, 0, 0, -1, 0, 1, 0, 0); break;
    case QS_GATE_Z: set(1, 0, 0, 0, 0, 0, -1, 0); break;
    case QS_GATE_H: set(h, 0, h, 0, h, 0, -h, 0); break;
    case QS_GATE_S: set(1, 0, 0, 0, 0, 0, 0, 1); break;
    case QS_GATE_SDG: set(1, 0, 0, 0, 0, 0, 0, -1); break;
    case QS_GATE_T: set(1, 0, 0, 0, 0, 0, h, h); break;
    case QS_GATE_TDG: set(1, 0, 0, 0, 0, 0, h, -h); break;
    case QS_GATE_RX: set(c, 0, 0, -s, 0, -s, c, 0); break;
    case QS_GATE_RY: set(c, 0, -s, 0, s, 0, c, 0); break;
    case QS_GATE_RZ: set(c, -s, 0, 0, 0, 0, c, s); break;
    case QS_GATE_SHIFT: { double s2, c2; sincos(th, &s2, &c2); set(1, 0, 0, 0, 0, 0, c2, s2); break; }
    case QS_GATE_PHASE: { double s2, c2; sincos(th, &s2, &c2); set(c2, s2, 0, 0, 0, 0, c2, s2); break; }
    case QS_GATE_MATRIX: U[0] = gs.mat[0]; U[1] = gs.mat[1]; U[2] = gs.mat[2]; U[3] = gs.mat[3]; break;
    default: set(1, 0, 0, 0, 0, 0, 1, 0); break;
  }
}

__device__ __forceinline__ double2 zmul(double2 a, double2 b) {
  return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ double2 zadd(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }

// FP32 value of v and its correction v - hi (both components)
__device__ __forceinline__ float2 hi_of(double2 v) { return make_float2((float)v.x, (float)v.y); }
__device__ __forceinline__ float2 lo_of(double2 v) {
  const float2 h = hi_of(v);
  return make_float2((float)(v.x - (double)h.x), (float)(v.y - (double)h.y));
}

__global__ void k_batch_prep(PrepArgs a) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < a.nfop) {
    const FMem& fm = a.fmem[i];
    double2 A[4] = {make_double2(1, 0), make_double2(0, 0), make_double2(0, 0), make_double2(1, 0)};
    for (int k = 0; k < fm.count; ++k) {
      double2 U[4];
      gate_mat(a.gspec[fm.g[k]], a.params, U);
      const double2 C0 = zadd(zmul(U[0], A[0]), zmul(U[1], A[2]));
      const double2 C1 = zadd(zmul(U[0], A[1]), zmul(U[1], A[3]));
      const double2 C2 = zadd(zmul(U[2], A[0]), zmul(U[3], A[2]));
      const double2 C3 = zadd(zmul(U[2], A[1]), zmul(U[3], A[3]));
      A[0] = C0; A[1] = C1; A[2] = C2; A[3] = C3;
    }
    for (int k = 0; k < 4; ++k) a.fops[i].u[k] = hi_of(A[k]);
    if (a.flo)
      for (int k = 0; k < 4; ++k) a.flo[4 * i + k] = lo_of(A[k]);
  } else if (i < a.nfop + a.nbop) {
    const int j = i - a.nfop;
    const FMem& bm = a.bmem[j];
    double2 U[4];
    gate_mat(a.gspec[bm.g[bm.count - 1]], a.params, U);
    if (bm.count > 1) {
      // walk the run from its end: E is the product of the members passed, and a
      // member's generator H becomes E H E^dagger at the end of the run
      double2 E[4] = {make_double2(1, 0), make_double2(0, 0), make_double2(0, 0), make_double2(1, 0)};
      int rec = bm.rec0;
      for (int k = bm.count - 1; k >= 0; --k) {
        const GSpec& gs = a.gspec[bm.g[k]];
        if (bm.rec0 >= 0 && gs.param >= 0) {
          // E H E^dagger for H = [[h0, h1], [conj(h1), h3]]
          double f = 1.0, h0 = 0.0, h3 = 0.0;
          double2 h1 = make_double2(0, 0);
          switch (gs.kind) {
            case QS_GATE_RX: h1.x = 1.0; break;
            case QS_GATE_RY: h1.y = -1.0; break;
            case QS_GATE_RZ: h0 = 1.0; h3 = -1.0; break;
            case QS_GATE_SHIFT: f = -2.0; h3 = 1.0; break;
            default: f = -2.0; h0 = h3 = 1.0; break;  // PHASE
          }
          auto row = [&](double2 p, double2 q, double2& r0, double2& r1) {  // (p, q) H
            r0 = zadd(make_double2(p.x * h0, p.y * h0), zmul(q, make_double2(h1.x, -h1.y)));
            r1 = zadd(zmul(p, h1), make_double2(q.x * h3, q.y * h3));
          };
          auto dot = [&](double2 p, double2 q, double2 u, double2 v) {  // p conj(u) + q conj(v)
            return zadd(zmul(p, make_double2(u.x, -u.y)), zmul(q, make_double2(v.x, -v.y)));
          };
          double2 p0, p1, q0, q1;
          row(E[0], E[1], p0, p1);
          row(E[2], E[3], q0, q1);
          const double2 m00 = dot(p0, p1, E[0], E[1]), m01 = dot(p0, p1, E[2], E[3]), m11 = dot(q0, q1, E[2], E[3]);
          GMem& m = a.gmem[rec++];
          m.c[0] = (float)(f * m00.x);
          m.c[1] = (float)(f * m11.x);
          m.c[2] = (float)(f * m01.x);
          m.c[3] = (float)(-f * m01.y);
        }
        gate_mat(gs, a.params, U);
        const double2 C0 = zadd(zmul(E[0], U[0]), zmul(E[1], U[2])), C1 = zadd(zmul(E[0], U[1]), zmul(E[1], U[3]));
        const double2 C2 = zadd(zmul(E[2], U[0]), zmul(E[3], U[2])), C3 = zadd(zmul(E[2], U[1]), zmul(E[3], U[3]));
        E[0] = C0; E[1] = C1; E[2] = C2; E[3] = C3;
      }
      for (int k = 0; k < 4; ++k) U[k] = E[k];
    }
    // U^dagger
    const double2 D[4] = {make_double2(U[0].x, -U[0].y), make_double2(U[2].x, -U[2].y),
                          make_double2(U[1].x, -U[1].y), make_double2(U[3].x, -U[3].y)};
    for (int k = 0; k < 4; ++k) a.bops[j].u[k] = hi_of(D[k]);
    if (a.blo)
      for (int k = 0; k < 4; ++k) a.blo[4 * j + k] = lo_of(D[k]);
  } else if (i < a.nfop + a.nbop + a.ndiag) {
    // product of the member gates' diagonals on the 16 phase amplitudes
    const int d = i - a.nfop - a.nbop;
    double2 f[16];
    for (int j = 0; j < 16; ++j) f[j] = make_double2(1.0, 0.0);
    const DRef r = a.dref[d];
    for (int k = 0; k < r.count; ++k) {
      const DMem mb = a.dmem[r.mem0 + k];
      double2 U[4];
      gate_mat(a.gspec[mb.g], a.params, U);
      for (int j = 0; j < 16; ++j)
        if ((j & mb.cm) == mb.cv) f[j] = zmul(f[j], ((j >> mb.tb) & 1) ? U[3] : U[0]);
    }
    for (int j = 0; j < 16; ++j) a.dtab[16 * d + j] = hi_of(f[j]);
    if (a.dtlo)
      for (int j = 0; j < 16; ++j) a.dtlo[16 * d + j] = lo_of(f[j]);
  } else if (i < a.nfop + a.nbop + a.ndiag + a.ndrun) {
    DRun& e = a.druns[i - a.nfop - a.nbop - a.ndiag];
    double2 U[4];
    gate_mat(a.gspec[e.gate], a.params, U);
    e.u0 = hi_of(U[0]);
    e.u3 = hi_of(U[3]);
  } else if (i < a.nfop + a.nbop + a.ndiag + a.ndrun + a.nrun * kRunTab) {
    // an entry of a run's table: the products over the members whose controls hold at
    // this lane (or warp), formed in FP64 and rounded once
    const int k = i - a.nfop - a.nbop - a.ndiag - a.ndrun, run = k / kRunTab, at = k % kRunTab;
    const int4 t = a.tabs[run];
    const uint32_t bits = at < 32 ? at : at - 32;
    const int e0 = at < 32 ? t.x : t.x + t.y, n = at < 32 ? t.y : t.z;
    double2 p0 = make_double2(1.0, 0.0), p1 = p0;
    for (int q = 0; q < n; ++q) {
      const DRun& e = a.tabent[e0 + q];
      if ((bits & e.tmask) != e.tval) continue;
      double2 U[4];
      gate_mat(a.gspec[e.gate], a.params, U);
      const bool scalar = e.tq != 0xffffffffu, one = scalar && ((bits >> e.tq) & 1u);
      p0 = zmul(p0, one ? U[3] : U[0]);
      p1 = zmul(p1, scalar && !one ? U[0] : U[3]);
    }
    const float2 h0 = hi_of(p0), h1 = hi_of(p1);
    a.rtab[k] = make_float4(h0.x, h0.y, h1.x, h1.y);
  }
}

}  // namespace qs

// ------------------------------------------------------------------ host: the program object

struct qs_batch_program {
  int device = -1;                   // CUDA device that holds the tables below
  int nreg = 0;
  std::vector<int> nq;
  std::vector<int64_t> param_off;    // nreg + 1
  std::vector<int64_t> amp_off;      // nreg + 1
  int64_t work_elems = 0;
  // device tables (one allocation)
  void* tables = nullptr;
  qs::BReg* regs = nullptr;
  int32_t* order = nullptr;
  qs::TPass* passes = nullptr;
  qs::TPhase* phases = nullptr;
  qs::TOp* fops = nullptr;
  qs::TOp* bops = nullptr;
  qs::BTerm* terms = nullptr;
  qs::GSpec* gspec = nullptr;
  qs::FMem* fmem = nullptr;
  qs::FMem* bmem = nullptr;
  qs::GMem* gmem = nullptr;
  qs::DMem* dmem = nullptr;
  qs::DRef* dref = nullptr;
  float2* dtab = nullptr;
  int ndiag = 0;
  qs::DRun* druns = nullptr;  // TK_DIAGRUN entries
  int ndrun = 0;
  qs::DRun* tabent = nullptr;  // those formed into tables
  int4* tabs = nullptr;
  int2* runs = nullptr;
  float4* rtab = nullptr;
  int nrun = 0;
  int* counter = nullptr;
  float2* wpsi = nullptr;
  float2* wlam = nullptr;
  // phase width and the precise path (compensated forward, double-float uncompute)
  int rb = qs::kRB;
  int tile = 0;
  bool precise = false;
  bool forward_only = false;  // no tables and buffers for a backward pass
  float2* flo = nullptr;   // corrections of the forward ops (4 per op)
  float2* blo = nullptr;   // corrections of the backward ops (4 per op)
  float2* dtlo = nullptr;  // corrections of the diagonal tables (16 per table)
  float4* wpsif = nullptr;
  float4* wlamf = nullptr;
  int nfop = 0, nbop = 0;
  int64_t npass = 0, nphase = 0;
  int blocks = 0;
  size_t smem = 0;
  // single-register fused forward (no observable, no backward): host copies of
  // the pass table and a device parameter buffer
  bool fused_only = false;
  std::vector<qs::TPass> host_passes;
  double* dparams = nullptr;
  int64_t dparams_n = 0;
  // SWAP networks before and after the passes (k_bitswap), the phases' share of npass
  std::vector<std::pair<int, int>> pre_swaps, post_swaps;
};

namespace qs {

static int gen_of(int kind, float* cfac2) {
  switch (kind) {
    case QS_GATE_RX: *cfac2 = 1.f; return GEN_X;
    case QS_GATE_RY: *cfac2 = 1.f; return GEN_Y;
    case QS_GATE_RZ: *cfac2 = 1.f; return GEN_Z;
    case QS_GATE_SHIFT: *cfac2 = -2.f; return GEN_P1;
    case QS_GATE_PHASE: *cfac2 = -2.f; return GEN_I;
  }
  *cfac2 = 0.f;
  return GEN_NONE;
}

// The program's tables in one device allocation (an allocation and a free a table were a
// third of the time a program of 240 registers took to make)
struct TableSet {
  struct Item {
    void** dst;
    const void* src;  // NULL: written on the device
    size_t bytes, at;
  };
  std::vector<Item> items;
  size_t total = 0;
  template <typename T>
  void add(T** dst, const std::vector<T>& v) { put((void**)dst, v.empty() ? nullptr : v.data(), sizeof(T) * v.size()); }
  template <typename T>
  void room(T** dst, size_t count) { put((void**)dst, nullptr, sizeof(T) * count); }
  void put(void** dst, const void* src, size_t bytes) {
    items.push_back(Item{dst, src, bytes, total});
    total += (std::max<size_t>(bytes, 1) + 255) / 256 * 256;
  }
  int upload(void** base) {
    if (cudaMalloc(base, total) != cudaSuccess) {
      cudaGetLastError();
      *base = nullptr;
      return fail(QS_ENOMEM, "cudaMalloc of %zu program bytes failed", total);
    }
    for (const Item& i : items) {
      *i.dst = (char*)*base + i.at;
      if (i.src) QS_CUDA(cudaMemcpy(*i.dst, i.src, i.bytes, cudaMemcpyHostToDevice));
    }
    return QS_OK;
  }
};

static void free_program(qs_batch_program* p) {
  if (!p) return;
  // the tables live on the device that built them, which need not be the current one
  int cur = -1;
  const bool swap = p->device >= 0 && cudaGetDevice(&cur) == cudaSuccess && cur != p->device &&
                    cudaSetDevice(p->device) == cudaSuccess;
  void* ptrs[] = {p->tables, p->wpsi, p->wlam, p->dparams, p->flo, p->blo, p->dtlo, p->wpsif, p->wlamf};
  for (void* q : ptrs)
    if (q) cudaFree(q);
  if (swap) cudaSetDevice(cur);
  delete p;
}

// largest tile of the batched kernel for rb-bit phases: 512 threads x 2^rb amplitudes
static int max_tile(int rb) { return std::min(kBatchTile, 9 + rb); }

// TOp::var of a backward op (bwd_form): 13 t + form
static uint8_t bwd_variant(const TOp& b) {
  if (b.kind == TK_DIAGOUT) return 0xff;
  if (b.kind == TK_RUN) return b.var;  // set where the op is built
  int f;
  if (b.gen == GEN_NONE) f = b.kind == TK_SWAP ? 0 : b.kind == TK_DIAG ? 1 : 2;
  else f = 3 + 2 * (b.gen - GEN_X) + (b.cmask ? 1 : 0);
  return (uint8_t)(13 * b.t + f);
}

// TOp::var of a forward op (FV_* forms)
static uint8_t fwd_variant(const TOp& f) {
  switch (f.kind) {
    case TK_DIAGOUT: return FV_DIAGOUT;
    case TK_DIAG16: return FV_DIAG16;
    case TK_DIAGRUN: return FV_DIAGRUN;
    case TK_DENSEX: return f.var;  // set where the op is built
    case TK_SWAP: return (uint8_t)(FV_SWAP + f.t);
    case TK_DIAG: return (uint8_t)((f.cmask ? FV_DIAGC : FV_DIAG) + f.t);
    default: return (uint8_t)((f.cmask ? FV_DENSEC : FV_DENSE) + f.t);
  }
}

// gates whose product is a real 2x2
static bool real_gates(const std::vector<GSpec>& gspec, const FMem& fm) {
  for (int k = 0; k < fm.count; ++k) {
    const GSpec& gs = gspec[fm.g[k]];
    if (!(gs.kind == QS_GATE_H || gs.kind == QS_GATE_RY || gs.kind == QS_GATE_X || gs.kind == QS_GATE_Z ||
          gs.kind == QS_GATE_I ||
          (gs.kind == QS_GATE_MATRIX && gs.mat[0].y == 0 && gs.mat[1].y == 0 && gs.mat[2].y == 0 && gs.mat[3].y == 0)))
      return false;
  }
  return true;
}

// diagonal gates with the first entry exactly 1: factors on the target's 1 only
static bool unit_first(int kind) {
  return kind == QS_GATE_SHIFT || kind == QS_GATE_Z || kind == QS_GATE_S || kind == QS_GATE_SDG || kind == QS_GATE_T ||
         kind == QS_GATE_TDG || kind == QS_GATE_I;
}

// Gradient sums a phase may have.  The tiled gradient keeps them beside a double per
// parameter in shared memory: circuits that nearly fill it keep to one sum a gate.
static int phase_vals(int nparams) { return nparams > 11000 ? kMaxPhaseOps : kMaxPhaseVals; }

// uncompute kind of a gate on a phase bit: the generator picks the structured form
static uint8_t bwd_kind(int gen, bool diag, bool x) {
  if (gen == GEN_X) return TK_RX;
  if (gen == GEN_Y) return TK_RY;
  if (gen != GEN_NONE) return TK_DIAG;
  return x ? TK_SWAP : diag ? TK_DIAG : TK_DENSE;
}

// a run that TK_RUN takes: two gates or more, not all diagonal, one of them with a parameter
static bool is_run(const qs_circuit* c, const int* gates, int count) {
  bool diag = true, param = false;
  for (int k = 0; k < count; ++k) {
    diag = diag && gate_is_diagonal(c, c->gates[gates[k]]);
    param = param || c->gates[gates[k]].param >= 0;
  }
  return count > 1 && !diag && param;
}

// The backward ops of a phase while they are put together: a run of gates, with the X it
// takes along (gate x, -1: none; xop: as an op of its own), before or after it
struct BGroup {
  TOp op, xop;
  int gates[kMaxRun];
  int count, x;
  bool dead, pre;
};

// sizes of the program's tables (fmem and bmem go with the ops, runs with tabs)
struct Marks {
  size_t passes, phases, fops, bops, gspec, dmems, drefs, druns, tabent, tabs, gmem;
};

static int build_program(int nreg, const qs_circuit* const* circs, const qs_observable* const* obs, int tile_qubits,
                         qs_batch_program* P, int rb = kRB, bool precise = false, bool plain = false) {
  if (rb < kMinRB || rb > kRB) return fail(QS_EINVAL, "phase_qubits must be in %d..%d", kMinRB, kRB);
  if (precise && rb > 3) return fail(QS_EINVAL, "the precise path takes phases of at most 3 qubits");
  const int MT = max_tile(rb);
  const int M = tile_qubits > 0 ? tile_qubits : MT;
  // a tile holds register qubits 0..4 (contiguous rows) plus a phase's register bits
  if (M < kRowBits + rb || M > MT)
    return fail(QS_EINVAL, "tile_qubits must be in %d..%d for %d-qubit phases", kRowBits + rb, MT, rb);
  P->rb = rb;
  P->precise = precise;
  P->tile = M;
  QS_CUDA(cudaGetDevice(&P->device));
  std::vector<BReg> regs(nreg);
  std::vector<TPass> passes;
  std::vector<TPhase> phases;
  std::vector<TOp> fops, bops;
  std::vector<BTerm> terms;
  std::vector<GSpec> gspec;
  std::vector<FMem> fmem;
  std::vector<FMem> bmem;
  std::vector<GMem> gmem;
  std::vector<DMem> dmems;
  std::vector<DRef> drefs;
  std::vector<DRun> druns, tabent;
  std::vector<int4> tabs;
  std::vector<int2> runs;
  P->nreg = nreg;
  P->nq.resize(nreg);
  P->param_off.assign(nreg + 1, 0);
  P->amp_off.assign(nreg + 1, 0);
  int64_t work = 0;
  std::vector<TOp> pf;   // a phase's ops while they are put together: one that moves to a
  std::vector<FMem> pm;  // later place leaves a dead one behind
  std::vector<BGroup> pb;
  // registers of one circuit share its schedule: the tables of the first are copied
  // with their indices moved
  std::unordered_map<const qs_circuit*, int> first;
  std::vector<Marks> marks(nreg + 1);
  auto here = [&] {
    return Marks{passes.size(), phases.size(), fops.size(), bops.size(), gspec.size(), dmems.size(), drefs.size(),
                 druns.size(), tabent.size(), tabs.size(), gmem.size()};
  };
  for (int r = 0; r < nreg; ++r) {
    marks[r] = here();
    const qs_circuit* c = circs[r];
    const qs_observable* o = obs ? obs[r] : nullptr;
    if (!c || (!o && !P->fused_only)) return fail(QS_EINVAL, "register %d: null circuit or observable", r);
    const int n = c->nqubits;
    if (n < kRowBits || n > (P->fused_only ? 32 : 30))
      return fail(QS_EUNSUPPORTED, "register %d: %d qubits outside the tile engine's range", r, n);
    if (!P->fused_only && c->nparams > kMaxRegParams)
      return fail(QS_EUNSUPPORTED, "register %d: more than %d parameters", r, kMaxRegParams);
    P->nq[r] = n;
    P->param_off[r + 1] = P->param_off[r] + c->nparams;
    P->amp_off[r + 1] = P->amp_off[r] + (1ll << n);
    const int m = std::min(n, M);
    const auto seen = first.emplace(c, r);
    const int r0 = seen.second ? -1 : seen.first->second;
    std::vector<HostPass> hp;
    if (r0 < 0) QS_TRY(plan_passes(c, n, m, kMaxPhaseOps, hp, rb, plain));
    BReg& R = regs[r];
    memset(&R, 0, sizeof(R));
    R.n = n;
    R.m = m;
    R.npass = r0 < 0 ? (int)hp.size() : regs[r0].npass;
    R.pass0 = (int)passes.size();
    R.nparam = c->nparams;
    R.amp_off = P->amp_off[r];
    R.param_off = P->param_off[r];
    R.work_off = (n > m && !P->fused_only) ? work : -1;
    if (n > m && !P->fused_only) work += 1ll << n;
    // observable: diagonal Pauli strings only
    R.term0 = (int)terms.size();
    if (o) {
      for (const auto& t : o->terms) {
        if (t.x_mask) return fail(QS_EUNSUPPORTED, "register %d: batched observables must be diagonal (Z strings)", r);
        if (n < 64 && (t.z_mask >> n)) return fail(QS_EINVAL, "register %d: observable qubit out of range", r);
        terms.push_back({t.coeff, t.z_mask});
      }
    }
    R.nterm = o ? (int)o->terms.size() : 0;
    if (r0 >= 0) {
      const Marks &a = marks[r0], &z = marks[r0 + 1], d = marks[r];
      auto moved = [](size_t from, size_t to) { return (int)to - (int)from; };
      const int dg = moved(a.gspec, d.gspec), dm = moved(a.gmem, d.gmem);
      auto copy = [](auto& v, size_t i0, size_t i1, auto fix) {
        for (size_t i = i0; i < i1; ++i) {
          auto e = v[i];
          fix(e);
          v.push_back(e);
        }
      };
      copy(gspec, a.gspec, z.gspec, [&](GSpec& e) { if (e.param >= 0) e.param += (int)(P->param_off[r] - P->param_off[r0]); });
      copy(passes, a.passes, z.passes, [&](TPass& e) {
        e.phase0 += moved(a.phases, d.phases);
        e.drun0 += moved(a.druns, d.druns);
        e.run0 += moved(a.tabs, d.tabs);
        e.mem0 += dm;
        e.dt0 += moved(a.drefs, d.drefs);
      });
      copy(phases, a.phases, z.phases, [&](TPhase& e) {
        e.fop0 += moved(a.fops, d.fops);
        e.bop0 += moved(a.bops, d.bops);
      });
      auto mems = [&](FMem& e) {
        for (int k = 0; k < e.count; ++k) e.g[k] += dg;
        if (e.rec0 >= 0) e.rec0 += dm;
      };
      copy(fops, a.fops, z.fops, [&](TOp& e) { if (e.kind == TK_DIAG16) e.param += moved(a.drefs, d.drefs); });
      copy(fmem, a.fops, z.fops, mems);
      copy(bops, a.bops, z.bops, [&](TOp& e) { if (e.count) e.param += dm; });
      copy(bmem, a.bops, z.bops, mems);
      copy(dmems, a.dmems, z.dmems, [&](DMem& e) { e.g += dg; });
      copy(drefs, a.drefs, z.drefs, [&](DRef& e) { e.mem0 += moved(a.dmems, d.dmems); });
      copy(druns, a.druns, z.druns, [&](DRun& e) { e.gate += dg; });
      copy(tabent, a.tabent, z.tabent, [&](DRun& e) { e.gate += dg; });
      copy(tabs, a.tabs, z.tabs, [&](int4& e) { e.x += moved(a.tabent, d.tabent); });
      copy(runs, a.tabs, z.tabs, [](int2&) {});
      copy(gmem, a.gmem, z.gmem, [](GMem&) {});
      R.cost = regs[r0].cost;
      marks[r + 1] = here();
      continue;
    }
    // gate specs of this register
    const int g0 = (int)gspec.size();
    for (const auto& g : c->gates) {
      GSpec s;
      memset(&s, 0, sizeof(s));
      s.kind = g.kind;
      s.param = g.param >= 0 ? (int)(P->param_off[r] + g.param) : -1;
      s.theta = g.theta;
      if (g.kind == QS_GATE_MATRIX) {
        if (g.nlocs != 1) return fail(QS_EUNSUPPORTED, "register %d: multi-qubit matrices in a batch", r);
        for (int k = 0; k < 4; ++k) s.mat[k] = make_double2(c->mats[g.mat_offset + k].real(), c->mats[g.mat_offset + k].imag());
      }
      if (g.kind == QS_GATE_ROT || g.kind == QS_GATE_SWAP)
        return fail(QS_EUNSUPPORTED, "register %d: ROT / SWAP gates in a batch", r);
      gspec.push_back(s);
    }
    double cost = 0;
    for (const HostPass& p : hp) {
      TPass tp;
      memset(&tp, 0, sizeof(tp));
      for (int k = 0; k < m; ++k) tp.tbits[k] = (uint8_t)p.tbits[k];
      int ng = 0;
      for (int qb = 0; qb < n; ++qb)
        if (std::find(p.tbits.begin(), p.tbits.end(), qb) == p.tbits.end()) tp.gbits[ng++] = (uint8_t)qb;
      tp.phase0 = (int)phases.size();
      tp.drun0 = (int)druns.size();
      tp.run0 = (int)runs.size();
      tp.mem0 = (int)gmem.size();
      tp.dt0 = (int)drefs.size();
      tp.nphase = (int)p.phases.size();
      for (const HostPhase& ph : p.phases) {
        TPhase t;
        phase_positions(p, ph, &t, rb);
        // register qubit -> phase bit index
        auto pbit = [&](int qb) {
          for (int k = 0; k < rb; ++k)
            if (ph.rbits[k] == qb) return k;
          return -1;
        };
        t.bop0 = (int)bops.size();
        t.fop0 = (int)fops.size();
        pf.clear();
        pm.clear();
        pb.clear();
        constexpr uint8_t kDead = 0xff;
        int last[kRB], lastx[kRB], xlast[kRB], blast[kRB];
        for (int k = 0; k < kRB; ++k) {
          last[k] = -1;   // forward op (in pf) open for fusion per phase bit
          lastx[k] = -1;  // forward op (in pf) of the X that was the last gate on a phase bit
          xlast[k] = 0;   // and its form
          blast[k] = -1;  // backward run (in pb) open per phase bit
        }
        // the run on bit tb comes to the place of the X before it (nothing in between has
        // touched the bit)
        auto join_x = [&](int tb, const FMem run) {
          if (last[tb] >= 0) pf[last[tb]].kind = kDead;
          TOp& x = pf[lastx[tb]];
          x.kind = TK_DENSEX;
          x.cmask = x.cval = 0;
          x.var = (uint8_t)(FV_DENSEX + 10 * tb + 5 + xlast[tb]);
          pm[lastx[tb]] = run;
          last[tb] = lastx[tb];
          lastx[tb] = -1;
        };
        int dg = -1;                     // open TK_DIAG16 table of this phase
        int nval = 0;                    // gradient sums of the backward ops
        // TK_DIAGRUN runs of this phase (complex64 path): the op each opened,
        // its entries, the run open per phase bit and the latest run opened
        std::vector<int> run_op;
        std::vector<std::vector<DRun>> run_ent;
        std::vector<int> run_bit;
        std::vector<int> run_open(rb, -1);
        int run_last = -1;
        uint8_t nondiag = 0;             // phase bits touched by non-diagonal gates since it opened
        for (int gi : ph.gates) {
          const qs_gate_desc& g = c->gates[gi];
          const bool diag = gate_is_diagonal(c, g);
          const int tb = pbit(g.locs[0]);  // -1: target outside the phase (diagonal gates only)
          uint8_t cm = 0, cv = 0;          // controls inside the phase
          uint32_t tmask = 0, tval = 0;    // controls outside the phase (register qubits)
          for (int qb = 0; qb < n; ++qb)
            if ((g.ctrl_mask >> qb) & 1ull) {
              const int k = pbit(qb);
              const bool v = (g.ctrl_vals >> qb) & 1ull;
              if (k >= 0) {
                cm |= (uint8_t)(1 << k);
                if (v) cv |= (uint8_t)(1 << k);
              } else {
                tmask |= 1u << qb;
                if (v) tval |= 1u << qb;
              }
            }
          // X with one control in the phase (its value 1) and none outside, or with
          // controls outside only: renames the outputs of the run before it
          const bool renames = !plain && g.kind == QS_GATE_X && tb >= 0 && (cm || tmask) &&
                               (cm == 0 || (tmask == 0 && !(cm & (cm - 1)) && cv == cm));
          const int xform = cm ? 1 + __builtin_ctz(cm) : 0;
          // backward op: uncontrolled gates on one phase bit collect in a run (no gate in
          // between touches the bit); others are ops of their own
          TOp b;
          memset(&b, 0, sizeof(b));
          b.t = (uint8_t)(tb >= 0 ? tb : g.locs[0]);
          b.cmask = cm;
          b.cval = cv;
          b.tmask = tmask;
          b.tval = tval;
          float cf2 = 0.f;
          b.gen = g.param >= 0 ? (uint8_t)gen_of(g.kind, &cf2) : GEN_NONE;
          // uncompute kind: the generator picks the structured form (Rx / Ry / diagonal)
          if (tb < 0) b.kind = TK_DIAGOUT;
          else b.kind = bwd_kind(b.gen, diag, g.kind == QS_GATE_X);
          if (g.param >= 0 && b.gen == GEN_NONE)
            return fail(QS_EUNSUPPORTED, "register %d gate %d: kind %d has no batched gradient", r, gi, g.kind);
          {
            const bool plain = tb >= 0 && !cm && !tmask && g.kind != QS_GATE_X;
            BGroup* run = tb >= 0 && blast[tb] >= 0 ? &pb[blast[tb]] : nullptr;
            auto take = [&](BGroup& u, bool pre) {
              u.op.cmask = cm ? 0 : 1;  // controls outside the phase: tmask / tval
              u.op.cval = 0;
              u.op.tmask = tmask;
              u.op.tval = tval;
              u.op.t = (uint8_t)tb;
              u.op.var = (uint8_t)(BV_RUN + 10 * tb + xform + (pre ? 5 : 0));
              u.x = gi;
              u.xop = b;
              u.pre = pre;
              pb.push_back(u);
            };
            if (plain && run && run->count < kMaxRun) {
              run->gates[run->count++] = gi;  // stays at the run's place: nothing since has touched the bit
            } else if (renames && run && run->x < 0 && is_run(c, run->gates, run->count)) {
              const BGroup u = *run;  // moves here with the X
              run->dead = true;
              BGroup v = u;
              take(v, false);
              blast[tb] = -1;
            } else if (renames) {
              BGroup u{b, b, {0}, 0, -1, false, false};  // the next run on the bit may come to this place
              take(u, true);
              blast[tb] = (int)pb.size() - 1;
            } else {
              pb.push_back(BGroup{b, b, {gi}, 1, -1, false, false});
              if (tb >= 0) blast[tb] = plain ? (int)pb.size() - 1 : -1;
            }
            for (int k = 0; k < rb; ++k)
              if ((cm >> k) & 1) blast[k] = -1;
          }
          // forward op.  A diagonal gate with its target outside the phase is a
          // per-thread factor.  Consecutive uncontrolled gates on one target fuse
          // into one 2x2; controlled diagonal gates inside the phase join its open
          // 16-entry table unless a non-diagonal op since the table opened shares a
          // qubit with them (diagonal gates commute with each other).
          TOp f;
          memset(&f, 0, sizeof(f));
          f.cmask = cm;
          f.cval = cv;
          f.tmask = tmask;
          f.tval = tval;
          f.param = -1;
          FMem fm;
          memset(&fm, 0, sizeof(fm));
          fm.count = 1;
          fm.g[0] = g0 + gi;
          if (tb < 0 && !precise && cm == 0 && run_last >= 0 && run_open[run_bit[run_last]] == run_last) {
            // a scalar for each thread: commutes with every op of the phase
            DRun e;
            memset(&e, 0, sizeof(e));
            e.tmask = tmask;
            e.tval = tval;
            e.gate = g0 + gi;
            e.tq = (uint32_t)g.locs[0];
            run_ent[run_last].push_back(e);
            continue;
          }
          if (tb < 0) {
            f.kind = TK_DIAGOUT;
            f.t = (uint8_t)g.locs[0];
            pf.push_back(f);
            pm.push_back(fm);
            for (int k = 0; k < rb; ++k)
              if ((cm >> k) & 1) last[k] = lastx[k] = -1;
            continue;
          }
          const bool fusable = cm == 0 && tmask == 0 && g.kind != QS_GATE_X;
          int xat = -1;  // this gate's op if it is an X that a run may come to
          const uint8_t gbits = (uint8_t)(cm | (1u << tb));
          if (!diag) nondiag |= gbits;
          if (!diag) run_open[tb] = -1;  // a run moves no later gate past this one
          if (fusable && last[tb] >= 0 && pm[last[tb]].count < kMaxRun) {
            FMem& fmo = pm[last[tb]];
            fmo.g[fmo.count++] = g0 + gi;
            if (!diag && pf[last[tb]].kind == TK_DIAG) {
              pf[last[tb]].kind = TK_DENSE;
              if (lastx[tb] >= 0) join_x(tb, pm[last[tb]]);
            }
          } else if (fusable && !diag && lastx[tb] >= 0 && last[tb] < 0) {
            join_x(tb, fm);
          } else if (renames && last[tb] >= 0 && pf[last[tb]].kind == TK_DENSE) {
            // the dense op moves here (nothing since has touched its bit) and takes the X along
            TOp x = pf[last[tb]];
            x.kind = TK_DENSEX;
            x.tmask = tmask;
            x.tval = tval;
            x.var = (uint8_t)(FV_DENSEX + 10 * tb + xform);
            pf[last[tb]].kind = kDead;
            pf.push_back(x);
            pm.push_back(FMem(pm[last[tb]]));
          } else if (!precise && diag && cm == 0 && tmask != 0) {
            // joins (or opens) the run on its target: diagonal gates commute, and
            // no non-diagonal op on this bit was emitted since the run opened
            if (run_open[tb] < 0) {
              f.kind = TK_DIAGRUN;
              f.t = (uint8_t)tb;
              f.tmask = f.tval = 0;
              fm.count = 0;
              run_open[tb] = (int)run_op.size();
              run_last = run_open[tb];
              run_op.push_back((int)pf.size());
              run_ent.emplace_back();
              run_bit.push_back(tb);
              pf.push_back(f);
              pm.push_back(fm);
            }
            DRun e;
            memset(&e, 0, sizeof(e));
            e.tmask = tmask;
            e.tval = tval;
            e.gate = g0 + gi;
            e.tq = 0xffffffffu;
            run_ent[run_open[tb]].push_back(e);
          } else if (diag && cm != 0 && tmask == 0) {
            if (dg < 0 || (gbits & nondiag)) {
              f.kind = TK_DIAG16;
              f.cmask = f.cval = 0;
              f.param = (int)drefs.size();
              fm.count = 0;
              pf.push_back(f);
              pm.push_back(fm);
              drefs.push_back({(int32_t)dmems.size(), 0});
              dg = (int)drefs.size() - 1;
              nondiag = 0;
            }
            DMem mb;
            memset(&mb, 0, sizeof(mb));
            mb.g = g0 + gi;
            mb.tb = (uint8_t)tb;
            mb.cm = cm;
            mb.cv = cv;
            dmems.push_back(mb);
            drefs[dg].count++;
          } else {
            f.kind = g.kind == QS_GATE_X ? TK_SWAP : diag ? TK_DIAG : TK_DENSE;
            f.t = (uint8_t)tb;
            pf.push_back(f);
            pm.push_back(fm);
            if (last[tb] >= 0) lastx[tb] = -1;  // a full run lies between
            last[tb] = fusable ? (int)pf.size() - 1 : -1;
            if (renames) {
              xat = (int)pf.size() - 1;
              xlast[tb] = xform;
            }
          }
          // a controlled gate closes fusion on its target and its phase-local controls
          if (cm || tmask) {
            for (int k = 0; k < rb; ++k)
              if ((cm >> k) & 1) last[k] = lastx[k] = -1;
            last[tb] = -1;
          }
          if (xat >= 0) lastx[tb] = xat;
          else if (!fusable) lastx[tb] = -1;
        }
        for (size_t r = 0; r < run_op.size(); ++r) {
          TOp& ro = pf[run_op[r]];
          if (run_ent[r].size() == 1) {
            // a run of one gate stays that gate's own op (its outside controls as tmask)
            const DRun& e = run_ent[r][0];
            ro.kind = TK_DIAG;
            ro.tmask = e.tmask;
            ro.tval = e.tval;
            ro.param = -1;
            pm[run_op[r]].count = 1;
            pm[run_op[r]].g[0] = e.gate;
            continue;
          }
          // entries by where their qubits lie: lane bits, warp bits, tile-id bits, several
          const int ntb = m - rb;
          uint32_t lanes = 0, warps = 0, tile = 0;
          for (int k = 0; k < ntb; ++k) (k < 5 ? lanes : warps) |= 1u << t.tq[k];
          for (int k = 0; k < ng; ++k) tile |= 1u << tp.gbits[k];
          auto local = [&](uint32_t q, int k0) {  // register qubits as table index bits
            uint32_t v = 0;
            for (int k = k0; k < std::min(ntb, k0 == 0 ? 5 : ntb); ++k) v |= ((q >> t.tq[k]) & 1u) << (k - k0);
            return v;
          };
          std::vector<DRun> part[4];
          for (const DRun& e : run_ent[r]) {
            const uint32_t q = e.tmask | (e.tq != 0xffffffffu ? 1u << e.tq : 0u);
            const int kind = !(q & ~lanes) ? 0 : !(q & ~warps) ? 1 : !(q & ~tile) ? 2 : 3;
            DRun f = e;
            if (kind < 2) {
              const int k0 = kind == 0 ? 0 : 5;
              f.tmask = local(e.tmask, k0);
              f.tval = local(e.tval, k0);
              if (e.tq != 0xffffffffu) f.tq = (uint32_t)__builtin_ctz(local(1u << e.tq, k0));
            }
            part[kind == 2 && part[2].size() >= 255 ? 3 : kind].push_back(f);
          }
          bool one0 = true;
          for (const DRun& e : run_ent[r]) one0 = one0 && e.tq == 0xffffffffu && unit_first(gspec[e.gate].kind);
          const int run = (int)runs.size() - tp.run0;
          ro.param = (int)druns.size() - tp.drun0;
          ro.count = (uint32_t)(part[2].size() + part[3].size());
          ro.shared = (uint8_t)part[2].size();
          ro.gen = one0 ? 1 : 0;
          std::memcpy(&ro.cfac2, &run, sizeof(run));
          runs.push_back(make_int2(ro.param, (int)part[2].size()));
          tabs.push_back(make_int4((int)tabent.size(), (int)part[0].size(), (int)part[1].size(), 0));
          for (int k = 0; k < 2; ++k) tabent.insert(tabent.end(), part[k].begin(), part[k].end());
          for (int k = 2; k < 4; ++k) druns.insert(druns.end(), part[k].begin(), part[k].end());
        }
        // tile engine: a real 2x2, a run on its bit and a table of gates on its bit, next to
        // each other, become one op when both multiply only where the bit is 1
        if (P->fused_only && rb == kRB) {
          int at = -1, tbl = -1, run = -1;  // the 2x2 and what follows it so far
          auto close = [&] {
            if (at >= 0 && run >= 0) {
              TOp& h = pf[at];
              const TOp& r = pf[run];
              h.kind = TK_REALRUN;
              h.param = r.param;
              h.count = r.count;
              h.shared = r.shared;
              h.cfac2 = r.cfac2;
              h.pad = tbl >= 0 ? pf[tbl].param + 1 : 0;
              pf[run].kind = kDead;
              if (tbl >= 0) pf[tbl].kind = kDead;
            }
            at = tbl = run = -1;
          };
          for (int k = 0; k < (int)pf.size(); ++k) {
            const TOp& o = pf[k];
            if (o.kind == kDead) continue;
            if (at >= 0 && run < 0 && o.kind == TK_DIAGRUN && o.t == pf[at].t && o.gen == 1) {
              run = k;
              continue;
            }
            if (at >= 0 && tbl < 0 && o.kind == TK_DIAG16) {
              const DRef d = drefs[o.param];
              const int bit = 1 << pf[at].t;
              bool on1 = true;
              for (int q = d.mem0; q < d.mem0 + d.count; ++q)
                on1 = on1 && ((dmems[q].cm & dmems[q].cv & bit) || (dmems[q].tb == pf[at].t && unit_first(gspec[dmems[q].g].kind)));
              if (on1) {
                tbl = k;
                continue;
              }
            }
            close();
            if (o.kind == TK_DENSE && !o.cmask && !o.tmask && real_gates(gspec, pm[k])) at = k;
          }
          close();
        }
        for (size_t k = 0; k < pf.size(); ++k) {
          if (pf[k].kind == kDead) continue;
          fops.push_back(pf[k]);
          fmem.push_back(pm[k]);
        }
        // backward ops: a run becomes one op (TK_RUN, or its plain product without
        // parameters), a run of diagonal gates or of one gate its gates' own ops, as does
        // a run whose four sums would leave no room for the gates still to come
        nval = 0;
        int left = 0;
        for (const BGroup& u : pb)
          for (int k = 0; k < u.count; ++k) left += !u.dead && c->gates[u.gates[k]].param >= 0;
        const int rec0 = (int)gmem.size();
        auto record = [&](int gi, float c0) {
          GMem q;
          memset(&q, 0, sizeof(q));
          q.param = c->gates[gi].param;
          q.c[0] = c0;
          for (int k = rec0; k < (int)gmem.size(); ++k)
            if (gmem[k].param == q.param) gmem[k].shared = q.shared = 1;
          gmem.push_back(q);
        };
        for (const BGroup& u : pb) {
          if (u.dead || plain) continue;  // a plain program runs forward only
          FMem fm;
          memset(&fm, 0, sizeof(fm));
          fm.rec0 = -1;
          bool diag = true, param = false;
          for (int k = 0; k < u.count; ++k) {
            const qs_gate_desc& g = c->gates[u.gates[k]];
            diag = diag && gate_is_diagonal(c, g);
            param = param || g.param >= 0;
            left -= g.param >= 0;
          }
          TOp b = u.op;
          const bool fits = !param || nval + 4 + left <= phase_vals(P->fused_only ? c->nparams : 0);
          if (u.count > 1 && !diag && fits && (param || u.x < 0)) {
            for (; fm.count < u.count; ++fm.count) fm.g[fm.count] = g0 + u.gates[fm.count];
            b.gen = GEN_NONE;
            b.kind = param ? TK_RUN : TK_DENSE;
            if (param) {
              if (u.x < 0) b.var = (uint8_t)(BV_RUN + 10 * b.t);
              fm.rec0 = b.param = (int)gmem.size();
              // in the order k_batch_prep meets them: from the run's end
              for (int k = u.count; k-- > 0;)
                if (c->gates[u.gates[k]].param >= 0) record(u.gates[k], 0.f);
              b.count = (uint32_t)((int)gmem.size() - b.param);
              b.val = (uint8_t)nval;
              nval += 4;
            }
            bops.push_back(b);
            bmem.push_back(fm);
            continue;
          }
          auto lone_x = [&] {  // the X the run would have taken along
            fm.count = 1;
            fm.g[0] = g0 + u.x;
            bops.push_back(u.xop);
            bmem.push_back(fm);
          };
          if (u.x >= 0 && u.pre) lone_x();
          for (int k = 0; k < u.count; ++k) {
            const int gi = u.gates[k];
            const qs_gate_desc& g = c->gates[gi];
            TOp o = u.op;
            float cf2 = 0.f;
            if (u.count > 1 || u.x >= 0) {  // a gate of a run: uncontrolled, on the run's bit
              o.cmask = o.cval = o.var = 0;
              o.tmask = o.tval = 0;
              o.gen = g.param >= 0 ? (uint8_t)gen_of(g.kind, &cf2) : GEN_NONE;
              o.kind = bwd_kind(o.gen, gate_is_diagonal(c, g), false);
            }
            if (o.gen != GEN_NONE) {
              gen_of(g.kind, &cf2);
              o.param = (int)gmem.size();
              o.count = 1;
              o.val = (uint8_t)nval++;
              record(gi, cf2);
            }
            fm.count = 1;
            fm.g[0] = g0 + gi;
            bops.push_back(o);
            bmem.push_back(fm);
          }
          if (u.x >= 0 && !u.pre) lone_x();
        }
        t.nbop = (int)bops.size() - t.bop0;
        t.nfop = (int)fops.size() - t.fop0;
        t.nshared = 0;
        for (int q = rec0; q < (int)gmem.size(); ++q) t.nshared += gmem[q].shared ? 1 : 0;
        phases.push_back(t);
        cost += (double)(1ll << n) * (1 + 0.02 * t.nbop);
      }
      tp.ndrun = (int)druns.size() - tp.drun0;
      tp.nrun = (int)runs.size() - tp.run0;
      tp.nmem = (int)gmem.size() - tp.mem0;
      tp.ndt = (int)drefs.size() - tp.dt0;
      passes.push_back(tp);
    }
    R.cost = cost;
    marks[r + 1] = here();
  }
  for (size_t i = 0; i < fops.size(); ++i) {
    TOp& f = fops[i];
    f.var = fwd_variant(f);
    if (!precise && f.kind == TK_DENSE && !f.cmask && real_gates(gspec, fmem[i])) f.var = (uint8_t)(FV_REAL + f.t);
  }
  for (TOp& b : bops) b.var = bwd_variant(b);
  // decreasing cost order
  std::vector<int32_t> order(nreg);
  std::iota(order.begin(), order.end(), 0);
  std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return regs[a].cost > regs[b].cost; });
  P->nfop = (int)fops.size();
  P->nbop = (int)bops.size();
  P->npass = (int64_t)passes.size();
  P->nphase = (int64_t)phases.size();
  P->work_elems = work;
  P->ndiag = (int)drefs.size();
  P->ndrun = (int)druns.size();
  P->nrun = (int)runs.size();
  TableSet tab;
  tab.add(&P->regs, regs);
  tab.add(&P->order, order);
  tab.add(&P->passes, passes);
  tab.add(&P->phases, phases);
  tab.add(&P->fops, fops);
  tab.add(&P->bops, bops);
  tab.add(&P->terms, terms);
  tab.add(&P->gspec, gspec);
  tab.add(&P->fmem, fmem);
  tab.add(&P->bmem, bmem);
  tab.add(&P->gmem, gmem);
  tab.add(&P->dmem, dmems);
  tab.add(&P->dref, drefs);
  tab.add(&P->druns, druns);
  tab.add(&P->tabent, tabent);
  tab.add(&P->tabs, tabs);
  tab.add(&P->runs, runs);
  tab.room(&P->rtab, (size_t)kRunTab * runs.size());
  tab.room(&P->dtab, 16 * drefs.size());
  tab.room(&P->counter, 1);
  QS_TRY(tab.upload(&P->tables));
  P->forward_only = plain;
  if (work > 0 && !precise && !plain) {
    if (cudaMalloc(&P->wpsi, sizeof(float2) * work) != cudaSuccess ||
        cudaMalloc(&P->wlam, sizeof(float2) * work) != cudaSuccess) {
      cudaGetLastError();
      return fail(QS_ENOMEM, "cudaMalloc of the backward work buffers failed");
    }
  }
  if (precise) {
    if ((work > 0 && (cudaMalloc(&P->wpsif, sizeof(float4) * work) != cudaSuccess ||
                      cudaMalloc(&P->wlamf, sizeof(float4) * work) != cudaSuccess)) ||
        cudaMalloc(&P->flo, sizeof(float2) * 4 * std::max<size_t>(1, fops.size())) != cudaSuccess ||
        cudaMalloc(&P->blo, sizeof(float2) * 4 * std::max<size_t>(1, bops.size())) != cudaSuccess ||
        cudaMalloc(&P->dtlo, sizeof(float2) * 16 * std::max<size_t>(1, drefs.size())) != cudaSuccess) {
      cudaGetLastError();
      return fail(QS_ENOMEM, "cudaMalloc of the precise path's buffers failed");
    }
  }
  P->host_passes = passes;
  if (P->fused_only) {
    P->smem = kFpBytes;
    QS_CUDA(cudaFuncSetAttribute(k_fused_pass, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)P->smem));
    int dev = 0, sms = 0, per_sm = 0;
    QS_CUDA(cudaGetDevice(&dev));
    QS_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    QS_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_fused_pass, kTileThreads, P->smem));
    if (per_sm < 1) return fail(QS_EDEVICE, "fused pass kernel does not fit on an SM");
    P->blocks = sms * per_sm;
    return QS_OK;
  }
  P->smem = batch_smem(rb, precise);
  const void* kfn = batch_kernel(rb, precise);
  QS_CUDA(cudaFuncSetAttribute(kfn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)P->smem));
  int dev = 0, sms = 0, per_sm = 0;
  QS_CUDA(cudaGetDevice(&dev));
  QS_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  QS_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kfn, kTileThreads, P->smem));
  if (per_sm < 1) return fail(QS_EDEVICE, "batched kernel does not fit on an SM");
  P->blocks = std::min(nreg, sms * per_sm);
  return QS_OK;
}

// matrices of the forward ops, U^dagger of the backward ops (when `bwd`) and the
// diagonal tables from the current parameters, on the device
static int launch_prep(const qs_batch_program* P, const double* dev_params, bool bwd, cudaStream_t st) {
  PrepArgs pa;
  pa.gspec = P->gspec;
  pa.fmem = P->fmem;
  pa.bmem = P->bmem;
  pa.gmem = P->gmem;
  pa.flo = P->flo;
  pa.blo = P->blo;
  pa.dtlo = P->dtlo;
  pa.dmem = P->dmem;
  pa.dref = P->dref;
  pa.fops = P->fops;
  pa.bops = P->bops;
  pa.dtab = P->dtab;
  pa.druns = P->druns;
  pa.tabent = P->tabent;
  pa.tabs = P->tabs;
  pa.rtab = P->rtab;
  pa.nrun = P->nrun;
  pa.params = dev_params;
  pa.nfop = P->nfop;
  pa.nbop = bwd ? P->nbop : 0;
  pa.ndiag = P->ndiag;
  pa.ndrun = P->ndrun;
  const int tot = pa.nfop + pa.nbop + pa.ndiag + pa.ndrun + pa.nrun * kRunTab;
  if (tot > 0) {
    k_batch_prep<<<(tot + 255) / 256, 256, 0, st>>>(pa);
    QS_LAUNCHED();
  }
  return QS_OK;
}

// ------------------------------------------------------------------ host: fused forward of one circuit

// SWAP(a, b) = CX(a->b) CX(b->a) CX(a->b), each also carrying the SWAP's own controls;
// gates first .. last - 1 of c
static void expand_swaps(const qs_circuit* c, size_t first, size_t last, qs_circuit* out) {
  out->nqubits = c->nqubits;
  out->nparams = c->nparams;
  out->mats = c->mats;
  out->gates.clear();
  for (size_t i = first; i < last; ++i) {
    const qs_gate_desc& g = c->gates[i];
    if (g.kind != QS_GATE_SWAP) {
      out->gates.push_back(g);
      continue;
    }
    const int a = g.locs[0], b = g.locs[1];
    for (int k = 0; k < 3; ++k) {
      qs_gate_desc x;
      memset(&x, 0, sizeof(x));
      x.kind = QS_GATE_X;
      x.nlocs = 1;
      x.param = -1;
      const int t = (k == 1) ? a : b, ctl = (k == 1) ? b : a;
      x.locs[0] = t;
      x.ctrl_mask = g.ctrl_mask | (1ull << ctl);
      x.ctrl_vals = (g.ctrl_vals & g.ctrl_mask) | (1ull << ctl);
      out->gates.push_back(x);
    }
  }
}

// The tile engine's plan of a circuit: SWAP networks (uncontrolled, on disjoint
// qubits) at its start and its end as passes of their own where that takes no more
// passes than their controlled X gates inside the others (a pass that only moves
// amplitudes runs at the copy rate, one that tests controls at half of it), and the
// tile passes of what lies between.
struct TilePlan {
  size_t first = 0, last = 0;  // gates of the tile passes
  std::vector<HostPass> passes;
  qs_circuit mid;              // those gates, SWAPs expanded
};

static int plan_tiles(const qs_circuit* c, int M, TilePlan* out) {
  const int n = c->nqubits, m = std::min(n, M);
  const size_t ng = c->gates.size();
  out->first = 0;
  out->last = ng;
  expand_swaps(c, 0, ng, &out->mid);
  QS_TRY(plan_passes(&out->mid, n, m, kMaxPhaseOps, out->passes));
  if (n < kBitSwapMinQubits) return QS_OK;
  uint64_t used = 0;
  auto network = [&](const qs_gate_desc& g) {
    const uint64_t q = g.kind == QS_GATE_SWAP && !g.ctrl_mask ? (1ull << g.locs[0]) | (1ull << g.locs[1]) : 0;
    if (!q || (q & used)) return false;
    used |= q;
    return true;
  };
  size_t first = 0, last = ng;
  while (last > 0 && network(c->gates[last - 1])) --last;
  used = 0;
  while (first < last && network(c->gates[first])) ++first;
  if (first == 0 && last == ng) return QS_OK;
  TilePlan t;
  t.first = first;
  t.last = last;
  expand_swaps(c, first, last, &t.mid);
  QS_TRY(plan_passes(&t.mid, n, m, kMaxPhaseOps, t.passes));
  if (t.passes.size() + (first > 0) + (last < ng) <= out->passes.size()) *out = t;
  return QS_OK;
}

// the circuit's tile-engine schedule for tiles of M qubits, built once and cached
// on the current device (a schedule built on another device is rebuilt here: its
// tables are that device's memory)
static int ensure_schedule(const qs_circuit* c, int M) {
  int dev = 0;
  QS_CUDA(cudaGetDevice(&dev));
  if (c->fused && c->fused_tile == M && c->fused->device == dev) return QS_OK;
  if (c->fused) {
    free_program(c->fused);
    c->fused = nullptr;
  }
  TilePlan plan;
  QS_TRY(plan_tiles(c, M, &plan));
  const qs_circuit* cp = &plan.mid;
  qs_batch_program* P = new qs_batch_program();
  P->fused_only = true;
  for (size_t i = 0; i < c->gates.size(); ++i)
    if (i < plan.first || i >= plan.last)
      (i < plan.first ? P->pre_swaps : P->post_swaps).emplace_back(c->gates[i].locs[0], c->gates[i].locs[1]);
  const int rc = build_program(1, &cp, nullptr, M, P);
  if (rc != QS_OK) {
    const std::string msg = qs_last_error();
    free_program(P);
    return fail(rc, "%s", msg.c_str());
  }
  c->fused = P;
  c->fused_tile = M;
  return QS_OK;
}

// Applies circuit c to the (uniform, complex64) registers of s with the tile
// engine: one launch of k_fused_pass per pass.  Returns QS_EUNSUPPORTED (with
// nothing launched) when the circuit does not fit the engine.
int fused_forward(qs_state* s, const qs_circuit* c, const double* host_params, int tile_qubits) {
  if (s->dtype != QS_C64 || !s->uniform || s->nq[0] != c->nqubits)
    return fail(QS_EUNSUPPORTED, "the tile engine runs uniform complex64 registers of the circuit's size");
  const int n = s->nq[0];
  const int M = tile_qubits > 0 ? tile_qubits : kBatchTile;
  QS_TRY(ensure_schedule(c, M));
  qs_batch_program* P = c->fused;
  cudaStream_t st = s->stream;
  if (c->nparams > 0) {
    if (P->dparams_n < c->nparams) {
      if (P->dparams) cudaFree(P->dparams);
      P->dparams = nullptr;
      P->dparams_n = 0;
      if (cudaMalloc(&P->dparams, sizeof(double) * c->nparams) != cudaSuccess) {
        cudaGetLastError();
        return fail(QS_ENOMEM, "cudaMalloc of the parameter buffer failed");
      }
      P->dparams_n = c->nparams;
    }
    QS_CUDA(cudaMemcpyAsync(P->dparams, host_params, sizeof(double) * c->nparams, cudaMemcpyHostToDevice, st));
  }
  QS_TRY(launch_prep(P, P->dparams, false, st));
  const int m = std::min(n, M), g = n - m;
  FArgs a;
  a.state = (float2*)s->data;
  a.phases = P->phases;
  a.fops = P->fops;
  a.dtab = P->dtab;
  a.druns = P->druns;
  a.rtab = P->rtab;
  a.runs = P->runs;
  a.m = m;
  a.g = g;
  a.ntile = 1ull << g;
  a.reg_stride = 1ull << n;
  a.nreg = s->nreg;
  const uint64_t tiles = a.ntile * (uint64_t)s->nreg;
  const unsigned grid = (unsigned)std::min<uint64_t>(tiles, (uint64_t)P->blocks);
  if (!P->pre_swaps.empty()) QS_TRY(launch_bitswap(a.state, n, s->nreg, P->pre_swaps, st));
  for (int64_t pi = 0; pi < P->npass; ++pi) {
    a.pass = P->passes + pi;
    k_fused_pass<<<grid, kTileThreads, P->smem, st>>>(a);
    QS_LAUNCHED();
  }
  if (!P->post_swaps.empty()) QS_TRY(launch_bitswap(a.state, n, s->nreg, P->post_swaps, st));
  return QS_OK;
}

void free_fused(qs_batch_program* p) { free_program(p); }

int schedule_info(const qs_circuit* c, int tile_qubits, int* npasses, int* nphases) {
  QS_TRY(ensure_schedule(c, tile_qubits > 0 ? tile_qubits : kBatchTile));
  if (npasses) *npasses = (int)c->fused->npass + !c->fused->pre_swaps.empty() + !c->fused->post_swaps.empty();
  if (nphases) *nphases = (int)c->fused->nphase;
  return QS_OK;
}

int tile_order(const qs_circuit* c, int tile_qubits, std::vector<int>& order, std::vector<int>& pass) {
  const int M = tile_qubits > 0 ? tile_qubits : kBatchTile;
  if (M < kRowBits + kRB || M > kBatchTile) return fail(QS_EINVAL, "tile_qubits must be in %d..%d", kRowBits + kRB, kBatchTile);
  const int n = c->nqubits;
  if (n < kRowBits || n > 32) return fail(QS_EUNSUPPORTED, "%d qubits outside the tile engine's range", n);
  TilePlan plan;
  QS_TRY(plan_tiles(c, M, &plan));
  order.clear();
  pass.clear();
  int at = 0, p = 0;  // place in the expanded list, pass
  auto network = [&](size_t first, size_t last) {
    if (first == last) return;
    for (size_t k = 0; k < 3 * (last - first); ++k) {
      order.push_back(at++);
      pass.push_back(p);
    }
    ++p;
  };
  network(0, plan.first);
  const int mid = at;
  for (const HostPass& hp : plan.passes) {
    for (const HostPhase& ph : hp.phases)
      for (int gi : ph.gates) {
        order.push_back(mid + gi);
        pass.push_back(p);
      }
    ++p;
  }
  at = mid + (int)plan.mid.gates.size();
  network(plan.last, c->gates.size());
  return QS_OK;
}

int expect_raw(const void* data, int dtype, int n, int nreg, const qs_observable* o, qs_state* ws_owner,
               double* host_out);

// Reversible gradient of one complex64 register with the tile engine: psi_N and
// lambda = O psi_N are copied into dev_work (2 x 2^n complex64), then the
// schedule's passes run backwards (FP32 uncompute, FP64 accumulation of the
// per-CTA gradient partials, folded in CTA order).
int fused_backward(qs_state* s, const qs_circuit* c, const double* host_params, const qs_observable* o,
                   void* dev_work, double* host_grad, double* host_loss, int tile_qubits) {
  if (s->dtype != QS_C64 || s->nreg != 1 || s->nq[0] != c->nqubits)
    return fail(QS_EUNSUPPORTED, "the tiled backward takes one complex64 register of the circuit's size");
  if (!dev_work) return fail(QS_EINVAL, "work buffer is NULL");
  const int n = s->nq[0];
  const int M = tile_qubits > 0 ? tile_qubits : kBatchTile;
  const int m = std::min(n, M), g = n - m;
  for (const auto& t : o->terms)
    if (n < 64 && ((t.x_mask | t.z_mask) >> n)) return fail(QS_EINVAL, "observable acts on a qubit >= n=%d", n);
  if (o->terms.size() > 64) return fail(QS_EUNSUPPORTED, "the tiled backward takes at most 64 observable terms");
  // schedule (shared with the fused forward) and parameter-dependent matrices
  QS_TRY(ensure_schedule(c, M));
  qs_batch_program* P = c->fused;
  cudaStream_t st = s->stream;
  const int np = c->nparams;
  size_t smem = sizeof(uint32_t) * (1 << (kMaxTileBits - kRowBits)) + sizeof(float) * phase_vals(c->nparams) * kWarps +
                sizeof(double) * ((np + 1) & ~1) + 2 * sizeof(float2) * (1ull << m);
  if (smem > kMaxSmem) return fail(QS_EUNSUPPORTED, "%d parameters do not fit the tiled backward's shared memory", np);
  // without room for the records those are read from global memory, once a phase
  const int stage = smem + kStageBytes + kStageMemBytes <= kMaxSmem ? kStageMems : smem + kStageBytes <= kMaxSmem ? 0 : -1;
  if (stage >= 0) smem += kStageBytes + sizeof(GMem) * stage;
  if (host_loss) QS_TRY(expect_raw(s->data, QS_C64, n, 1, o, s, host_loss));
  if (np > 0) {
    if (P->dparams_n < np) {
      if (P->dparams) cudaFree(P->dparams);
      P->dparams = nullptr;
      P->dparams_n = 0;
      if (cudaMalloc(&P->dparams, sizeof(double) * np) != cudaSuccess) {
        cudaGetLastError();
        return fail(QS_ENOMEM, "cudaMalloc of the parameter buffer failed");
      }
      P->dparams_n = np;
    }
    QS_CUDA(cudaMemcpyAsync(P->dparams, host_params, sizeof(double) * np, cudaMemcpyHostToDevice, st));
  }
  QS_TRY(launch_prep(P, P->dparams, true, st));
  // psi and lambda work copies
  const uint64_t dim = 1ull << n;
  float2* wpsi = (float2*)dev_work;
  float2* wlam = wpsi + dim;
  QS_CUDA(cudaMemcpyAsync(wpsi, s->data, sizeof(float2) * dim, cudaMemcpyDeviceToDevice, st));
  if (o->terms.empty()) {
    QS_CUDA(cudaMemsetAsync(wlam, 0, sizeof(float2) * dim, st));
  } else {
    ObsC64 ob;
    memset(&ob, 0, sizeof(ob));
    ob.nt = (int)o->terms.size();
    for (int t = 0; t < ob.nt; ++t) {
      ob.x[t] = o->terms[t].x_mask;
      ob.z[t] = o->terms[t].z_mask;
      ob.ny[t] = __builtin_popcountll(o->terms[t].x_mask & o->terms[t].z_mask) & 3;
      ob.c[t] = (float)o->terms[t].coeff;
    }
    k_apply_obs_c64<<<(unsigned)((dim + 255) / 256), 256, 0, st>>>(wpsi, wlam, dim, 0, ob);
    QS_LAUNCHED();
  }
  // per-CTA partials and the gradient accumulator in the state's scratch
  // the limit belongs to the function: the same for every circuit, as other threads launch theirs
  QS_CUDA(cudaFuncSetAttribute(k_fused_bwd_pass, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem));
  int dev = 0, sms = 0, per_sm = 0;
  QS_CUDA(cudaGetDevice(&dev));
  QS_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  QS_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_fused_bwd_pass, kTileThreads, smem));
  if (per_sm < 1) return fail(QS_EDEVICE, "tiled backward kernel does not fit on an SM");
  const uint64_t ntile = 1ull << g;
  const int grid = (int)std::min<uint64_t>(ntile, (uint64_t)sms * per_sm);
  const size_t npad = (size_t)std::max(1, np);
  QS_TRY(ensure_ws(s, s->ws, sizeof(double) * (npad + (size_t)grid * npad)));
  double* dgrad = (double*)s->ws.ptr;
  double* partials = dgrad + npad;
  QS_CUDA(cudaMemsetAsync(dgrad, 0, sizeof(double) * npad, st));
  FBArgs a;
  a.wpsi = wpsi;
  a.wlam = wlam;
  a.phases = P->phases;
  a.bops = P->bops;
  a.gmem = P->gmem;
  a.vals = phase_vals(np);
  a.m = m;
  a.g = g;
  a.nparam = np;
  a.stage = stage;
  a.ntile = ntile;
  a.partials = partials;
  auto swaps = [&](const std::vector<std::pair<int, int>>& net) -> int {  // its own inverse, on psi and lambda
    return net.empty() ? QS_OK : launch_bitswap(wpsi, n, 2, net, st);
  };
  QS_TRY(swaps(P->post_swaps));
  for (int64_t pi = P->npass - 1; pi >= 0; --pi) {
    a.pass = P->passes + pi;
    k_fused_bwd_pass<<<grid, kTileThreads, smem, st>>>(a);
    QS_LAUNCHED();
    if (np > 0) {
      k_fold_partials<<<(np + 255) / 256, 256, 0, st>>>(partials, grid, np, dgrad);
      QS_LAUNCHED();
    }
  }
  if (np > 0) QS_CUDA(cudaMemcpyAsync(host_grad, dgrad, sizeof(double) * np, cudaMemcpyDeviceToHost, st));
  QS_CUDA(cudaStreamSynchronize(st));
  return QS_OK;
}

}  // namespace qs

using namespace qs;

extern "C" {

int qs_batch_autotune(int nreg, const qs_circuit* const* circuits, const qs_observable* const* observables,
                      qs_state* s, const double* dev_params, double* dev_loss, double* dev_grad, int reps,
                      int* best_tile, int* ncand, int32_t* host_tiles, double* host_ms) {
  if (!circuits || !observables || !s || !dev_params || !dev_loss || !best_tile) return fail(QS_EINVAL, "null argument");
  if (reps < 1) reps = 1;
  const int flags = QS_BATCH_RESET | (dev_grad ? QS_BATCH_GRAD : 0);
  int best = -1, nc = 0;
  double best_ms = 0;
  cudaEvent_t e0, e1;
  QS_CUDA(cudaEventCreate(&e0));
  QS_CUDA(cudaEventCreate(&e1));
  int rc = QS_OK;
  for (int m = kBatchTile; m >= kRowBits + kRB + 2 && rc == QS_OK; --m) {
    qs_batch_program* P = nullptr;
    double ms = -1;
    const int crc = qs_batch_program_create(nreg, circuits, observables, m, &P);
    if (crc == QS_OK) {
      rc = qs_batch_run(s, P, dev_params, dev_loss, dev_grad, flags);  // warm-up
      if (rc == QS_OK && cudaEventRecord(e0, s->stream) != cudaSuccess) rc = fail(QS_EDEVICE, "event record");
      for (int r = 0; r < reps && rc == QS_OK; ++r) rc = qs_batch_run(s, P, dev_params, dev_loss, dev_grad, flags);
      if (rc == QS_OK && cudaEventRecord(e1, s->stream) != cudaSuccess) rc = fail(QS_EDEVICE, "event record");
      if (rc == QS_OK && cudaEventSynchronize(e1) != cudaSuccess) rc = fail(QS_EDEVICE, "event sync");
      float t = 0;
      if (rc == QS_OK && cudaEventElapsedTime(&t, e0, e1) == cudaSuccess) ms = (double)t / reps;
      qs_batch_program_destroy(P);
    } else if (crc != QS_EUNSUPPORTED && crc != QS_EINVAL) {
      rc = crc;
    }
    if (ncand && nc < *ncand) {
      if (host_tiles) host_tiles[nc] = m;
      if (host_ms) host_ms[nc] = ms;
    }
    ++nc;
    if (ms >= 0 && (best < 0 || ms < best_ms)) {
      best = m;
      best_ms = ms;
    }
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  if (rc != QS_OK) return rc;
  if (ncand) *ncand = nc;
  if (best < 0) return fail(QS_EUNSUPPORTED, "no tile size ran the batch");
  *best_tile = best;
  return QS_OK;
}

int qs_batch_program_create(int nreg, const qs_circuit* const* circuits, const qs_observable* const* observables,
                            int tile_qubits, qs_batch_program** out) {
  if (!out || nreg < 1 || !circuits || !observables) return fail(QS_EINVAL, "bad arguments");
  *out = nullptr;
  qs_batch_program* P = new qs_batch_program();
  const int rc = build_program(nreg, circuits, observables, tile_qubits, P);
  if (rc != QS_OK) {
    const std::string msg = qs_last_error();
    free_program(P);
    return fail(rc, "%s", msg.c_str());
  }
  *out = P;
  return QS_OK;
}

}  // extern "C"

// A forward-only program that applies the gates without moving a run past gates on other
// qubits to an X that it could take along, in phases cut at the same gates whatever the
// later engine's limits: the last bits of its amplitudes, and with them the samples that a
// shot-based estimate counts, are those of the plain order.
int qs::batch_program_plain(int nreg, const qs_circuit* const* circuits, const qs_observable* const* observables,
                            qs_batch_program** out) {
  *out = nullptr;
  qs_batch_program* P = new qs_batch_program();
  const int rc = build_program(nreg, circuits, observables, 0, P, kRB, false, true);
  if (rc != QS_OK) {
    const std::string msg = qs_last_error();
    free_program(P);
    return fail(rc, "%s", msg.c_str());
  }
  *out = P;
  return QS_OK;
}

extern "C" {

int qs_batch_program_create_ex(int nreg, const qs_circuit* const* circuits, const qs_observable* const* observables,
                               int tile_qubits, int phase_qubits, int flags, qs_batch_program** out) {
  if (!out || nreg < 1 || !circuits || !observables) return fail(QS_EINVAL, "bad arguments");
  if (flags & ~QS_BATCH_PRECISE) return fail(QS_EINVAL, "unknown program flags 0x%x", flags);
  *out = nullptr;
  qs_batch_program* P = new qs_batch_program();
  const bool precise = (flags & QS_BATCH_PRECISE) != 0;
  const int rb = phase_qubits > 0 ? phase_qubits : (precise ? 3 : kRB);  // the widest phase of the path
  const int rc = build_program(nreg, circuits, observables, tile_qubits, P, rb, precise);
  if (rc != QS_OK) {
    const std::string msg = qs_last_error();
    free_program(P);
    return fail(rc, "%s", msg.c_str());
  }
  *out = P;
  return QS_OK;
}

int qs_batch_program_shape(const qs_batch_program* p, int* tile_qubits, int* phase_qubits, int* flags) {
  if (!p) return fail(QS_EINVAL, "null program");
  if (tile_qubits) *tile_qubits = p->tile;
  if (phase_qubits) *phase_qubits = p->rb;
  if (flags) *flags = p->precise ? QS_BATCH_PRECISE : 0;
  return QS_OK;
}

int qs_batch_autotune_ex(int nreg, const qs_circuit* const* circuits, const qs_observable* const* observables,
                         int flags, qs_state* s, const double* dev_params, double* dev_loss, double* dev_grad,
                         int reps, int* best_tile, int* best_phase, int* ncand, int32_t* host_tiles,
                         int32_t* host_phases, double* host_ms) {
  if (!circuits || !observables || !s || !dev_params || !dev_loss || !best_tile || !best_phase)
    return fail(QS_EINVAL, "null argument");
  if (flags & ~QS_BATCH_PRECISE) return fail(QS_EINVAL, "unknown program flags 0x%x", flags);
  if (reps < 1) reps = 1;
  const bool precise = (flags & QS_BATCH_PRECISE) != 0;
  const int rflags = QS_BATCH_RESET | (dev_grad ? QS_BATCH_GRAD : 0);
  int best = -1, bestrb = -1, nc = 0;
  double best_ms = 0;
  cudaEvent_t e0, e1;
  QS_CUDA(cudaEventCreate(&e0));
  QS_CUDA(cudaEventCreate(&e1));
  int rc = QS_OK;
  for (int rb = precise ? 3 : kRB; rb >= kMinRB && rc == QS_OK; --rb) {
    const int mt = max_tile(rb);
    for (int m = mt; m >= std::max(kRowBits + rb + 2, mt - 2) && rc == QS_OK; --m) {
      qs_batch_program* P = nullptr;
      double ms = -1;
      const int crc = qs_batch_program_create_ex(nreg, circuits, observables, m, rb, flags, &P);
      if (crc == QS_OK) {
        rc = qs_batch_run(s, P, dev_params, dev_loss, dev_grad, rflags);  // warm-up
        if (rc == QS_OK && cudaEventRecord(e0, s->stream) != cudaSuccess) rc = fail(QS_EDEVICE, "event record");
        for (int r = 0; r < reps && rc == QS_OK; ++r) rc = qs_batch_run(s, P, dev_params, dev_loss, dev_grad, rflags);
        if (rc == QS_OK && cudaEventRecord(e1, s->stream) != cudaSuccess) rc = fail(QS_EDEVICE, "event record");
        if (rc == QS_OK && cudaEventSynchronize(e1) != cudaSuccess) rc = fail(QS_EDEVICE, "event sync");
        float t = 0;
        if (rc == QS_OK && cudaEventElapsedTime(&t, e0, e1) == cudaSuccess) ms = (double)t / reps;
        qs_batch_program_destroy(P);
      } else if (crc != QS_EUNSUPPORTED && crc != QS_EINVAL) {
        rc = crc;
      }
      if (ncand && nc < *ncand) {
        if (host_tiles) host_tiles[nc] = m;
        if (host_phases) host_phases[nc] = rb;
        if (host_ms) host_ms[nc] = ms;
      }
      ++nc;
      if (ms >= 0 && (best < 0 || ms < best_ms)) {
        best = m;
        bestrb = rb;
        best_ms = ms;
      }
    }
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  if (rc != QS_OK) return rc;
  if (ncand) *ncand = nc;
  if (best < 0) return fail(QS_EUNSUPPORTED, "no program shape ran the batch");
  *best_tile = best;
  *best_phase = bestrb;
  return QS_OK;
}

int qs_batch_program_destroy(qs_batch_program* p) {
  free_program(p);
  return QS_OK;
}

int qs_batch_program_info(const qs_batch_program* p, int* nreg, int64_t* nparams_total, int64_t* host_param_offsets,
                          int64_t* host_amp_offsets) {
  if (!p) return fail(QS_EINVAL, "null program");
  if (nreg) *nreg = p->nreg;
  if (nparams_total) *nparams_total = p->param_off[p->nreg];
  if (host_param_offsets) std::copy(p->param_off.begin(), p->param_off.end(), host_param_offsets);
  if (host_amp_offsets) std::copy(p->amp_off.begin(), p->amp_off.end(), host_amp_offsets);
  return QS_OK;
}

int qs_batch_run(qs_state* s, const qs_batch_program* p, const double* dev_params, double* dev_loss,
                 double* dev_grad, int flags) {
  if (!s || !p || !dev_loss) return fail(QS_EINVAL, "null argument");
  if (s->dtype != QS_C64) return fail(QS_EUNSUPPORTED, "the batched engine runs complex64 states");
  if (s->nreg != p->nreg) return fail(QS_EINVAL, "state has %d registers, program %d", s->nreg, p->nreg);
  for (int r = 0; r < s->nreg; ++r)
    if (s->nq[r] != p->nq[r]) return fail(QS_EINVAL, "register %d: %d qubits in the state, %d in the program", r, s->nq[r], p->nq[r]);
  if (p->param_off[p->nreg] > 0 && !dev_params) return fail(QS_EINVAL, "params is NULL");
  const bool grad = (flags & QS_BATCH_GRAD) != 0;
  if (grad && !dev_grad) return fail(QS_EINVAL, "grad is NULL");
  if (grad && p->forward_only) return fail(QS_EINVAL, "a forward-only program has no gradient");
  int dev = 0;
  QS_CUDA(cudaGetDevice(&dev));
  if (dev != p->device)
    return fail(QS_EINVAL, "the program was built on device %d; the current device is %d", p->device, dev);
  cudaStream_t st = s->stream;
  QS_TRY(launch_prep(p, dev_params, grad, st));  // without gradients the backward's records are not read
  QS_CUDA(cudaMemsetAsync(p->counter, 0, sizeof(int), st));
  BArgs a;
  a.state = (float2*)s->data;
  a.dtab = p->dtab;
  a.druns = p->druns;
  a.rtab = p->rtab;
  a.wpsi = p->wpsi;
  a.wlam = p->wlam;
  a.wpsif = p->wpsif;
  a.wlamf = p->wlamf;
  a.flo = p->flo;
  a.blo = p->blo;
  a.dtlo = p->dtlo;
  a.regs = p->regs;
  a.order = p->order;
  a.passes = p->passes;
  a.phases = p->phases;
  a.fops = p->fops;
  a.bops = p->bops;
  a.gmem = p->gmem;
  a.terms = p->terms;
  a.loss = dev_loss;
  a.grad = dev_grad;
  a.counter = p->counter;
  a.nreg = p->nreg;
  a.flags = ((flags & QS_BATCH_RESET) ? BF_RESET : 0) | (grad ? BF_GRAD : 0);
  if (p->precise) {
    if (p->rb == 2) k_batch<2, true><<<p->blocks, kTileThreads, p->smem, st>>>(a);
    else k_batch<3, true><<<p->blocks, kTileThreads, p->smem, st>>>(a);
  } else {
    switch (p->rb) {
      case 2: k_batch<2, false><<<p->blocks, kTileThreads, p->smem, st>>>(a); break;
      case 3: k_batch<3, false><<<p->blocks, kTileThreads, p->smem, st>>>(a); break;
      default: k_batch<4, false><<<p->blocks, kTileThreads, p->smem, st>>>(a); break;
    }
  }
  QS_LAUNCHED();
  return QS_OK;
}

}  // extern "C"
