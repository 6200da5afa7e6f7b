// reduce.cu -- expectation values, lambda = O psi, measurement sampling, reset
// and collapse (sm_103a).
//
// expect (Sec. "Forward Mode"): O = sum_t c_t P_t with P_t a Pauli string.
// For a basis state, P|i> = i^{nY} (-1)^{popc(i & z)} |i ^ x>, so
// <psi|P|psi> = sum_i ph(i) conj(psi_{i^x}) psi_i.  Terms are grouped by their
// x mask; each group reads each amplitude (or each pair (i, i^x) once, counting
// it twice) and adds it weighted with the group's coefficients in FP64.  The sum
// is pairwise: a thread adds at most 16 items in order to each of its sums (32
// where a unit has odd and even numbers of Y factors; the serial base case),
// threads, warps and blocks combine by balanced trees, and a second kernel folds
// the per-block partials (16 at most in order) and the groups by balanced trees
// as well (fixed shapes, so results are reproducible run to run).  qs_expect_static
// has room for 65536 partial sums: with nblk blocks for 2^n amplitudes a thread
// adds 16 ceil(2^n / kBlockAmps / nblk) items in order.
//
// measure (Sec. "Instructions on Quantum Registers"): the deterministic
// contract of qsim.h -- FP64 probabilities with separately rounded multiply
// and add, left folds over level-0 blocks of 1024 probabilities and level-1
// blocks of 1024 level-0 sums, and a three-level walk per shot.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "common.cuh"

namespace qs {

constexpr int kRedThreads = 256;
constexpr int kObsChunk = 64;     // terms per lambda = O psi launch

// A float as a double without the conversion instruction, which runs on the FP64
// unit, this part's scarcest (1/64 of the FP32 rate): the exponent is rebased and
// the mantissa moved by integer instructions, a subnormal scaled to a normal one
// first.
__device__ __forceinline__ double widen(float x) {
  const uint32_t sign = __float_as_uint(x) & 0x80000000u;
  const bool tiny = (__float_as_uint(x) & 0x7fffffffu) < 0x00800000u;
  const uint32_t m = __float_as_uint(tiny ? __fmul_rn(x, 16777216.f) : x) & 0x7fffffffu;
  const uint32_t bias = tiny ? 0x38000000u - (24u << 20) : m >= 0x7f800000u ? 0x70000000u : 0x38000000u;
  const uint32_t hi = m ? (m >> 3) + bias : 0u;
  return __hiloint2double((int)(hi | sign), (int)(m << 29));
}

__device__ __forceinline__ double2 widen(float2 v) { return make_double2(widen(v.x), widen(v.y)); }
__device__ __forceinline__ double2 widen(double2 v) { return v; }
template <typename T>
__device__ __forceinline__ double2 ld_amp(const T* p, uint64_t i) { return widen(p[i]); }

// Expectation sums: a block of 256 threads covers kBlockAmps amplitudes (64 a
// thread, or 32 pairs), the terms' coefficients inside the sum, and writes one
// partial sum for each slot (a launch's unit).  FP64 products of this part run
// at 1/64 of the FP32 rate, so both kernels are written for their FP64
// operations: floats are widened by integer instructions, the signs of a term
// are bit patterns of the index whose low bits a thread keeps for all its items
// and whose high bits are worked out once a block.
constexpr int kBlockAmps = 16384;
constexpr int kZLo = 10;     // index bits a thread of k_expect_z keeps fixed
constexpr int kZTerms = 64;  // terms of a k_expect_z launch
constexpr int kZMixed = 32;  // of them, terms with qubits on both sides of bit kZLo

__device__ __forceinline__ double flip(double c, uint32_t neg) {  // neg & 1: -c
  return __hiloint2double(__double2hiint(c) ^ (int)(neg << 31), __double2loint(c));
}

__device__ __forceinline__ void block_partial(double acc, double* out) {
  __shared__ double red[kRedThreads / 32];
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    static_assert(kRedThreads / 32 == 8, "block tree below is written for 8 warps");
    *out = ((red[0] + red[1]) + (red[2] + red[3])) + ((red[4] + red[5]) + (red[6] + red[7]));
  }
}

// Z strings: sum_i W(i) |psi_i|^2 with W(i) = sum_t c_t (-1)^popcount(i & z_t).
// Terms on qubits below kZLo are a constant of the thread's item, terms above a
// value of the chunk of 2^kZLo amplitudes; only those that span both are added
// item by item.  4 FP64 operations an amplitude and one a mixed term, where a sum a
// term took 2 and one for every term.  Bound by them: 24 strings Z_i Z_{i+1} at
// n = 25 complex64 368 us (two launches of 610 us before).
struct ZTerms {
  int nlo, nhi, nmix;
  uint64_t z[kZTerms];  // low terms, high ones, mixed ones
  double c[kZTerms];
};

template <typename T>
__global__ void __launch_bounds__(kRedThreads)
k_expect_z(const T* __restrict__ psi, int n, const __grid_constant__ ZTerms g, double* __restrict__ partials,
           int nslots, int slot) {
  constexpr int CH = kBlockAmps >> kZLo;         // chunks of a block
  constexpr int I = (1 << kZLo) / kRedThreads;   // items of a thread in a chunk
  __shared__ double high[CH];
  __shared__ uint32_t mixhi[CH];
  const uint64_t dim = 1ull << n, nvb = (dim + kBlockAmps - 1) / kBlockAmps;
  const T* p = psi + blockIdx.y * dim;
  const int tid = threadIdx.x, nl = g.nlo + g.nhi, nt = nl + g.nmix;
  double low[I], acc[I];
  uint32_t mixlo[I];
#pragma unroll
  for (int k = 0; k < I; ++k) {
    const uint32_t lo = tid + k * kRedThreads;
    low[k] = acc[k] = 0.0;
    mixlo[k] = 0;
    for (int t = 0; t < g.nlo; ++t) low[k] += flip(g.c[t], __popc(lo & (uint32_t)g.z[t]));
    for (int t = nl; t < nt; ++t) mixlo[k] |= (__popc(lo & (uint32_t)g.z[t] & ((1u << kZLo) - 1)) & 1u) << (t - nl);
  }
  for (uint64_t vb = blockIdx.x; vb < nvb; vb += gridDim.x) {
    __syncthreads();
    if (tid < 2 * CH) {
      const int ch = tid & (CH - 1);
      const uint64_t hi = (vb * CH + ch) << kZLo;
      if (tid < CH) {
        double w = 0.0;
        for (int t = g.nlo; t < nl; ++t) w += flip(g.c[t], __popcll(hi & g.z[t]));
        high[ch] = w;
      } else {
        uint32_t m = 0;
        for (int t = nl; t < nt; ++t) m |= (__popcll(hi & g.z[t]) & 1u) << (t - nl);
        mixhi[ch] = m;
      }
    }
    __syncthreads();
    const uint64_t i0 = vb * kBlockAmps + tid;
    const int chunks = dim >= kBlockAmps ? CH : (int)((dim + (1 << kZLo) - 1) >> kZLo);
#pragma unroll 2
    for (int ch = 0; ch < chunks; ++ch) {
      const double h = high[ch];
      const uint32_t mh = mixhi[ch];
#pragma unroll
      for (int k = 0; k < I; ++k) {
        const uint64_t i = i0 + ((uint64_t)ch << kZLo) + k * kRedThreads;
        if (i >= dim) continue;
        const double2 a = ld_amp(p, i);
        double w = low[k] + h;
        const uint32_t m = mixlo[k] ^ mh;
        for (int t = 0; t < g.nmix; ++t) w += flip(g.c[nl + t], m >> t);
        acc[k] = fma(w, fma(a.x, a.x, a.y * a.y), acc[k]);
      }
    }
  }
  double v = 0.0;
  static_assert(I == 4, "the thread's tree below is written for 4 items");
  v = (acc[0] + acc[1]) + (acc[2] + acc[3]);
  block_partial(v, partials + ((size_t)blockIdx.y * nslots + slot) * gridDim.x + blockIdx.x);
}

// Strings with X or Y factors.  The terms of one x mask share their pairs (i, i ^ x),
// i without x's highest bit h: with zr + i zi = conj(psi_{i^x}) psi_i a pair adds
// 2 (Wr zr + Wi zi), where a term puts its +-c into Wr (an even number of Y factors)
// or Wi (an odd one).  A unit is up to kXTerms terms of one mask: their signs index a
// table of Wr and Wi, and a lone term without sign (an X string) needs 2 FP64
// operations a pair.  The units of an observable run in one launch (blockIdx.z).
// Bound by the FP64 operations: 25 strings X_i at n = 25 complex64 1.63 ms, 65 us
// each (610 us each as launches that ran 16 predicated terms a pair).
constexpr int kXTerms = 4;
constexpr int kXUnits = 36;
struct XUnit {
  uint64_t x;
  uint64_t z[kXTerms];  // over pair numbers: bit h taken out
  double c[kXTerms];
  int8_t ny[kXTerms];   // number of Y factors mod 4
  int16_t h, nt;
};
struct XUnits {
  XUnit u[kXUnits];
};

template <typename T> struct Pairs { double2 a0, b0, a1, b1; };  // pairs j and j + 1

// vec: the registers start on 16-byte boundaries
template <typename T>
__device__ __forceinline__ Pairs<T> ld_pairs(const T* __restrict__ p, uint64_t j, int h, uint64_t x, bool vec) {
  Pairs<T> r;
  const uint64_t i = ((j >> h) << (h + 1)) | (j & ((1ull << h) - 1ull));
  const uint64_t step = h ? 1 : 2;  // from pair j to j + 1
  if constexpr (sizeof(T) == 8) {
    if (vec) {
      const float4 u = *reinterpret_cast<const float4*>(p + i);
      const float4 v = *reinterpret_cast<const float4*>(p + (h ? ((i ^ x) & ~1ull) : i + 2));
      const double2 u0 = widen(make_float2(u.x, u.y)), u1 = widen(make_float2(u.z, u.w));
      const double2 v0 = widen(make_float2(v.x, v.y)), v1 = widen(make_float2(v.z, v.w));
      if (h == 0) return {u0, u1, v0, v1};
      return (x & 1) ? Pairs<T>{u0, v1, u1, v0} : Pairs<T>{u0, v0, u1, v1};
    }
  }
  r.a0 = ld_amp(p, i);
  r.b0 = ld_amp(p, i ^ x);
  r.a1 = ld_amp(p, i + step);
  r.b1 = ld_amp(p, (i + step) ^ x);
  return r;
}

template <typename T>
__global__ void __launch_bounds__(kRedThreads)
k_expect_x(const T* __restrict__ psi, int n, const __grid_constant__ XUnits g, double* __restrict__ partials,
           int nslots, int slot0, int vec) {
  constexpr int STEPS = kBlockAmps / 2 / (2 * kRedThreads);
  __shared__ double tabr[1 << kXTerms], tabi[1 << kXTerms];
  __shared__ uint32_t pathi[STEPS];
  const XUnit& U = g.u[blockIdx.z];
  const int tid = threadIdx.x, h = U.h, nt = U.nt;
  const uint64_t x = U.x, dim = 1ull << n, items = dim >> 1, nvb = (dim + kBlockAmps - 1) / kBlockAmps;
  const T* p = psi + blockIdx.y * dim;
  bool real = false, imag = false;
  for (int t = 0; t < nt; ++t) ((U.ny[t] & 1) ? imag : real) = true;
  const bool plain = nt == 1 && !imag && U.z[0] == 0;
  if (tid < (1 << kXTerms)) {
    double wr = 0.0, wi = 0.0;
    for (int t = 0; t < nt; ++t) {
      // i^ny z: zr, -zi, -zr, zi
      const double c = flip(U.c[t], ((uint32_t)tid >> t) ^ (U.ny[t] == 1 || U.ny[t] == 2));
      if (U.ny[t] & 1) wi += c;
      else wr += c;
    }
    tabr[tid] = wr;
    tabi[tid] = wi;
  }
  uint32_t lo0 = 0, lo1 = 0;  // sign patterns of the thread's two pairs of a step
  for (int t = 0; t < nt; ++t) {
    lo0 |= (__popc((uint32_t)(2 * tid) & (uint32_t)U.z[t]) & 1u) << t;
    lo1 |= (__popc((uint32_t)(2 * tid + 1) & (uint32_t)U.z[t]) & 1u) << t;
  }
  double acc0 = 0.0, acc1 = 0.0;
  for (uint64_t vb = blockIdx.x; vb < nvb; vb += gridDim.x) {
    const uint64_t j0 = vb * (kBlockAmps / 2);
    __syncthreads();
    if (tid < STEPS) {
      uint32_t m = 0;
      for (int t = 0; t < nt; ++t) m |= (__popcll((j0 + (uint64_t)tid * 2 * kRedThreads) & U.z[t]) & 1u) << t;
      pathi[tid] = m;
    }
    __syncthreads();
    if (items == 1) {  // a one-qubit register: one pair
      if (tid == 0) {
        const double2 a = ld_amp(p, 0), b = ld_amp(p, 1);
        acc0 = tabr[0] * (b.x * a.x + b.y * a.y) + tabi[0] * (b.x * a.y - b.y * a.x);
      }
      continue;
    }
    const int steps = items >= kBlockAmps / 2 ? STEPS : (int)((items + 2 * kRedThreads - 1) / (2 * kRedThreads));
    auto load = [&](int s) { return ld_pairs(p, j0 + (uint64_t)(s * 2 * kRedThreads + 2 * tid), h, x, vec != 0); };
    auto on = [&](int s) { return j0 + (uint64_t)(s * 2 * kRedThreads + 2 * tid) < items; };
    if (plain) {
#pragma unroll 4
      for (int s = 0; s < steps; ++s) {
        if (!on(s)) continue;
        const Pairs<T> q = load(s);
        acc0 = fma(q.b0.x, q.a0.x, fma(q.b0.y, q.a0.y, acc0));
        acc1 = fma(q.b1.x, q.a1.x, fma(q.b1.y, q.a1.y, acc1));
      }
    } else {
#pragma unroll 4
      for (int s = 0; s < steps; ++s) {
        if (!on(s)) continue;
        const Pairs<T> q = load(s);
        const uint32_t m0 = lo0 ^ pathi[s], m1 = lo1 ^ pathi[s];
        if (real) {
          acc0 = fma(tabr[m0], fma(q.b0.x, q.a0.x, q.b0.y * q.a0.y), acc0);
          acc1 = fma(tabr[m1], fma(q.b1.x, q.a1.x, q.b1.y * q.a1.y), acc1);
        }
        if (imag) {
          acc0 = fma(tabi[m0], fma(q.b0.x, q.a0.y, -q.b0.y * q.a0.x), acc0);
          acc1 = fma(tabi[m1], fma(q.b1.x, q.a1.y, -q.b1.y * q.a1.x), acc1);
        }
      }
    }
  }
  const double c = plain && items > 1 ? 2.0 * U.c[0] : 2.0;
  block_partial(c * (acc0 + acc1),
                partials + ((size_t)blockIdx.y * nslots + slot0 + blockIdx.z) * gridDim.x + blockIdx.x);
}

// Pairwise sum in index order of the values add()ed one by one: a binary
// counter of partial sums, so 2^k values form a balanced tree.
struct PairwiseAcc {
  double stk[40];
  uint64_t cnt = 0;
  __device__ void add(double v) {
    int lvl = 0;
    while ((cnt >> lvl) & 1ull) {
      v = stk[lvl] + v;
      ++lvl;
    }
    stk[lvl] = v;
    ++cnt;
  }
  __device__ double total() const {
    double r = 0.0;
    bool any = false;
    for (int lvl = 0; lvl < 40; ++lvl)
      if ((cnt >> lvl) & 1ull) {
        r = any ? stk[lvl] + r : stk[lvl];
        any = true;
      }
    return r;
  }
};

constexpr int kFoldThreads = 1024;
constexpr int kFoldRow = 2048;  // partial sums a warp takes at a time

// one CTA per register, one warp per slot: the slot's block partials in rows of
// kFoldRow (64 a lane in four chains, then a tree), the rows pairwise; then the
// warps' slots (one CTA summing every term's partials in turn took 180 us for 49
// terms at n = 25; this 21 us for their 26 slots)
__global__ void __launch_bounds__(kFoldThreads)
k_expect_final(const double* __restrict__ partials, int nblk, int nslots, double* __restrict__ out) {
  __shared__ double sh[kFoldThreads / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  PairwiseAcc slots;
  for (int t = warp; t < nslots; t += kFoldThreads / 32) {
    const double* row = partials + ((size_t)blockIdx.x * nslots + t) * nblk;
    PairwiseAcc rows;
    double v = 0.0;
    for (int64_t r0 = 0; r0 < nblk; r0 += kFoldRow) {
      double a[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 4
      for (int k = 0; k < kFoldRow / 32 / 4; ++k)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int64_t i = r0 + (k * 4 + q) * 32 + lane;
          if (i < nblk) a[q] += row[i];
        }
      v = (a[0] + a[1]) + (a[2] + a[3]);
      for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      if (nblk > kFoldRow) rows.add(v);
    }
    slots.add(nblk > kFoldRow ? rows.total() : v);
  }
  if (lane == 0) sh[warp] = slots.total();
  __syncthreads();
  if (warp == 0) {
    double v = sh[lane];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0) out[blockIdx.x] = v;
  }
}

// blocks per register for the pairwise expectation
static int expect_blocks(uint64_t dim) { return (int)std::max<uint64_t>(1, (dim + kBlockAmps - 1) / kBlockAmps); }

// Slots (partial sums per block) of terms ordered by x mask, and their launches into
// partials[nreg][slots][nblk]; partials == NULL: only the count
static int expect_launch(const void* psi, int dtype, int n, int nreg, const qs_pauli_term* const* terms, int nt,
                         double* partials, int nblk, int nslots, int* slots, cudaStream_t st) {
  const dim3 grid((unsigned)nblk, (unsigned)nreg);
  int slot = 0, t = 0;
  // Z strings
  while (t < nt && !terms[t]->x_mask) {
    ZTerms g;
    memset(&g, 0, sizeof(g));
    const int t0 = t;
    const uint64_t lo = (1ull << kZLo) - 1;
    auto kind = [&](const qs_pauli_term* q) { return !(q->z_mask & ~lo) ? 0 : !(q->z_mask & lo) ? 1 : 2; };
    while (t < nt && !terms[t]->x_mask && t - t0 < kZTerms && (kind(terms[t]) != 2 || g.nmix < kZMixed))
      g.nmix += kind(terms[t++]) == 2;
    int at = 0;
    g.nmix = 0;
    for (int k = 0; k < 3; ++k)
      for (int q = t0; q < t; ++q) {
        if (kind(terms[q]) != k) continue;
        g.z[at] = terms[q]->z_mask;
        g.c[at++] = terms[q]->coeff;
        ++(k == 0 ? g.nlo : k == 1 ? g.nhi : g.nmix);
      }
    if (partials) {
      if (dtype == QS_C64)
        k_expect_z<float2><<<grid, kRedThreads, 0, st>>>((const float2*)psi, n, g, partials, nslots, slot);
      else
        k_expect_z<double2><<<grid, kRedThreads, 0, st>>>((const double2*)psi, n, g, partials, nslots, slot);
      QS_LAUNCHED();
    }
    ++slot;
  }
  // the others
  const int vec = ((uintptr_t)psi & 15) == 0;
  while (t < nt) {
    XUnits g;
    memset(&g, 0, sizeof(g));
    int nu = 0;
    for (; t < nt && nu < kXUnits; ++nu) {
      XUnit& u = g.u[nu];
      u.x = terms[t]->x_mask;
      u.h = (int16_t)(63 - __builtin_clzll(u.x));
      for (; t < nt && terms[t]->x_mask == u.x && u.nt < kXTerms; ++t, ++u.nt) {
        const uint64_t z = terms[t]->z_mask, low = (1ull << u.h) - 1;
        u.z[u.nt] = (z & low) | ((z >> 1) & ~low);
        u.c[u.nt] = terms[t]->coeff;
        u.ny[u.nt] = (int8_t)(__builtin_popcountll(u.x & z) & 3);
      }
    }
    if (partials) {
      const dim3 gx(grid.x, grid.y, (unsigned)nu);
      if (dtype == QS_C64)
        k_expect_x<float2><<<gx, kRedThreads, 0, st>>>((const float2*)psi, n, g, partials, nslots, slot, vec);
      else
        k_expect_x<double2><<<gx, kRedThreads, 0, st>>>((const double2*)psi, n, g, partials, nslots, slot, vec);
      QS_LAUNCHED();
    }
    slot += nu;
  }
  *slots = slot;
  return QS_OK;
}

struct ObsChunk {
  int nt;
  uint64_t x[kObsChunk];
  uint64_t z[kObsChunk];
  int ny[kObsChunk];
  double c[kObsChunk];
};

// lam (+)= sum_t c_t P_t psi, FP64 (complex128 buffers), one amplitude per thread
__global__ void __launch_bounds__(256)
k_apply_obs(const double2* __restrict__ psi, double2* __restrict__ lam, uint64_t dim, int accumulate,
            const __grid_constant__ ObsChunk o) {
  const uint64_t i = (uint64_t)blockIdx.x * 256 + threadIdx.x;
  if (i >= dim) return;
  double2 acc = accumulate ? lam[i] : make_double2(0.0, 0.0);
  for (int t = 0; t < o.nt; ++t) {
    const uint64_t j = i ^ o.x[t];          // (P psi)_i = ph(j) psi_j, j = i ^ x
    const double2 v = psi[j];
    const double s = (__popcll(j & o.z[t]) & 1) ? -o.c[t] : o.c[t];
    double re, im;
    switch (o.ny[t] & 3) {
      case 0: re = v.x; im = v.y; break;
      case 1: re = -v.y; im = v.x; break;   // * i
      case 2: re = -v.x; im = -v.y; break;  // * -1
      default: re = v.y; im = -v.x; break;  // * -i
    }
    acc.x += s * re;
    acc.y += s * im;
  }
  lam[i] = acc;
}

// ------------------------------------------------------------------ host side

// expectation of registers stored at `data` (uniform: nreg x 2^n, else one register)
int expect_raw(const void* data, int dtype, int n, int nreg, const qs_observable* o, qs_state* ws_owner,
               double* host_out) {
  cudaStream_t st = ws_owner->stream;
  std::vector<const qs_pauli_term*> terms;
  for (const auto& t : o->terms) {
    if (n < 64 && ((t.x_mask | t.z_mask) >> n)) return fail(QS_EINVAL, "observable acts on a qubit >= n=%d", n);
    terms.push_back(&t);
  }
  std::stable_sort(terms.begin(), terms.end(),
                   [](const qs_pauli_term* a, const qs_pauli_term* b) { return a->x_mask < b->x_mask; });
  const int nt = (int)terms.size(), nblk = expect_blocks(1ull << n), group = std::min(nreg, 65535);
  int nslots = 0;
  QS_TRY(expect_launch(data, dtype, n, nreg, terms.data(), nt, nullptr, nblk, 0, &nslots, st));
  const size_t out_off = (sizeof(double) * (size_t)group * std::max(1, nslots) * nblk + 255) / 256 * 256;
  QS_TRY(ensure_ws(ws_owner, ws_owner->ws, out_off + sizeof(double) * nreg));
  double* partials = (double*)ws_owner->ws.ptr;
  double* dev_out = (double*)((char*)ws_owner->ws.ptr + out_off);
  if (nt == 0) QS_CUDA(cudaMemsetAsync(dev_out, 0, sizeof(double) * nreg, st));
  for (int r = 0; nt > 0 && r < nreg; r += group) {
    const int k = std::min(group, nreg - r);
    const char* p = (const char*)data + ((amp_bytes(dtype) * (size_t)r) << n);
    QS_TRY(expect_launch(p, dtype, n, k, terms.data(), nt, partials, nblk, nslots, &nslots, st));
    k_expect_final<<<k, kFoldThreads, 0, st>>>(partials, nblk, nslots, dev_out + r);
    QS_LAUNCHED();
  }
  QS_CUDA(cudaMemcpyAsync(host_out, dev_out, sizeof(double) * nreg, cudaMemcpyDeviceToHost, st));
  QS_CUDA(cudaStreamSynchronize(st));
  return QS_OK;
}

int apply_observable_c128(const double2* psi, double2* lam, int n, const qs_observable* o, cudaStream_t st) {
  const uint64_t dim = 1ull << n;
  const int nt = (int)o->terms.size();
  if (nt == 0) {
    QS_CUDA(cudaMemsetAsync(lam, 0, sizeof(double2) * dim, st));
    return QS_OK;
  }
  for (int c0 = 0; c0 < nt; c0 += kObsChunk) {
    ObsChunk ch;
    memset(&ch, 0, sizeof(ch));
    ch.nt = std::min(kObsChunk, nt - c0);
    for (int t = 0; t < ch.nt; ++t) {
      const auto& term = o->terms[c0 + t];
      ch.x[t] = term.x_mask;
      ch.z[t] = term.z_mask;
      ch.ny[t] = __builtin_popcountll(term.x_mask & term.z_mask) & 3;
      ch.c[t] = term.coeff;
    }
    k_apply_obs<<<(unsigned)((dim + 255) / 256), 256, 0, st>>>(psi, lam, dim, c0 > 0, ch);
    QS_LAUNCHED();
  }
  return QS_OK;
}

// ------------------------------------------------------------------ sampling

constexpr int kF = 1024;

// What a fold adds up: |amplitude|^2 by the contract, or a level's sums.  The
// square of a float is exact in FP64, so one fused multiply-add rounds re*re +
// im*im once, as the contract's multiply, multiply and add do: 2 FP64
// operations instead of 5 with the conversions.
__device__ __forceinline__ double prob(float2 v) {
  const double2 w = widen(v);
  return __fma_rn(w.x, w.x, __dmul_rn(w.y, w.y));
}
__device__ __forceinline__ double prob(double2 v) { return __dadd_rn(__dmul_rn(v.x, v.x), __dmul_rn(v.y, v.y)); }
__device__ __forceinline__ double prob(double v) { return v; }

// Left folds of equal blocks.  A block's fold is one chain of dependent FP64
// adds, so a CTA gives each of up to 32 blocks a lane of one warp and lets all
// its warps load the values (coalesced, the next chunk while the present one
// is folded), form the probabilities and put them in shared memory.
//   bound: the FP64 rate (3 operations an amplitude) when the blocks fill the
//   GPU, the chain's latency (1024 adds of 87 clocks) when they do not; the
//   fold warp differs between the CTAs of an SM so that each of its FP64 units
//   gets its share.  Measured, n = 25 complex64: 210 us (a thread a block reading
//   the state directly: 449 us; with conversion instructions here: 346 us).  One
//   block, n = 10: 58 us (198 us).
// `start`: the value a block's fold begins with; RUN: also every running sum.
constexpr int kFoldCta = 128;
constexpr int kFoldElems = 1024;  // values of a chunk over all blocks of the CTA

// the exclusive prefix of block b of a register that has `per` of them: inner[b - 1],
// or outer[g - 1] for the first block of group g of 1024 (mask: the bits of a block's
// place in its group), 0 for the register's first
struct FoldStart {
  const double* inner;
  const double* outer;
  uint64_t per, mask, outer_per;
};
__device__ __forceinline__ double start_of(const FoldStart& s, uint64_t b) {
  const uint64_t r = b / s.per, k = b - r * s.per;
  if (s.inner && (k & s.mask)) return s.inner[b - 1];
  if (!s.outer || k < kF) return 0.0;
  return s.outer[r * s.outer_per + k / kF - 1];
}

template <typename T>
struct FoldChunk {
  T v[kFoldElems / kFoldCta];
};

// values j0 .. j0 + 2^chl - 1 of blocks first[g] (in units of len values), thread by thread
template <typename T, typename First>
__device__ __forceinline__ void fold_load(FoldChunk<T>& c, const T* __restrict__ src, First first, int elems, int chl,
                                          uint64_t len, uint64_t j0) {
#pragma unroll
  for (int k = 0; k < kFoldElems / kFoldCta; ++k) {
    const int e = threadIdx.x + k * kFoldCta;
    if (e < elems) c.v[k] = src[first(e >> chl) * len + j0 + (uint64_t)(e & ((1 << chl) - 1))];
  }
}
template <typename T>
__device__ __forceinline__ void fold_put(double* buf, const FoldChunk<T>& c, int elems, int chl) {
#pragma unroll
  for (int k = 0; k < kFoldElems / kFoldCta; ++k) {
    const int e = threadIdx.x + k * kFoldCta;
    if (e < elems) buf[(e >> chl) * ((1 << chl) + 1) + (e & ((1 << chl) - 1))] = prob(c.v[k]);
  }
}

// B: values read ahead of the adds (a divisor of the chunk)
template <typename T, bool RUN, int B>
__global__ void __launch_bounds__(kFoldCta)
k_fold(const T* __restrict__ src, uint64_t nblocks, uint64_t len, int gl, int chl, const FoldStart st,
       double* __restrict__ sums, double* __restrict__ run) {
  __shared__ double buf[2][kFoldElems + 32];
  const uint64_t b0 = (uint64_t)blockIdx.x << gl;
  const int G = (int)(nblocks - b0 < (1ull << gl) ? nblocks - b0 : (1ull << gl)), elems = G << chl;
  const int pitch = (1 << chl) + 1, lane = threadIdx.x & 31;
  const bool folds = (int)(threadIdx.x >> 5) == (int)(blockIdx.x % (kFoldCta / 32)) && lane < G;
  auto first = [&](int g) { return b0 + (uint64_t)g; };
  double a = folds ? start_of(st, b0 + lane) : 0.0;
  FoldChunk<T> c;
  fold_load(c, src, first, elems, chl, len, 0);
  fold_put(buf[0], c, elems, chl);
  __syncthreads();
  const uint64_t nch = len >> chl;
  // running sums replace their values in the chunk's buffer; a thread stores
  // the slots of the chunk before the last that it then refills itself
  auto flush = [&](const double* b, uint64_t ch) {
#pragma unroll
    for (int k = 0; k < kFoldElems / kFoldCta; ++k) {
      const int e = threadIdx.x + k * kFoldCta, g = e >> chl, j = e & ((1 << chl) - 1);
      if (e < elems) run[(b0 + g) * len + (ch << chl) + j] = b[g * pitch + j];
    }
  };
  for (uint64_t ch = 0; ch < nch; ++ch) {
    double* cur = buf[ch & 1];
    double* nxt = buf[(ch + 1) & 1];
    if (ch + 1 < nch) fold_load(c, src, first, elems, chl, len, (ch + 1) << chl);
    if (folds) {
      double* row = cur + lane * pitch;
      for (int j = 0; j < (1 << chl); j += B) {
        double v[B];
#pragma unroll
        for (int k = 0; k < B; ++k) v[k] = row[j + k];
#pragma unroll
        for (int k = 0; k < B; ++k) v[k] = a = __dadd_rn(a, v[k]);
        if (RUN) {
#pragma unroll
          for (int k = 0; k < B; ++k) row[j + k] = v[k];
        }
      }
    }
    if (RUN && ch > 0) flush(nxt, ch - 1);
    if (ch + 1 < nch) fold_put(nxt, c, elems, chl);
    __syncthreads();
  }
  if (RUN) flush(buf[(nch - 1) & 1], nch - 1);
  if (sums && folds) sums[b0 + lane] = a;
}

// Where the running sums of the three levels lie.  r2 is over the level-1 sums
// (NULL: one level-1 block, whose prefix is 0), r1 over the level-0 sums (NULL:
// one level-0 block), r0 over the probabilities (NULL: folded per shot).
struct SampleArgs {
  const double *s1, *s0, *r2, *r1, *r0, *u;
  int64_t* out;
  uint64_t dim, nb0, nb1;
  int nshots;
  uint64_t total;  // shots of all registers
};

// The walk of the contract: the first value whose running sum exceeds t, else the
// last positive one, else the last.  The running sums of non-negative values do
// not decrease, so the first is found by bisection (a sum that is not finite
// makes the total and t so as well, and no sum exceeds that).
template <typename V>
__device__ __forceinline__ uint64_t walk(const double* __restrict__ run, uint64_t len, double t, V value) {
  uint64_t lo = 0, hi = len;
  while (lo < hi) {
    const uint64_t mid = (lo + hi) >> 1;
    if (run[mid] > t) hi = mid;
    else lo = mid + 1;
  }
  if (lo < len) return lo;
  for (uint64_t j = len; j-- > 0;)
    if (value(j) > 0.0) return j;
  return len - 1;
}

// level-0 block of shot s (of its register r) and the target t
__device__ __forceinline__ uint64_t shot_block(const SampleArgs& a, uint64_t r, double t) {
  uint64_t c = 0;
  if (a.r2) c = walk(a.r2 + r * a.nb1, a.nb1, t, [&](uint64_t j) { return a.s1[r * a.nb1 + j]; });
  if (!a.r1) return 0;
  const uint64_t k0 = c * kF, k1 = k0 + kF < a.nb0 ? k0 + kF : a.nb0;
  return k0 + walk(a.r1 + r * a.nb0 + k0, k1 - k0, t, [&](uint64_t j) { return a.s0[r * a.nb0 + k0 + j]; });
}
__device__ __forceinline__ double shot_target(const SampleArgs& a, uint64_t s, uint64_t r) {
  const double total = a.r2   ? a.r2[(r + 1) * a.nb1 - 1]
                       : a.r1 ? a.r1[(r + 1) * a.nb0 - 1]
                              : a.r0[(r + 1) * a.dim - 1];
  return __dmul_rn(a.u[s], total);
}

// every running sum at hand: three bisections a shot (240 registers x 1024 shots at
// n = 10: 9.5 us; a serial walk a shot, one launch a register, took 366 us each)
template <typename T>
__global__ void __launch_bounds__(128) k_sample(const T* __restrict__ psi, const SampleArgs a) {
  const uint64_t s = (uint64_t)blockIdx.x * 128 + threadIdx.x;
  if (s >= a.total) return;
  const uint64_t r = s / a.nshots;
  const double t = shot_target(a, s, r);
  const uint64_t b = shot_block(a, r, t), i0 = b * kF, i1 = i0 + kF < a.dim ? i0 + kF : a.dim;
  const T* p = psi + r * a.dim + i0;
  a.out[s] = (int64_t)(i0 + walk(a.r0 + r * a.dim + i0, i1 - i0, t, [&](uint64_t j) { return prob(p[j]); }));
}

// fewer shots than blocks: a lane a shot folds its own block of probabilities
// from the block's prefix (k_fold's layout, with the blocks that the shots fall into;
// 4096 shots at n = 25: 112 us, 621 us as a serial walk of every level a thread)
template <typename T>
__global__ void __launch_bounds__(kFoldCta) k_sample_fold(const T* __restrict__ psi, const FoldStart st, const SampleArgs a) {
  __shared__ double buf[2][kFoldElems + 32];
  __shared__ uint64_t blk[32];
  constexpr int CHL = 5;
  const uint64_t s0 = (uint64_t)blockIdx.x * 32;
  const int G = (int)(a.total - s0 < 32 ? a.total - s0 : 32), elems = G << CHL;
  const int lane = threadIdx.x & 31;
  const bool folds = (int)(threadIdx.x >> 5) == (int)(blockIdx.x % (kFoldCta / 32)) && lane < G;
  uint64_t r = 0, b = 0;
  // the target's bit pattern: sums and values have no sign, so that theirs are in order as
  // integers, above the pattern of any smaller target.  A target of -0 is 0; infinities and NaNs
  // of either sign are never exceeded
  long long tb = 0;
  double acc = 0.0;
  if (folds) {
    r = (s0 + lane) / a.nshots;
    const double t = shot_target(a, s0 + lane, r);
    b = shot_block(a, r, t);
    blk[lane] = r * a.nb0 + b;
    acc = start_of(st, r * a.nb0 + b);
    tb = t == 0.0 ? 0 : t <= 0x1.fffffffffffffp1023 ? __double_as_longlong(t) : 0x7fffffffffffffffll;
  }
  __syncthreads();
  auto first = [&](int g) { return blk[g]; };
  FoldChunk<T> c;
  fold_load(c, psi, first, elems, CHL, kF, 0);
  fold_put(buf[0], c, elems, CHL);
  __syncthreads();
  int found = -1, last = -1;
  for (int ch = 0; ch < kF / 32; ++ch) {
    if (ch + 1 < kF / 32) fold_load(c, psi, first, elems, CHL, kF, (uint64_t)(ch + 1) << CHL);
    if (folds) {
      const double* row = buf[ch & 1] + lane * 33;
#pragma unroll 8
      for (int j = 0; j < 32; ++j) {
        const double v = row[j];
        acc = __dadd_rn(acc, v);
        // compared by the bit patterns, off the FP64 unit
        if (found < 0 && __double_as_longlong(acc) > tb) found = ch * 32 + j;
        const long long vb = __double_as_longlong(v);
        if (vb > 0 && vb <= 0x7ff0000000000000ll) last = ch * 32 + j;
      }
    }
    if (ch + 1 < kF / 32) fold_put(buf[(ch + 1) & 1], c, elems, CHL);
    __syncthreads();
  }
  if (folds) a.out[s0 + lane] = (int64_t)(b * kF + (found >= 0 ? found : last >= 0 ? last : kF - 1));
}

template <typename T>
__global__ void k_collapse_scale(T* psi, int64_t x, double2* keep) {
  const double2 a = ld_amp(psi, (uint64_t)x);
  const double r = sqrt(a.x * a.x + a.y * a.y);
  *keep = r > 0.0 ? make_double2(a.x / r, a.y / r) : make_double2(1.0, 0.0);
}

__device__ __forceinline__ void st_amp(float2* p, uint64_t i, double2 v) { p[i] = make_float2((float)v.x, (float)v.y); }
__device__ __forceinline__ void st_amp(double2* p, uint64_t i, double2 v) { p[i] = v; }

template <typename T>
__global__ void k_collapse_write(T* psi, uint64_t dim, int64_t x, const double2* keep) {
  const uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= dim) return;
  st_amp(psi, i, i == (uint64_t)x ? *keep : make_double2(0.0, 0.0));
}

// samples of nreg registers of 2^n amplitudes (back to back) with device uniforms
// [nreg][nshots] into device indices; scratch: sample_scratch_doubles() doubles.  lean: for a
// device that has no room for the running sums of the probabilities; same samples
constexpr uint64_t kRunDoubles = 1ull << 25;   // running sums of the probabilities in scratch: at most 256 MiB
constexpr uint64_t kLeanDoubles = 1ull << 17;  // lean: 1 MiB, those of single-block registers only

// The running sums of every probability cost a second pass over the state and
// 8 bytes an amplitude, a shot without them folds 1024 probabilities: they are
// formed once a level-0 block gets a shot or more on the average, or when a
// register is a single block (whose fold is the running sum).
static bool keep_runs(int n, int nshots, bool lean) {
  const uint64_t dim = 1ull << n, nb0 = (dim + kF - 1) / kF;
  return nb0 == 1 || (!lean && nb0 <= (uint64_t)nshots && dim <= kRunDoubles);
}
// registers sampled together
static int sample_group(int n, int nreg, bool lean) {
  return (int)std::min<uint64_t>((uint64_t)nreg, std::max<uint64_t>(1, (lean ? kLeanDoubles : kRunDoubles) >> n));
}

size_t sample_scratch_doubles(int n, int nreg, int nshots, bool lean) {
  const uint64_t dim = 1ull << n, nb0 = (dim + kF - 1) / kF, nb1 = (nb0 + kF - 1) / kF;
  const uint64_t levels = (nb0 > 1 ? 2 * nb0 : 0) + (nb1 > 1 ? 2 * nb1 : 0);
  return (size_t)((levels + (keep_runs(n, nshots, lean) ? dim : 0)) * (uint64_t)sample_group(n, nreg, lean));
}

template <typename T, bool RUN>
static int launch_fold(const T* src, uint64_t nblocks, uint64_t len, const FoldStart& st, double* sums, double* run,
                       cudaStream_t stream) {
  // as many blocks a CTA (up to a warp of chains) as leave two CTAs an SM
  int gl = 0;
  while (gl < 5 && (nblocks >> (gl + 1)) >= 304) ++gl;
  int chl = 10 - gl;
  while ((1ull << chl) > len) --chl;
  const uint64_t grid = (nblocks + (1ull << gl) - 1) >> gl;
  if (grid > 0x7fffffffull) return fail(QS_EUNSUPPORTED, "register too large to sample");
  if (chl >= 3) k_fold<T, RUN, 8><<<(unsigned)grid, kFoldCta, 0, stream>>>(src, nblocks, len, gl, chl, st, sums, run);
  else k_fold<T, RUN, 1><<<(unsigned)grid, kFoldCta, 0, stream>>>(src, nblocks, len, gl, chl, st, sums, run);
  QS_LAUNCHED();
  return QS_OK;
}

template <typename T>
static int sample_regs(const T* psi, int n, int nreg, const double* dev_u, int nshots, int64_t* dev_out, double* scratch,
                       bool lean, cudaStream_t st) {
  const uint64_t dim = 1ull << n, R = (uint64_t)nreg;
  const uint64_t nb0 = (dim + kF - 1) / kF, nb1 = (nb0 + kF - 1) / kF, len0 = std::min<uint64_t>(dim, kF);
  const bool runs = keep_runs(n, nshots, lean);
  SampleArgs a;
  memset(&a, 0, sizeof(a));
  a.u = dev_u;
  a.out = dev_out;
  a.dim = dim;
  a.nb0 = nb0;
  a.nb1 = nb1;
  a.nshots = nshots;
  a.total = R * (uint64_t)nshots;
  FoldStart zero;
  memset(&zero, 0, sizeof(zero));
  zero.per = 1;
  FoldStart st0 = zero;  // prefixes of the level-0 blocks
  if (nb0 > 1) {
    double* s0 = scratch;
    double* r1 = s0 + R * nb0;
    scratch = r1 + R * nb0;
    QS_TRY((launch_fold<T, false>(psi, R * nb0, len0, zero, s0, nullptr, st)));
    FoldStart st1 = zero;  // prefixes of the level-1 blocks
    if (nb1 > 1) {
      double* s1 = scratch;
      double* r2 = s1 + R * nb1;
      scratch = r2 + R * nb1;
      QS_TRY((launch_fold<double, false>(s0, R * nb1, kF, zero, s1, nullptr, st)));
      QS_TRY((launch_fold<double, true>(s1, R, nb1, zero, nullptr, r2, st)));
      a.s1 = s1;
      a.r2 = r2;
      st1 = FoldStart{r2, nullptr, nb1, ~0ull, 0};
    }
    QS_TRY((launch_fold<double, true>(s0, R * nb1, std::min<uint64_t>(nb0, kF), st1, nullptr, r1, st)));
    a.s0 = s0;
    a.r1 = r1;
    st0 = FoldStart{r1, a.r2, nb0, kF - 1, nb1};
  }
  if (runs) {
    QS_TRY((launch_fold<T, true>(psi, R * nb0, len0, st0, nullptr, scratch, st)));
    a.r0 = scratch;
    k_sample<T><<<(unsigned)((a.total + 127) / 128), 128, 0, st>>>(psi, a);
  } else {
    k_sample_fold<T><<<(unsigned)((a.total + 31) / 32), kFoldCta, 0, st>>>(psi, st0, a);
  }
  QS_LAUNCHED();
  return QS_OK;
}

int sample_dev(const void* data, int dtype, int n, int nreg, const double* dev_u, int nshots, int64_t* dev_out,
               double* scratch, bool lean, cudaStream_t st) {
  const int group = sample_group(n, nreg, lean);
  for (int r = 0; r < nreg; r += group) {
    const int k = std::min(group, nreg - r);
    const char* p = (const char*)data + ((amp_bytes(dtype) * (size_t)r) << n);
    const double* u = dev_u + (size_t)r * nshots;
    int64_t* out = dev_out + (size_t)r * nshots;
    if (dtype == QS_C64) QS_TRY(sample_regs((const float2*)p, n, k, u, nshots, out, scratch, lean, st));
    else QS_TRY(sample_regs((const double2*)p, n, k, u, nshots, out, scratch, lean, st));
  }
  return QS_OK;
}

// Uniforms of the seeded measurement: draw k of SplitMix64 started from `seed`
// (Steele, Lea and Flood 2014): state seed + k * 0x9E3779B97F4A7C15, then the
// 64-bit finaliser (xor-shift 30, multiply, xor-shift 27, multiply, xor-shift
// 31); u = top 53 bits / 2^53.  Shot j of this call is draw k0 + j + 1.
__global__ void k_seeded_uniforms(uint64_t seed, uint64_t k0, uint64_t nshots, double* __restrict__ u) {
  const uint64_t j = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= nshots) return;
  uint64_t x = seed + (k0 + j + 1ull) * 0x9E3779B97F4A7C15ull;
  x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ull;
  x = (x ^ (x >> 27)) * 0x94D049BB133111EBull;
  x ^= x >> 31;
  u[j] = (double)(x >> 11) * 0x1.0p-53;
}

// nreg registers of 2^n amplitudes back to back; the uniforms are host_u or drawn
// from seed (shot j of register r: draw k0 + r nshots + j + 1).  Scratch that the device
// has no room for: without the running sums, then half the registers at a time.
int measure_regs(void* data, int dtype, int n, int nreg, const double* host_u, int nshots, int64_t* host_out,
                 int collapse, qs_state* owner, const uint64_t* seed, uint64_t k0) {
  cudaStream_t st = owner->stream;
  const uint64_t dim = 1ull << n;
  const size_t shots = (size_t)nreg * nshots;
  bool lean = false;
  auto room = [&] {
    return ensure_ws(owner, owner->ws, sizeof(double) * (sample_scratch_doubles(n, nreg, nshots, lean) + shots) +
                                           sizeof(int64_t) * shots + sizeof(double2) + 256);
  };
  int rc = room();
  if (rc == QS_ENOMEM) {
    lean = true;
    rc = room();
  }
  if (rc == QS_ENOMEM && nreg > 1) {
    const int h = nreg / 2;
    const size_t k = (size_t)h * nshots;
    QS_TRY(measure_regs(data, dtype, n, h, host_u, nshots, host_out, collapse, owner, seed, k0));
    return measure_regs((char*)data + ((amp_bytes(dtype) * (size_t)h) << n), dtype, n, nreg - h,
                        host_u ? host_u + k : nullptr, nshots, host_out + k, collapse, owner, seed, k0 + k);
  }
  QS_TRY(rc);
  const size_t scr = sample_scratch_doubles(n, nreg, nshots, lean);
  double* dscr = (double*)owner->ws.ptr;
  double* du = dscr + scr;
  int64_t* dout = (int64_t*)(du + shots);
  double2* keep = (double2*)(((uintptr_t)(dout + shots) + 15) & ~(uintptr_t)15);
  if (seed) {
    k_seeded_uniforms<<<(unsigned)((shots + 127) / 128), 128, 0, st>>>(*seed, k0, shots, du);
    QS_LAUNCHED();
  } else {
    QS_CUDA(cudaMemcpyAsync(du, host_u, sizeof(double) * shots, cudaMemcpyHostToDevice, st));
  }
  QS_TRY(sample_dev(data, dtype, n, nreg, du, nshots, dout, dscr, lean, st));
  QS_CUDA(cudaMemcpyAsync(host_out, dout, sizeof(int64_t) * shots, cudaMemcpyDeviceToHost, st));
  QS_CUDA(cudaStreamSynchronize(st));
  if (!collapse) return QS_OK;
  for (int r = 0; r < nreg; ++r) {
    const int64_t x = host_out[r];
    char* reg = (char*)data + amp_bytes(dtype) * dim * r;
    if (dtype == QS_C64) {
      k_collapse_scale<float2><<<1, 1, 0, st>>>((float2*)reg, x, keep);
      k_collapse_write<float2><<<(unsigned)((dim + 255) / 256), 256, 0, st>>>((float2*)reg, dim, x, keep);
    } else {
      k_collapse_scale<double2><<<1, 1, 0, st>>>((double2*)reg, x, keep);
      k_collapse_write<double2><<<(unsigned)((dim + 255) / 256), 256, 0, st>>>((double2*)reg, dim, x, keep);
    }
    QS_LAUNCHED();
  }
  QS_CUDA(cudaStreamSynchronize(st));
  return QS_OK;
}

// ------------------------------------------------------------------ reset / promote

__global__ void k_set_ones(char* data, int dtype, const int64_t* __restrict__ pos, int count) {
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= count) return;
  if (dtype == QS_C64) ((float2*)data)[pos[r]] = make_float2(1.f, 0.f);
  else ((double2*)data)[pos[r]] = make_double2(1.0, 0.0);
}

int reset_basis(qs_state* s, const uint64_t* host_basis) {
  cudaStream_t st = s->stream;
  std::vector<int64_t> pos(s->nreg);
  for (int r = 0; r < s->nreg; ++r) {
    const uint64_t x = host_basis ? host_basis[r] : 0;
    if (s->nq[r] < 64 && (x >> s->nq[r])) return fail(QS_EINVAL, "basis index %llu out of range for register %d",
                                                     (unsigned long long)x, r);
    pos[r] = s->off[r] + (int64_t)x;
  }
  QS_TRY(ensure_ws(s, s->ws, sizeof(int64_t) * s->nreg));
  QS_CUDA(cudaMemsetAsync(s->data, 0, s->bytes, st));
  QS_CUDA(cudaMemcpyAsync(s->ws.ptr, pos.data(), sizeof(int64_t) * s->nreg, cudaMemcpyHostToDevice, st));
  k_set_ones<<<(s->nreg + 127) / 128, 128, 0, st>>>((char*)s->data, s->dtype, (const int64_t*)s->ws.ptr, s->nreg);
  QS_LAUNCHED();
  return QS_OK;
}

template <typename C, bool SCALE>
__global__ void k_promote(const C* __restrict__ in, double2* __restrict__ out, uint64_t dim, double2 f) {
  const uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= dim) return;
  const C v = in[i];
  const double2 w = make_double2(v.x, v.y);
  out[i] = SCALE ? cmul(f, w) : w;
}

// out = f in
int promote_to_c128(const void* in, int dtype, double2* out, uint64_t dim, cd f, cudaStream_t st) {
  const unsigned nb = (unsigned)((dim + 255) / 256);
  const double2 d = make_double2(f.real(), f.imag());
  const bool one = f == cd(1, 0);
  if (dtype == QS_C128 && one) {
    QS_CUDA(cudaMemcpyAsync(out, in, sizeof(double2) * dim, cudaMemcpyDeviceToDevice, st));
    return QS_OK;
  }
  if (dtype == QS_C128) k_promote<double2, true><<<nb, 256, 0, st>>>((const double2*)in, out, dim, d);
  else if (one) k_promote<float2, false><<<nb, 256, 0, st>>>((const float2*)in, out, dim, d);
  else k_promote<float2, true><<<nb, 256, 0, st>>>((const float2*)in, out, dim, d);
  QS_LAUNCHED();
  return QS_OK;
}

}  // namespace qs

// ------------------------------------------------------------------ expectation without allocation
//
// qs_expect_static: the expectation reduction above with its scratch in a
// fixed, file-scope device array instead of memory obtained from cudaMalloc,
// for callers that cannot allocate device memory.  Every GPU that loads the
// library holds this array (512 KiB) until the process exits.  All calls
// share it, so calls whose kernels overlap on the GPU race on it.

namespace qs {

constexpr int kStaticPartials = 1 << 16;  // FP64 partial sums (512 KiB)
constexpr int kStaticTerms = 64;
constexpr int kStaticMaxDevices = 64;

static __device__ __align__(256) double g_static_partials[kStaticPartials];

// device address of g_static_partials on the current device, resolved once per
// device (host code must not use the symbol's host-side name as an address)
static double* g_static_addr[kStaticMaxDevices];

static int static_partials(double** out) {
  int dev = 0;
  QS_CUDA(cudaGetDevice(&dev));
  if (dev < 0 || dev >= kStaticMaxDevices) return fail(QS_EUNSUPPORTED, "device ordinal %d >= %d", dev, kStaticMaxDevices);
  if (!g_static_addr[dev]) {
    void* p = nullptr;
    const cudaError_t e = cudaGetSymbolAddress(&p, g_static_partials);
    if (e != cudaSuccess || !p)
      return fail(QS_EDEVICE, "cudaGetSymbolAddress of the static scratch failed: %s", cudaGetErrorString(e));
    g_static_addr[dev] = (double*)p;
  }
  *out = g_static_addr[dev];
  return QS_OK;
}

}  // namespace qs

extern "C" int qs_expect_static(const void* dev_amps, int dtype, int nqubits, int nreg, const qs_pauli_term* host_terms,
                                int nterms, double* dev_out, void* stream) {
  using namespace qs;
  if (!dev_amps || !dev_out || (nterms > 0 && !host_terms)) return fail(QS_EINVAL, "null argument");
  if (dtype != QS_C64 && dtype != QS_C128) return fail(QS_EINVAL, "dtype must be QS_C64 or QS_C128");
  if (((uintptr_t)dev_amps % amp_bytes(dtype)) || ((uintptr_t)dev_out % sizeof(double)))
    return fail(QS_EINVAL, "misaligned amplitude or output pointer");
  if (nqubits < 1 || nqubits > QS_MAXQ) return fail(QS_EINVAL, "nqubits %d not in 1..%d", nqubits, QS_MAXQ);
  if (nreg < 1 || nreg > 65535) return fail(QS_EINVAL, "nreg %d not in 1..65535", nreg);
  if (nterms < 0 || nterms > kStaticTerms)
    return fail(QS_EINVAL, "nterms %d exceeds the static limit of %d terms", nterms, kStaticTerms);
  if ((long long)nreg * nterms > kStaticPartials)
    return fail(QS_EINVAL, "nreg * nterms = %lld exceeds the static scratch of %d partial sums",
                (long long)nreg * nterms, kStaticPartials);
  for (int t = 0; t < nterms; ++t)
    if (nqubits < 64 && ((host_terms[t].x_mask | host_terms[t].z_mask) >> nqubits))
      return fail(QS_EINVAL, "term %d acts on a qubit >= n=%d", t, nqubits);
  cudaStream_t st = (cudaStream_t)stream;
  if (nterms == 0) {
    QS_CUDA(cudaMemsetAsync(dev_out, 0, sizeof(double) * nreg, st));
    return QS_OK;
  }
  double* partials = nullptr;
  QS_TRY(static_partials(&partials));
  int cur_dev = 0;
  cudaGetDevice(&cur_dev);
  // terms ordered by x mask (insertion sort on the stack, stable)
  int order[kStaticTerms];
  for (int t = 0; t < nterms; ++t) {
    int j = t;
    while (j > 0 && host_terms[order[j - 1]].x_mask > host_terms[t].x_mask) {
      order[j] = order[j - 1];
      --j;
    }
    order[j] = t;
  }
  const uint64_t dim = 1ull << nqubits;
  const qs_pauli_term* terms[kStaticTerms];
  for (int t = 0; t < nterms; ++t) terms[t] = &host_terms[order[t]];
  int nslots = 0;
  QS_TRY(expect_launch(dev_amps, dtype, nqubits, nreg, terms, nterms, nullptr, 1, 0, &nslots, st));
  const int nblk = (int)std::max<long long>(
      1, std::min<long long>(expect_blocks(dim), (long long)kStaticPartials / ((long long)nreg * nslots)));
  QS_TRY(expect_launch(dev_amps, dtype, nqubits, nreg, terms, nterms, partials, nblk, nslots, &nslots, st));
  k_expect_final<<<nreg, kFoldThreads, 0, st>>>(partials, nblk, nslots, dev_out);
  if (cudaPeekAtLastError() != cudaSuccess) g_static_addr[cur_dev] = nullptr;  // resolve again next call
  QS_LAUNCHED();
  return QS_OK;
}
