// reduce.cu -- expectation values, lambda = O psi, measurement sampling, reset
// and collapse (sm_103a).
//
// expect (Sec. "Forward Mode"): O = sum_t c_t P_t with P_t a Pauli string.
// For a basis state, P|i> = i^{nY} (-1)^{popc(i & z)} |i ^ x>, so
// <psi|P|psi> = sum_i ph(i) conj(psi_{i^x}) psi_i.  Terms are grouped by their
// x mask; one streaming pass per group reads each amplitude (or each pair
// (i, i^x) once, counting it twice) and accumulates every term of the group in
// FP64.  The sum is pairwise: a thread adds at most kSerialItems items in
// order (the serial base case), warps and blocks combine by balanced trees,
// and a second kernel folds the per-block partials of every term by a
// balanced tree as well (fixed shapes, so results are reproducible run to
// run).  Error bound: (kSerialItems + log2 of the item count) * 2^-53 of the
// sum of the absolute terms.
//
// measure (Sec. "Instructions on Quantum Registers"): the deterministic
// contract of qsim.h -- FP64 probabilities with separately rounded multiply
// and add, left folds over level-0 blocks of 1024 probabilities and level-1
// blocks of 1024 level-0 sums, and a three-level walk per shot.
#include <cmath>
#include <cstring>
#include <map>

#include "common.cuh"

namespace qs {

constexpr int kRedThreads = 256;
constexpr int kSerialItems = 64;  // serial base case of the pairwise expectation sums
constexpr int kGroupTerms = 16;   // terms of one x-mask group handled per launch
constexpr int kObsChunk = 64;     // terms per lambda = O psi launch

struct TermGroup {
  int nt;
  int item_log2;
  int h;                 // highest bit of x (-1 if x == 0)
  uint64_t x;
  uint64_t z[kGroupTerms];
  int ny[kGroupTerms];   // number of Y factors mod 4
};

__device__ __forceinline__ double2 ld_amp(const float2* p, uint64_t i) {
  const float2 v = p[i];
  return make_double2((double)v.x, (double)v.y);
}
__device__ __forceinline__ double2 ld_amp(const double2* p, uint64_t i) { return p[i]; }

__device__ __forceinline__ double term_value(int ny, double s, double zr, double zi) {
  switch (ny & 3) {
    case 0: return s * zr;
    case 1: return -s * zi;
    case 2: return -s * zr;
    default: return s * zi;
  }
}

// grid (blocks_per_reg, nreg); partials[(reg * nt_total + term_base + t) * nblk + block]
template <typename T>
__global__ void __launch_bounds__(kRedThreads)
k_expect_group(const T* __restrict__ psi, uint64_t reg_stride, TermGroup g, double* __restrict__ partials,
               int nt_total, int term_base) {
  const int nblk = gridDim.x;
  const uint64_t r = blockIdx.y;
  const T* p = psi + r * reg_stride;
  const uint64_t items = 1ull << g.item_log2;
  double acc[kGroupTerms];
#pragma unroll
  for (int t = 0; t < kGroupTerms; ++t) acc[t] = 0.0;
  for (uint64_t j = (uint64_t)blockIdx.x * kRedThreads + threadIdx.x; j < items;
       j += (uint64_t)nblk * kRedThreads) {
    uint64_t i = j;
    if (g.h >= 0) i = ((j >> g.h) << (g.h + 1)) | (j & ((1ull << g.h) - 1ull));
    const double2 a = ld_amp(p, i);
    double zr, zi;
    if (g.h >= 0) {
      const double2 b = ld_amp(p, i ^ g.x);
      zr = b.x * a.x + b.y * a.y;
      zi = b.x * a.y - b.y * a.x;
    } else {
      zr = a.x * a.x + a.y * a.y;
      zi = 0.0;
    }
#pragma unroll
    for (int t = 0; t < kGroupTerms; ++t) {
      if (t < g.nt) {
        const double s = (__popcll(i & g.z[t]) & 1) ? -1.0 : 1.0;
        acc[t] += term_value(g.ny[t], s, zr, zi);
      }
    }
  }
  __shared__ double red[kRedThreads / 32][kGroupTerms];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int t = 0; t < kGroupTerms; ++t) {
    double v = acc[t];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0) red[warp][t] = v;
  }
  __syncthreads();
  if (threadIdx.x < g.nt) {
    static_assert(kRedThreads / 32 == 8, "block tree below is written for 8 warps");
    const int t = threadIdx.x;
    const double v = ((red[0][t] + red[1][t]) + (red[2][t] + red[3][t])) +
                     ((red[4][t] + red[5][t]) + (red[6][t] + red[7][t]));
    const double f = g.h >= 0 ? 2.0 : 1.0;
    partials[((r * nt_total) + term_base + threadIdx.x) * nblk + blockIdx.x] = f * v;
  }
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

constexpr int kFoldThreads = 256;

// Pairwise sum of v[0..len) by one CTA of kFoldThreads threads: contiguous
// chunks per thread (binary counter), then a shared-memory tree.  Every thread
// receives the result.
__device__ double block_pairwise(const double* __restrict__ v, int64_t len, double* sh) {
  const int64_t chunk = (len + kFoldThreads - 1) / kFoldThreads;
  const int64_t lo = (int64_t)threadIdx.x * chunk, hi = lo + chunk < len ? lo + chunk : len;
  PairwiseAcc acc;
  for (int64_t i = lo; i < hi; ++i) acc.add(v[i]);
  sh[threadIdx.x] = acc.total();
  __syncthreads();
  for (int w = kFoldThreads / 2; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w) sh[threadIdx.x] = sh[threadIdx.x] + sh[threadIdx.x + w];
    __syncthreads();
  }
  const double r = sh[0];
  __syncthreads();
  return r;
}

// one CTA per register: every term's block partials folded pairwise, then the
// terms' c_t * v_t pairwise in term order.
__global__ void __launch_bounds__(kFoldThreads)
k_expect_final(const double* __restrict__ partials, int nblk, int nt_total, const double* __restrict__ coeff,
               double* __restrict__ out) {
  __shared__ double sh[kFoldThreads];
  const int r = blockIdx.x;
  PairwiseAcc terms;
  for (int t = 0; t < nt_total; ++t) {
    const double v = block_pairwise(partials + ((size_t)r * nt_total + t) * nblk, nblk, sh);
    terms.add(coeff[t] * v);
  }
  if (threadIdx.x == 0) out[r] = terms.total();
}

// blocks per register for the pairwise expectation: at most kSerialItems items per thread
static int expect_blocks(uint64_t items) {
  const uint64_t per_block = (uint64_t)kRedThreads * kSerialItems;
  return (int)std::max<uint64_t>(1, (items + per_block - 1) / per_block);
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

static int grouped(const qs_observable* o, std::vector<std::pair<uint64_t, std::vector<int>>>& groups) {
  std::map<uint64_t, std::vector<int>> m;
  for (int t = 0; t < (int)o->terms.size(); ++t) m[o->terms[t].x_mask].push_back(t);
  groups.assign(m.begin(), m.end());
  return QS_OK;
}

// expectation of registers stored at `data` (uniform: nreg x 2^n, else one register)
int expect_raw(const void* data, int dtype, int n, int nreg, const qs_observable* o, qs_state* ws_owner,
               double* host_out) {
  cudaStream_t st = ws_owner->stream;
  const int nt_total = (int)o->terms.size();
  for (const auto& t : o->terms) {
    if (n < 64 && ((t.x_mask | t.z_mask) >> n)) return fail(QS_EINVAL, "observable acts on a qubit >= n=%d", n);
  }
  std::vector<std::pair<uint64_t, std::vector<int>>> groups;
  grouped(o, groups);
  const uint64_t dim = 1ull << n;
  // every group's items: 2^n (x = 0) or 2^(n-1) pairs; the grid covers the larger
  const int nblk = expect_blocks(dim);
  const size_t part_bytes = sizeof(double) * (size_t)nreg * std::max(1, nt_total) * nblk;
  const size_t coeff_off = (part_bytes + 255) / 256 * 256;
  const size_t out_off = coeff_off + (sizeof(double) * std::max(1, nt_total) + 255) / 256 * 256;
  QS_TRY(ensure_ws(ws_owner, ws_owner->ws, out_off + sizeof(double) * nreg));
  double* partials = (double*)ws_owner->ws.ptr;
  double* dcoeff = (double*)((char*)ws_owner->ws.ptr + coeff_off);
  double* dev_out = (double*)((char*)ws_owner->ws.ptr + out_off);
  // coefficients in the global term order of the partials layout below
  std::vector<double> coeff;
  std::vector<int> order;
  for (auto& g : groups)
    for (int t : g.second) { order.push_back(t); coeff.push_back(o->terms[t].coeff); }
  if (nt_total > 0)
    QS_CUDA(cudaMemcpyAsync(dcoeff, coeff.data(), sizeof(double) * nt_total, cudaMemcpyHostToDevice, st));
  int base = 0;
  for (auto& g : groups) {
    const auto& ids = g.second;
    for (size_t c0 = 0; c0 < ids.size(); c0 += kGroupTerms) {
      TermGroup tg;
      memset(&tg, 0, sizeof(tg));
      tg.x = g.first;
      tg.h = g.first ? 63 - __builtin_clzll(g.first) : -1;
      tg.item_log2 = g.first ? n - 1 : n;
      tg.nt = (int)std::min<size_t>(kGroupTerms, ids.size() - c0);
      for (int t = 0; t < tg.nt; ++t) {
        const auto& term = o->terms[ids[c0 + t]];
        tg.z[t] = term.z_mask;
        tg.ny[t] = __builtin_popcountll(term.x_mask & term.z_mask) & 3;
      }
      dim3 grid(nblk, nreg);
      if (dtype == QS_C64)
        k_expect_group<float2><<<grid, kRedThreads, 0, st>>>((const float2*)data, dim, tg, partials, nt_total, base);
      else
        k_expect_group<double2><<<grid, kRedThreads, 0, st>>>((const double2*)data, dim, tg, partials, nt_total, base);
      QS_LAUNCHED();
      base += tg.nt;
    }
  }
  if (nt_total == 0) {
    QS_CUDA(cudaMemsetAsync(dev_out, 0, sizeof(double) * nreg, st));
  } else {
    k_expect_final<<<nreg, kFoldThreads, 0, st>>>(partials, nblk, nt_total, dcoeff, dev_out);
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

// What a fold adds up: |amplitude|^2 by the contract, or a level's sums.  The
// square of a float is exact in FP64, so one fused multiply-add rounds re*re +
// im*im once, as the contract's multiply, multiply and add do: 2 FP64
// operations instead of 5 with the conversions.
__device__ __forceinline__ double prob(float2 v) {
  const double x = widen(v.x), y = widen(v.y);
  return __fma_rn(x, x, __dmul_rn(y, y));
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
  double t = 0.0, acc = 0.0;
  if (folds) {
    r = (s0 + lane) / a.nshots;
    t = shot_target(a, s0 + lane, r);
    b = shot_block(a, r, t);
    blk[lane] = r * a.nb0 + b;
    acc = start_of(st, r * a.nb0 + b);
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
        // signs of the comparisons by the bit patterns (none is negative), off the FP64 unit;
        // a t that is not finite is never exceeded
        if (found < 0 && __double_as_longlong(acc) > __double_as_longlong(t) && !(__double2hiint(t) >= 0x7ff00000))
          found = ch * 32 + j;
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
// [nreg][nshots] into device indices; scratch: sample_scratch_doubles() doubles
constexpr uint64_t kRunDoubles = 1ull << 25;  // running sums of the probabilities in scratch: at most 256 MiB

// The running sums of every probability cost a second pass over the state and
// 8 bytes an amplitude, a shot without them folds 1024 probabilities: they are
// formed once a level-0 block gets a shot or more on the average, or when a
// register is a single block (whose fold is the running sum).
static bool keep_runs(int n, int nshots) {
  const uint64_t dim = 1ull << n, nb0 = (dim + kF - 1) / kF;
  return nb0 == 1 || (nb0 <= (uint64_t)nshots && dim <= kRunDoubles);
}
// registers sampled together
static int sample_group(int n, int nreg) {
  return (int)std::min<uint64_t>((uint64_t)nreg, std::max<uint64_t>(1, kRunDoubles >> n));
}

size_t sample_scratch_doubles(int n, int nreg, int nshots) {
  const uint64_t dim = 1ull << n, nb0 = (dim + kF - 1) / kF, nb1 = (nb0 + kF - 1) / kF;
  const uint64_t levels = (nb0 > 1 ? 2 * nb0 : 0) + (nb1 > 1 ? 2 * nb1 : 0);
  return (size_t)((levels + (keep_runs(n, nshots) ? dim : 0)) * (uint64_t)sample_group(n, nreg));
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
                       cudaStream_t st) {
  const uint64_t dim = 1ull << n, R = (uint64_t)nreg;
  const uint64_t nb0 = (dim + kF - 1) / kF, nb1 = (nb0 + kF - 1) / kF, len0 = std::min<uint64_t>(dim, kF);
  const bool runs = keep_runs(n, nshots);
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
               double* scratch, cudaStream_t st) {
  const int group = sample_group(n, nreg);
  for (int r = 0; r < nreg; r += group) {
    const int k = std::min(group, nreg - r);
    const char* p = (const char*)data + ((amp_bytes(dtype) * (size_t)r) << n);
    const double* u = dev_u + (size_t)r * nshots;
    int64_t* out = dev_out + (size_t)r * nshots;
    if (dtype == QS_C64) QS_TRY(sample_regs((const float2*)p, n, k, u, nshots, out, scratch, st));
    else QS_TRY(sample_regs((const double2*)p, n, k, u, nshots, out, scratch, st));
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
// from seed (shot j of register r: draw k0 + r nshots + j + 1)
int measure_regs(void* data, int dtype, int n, int nreg, const double* host_u, int nshots, int64_t* host_out,
                 int collapse, qs_state* owner, const uint64_t* seed, uint64_t k0) {
  cudaStream_t st = owner->stream;
  const uint64_t dim = 1ull << n;
  const size_t shots = (size_t)nreg * nshots, scr = sample_scratch_doubles(n, nreg, nshots);
  QS_TRY(ensure_ws(owner, owner->ws, sizeof(double) * (scr + shots) + sizeof(int64_t) * shots + sizeof(double2) + 256));
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
  QS_TRY(sample_dev(data, dtype, n, nreg, du, nshots, dout, dscr, st));
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

__global__ void k_promote(const float2* __restrict__ in, double2* __restrict__ out, uint64_t dim) {
  const uint64_t i = (uint64_t)blockIdx.x * 256 + threadIdx.x;
  if (i >= dim) return;
  const float2 v = in[i];
  out[i] = make_double2((double)v.x, (double)v.y);
}

int promote_to_c128(const void* in, int dtype, double2* out, uint64_t dim, cudaStream_t st) {
  if (dtype == QS_C128) {
    QS_CUDA(cudaMemcpyAsync(out, in, sizeof(double2) * dim, cudaMemcpyDeviceToDevice, st));
    return QS_OK;
  }
  k_promote<<<(unsigned)((dim + 255) / 256), 256, 0, st>>>((const float2*)in, out, dim);
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

struct StaticCoeffs {
  double c[kStaticTerms];
};

__global__ void __launch_bounds__(kFoldThreads)
k_expect_final_static(const double* __restrict__ partials, int nblk, int nt_total,
                      const __grid_constant__ StaticCoeffs co, double* __restrict__ out) {
  __shared__ double sh[kFoldThreads];
  const int r = blockIdx.x;
  PairwiseAcc terms;
  for (int t = 0; t < nt_total; ++t) {
    const double v = block_pairwise(partials + ((size_t)r * nt_total + t) * nblk, nblk, sh);
    terms.add(co.c[t] * v);
  }
  if (threadIdx.x == 0) out[r] = terms.total();
}

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
  long long nblk = expect_blocks(dim);
  nblk = std::max(1LL, std::min(nblk, (long long)kStaticPartials / ((long long)nreg * nterms)));
  StaticCoeffs co;
  memset(&co, 0, sizeof(co));
  int base = 0;
  while (base < nterms) {
    const uint64_t x = host_terms[order[base]].x_mask;
    TermGroup tg;
    memset(&tg, 0, sizeof(tg));
    tg.x = x;
    tg.h = x ? 63 - __builtin_clzll(x) : -1;
    tg.item_log2 = x ? nqubits - 1 : nqubits;
    while (base + tg.nt < nterms && tg.nt < kGroupTerms && host_terms[order[base + tg.nt]].x_mask == x) {
      const qs_pauli_term& term = host_terms[order[base + tg.nt]];
      tg.z[tg.nt] = term.z_mask;
      tg.ny[tg.nt] = __builtin_popcountll(term.x_mask & term.z_mask) & 3;
      co.c[base + tg.nt] = term.coeff;
      ++tg.nt;
    }
    dim3 grid((unsigned)nblk, nreg);
    if (dtype == QS_C64)
      k_expect_group<float2><<<grid, kRedThreads, 0, st>>>((const float2*)dev_amps, dim, tg, partials, nterms, base);
    else
      k_expect_group<double2><<<grid, kRedThreads, 0, st>>>((const double2*)dev_amps, dim, tg, partials, nterms, base);
    QS_LAUNCHED();
    base += tg.nt;
  }
  k_expect_final_static<<<nreg, kFoldThreads, 0, st>>>(partials, (int)nblk, nterms, co, dev_out);
  if (cudaPeekAtLastError() != cudaSuccess) g_static_addr[cur_dev] = nullptr;  // resolve again next call
  QS_LAUNCHED();
  return QS_OK;
}
