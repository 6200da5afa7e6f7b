// sparse.cu -- sparse (CSR) matrix of a sum of Pauli strings, the matrix
// representation of a Hamiltonian block (Sec. "Matrix Representation";
// App. "Matrix Types": sums of Pauli strings are sparse; benchmarked in
// Sec. "Matrix Representation and AD Performance" as mat(heisenberg(20))).
//
// A term c P with P = i^{popcount(x&z)} X^x Z^z (the convention of qs_expect)
// maps |j> to c i^{popcount(x&z)} (-1)^{popcount(j&z)} |j ^ x>.  Row i of the
// matrix therefore has one candidate column j = i ^ x per distinct x among the
// terms, with value sum over the terms t with x_t = x of
// c_t i^{popcount(x_t & z_t)} (-1)^{popcount(j & z_t)}.  Entries that sum to
// exactly zero are dropped; columns are ascending within a row.
//
// Two passes with a scan between them: the rows' nonzero counts with their
// prefixes inside blocks of 1024 rows, a scan of the block totals, the offsets
// added; then a fill that works out each row again and writes it in column
// order.  FP64 adds are the scarce operation of this part (1/64 of the FP32
// rate), scattered 8-byte stores the wasteful one:
//  - a group of at most kSmallTerms terms takes its value from a table indexed
//    by the terms' signs (formed on the host in the terms' order);
//  - for the other groups (the diagonal of a chain) a thread takes kSegs rows
//    that differ in the top bits only, which share the sum of the leading terms
//    that do not touch those bits;
//  - a row's column order follows from a binary trie of the x masks, walked with
//    the children swapped where the row's bit is 1;
//  - a warp stages its rows' entries as 2-byte codes in shared memory and writes
//    columns and values in order.
// heisenberg(20) (11.2 M nonzeros, 276 MB): counts 40 us, scan 10, fill 135 (bound by
// the walks' chains of dependent shared-memory loads; its stores alone would take
// 42).  Before, with every sum in FP64, a selection of the next column among all and
// a thread's rows stored one by one: 313, 80 and 629 us.
#include <algorithm>
#include <cstring>

#include "common.cuh"

namespace qs {

namespace {

constexpr int kSpMaxGroups = 64;   // distinct x masks (entries per row at most)
constexpr int kSpMaxTerms = 256;
constexpr int kSmallTerms = 3;     // terms of a group with a table of values
constexpr int kTab = 1 << kSmallTerms;
constexpr int kScanThreads = 1024;
constexpr int kSegBits = 2, kSegs = 1 << kSegBits;
constexpr int kFillWarps = 4;

struct SpGroup {
  uint64_t x;
  uint64_t z[kSmallTerms];  // small group: its terms' z masks
  int32_t t0, nt;           // its terms in SpTerms::z / cre / cim
  int32_t lead;             // large group: leading terms without the top kSegBits qubits
  int16_t large;            // large group: its index among them, else -1
  uint16_t nz;              // small group: bit p set if the value of sign pattern p is not zero
  uint64_t seg;             // small group: kSmallTerms bits a segment, the signs of its top bits
};
static_assert(sizeof(SpGroup) % 8 == 0, "records in shared memory");
struct SpTerms {
  int ngroups, nlarge;
  int imag;                        // a large group has a term with an imaginary coefficient
  int root;                        // trie: a node, or 0x80 | group
  SpGroup g[kSpMaxGroups];
  uint32_t node[kSpMaxGroups];     // bit | child with the bit 0 << 8 | child with the bit 1 << 16
  uint64_t z[kSpMaxTerms];
  double cre[kSpMaxTerms], cim[kSpMaxTerms];  // c i^{popcount(x&z)}
};
struct SpTable {
  double2 v[kSpMaxGroups * kTab];
};

__device__ __forceinline__ uint32_t parity(uint64_t v) {
  return __popc((uint32_t)v ^ (uint32_t)(v >> 32)) & 1u;
}
// v + the terms t0 .. t1 - 1 of a large group at column j, in their order
__device__ __forceinline__ double2 add_terms(const SpTerms& T, int t0, int t1, uint64_t j, double2 v) {
  for (int t = t0; t < t1; ++t) {
    const int neg = (int)(parity(j & T.z[t]) << 31);
    v.x += __hiloint2double(__double2hiint(T.cre[t]) ^ neg, __double2loint(T.cre[t]));
    if (T.imag) v.y += __hiloint2double(__double2hiint(T.cim[t]) ^ neg, __double2loint(T.cim[t]));
  }
  return v;
}
// sign pattern of a small group's terms at column j
__device__ __forceinline__ uint32_t signs(const SpGroup& G, uint64_t j) {
  uint32_t p = 0;
#pragma unroll
  for (int t = 0; t < kSmallTerms; ++t)
    if (G.z[t]) p |= parity(j & G.z[t]) << t;
  return p;
}
__device__ __forceinline__ uint32_t seg_signs(const SpGroup& G, int s) {
  return (uint32_t)(G.seg >> (kSmallTerms * s)) & (kTab - 1);
}

// counts of 1024 consecutive rows in each of `segs` segments of the rows, their
// exclusive prefixes inside the block to rowptr and the block totals to sums
__global__ void __launch_bounds__(kScanThreads)
k_sp_rows(const __grid_constant__ SpTerms T, uint64_t dim, int segs, int64_t* __restrict__ rowptr,
          int64_t* __restrict__ sums) {
  __shared__ int wsum[kSegs][kScanThreads / 32];
  const uint64_t seg = dim / segs, low = (uint64_t)blockIdx.x * kScanThreads + threadIdx.x;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int c[kSegs];
#pragma unroll
  for (int s = 0; s < kSegs; ++s) c[s] = 0;
  // a warp without rows does not queue for the FP64 unit (one qubit, 40 terms in two large groups:
  // the call 56 us, 34 without its 31 idle warps)
  const int ngroups = low - lane < dim ? T.ngroups : 0;
  for (int g = 0; g < ngroups; ++g) {
    const SpGroup& G = T.g[g];
    if (G.large < 0) {
      const uint32_t p = signs(G, low ^ G.x);
#pragma unroll
      for (int s = 0; s < kSegs; ++s) c[s] += (G.nz >> (p ^ seg_signs(G, s))) & 1;
    } else {
      const double2 lead = add_terms(T, G.t0, G.t0 + G.lead, low ^ G.x, make_double2(0.0, 0.0));
#pragma unroll
      for (int s = 0; s < kSegs; ++s) {
        if (s >= segs) continue;
        const double2 v = add_terms(T, G.t0 + G.lead, G.t0 + G.nt, (s * seg + low) ^ G.x, lead);
        c[s] += v.x != 0.0 || v.y != 0.0;
      }
    }
  }
  int inc[kSegs];
#pragma unroll
  for (int s = 0; s < kSegs; ++s) {
    if (low >= dim) c[s] = 0;
    inc[s] = c[s];
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, inc[s], o);
      if (lane >= o) inc[s] += v;
    }
    if (lane == 31) wsum[s][warp] = inc[s];
  }
  __syncthreads();
  if (warp < kSegs) {
    const int own = wsum[warp][lane];
    int v = own;
    for (int o = 1; o < 32; o <<= 1) {
      const int u = __shfl_up_sync(0xffffffffu, v, o);
      if (lane >= o) v += u;
    }
    wsum[warp][lane] = v - own;
    if (lane == 31 && warp < segs) sums[warp * (seg / kScanThreads) + blockIdx.x] = v;
  }
  __syncthreads();
#pragma unroll
  for (int s = 0; s < kSegs; ++s)
    if (s < segs && low < dim) rowptr[s * seg + low] = wsum[s][warp] + inc[s] - c[s];
}

// exclusive scan of the block totals by one CTA and the grand total at sums[nb]
__global__ void __launch_bounds__(kScanThreads) k_scan_sums(int64_t* __restrict__ sums, uint64_t nb) {
  __shared__ int64_t wsum[kScanThreads / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int64_t carry = 0;
  for (uint64_t b0 = 0; b0 < nb; b0 += kScanThreads) {
    const uint64_t b = b0 + threadIdx.x;
    const int64_t own = b < nb ? sums[b] : 0;
    int64_t v = own;
    for (int o = 1; o < 32; o <<= 1) {
      const int64_t u = __shfl_up_sync(0xffffffffu, v, o);
      if (lane >= o) v += u;
    }
    if (lane == 31) wsum[warp] = v;
    __syncthreads();
    int64_t before = 0, all = 0;
    for (int w = 0; w < kScanThreads / 32; ++w) {
      if (w < warp) before += wsum[w];
      all += wsum[w];
    }
    if (b < nb) sums[b] = carry + before + v - own;
    carry += all;
    __syncthreads();
  }
  if (threadIdx.x == 0) sums[nb] = carry;
}

__global__ void k_scan_add(int64_t* __restrict__ a, uint64_t n, const int64_t* __restrict__ sums) {
  const uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) a[i] += sums[i / kScanThreads];
  if (i == n - 1) a[n] = sums[(n + kScanThreads - 1) / kScanThreads];
}

// shared memory of k_sp_fill: the groups' records, the trie, the tables; then per
// warp the large groups' leading sums and row values, the entry codes and the small
// groups' sign patterns of the rows' low bits
__host__ __device__ constexpr size_t fill_common(int ngroups) {
  return ((size_t)ngroups * (sizeof(SpGroup) + sizeof(uint32_t) + kTab * sizeof(double2)) + 15) & ~(size_t)15;
}
__host__ __device__ constexpr size_t fill_per_warp(int ngroups, int nlarge) {
  return (size_t)nlarge * 32 * 2 * sizeof(double2) + (size_t)ngroups * 32 * (sizeof(uint16_t) + 1);
}
constexpr size_t kFillSmem = 100 * 1024;  // of a CTA: two an SM
static_assert(fill_common(kSpMaxGroups) + fill_per_warp(kSpMaxGroups, kSpMaxGroups) <= kFillSmem, "one warp always fits");

__global__ void __launch_bounds__(32 * kFillWarps)
k_sp_fill(const __grid_constant__ SpTerms T, const __grid_constant__ SpTable tables, uint64_t dim, int segs,
          const int64_t* __restrict__ rowptr, int64_t* __restrict__ cols, double2* __restrict__ vals) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, ng = T.ngroups, nl = T.nlarge;
  double2* tab = reinterpret_cast<double2*>(smem);
  SpGroup* grp = reinterpret_cast<SpGroup*>(tab + ng * kTab);
  uint32_t* node = reinterpret_cast<uint32_t*>(grp + ng);
  for (int k = threadIdx.x; k < ng * kTab; k += blockDim.x) tab[k] = tables.v[k];
  for (int k = threadIdx.x; k < ng; k += blockDim.x) {
    grp[k] = T.g[k];
    node[k] = T.node[k];
  }
  __syncthreads();
  double2* lead = reinterpret_cast<double2*>(smem + fill_common(ng) + warp * fill_per_warp(ng, nl));
  double2* val = lead + nl * 32;
  uint16_t* code = reinterpret_cast<uint16_t*>(val + nl * 32);
  uint8_t* pat = reinterpret_cast<uint8_t*>(code + ng * 32) + lane;
  const uint64_t seg = dim / segs, row0 = ((uint64_t)blockIdx.x * (blockDim.x >> 5) + warp) * 32;
  if (row0 >= seg) return;
  const bool on = row0 + lane < seg;
  for (int g = 0; g < ng; ++g) {
    const SpGroup& G = T.g[g];
    if (G.large >= 0)
      lead[G.large * 32 + lane] = add_terms(T, G.t0, G.t0 + G.lead, (row0 + lane) ^ G.x, make_double2(0.0, 0.0));
    else
      pat[g * 32] = (uint8_t)signs(G, (row0 + lane) ^ G.x);
  }
  for (int s = 0; s < segs; ++s) {
    const uint64_t r0 = s * seg + row0, i = r0 + lane;
    for (int g = 0; g < ng; ++g) {
      const SpGroup& G = T.g[g];
      if (G.large >= 0)
        val[G.large * 32 + lane] = add_terms(T, G.t0 + G.lead, G.t0 + G.nt, i ^ G.x, lead[G.large * 32 + lane]);
    }
    const int64_t base = rowptr[r0];
    const int total = (int)(rowptr[r0 + 32 < s * seg + seg ? r0 + 32 : s * seg + seg] - base);
    if (on) {
      // the nodes whose second child is still to come are ancestors of one another,
      // numbered from the root down: the next one is the highest bit of `pend`
      int w = (int)(rowptr[i] - base), cur = T.root;
      uint64_t pend = 0;
      for (;;) {
        while (!(cur & 0x80)) {
          const uint32_t nd = node[cur];
          pend |= 1ull << cur;
          cur = (int)(((i >> (nd & 0xffu)) & 1 ? nd >> 16 : nd >> 8) & 0xffu);
        }
        const int g = cur & 0x7f;
        const SpGroup& G = grp[g];
        uint32_t p = 0;
        bool nz;
        if (G.large < 0) {
          p = pat[g * 32] ^ seg_signs(G, s);
          nz = (G.nz >> p) & 1;
        } else {
          const double2 v = val[G.large * 32 + lane];
          nz = v.x != 0.0 || v.y != 0.0;
        }
        if (nz) code[w++] = (uint16_t)(g | (lane << 6) | (p << 11));
        if (!pend) break;
        const int up = 63 - __clzll(pend);
        pend ^= 1ull << up;
        const uint32_t nd = node[up];
        cur = (int)(((i >> (nd & 0xffu)) & 1 ? nd >> 8 : nd >> 16) & 0xffu);
      }
    }
    __syncwarp();
    for (int e = lane; e < total; e += 32) {
      const uint32_t cd = code[e];
      const int g = cd & 63, r = (cd >> 6) & 31;
      const SpGroup& G = grp[g];
      cols[base + e] = (int64_t)((r0 + r) ^ G.x);
      vals[base + e] = G.large < 0 ? tab[g * kTab + (cd >> 11)] : val[G.large * 32 + r];
    }
    __syncwarp();
  }
}

// trie over the x masks of groups idx[a..b) (ascending): a leaf, or a node that
// splits them at their highest differing bit
int build_trie(SpTerms* T, const std::vector<int>& idx, int a, int b, int* count) {
  if (b - a == 1) return 0x80 | idx[a];
  const int bit = 63 - __builtin_clzll(T->g[idx[a]].x ^ T->g[idx[b - 1]].x), me = (*count)++;
  int m = a;
  while (!((T->g[idx[m]].x >> bit) & 1)) ++m;
  const uint32_t l = (uint32_t)build_trie(T, idx, a, m, count), r = (uint32_t)build_trie(T, idx, m, b, count);
  T->node[me] = (uint32_t)bit | (l << 8) | (r << 16);
  return me;
}

// Segments of the rows: below 2^18 rows the GPU is not full and a thread's rows one
// after the other only add latency (eight
// segments at n = 14: counts 85 us and fill 68 us, one: 13 and 14)
int segments(int n) { return n >= 18 ? kSegs : 1; }

int build_terms(const qs_observable* o, int n, SpTerms* T, SpTable* tab) {
  std::memset(T, 0, sizeof(*T));
  std::vector<uint64_t> xs;
  for (const qs_pauli_term& p : o->terms) {
    if (n < 64 && ((p.x_mask | p.z_mask) >> n)) return fail(QS_EINVAL, "a term acts beyond qubit %d", n - 1);
    if (std::find(xs.begin(), xs.end(), p.x_mask) == xs.end()) xs.push_back(p.x_mask);
  }
  if ((int)xs.size() > kSpMaxGroups) return fail(QS_EUNSUPPORTED, "more than %d distinct X patterns", kSpMaxGroups);
  if ((int)o->terms.size() > kSpMaxTerms) return fail(QS_EUNSUPPORTED, "more than %d terms", kSpMaxTerms);
  T->ngroups = (int)xs.size();
  const uint64_t top = segments(n) > 1 ? ~0ull << (n - kSegBits) : 0;
  int t = 0;
  std::vector<int> idx(T->ngroups);
  for (int g = 0; g < T->ngroups; ++g) {
    SpGroup& G = T->g[g];
    idx[g] = g;
    G.x = xs[g];
    G.t0 = t;
    for (const qs_pauli_term& p : o->terms) {
      if (p.x_mask != xs[g]) continue;
      T->z[t] = p.z_mask;
      // c * i^{popcount(x & z)}
      const int ny = __builtin_popcountll(p.x_mask & p.z_mask) & 3;
      const double re[4] = {1, 0, -1, 0}, im[4] = {0, 1, 0, -1};
      T->cre[t] = p.coeff * re[ny];
      T->cim[t] = p.coeff * im[ny];
      ++t;
    }
    G.nt = t - G.t0;
    G.large = -1;
    if (G.nt > kSmallTerms) {
      G.large = (int16_t)T->nlarge++;
      while (G.lead < G.nt && !(T->z[G.t0 + G.lead] & top)) ++G.lead;
      for (int k = G.t0; k < t; ++k) T->imag |= T->cim[k] != 0.0;
      continue;
    }
    for (int k = 0; k < G.nt; ++k) G.z[k] = T->z[G.t0 + k];
    for (int q = 1; q < segments(n); ++q)  // segment 0 has no top bits
      for (int k = 0; k < G.nt; ++k)
        G.seg |= (uint64_t)(__builtin_popcountll(((uint64_t)q << (n - kSegBits)) & G.z[k] & top) & 1) << (kSmallTerms * q + k);
    for (int p = 0; p < kTab; ++p) {
      double re = 0.0, im = 0.0;
      for (int k = 0; k < G.nt; ++k) {
        const double s = (p >> k) & 1 ? -1.0 : 1.0;
        re += s * T->cre[G.t0 + k];
        im += s * T->cim[G.t0 + k];
      }
      tab->v[g * kTab + p] = make_double2(re, im);
      if (re != 0.0 || im != 0.0) G.nz |= (uint16_t)(1 << p);
    }
  }
  std::sort(idx.begin(), idx.end(), [&](int a, int b) { return T->g[a].x < T->g[b].x; });
  int count = 0;
  if (T->ngroups) T->root = build_trie(T, idx, 0, T->ngroups, &count);
  return QS_OK;
}

}  // namespace

}  // namespace qs

using namespace qs;

extern "C" {

int qs_observable_csr_rows(const qs_observable* o, int nqubits, int64_t* dev_rowptr, int64_t* dev_scratch,
                           int64_t* host_nnz, void* stream) {
  if (!o || !dev_rowptr || !dev_scratch || !host_nnz) return fail(QS_EINVAL, "null argument");
  if (nqubits < 1 || nqubits > 34) return fail(QS_EINVAL, "nqubits must be in 1..34");
  SpTerms T;
  SpTable tab;
  QS_TRY(build_terms(o, nqubits, &T, &tab));
  cudaStream_t st = (cudaStream_t)stream;
  const uint64_t dim = 1ull << nqubits, nb = (dim + kScanThreads - 1) / kScanThreads;
  const int segs = segments(nqubits);
  k_sp_rows<<<(unsigned)((dim / segs + kScanThreads - 1) / kScanThreads), kScanThreads, 0, st>>>(T, dim, segs, dev_rowptr,
                                                                                              dev_scratch);
  QS_LAUNCHED();
  k_scan_sums<<<1, kScanThreads, 0, st>>>(dev_scratch, nb);
  QS_LAUNCHED();
  k_scan_add<<<(unsigned)((dim + 255) / 256), 256, 0, st>>>(dev_rowptr, dim, dev_scratch);
  QS_LAUNCHED();
  QS_CUDA(cudaMemcpyAsync(host_nnz, dev_rowptr + dim, sizeof(int64_t), cudaMemcpyDeviceToHost, st));
  QS_CUDA(cudaStreamSynchronize(st));
  return QS_OK;
}

int qs_observable_csr_fill(const qs_observable* o, int nqubits, const int64_t* dev_rowptr, int64_t* dev_cols,
                           double* dev_vals, void* stream) {
  if (!o || !dev_rowptr || !dev_cols || !dev_vals) return fail(QS_EINVAL, "null argument");
  if (nqubits < 1 || nqubits > 34) return fail(QS_EINVAL, "nqubits must be in 1..34");
  SpTerms T;
  SpTable tab;
  QS_TRY(build_terms(o, nqubits, &T, &tab));
  if (T.ngroups == 0) return QS_OK;
  cudaStream_t st = (cudaStream_t)stream;
  const uint64_t dim = 1ull << nqubits;
  const int segs = segments(nqubits);
  // warps of a CTA: as many as keep two CTAs on an SM, at least one
  const size_t common = fill_common(T.ngroups), per = fill_per_warp(T.ngroups, T.nlarge);
  int warps = kFillWarps;
  while (warps > 1 && common + warps * per > kFillSmem) warps >>= 1;
  const size_t smem = common + warps * per;
  // the limit belongs to the function: the same for every observable, as other threads launch theirs
  if (smem > 48 * 1024) QS_CUDA(cudaFuncSetAttribute(k_sp_fill, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kFillSmem));
  const uint64_t rows = (dim / segs + 31) / 32;
  k_sp_fill<<<(unsigned)((rows + warps - 1) / warps), 32 * warps, smem, st>>>(T, tab, dim, segs, dev_rowptr, dev_cols,
                                                                           (double2*)dev_vals);
  QS_LAUNCHED();
  return QS_OK;
}

}  // extern "C"
