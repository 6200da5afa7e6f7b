// bitswap.cu -- a network of SWAP gates on disjoint qubit pairs as one pass over the
// state (sm_103a): the final swap network of a QFT (App. "Extending QBIR").
//
// The network is an involution s of the index bits: amplitude i trades places with
// amplitude s(i).  The index is cut into tile bits (the lowest five and whatever
// they are swapped with, then further bits with their partners up to 2^11
// amplitudes, so that s maps tile bits to tile bits) and outer bits.  The tiles of
// outer index o and s(o) are read into shared memory in rows of 32 amplitudes (256
// bytes) and written to each other's place with their bits swapped; slots are
// XOR-swizzled, as the swapped read walks them with a power-of-two stride.
//
// Bound by HBM: the state once in and once out.  As three controlled X gates a SWAP
// inside tile passes the network of 29 qubits took two further passes of 3.7 ms and
// half of a third; this takes 2.3 ms (3.7 TB/s; 2.6 ms with the slots' banks in conflict,
// 2.9 ms with 512 threads).
#include <algorithm>
#include <cstring>

#include "tiles.cuh"

namespace qs {

namespace {

constexpr int kSwapThreads = 256;
constexpr int kSwapTile = 11;             // tile bits wanted
constexpr int kSwapTileMax = kSwapTile + 1;  // a bit and its partner may overshoot by one

struct SwapArgs {
  float2* psi;
  uint64_t reg_stride, nouter;
  int m;                       // tile bits
  int nseg;                    // runs of consecutive outer bits
  uint8_t tbit[kSwapTileMax];  // register qubit of each tile bit (ascending; the first five are 0..4)
  uint8_t tperm[kSwapTileMax]; // tile bit that each tile bit is swapped with (itself: none)
  uint8_t seg_from[40], seg_to[40], seg_len[40];  // outer index bits -> register qubits
  int npair;
  uint8_t pa[32], pb[32];      // swapped outer index bits
};

// Half a warp reads or writes 16 amplitudes of 8 bytes at a time, one in each pair of
// banks: the lowest four bits of a slot take the XOR of every nibble, so that four lane bits
// that a network sends to neighbouring high bits spread over the banks as they do at home
__device__ __forceinline__ uint32_t swap_slot(uint32_t l) { return l ^ (((l >> 4) ^ (l >> 8)) & 15u); }

__global__ void __launch_bounds__(kSwapThreads) k_bitswap(const __grid_constant__ SwapArgs a) {
  extern __shared__ __align__(16) float2 sm[];
  __shared__ uint32_t rowoff[1 << (kSwapTileMax - 5)];
  __shared__ uint16_t rowperm[1 << (kSwapTileMax - 5)], colperm[32];
  const int m = a.m, rows = 1 << (m - 5);
  auto perm = [&](uint32_t l) {
    uint32_t r = 0;
    for (int k = 0; k < m; ++k) r |= ((l >> k) & 1u) << a.tperm[k];
    return r;
  };
  for (int r = threadIdx.x; r < rows; r += kSwapThreads) {
    uint32_t o = 0;
    for (int k = 5; k < m; ++k) o |= ((uint32_t)(r >> (k - 5)) & 1u) << a.tbit[k];
    rowoff[r] = o;
    rowperm[r] = (uint16_t)perm((uint32_t)r << 5);
  }
  if (threadIdx.x < 32) colperm[threadIdx.x] = (uint16_t)perm(threadIdx.x);
  __syncthreads();
  float2* reg = a.psi + blockIdx.y * a.reg_stride;
  float2* t0 = sm;
  float2* t1 = sm + (1u << m);
  const uint32_t nq = 1u << (m - 1);  // float4 of a tile
  auto base = [&](uint64_t o) {
    uint64_t b = 0;
    for (int s = 0; s < a.nseg; ++s) b |= ((o >> a.seg_from[s]) & ((1ull << a.seg_len[s]) - 1)) << a.seg_to[s];
    return b;
  };
  auto store = [&](float2* dst, const float2* src) {
#pragma unroll 4
    for (uint32_t q = threadIdx.x; q < nq; q += kSwapThreads) {
      const uint32_t l = 2 * q, row = rowperm[l >> 5];
      const float2 u = src[swap_slot(row | colperm[l & 31])], v = src[swap_slot(row | colperm[(l + 1) & 31])];
      *reinterpret_cast<float4*>(dst + rowoff[l >> 5] + (l & 31)) = make_float4(u.x, u.y, v.x, v.y);
    }
  };
  for (uint64_t o = blockIdx.x; o < a.nouter; o += gridDim.x) {
    uint64_t p = o;
    for (int k = 0; k < a.npair; ++k) {
      const uint64_t d = ((o >> a.pa[k]) ^ (o >> a.pb[k])) & 1ull;
      p ^= (d << a.pa[k]) | (d << a.pb[k]);
    }
    if (p < o) continue;  // the CTA of p moves both tiles
    float2* g0 = reg + base(o);
    float2* g1 = reg + base(p);
    constexpr int C = 8;
    for (uint32_t q0 = 0; q0 < nq; q0 += C / 2 * kSwapThreads) {
      float4 v[C];
#pragma unroll
      for (int k = 0; k < C; ++k) {
        const uint32_t q = q0 + threadIdx.x + (k >> 1) * kSwapThreads, l = 2 * q;
        if (q < nq && !((k & 1) && p == o))
          v[k] = *reinterpret_cast<const float4*>(((k & 1) ? g1 : g0) + rowoff[l >> 5] + (l & 31));
      }
#pragma unroll
      for (int k = 0; k < C; ++k) {
        const uint32_t q = q0 + threadIdx.x + (k >> 1) * kSwapThreads, l = 2 * q;
        if (q >= nq || ((k & 1) && p == o)) continue;
        float2* t = (k & 1) ? t1 : t0;
        t[swap_slot(l)] = make_float2(v[k].x, v[k].y);
        t[swap_slot(l + 1)] = make_float2(v[k].z, v[k].w);
      }
    }
    __syncthreads();
    store(g1, t0);
    if (p != o) store(g0, t1);
    __syncthreads();
  }
}

}  // namespace

// SWAP gates (pairs of qubits, disjoint) on nreg registers of 2^n complex64
// amplitudes, n >= kBitSwapMinQubits
int launch_bitswap(float2* psi, int n, int nreg, const std::vector<std::pair<int, int>>& swaps, cudaStream_t st) {
  int partner[QS_MAXQ];
  for (int q = 0; q < QS_MAXQ; ++q) partner[q] = q;
  for (const auto& s : swaps) {
    partner[s.first] = s.second;
    partner[s.second] = s.first;
  }
  if (n < kBitSwapMinQubits || n > 32) return fail(QS_EINVAL, "swap pass over %d qubits", n);
  SwapArgs a;
  std::memset(&a, 0, sizeof(a));
  uint64_t tile = 0;
  for (int q = 0; q < n; ++q)
    if (q < 5 || __builtin_popcountll(tile) < kSwapTile) tile |= (1ull << q) | (1ull << partner[q]);
  int tidx[QS_MAXQ], oidx[QS_MAXQ], no = 0;
  for (int q = 0; q < n; ++q) {
    if ((tile >> q) & 1) {
      tidx[q] = a.m;
      a.tbit[a.m++] = (uint8_t)q;
    } else {
      if (no == 0 || ((tile >> (q - 1)) & 1)) {
        a.seg_from[a.nseg] = (uint8_t)no;
        a.seg_to[a.nseg++] = (uint8_t)q;
      }
      ++a.seg_len[a.nseg - 1];
      oidx[q] = no++;
    }
  }
  for (int k = 0; k < a.m; ++k) a.tperm[k] = (uint8_t)tidx[partner[a.tbit[k]]];
  for (int q = 0; q < n; ++q)
    if (!((tile >> q) & 1) && partner[q] > q) {
      a.pa[a.npair] = (uint8_t)oidx[q];
      a.pb[a.npair++] = (uint8_t)oidx[partner[q]];
    }
  a.psi = psi;
  a.reg_stride = 1ull << n;
  a.nouter = 1ull << no;
  const size_t smem = sizeof(float2) * 2 << a.m;
  // the limit belongs to the function: always the largest tile's, never one that another thread's
  // launch exceeds
  if (smem > 48 * 1024)
    QS_CUDA(cudaFuncSetAttribute(k_bitswap, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)(sizeof(float2) * 2 << kSwapTileMax)));
  int dev = 0, sms = 0, per_sm = 0;
  QS_CUDA(cudaGetDevice(&dev));
  QS_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  QS_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_bitswap, kSwapThreads, smem));
  const unsigned grid = (unsigned)std::min<uint64_t>(a.nouter, (uint64_t)sms * std::max(1, per_sm));
  for (int r = 0; r < nreg; r += 65535) {
    SwapArgs b = a;
    b.psi = psi + ((uint64_t)r << n);
    k_bitswap<<<dim3(grid, (unsigned)std::min(65535, nreg - r)), kSwapThreads, smem, st>>>(b);
    QS_LAUNCHED();
  }
  return QS_OK;
}

}  // namespace qs
