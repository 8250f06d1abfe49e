// sv.cu -- the uncompressed state vector (sm_103a): several gates per pass over memory.
//
// A CTA owns a tile of 2^T amplitudes in shared memory: the tile's index bits are the
// low L qubits (contiguous 2^L * 16 byte runs in memory) and up to T - L higher ones, the
// targets of the group's non-diagonal gates.  It loads the tile, applies every gate of
// the group in order and stores it.  A diagonal gate needs no partner, so its target may
// be any qubit; controls may be anywhere.
//
// Bound: FP64 (two multiply-adds a clock and SM).  A dense gate costs 16 FP64 operations a
// pair in the kept-term sums and 10 in the +-2^k form below; the tile's 32 bytes of
// traffic per amplitude are paid once per group.  27 qubits, one random-circuit layer (36
// gates, 17 of them sqrt(X) / sqrt(Y)): one launch and one pass per gate 54.4 ms, grouped
// 33.6 ms (the FP64 operations alone take 25 ms).
#include "launch.h"
#include "gate_common.cuh"

namespace qc {

constexpr int kSvThreads = 256;

// State index of tile index i, less the tile's base.
__device__ __forceinline__ unsigned long long sv_offset(const SvGroup& G, uint32_t i) {
  unsigned long long o = i & ((1u << G.L) - 1u);
  for (int j = 0; j < G.nhi; ++j) o |= (unsigned long long)((i >> (G.L + j)) & 1u) << G.hi[j];
  return o;
}

__global__ void __launch_bounds__(kSvThreads) k_sv_group(double2* psi, const __grid_constant__ SvGroup G) {
  extern __shared__ __align__(16) double2 s_tile[];
  unsigned long long base = (unsigned long long)blockIdx.x << G.L;
  for (int j = 0; j < G.nhi; ++j) {  // a zero bit at each of the tile's high qubits, lowest first
    const unsigned long long low = (1ull << G.hi[j]) - 1ull;
    base = ((base & ~low) << 1) | (base & low);
  }
  const uint32_t A = 1u << G.T;
  // the gates that change anything in this tile (kSvMaxGates = 32 bits)
  uint32_t todo = 0u;
  for (int k = 0; k < G.ngates; ++k) {
    const SvGate& g = G.g[k];
    const uint32_t row = g.target < 0 ? (uint32_t)(base >> g.tbit) & 1u : 0u;
    if ((base & g.out_mask) == g.out_vals && (g.target >= 0 || !((g.copy >> row) & 1u))) todo |= 1u << k;
  }
  if (!todo) return;
  for (uint32_t i = threadIdx.x; i < A; i += kSvThreads)
    if ((i & G.need_mask) == G.need_vals) cp_async16(s_tile + i, psi + (base | sv_offset(G, i)));
  cp_async_commit();
  cp_async_wait_all();
  __syncthreads();
  for (; todo; todo &= todo - 1u) {
    const SvGate& g = G.g[__ffs((int)todo) - 1];
    if (g.form == 2) {  // diagonal: each amplitude by itself
      const double2 z = make_double2(0.0, 0.0);
      if (g.target < 0) {
        const bool second = (base >> g.tbit) & 1ull;
        for (uint32_t i = threadIdx.x; i < A; i += kSvThreads)
          if ((i & g.lo_mask) == g.lo_vals)
            s_tile[i] = second ? apply_rows23(g.g, z, s_tile[i]) : apply_rows01(g.g, s_tile[i], z);
      } else {
        const uint32_t tb = 1u << g.target, lowm = tb - 1u;
        for (uint32_t p = threadIdx.x; p < A / 2u; p += kSvThreads) {
          const uint32_t i = ((p & ~lowm) << 1) | (p & lowm);
          if ((i & g.lo_mask) != g.lo_vals) continue;
          if (!(g.copy & 1u)) s_tile[i] = apply_rows01(g.g, s_tile[i], z);
          if (!(g.copy & 2u)) s_tile[i | tb] = apply_rows23(g.g, z, s_tile[i | tb]);
        }
      }
    } else {
      const uint32_t tb = 1u << g.target, lowm = tb - 1u;
      for (uint32_t p = threadIdx.x; p < A / 2u; p += kSvThreads) {
        const uint32_t i = ((p & ~lowm) << 1) | (p & lowm);
        if ((i & g.lo_mask) != g.lo_vals) continue;
        double2 a = s_tile[i], b = s_tile[i | tb];
        if (g.form != 1 || !pow2_pair(g.sgn, g.sk, a, b)) apply_pair(g.g, a, b);
        s_tile[i] = a;
        s_tile[i | tb] = b;
      }
    }
    __syncthreads();
  }
  for (uint32_t i = threadIdx.x; i < A; i += kSvThreads)
    if ((i & G.need_mask) == G.need_vals) psi[base | sv_offset(G, i)] = s_tile[i];
}

// Tile bits: 2^12 amplitudes (64 KB, three CTAs an SM) where that leaves 2^9 CTAs or more,
// down to 2^9, below which a CTA's share of a gate is shorter than a launch.
int sv_tile_log2(int n) {
  const int t = n - 9 < 9 ? 9 : (n - 9 > kSvMaxTile ? kSvMaxTile : n - 9);
  return t < n ? t : n;
}
// Of them the low qubits: runs of 512 bytes in the largest tiles, 256 in the others.
int sv_low_bits(int T) {
  const int l = T - 7 < 4 ? 4 : T - 7;
  return l < T ? l : T;
}

cudaError_t launch_sv_group(double* psi, int n, const SvGroup& G, cudaStream_t st) {
  const size_t smem = sizeof(double2) << G.T;
  const cudaError_t e = cudaFuncSetAttribute(k_sv_group, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  k_sv_group<<<1u << (n - G.T), kSvThreads, smem, st>>>(reinterpret_cast<double2*>(psi), G);
  return cudaGetLastError();
}

}  // namespace qc
