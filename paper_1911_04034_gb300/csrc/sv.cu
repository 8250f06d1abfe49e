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

// The four sums of a dense gate whose coefficient parts are all +-2^k (k <= 0): every
// product is exact, so a chain of four equals 2^k times the chain of the signed inputs in
// the same order while no partial sum leaves the normal range.  The first sums of the four
// chains are +-(ar + ai) and +-(ar - ai), so two additions serve all four: 10 instead of
// 16 FP64 operations.  False (nothing done) if an input is nonzero below 2^-959 or above
// 2^1020: inputs of at least 2^-959 are multiples of 2^-1011, so a nonzero sum times 2^k
// (k >= -10) stays normal, and no sum overflows.
__device__ __forceinline__ bool sv_pow2_pair(uint32_t sgn, int sk, double2& a, double2& b) {
  auto bad = [](double v) {
    const uint64_t u = (uint64_t)__double_as_longlong(v);
    const uint32_t h = (uint32_t)(u >> 32) & 0x7fffffffu;
    return (h - (64u << 20)) >= ((0x7fcu - 64u) << 20) && (h | (uint32_t)u) != 0u;
  };
  if (bad(a.x) | bad(a.y) | bad(b.x) | bad(b.y)) return false;
  auto hi = [](double v) { return (uint32_t)__double2hiint(v); };
  auto sbit = [sgn](int q) { return ((sgn >> q) & 1u) << 31; };
  auto sg = [&](int q, double v) { return __hiloint2double((int)(hi(v) ^ sbit(q)), __double2loint(v)); };
  const double sum = __dadd_rn(a.x, a.y), dif = __dsub_rn(a.x, a.y);
  // Zero tests on the words: a double comparison would take the FP64 pipe.
  const bool zs = ((hi(sum) << 1) | (uint32_t)__double2loint(sum)) == 0u;
  const bool zd = ((hi(dif) << 1) | (uint32_t)__double2loint(dif)) == 0u;
  // (+-x) + (+-y) for the chain whose first term is coefficient q: x = a.x, y = a.y for the
  // real chains, the other way round for the imaginary ones.  A zero sum is +0 unless both
  // its terms are -0.
  auto first = [&](int q, bool im) {
    const uint32_t sx = sbit(im ? q + 1 : q), sy = sbit(im ? q : q + 1);  // the signs of a.x and a.y
    const bool same = sx == sy;
    const double m = same ? sum : dif;
    const uint32_t h = (same ? zs : zd) ? ((hi(a.x) ^ sx) & (hi(a.y) ^ sy) & 0x80000000u) : hi(m) ^ sx;
    return __hiloint2double((int)h, __double2loint(m));
  };
  auto scaled = [&](double y) {
    const uint32_t h = hi(y);
    const bool zero = ((h << 1) | (uint32_t)__double2loint(y)) == 0u;
    return zero ? y : __hiloint2double((int)(h + ((uint32_t)sk << 20)), __double2loint(y));
  };
  const double re0 = __dadd_rn(__dadd_rn(first(0, false), sg(2, b.x)), sg(3, b.y));
  const double im0 = __dadd_rn(__dadd_rn(first(4, true), sg(6, b.y)), sg(7, b.x));
  const double re1 = __dadd_rn(__dadd_rn(first(8, false), sg(10, b.x)), sg(11, b.y));
  const double im1 = __dadd_rn(__dadd_rn(first(12, true), sg(14, b.y)), sg(15, b.x));
  a = make_double2(scaled(re0), scaled(im0));
  b = make_double2(scaled(re1), scaled(im1));
  return true;
}

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
        if (g.form != 1 || !sv_pow2_pair(g.sgn, g.sk, a, b)) apply_pair(g.g, a, b);
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
