// gate_common.cuh -- device helpers shared by the two gate kernels (kernels.cu, fast.cu).
#pragma once
#include "launch.h"

namespace qc {

// Asynchronous 16-byte global -> shared copies (the next item's directory entries).
__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
  const uint32_t a = (uint32_t)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(a), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_group 0;\n" ::: "memory"); }
// Waits until at most N of this thread's most recent copy groups are still in flight.
template <int N>
__device__ __forceinline__ void cp_async_wait_group() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory"); }
// Section 3.7: the bound of the running gate, from E after the previous gate.  Every
// CTA evaluates the same rule on the same values (only the post kernel writes them).
__device__ __forceinline__ uint32_t gate_bits(const GateLaunch& L) {
  return (uint32_t)level_bits(L.ctl, next_level(L.ctl, L.P.ctl->E, L.P.ctl->level, L.P.ctl->n64));
}

// The chunk index of the k-th active chunk (or pair): the bits of k deposited into the
// free chunk-index bits, run by run.
__device__ __forceinline__ unsigned long long item_chunk(const GateLaunch& L, unsigned long long k) {
  if (L.nruns < 0) return deposit_bits(k, L.free_mask);
  unsigned long long out = 0;
  for (int i = 0; i < L.nruns; ++i) out |= (k << L.run_shift[i]) & L.run_mask[i];
  return out;
}

// True if the chunk's image is what the encoder would write of its values at S bits under
// `modes`: rewriting it unchanged can be left out.  Word 2 of a directory entry holds the
// mode set its image was chosen from (0: unknown); the smallest image of a larger set is
// the smallest of any subset that has it, and coding decoded values again at the same
// width gives the same bytes.  `hdr`: the image's first header word.
__device__ __forceinline__ bool entry_stands(const Pool& P, const uint32_t* e, uint32_t S, uint32_t modes,
                                             uint32_t& hdr) {
  const uint4 h = *reinterpret_cast<const uint4*>(e);
  const uint32_t first = e[4];
  hdr = first;
  if ((modes & kDefaultModes) != kDefaultModes || (h.z & modes) != modes) return false;
  if (h.y != 0u) {
    if (first >= P.npages) return false;
    hdr = *reinterpret_cast<const uint32_t*>(P.pages + (unsigned long long)first * kPage);
  }
  const uint32_t mode = hdr & 0xffu;
  return mode < M_NMODES && ((modes >> mode) & 1u) != 0u && (mode == M_ZERO || ((hdr >> 8) & 0xffu) == S);
}
__device__ __forceinline__ bool image_stands(const Pool& P, unsigned long long chunk, uint32_t S, uint32_t modes) {
  uint32_t hdr;
  return entry_stands(P, dir_entry(P, chunk), S, modes, hdr);
}

// The four sums of a dense gate whose coefficient parts are all +-2^k (k <= 0): every
// product is exact, so a chain of four equals 2^k times the chain of the signed inputs in
// the same order while no partial sum leaves the normal range.  The first sums of the four
// chains are +-(ar + ai) and +-(ar - ai), so two additions serve all four: 10 instead of
// 16 FP64 operations.  False (nothing done) if an input is nonzero below 2^-959 or at least
// 2^1021: inputs of at least 2^-959 are multiples of 2^-1011, so a nonzero sum times 2^k
// (k >= -10) stays normal, and no sum overflows.
__device__ __forceinline__ bool pow2_pair(uint32_t sgn, int sk, double2& a, double2& b) {
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

}  // namespace qc
