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

}  // namespace qc
