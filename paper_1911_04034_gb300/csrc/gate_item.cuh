// gate_item.cuh -- one work item of the general gate path, and the bookkeeping after a gate:
// what k_gate and k_gate_batch (kernels.cu) and k_run (run.cu) share.
#pragma once
#include "launch.h"
#include "gate_common.cuh"

// Resident CTAs per SM that the fused kernel's register budget is sized for (the grid
// follows the occupancy the build achieves).
#ifndef QC_GATE_MIN_CTAS
#define QC_GATE_MIN_CTAS 3
#endif

namespace qc {

__host__ __device__ __forceinline__ uint32_t imgcap(int kc) { return round16(max_image_bytes(kc)); }
// staging buffer of the codec entry points: any forced image fits
__host__ __device__ __forceinline__ uint32_t codedcap(int kc) { return round16(max_coded_bytes(kc)); }
__host__ __device__ __forceinline__ uint32_t pagelist_words(int kc) { return (max_pages(kc) + 3u) & ~3u; }

// Each image buffer keeps 16 spare bytes: the decoder's bit window reads up to 8 bytes
// past the end of a residual stream.
__host__ __device__ __forceinline__ uint32_t imgbuf(int kc) { return imgcap(kc) + 16u; }

// ------------------------------------------------------------- the gate -- //
// Shared-memory layout of the fused kernel and the per-CTA state it carries between
// work items (page cache, byte counters, scan-buffer parity).
struct GateSmem {
  uint64_t *tile0, *tile1;
  uint8_t *img0, *img1;
  uint32_t* ent[2][2];    // two sets of copies of the two directory entries (header, page
                          // ids or image): the current item's and the next item's
  ScanSmem* s;
  long long* ph;          // per-phase cycles, [6] = last clock (profiling)
  int* oom;
  uint32_t* np;
};
// Per-CTA counters that only thread 0 updates (kept in shared memory so that they
// hold no registers during the codec phases).
struct CtaAcc {
  long long dE;
  long long dn64;          // change in the number of images at S = 64
  unsigned long long rd, wr;
  unsigned long long key;  // block-cache key of the running item
  unsigned long long fast, rest;  // items at S <= 32 encoded as a pair of STREAM images or alone, and the others
};
struct GateCta {
  CtaCache cc;
  CtaAcc* acc;
  unsigned int err;        // thread 0: the error word as read during the previous item
  int pp;
  int cur;                        // directory-entry buffer set of the current item
  unsigned long long next_item;   // item whose entries were prefetched into set cur ^ 1
};

// Bulk asynchronous shared -> global copy (one page of a new image); the issuing thread
// later waits until the source has been read before the buffer is reused.
__device__ __forceinline__ void bulk_store(void* gmem, const void* smem, uint32_t bytes) {
  const uint32_t a = (uint32_t)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;\n" ::"l"(gmem), "r"(a), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_read() { asm volatile("cp.async.bulk.wait_group.read 0;\n" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;\n" ::: "memory"); }
// Makes this thread's earlier shared-memory writes visible to bulk copies.
__device__ __forceinline__ void fence_to_bulk() { asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory"); }

// Writes the two new images of a work item: pages by bulk copies (a lane of warp 0 per
// page), inline images and the directory entries by plain stores (warp 1).  All threads
// call it; the images in shared memory must stay untouched until bulk_wait_read.
__device__ __forceinline__ void commit_images(const Pool& P, unsigned long long c0, const uint8_t* img0, uint32_t n0,
                                              const uint32_t* pg0, uint32_t np0, bool has1, unsigned long long c1,
                                              const uint8_t* img1, uint32_t n1, const uint32_t* pg1, uint32_t np1,
                                              uint32_t md0, uint32_t md1) {
  if (threadIdx.x < 32u) {
    const uint32_t tot = np0 + (has1 ? np1 : 0u);
    bool issued = false;
    for (uint32_t k = threadIdx.x; k < tot; k += 32u) {
      const bool second = k >= np0;
      const uint32_t q = second ? k - np0 : k, bytes = second ? n1 : n0;
      const uint32_t len = min((uint32_t)kPage, bytes - q * kPage);
      if (!issued) fence_to_bulk();
      bulk_store(P.pages + (unsigned long long)(second ? pg1[q] : pg0[q]) * kPage,
                 (second ? img1 : img0) + q * kPage, len);
      issued = true;
    }
    if (issued) bulk_commit();
  } else if (threadIdx.x < 64u) {
    const uint32_t lane = threadIdx.x - 32u;
    for (int w = 0; w < (has1 ? 2 : 1); ++w) {
      uint32_t* e = dir_entry(P, w ? c1 : c0);
      const uint32_t bytes = w ? n1 : n0, np = w ? np1 : np0;
      const uint32_t* pg = w ? pg1 : pg0;
      if (np == 0u) {
        const uint4* src = reinterpret_cast<const uint4*>(w ? img1 : img0);
        for (uint32_t u = lane; u < bytes / 16u; u += 32u) reinterpret_cast<uint4*>(e + 4)[u] = src[u];
      } else {
        for (uint32_t q = lane; q < np; q += 32u) e[4 + q] = pg[q];
      }
      if (lane == 0) *reinterpret_cast<uint4*>(e) = make_uint4(bytes, np, w ? md1 : md0, 0u);
    }
  }
}

// Pulls one page of a later item's image into L2 (no data returned to the SM).
__device__ __forceinline__ void prefetch_l2_page(const void* gmem) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;\n" ::"l"(gmem), "r"((uint32_t)kPage) : "memory");
}

__device__ __forceinline__ GateSmem gate_smem(uint8_t* smem, int kc, uint32_t dir_words, long long* ph, int* oom,
                                               uint32_t* np) {
  GateSmem m;
  m.tile0 = reinterpret_cast<uint64_t*>(smem);
  m.tile1 = m.tile0 + tile_words(kc);
  m.img0 = reinterpret_cast<uint8_t*>(m.tile1 + tile_words(kc));
  m.img1 = m.img0 + imgbuf(kc);
  m.ent[0][0] = reinterpret_cast<uint32_t*>(m.img1 + imgbuf(kc));
  m.ent[0][1] = m.ent[0][0] + dir_words;
  m.ent[1][0] = m.ent[0][1] + dir_words;
  m.ent[1][1] = m.ent[1][0] + dir_words;
  m.s = reinterpret_cast<ScanSmem*>(m.ent[1][1] + dir_words);
  m.ph = ph;
  m.oom = oom;
  m.np = np;
  return m;
}

// Warp 0 loads this CTA's page cache of the simulator into shared memory (empty
// unless this CTA already worked for it in the same launch).
__device__ __forceinline__ void cta_begin(const Pool& P, GateCta& st, bool prof, long long* ph) {
  if (threadIdx.x < 32u) {
    const uint32_t n = P.cache_n[blockIdx.x];
    for (uint32_t q = threadIdx.x; q < n; q += 32u) st.cc.ids[q] = P.cache[(size_t)blockIdx.x * kCacheCap + q];
    if (threadIdx.x == 0) *st.cc.n = n;
    __syncwarp();
  }
  if (threadIdx.x == 0) {
    st.acc->dE = 0;
    st.acc->dn64 = 0;
    st.acc->rd = st.acc->wr = 0;
    st.acc->fast = st.acc->rest = 0;
  }
  // the error word as the launch finds it: after a device error even a CTA's first item
  // stops before it touches the pool
  st.err = threadIdx.x == 0 ? *(volatile unsigned int*)&P.ctl->err : 0u;
  st.pp = 0;
  st.cur = 0;
  st.next_item = ~0ull;
  if (prof && threadIdx.x == 0) {
    for (int k = 0; k < 6; ++k) ph[k] = 0;
    ph[6] = clock64();
  }
}

// Warp 0: hands the CTA's page cache and counters back to the simulator.
__device__ __forceinline__ void cta_end(const GateLaunch& L, GateCta& st, const long long* ph) {
  if (threadIdx.x >= 32u) return;
  const uint32_t n = *st.cc.n;
  for (uint32_t q = threadIdx.x; q < n; q += 32u) L.P.cache[(size_t)blockIdx.x * kCacheCap + q] = st.cc.ids[q];
  if (threadIdx.x != 0) return;
  DevCtl* ctl = L.P.ctl;
  if (L.prof)
    for (int k = 0; k < 6; ++k)
      if (ph[k]) atomicAdd(&ctl->phase_cycles[k], (unsigned long long)ph[k]);
  L.P.cache_n[blockIdx.x] = n;
  if (st.acc->dE) atomicAdd(&ctl->dE, (unsigned long long)st.acc->dE);
  if (st.acc->dn64) atomicAdd(reinterpret_cast<unsigned long long*>(&ctl->dn64), (unsigned long long)st.acc->dn64);
  if (st.acc->rd) atomicAdd(&ctl->bytes_in, st.acc->rd);
  if (st.acc->wr) atomicAdd(&ctl->bytes_out, st.acc->wr);
}

// One work item (two chunks) of a gate: stage, decode, apply, encode, commit.
// Returns false if the simulator's error word is set (nothing more to do for it).
// PREF: nx is the CTA's next item of the same gate (~0 if none); its directory
// entries are fetched asynchronously during this item and its pages pulled into L2.
template <int VPT, bool PREF>
__device__ __forceinline__ bool gate_item(const GateLaunch& L, unsigned long long item, unsigned long long nx,
                                          uint32_t S, unsigned long long serial, bool bc_on, const GateSmem& m,
                                          GateCta& st) {
  const int kc = L.P.kc;
  const uint32_t A = 1u << kc;
  const uint32_t cap = imgcap(kc);
  const Pool& P = L.P;
  DevCtl* ctl = P.ctl;
  const uint32_t dw4 = P.dir_words / 4u;  // 16-byte units of a directory entry
#define QC_PHASE(k)                     \
  if (L.prof && threadIdx.x == 0) {     \
    const long long now_ = clock64();   \
    m.ph[k] += now_ - m.ph[6];          \
    m.ph[6] = now_;                     \
  }
  // one barrier that also broadcasts thread 0's view of the error word (and publishes
  // the entries prefetched during the previous item); the previous item's bulk page
  // stores must have read the image buffers before they are refilled
  bulk_wait_read();
  if (PREF) cp_async_wait_all();
  if (__syncthreads_or(threadIdx.x == 0 && st.err != 0u)) return false;
  const bool have_entries = PREF && st.next_item == item;
  if (PREF && st.next_item != ~0ull) st.cur ^= 1;
  st.next_item = ~0ull;
  uint32_t* ent0 = m.ent[st.cur][0];
  uint32_t* const ent1 = m.ent[st.cur][1];
  bool solo = false;  // only the chunk of row L.solo is rewritten: it takes the place of the first
  // the item's chunks (recomputed at commit rather than kept through the codec)
  auto chunks_of = [&](unsigned long long& x0, unsigned long long& x1) {
    if (L.pair) {
      x0 = item_chunk(L, item) | L.hi_vals;
      x1 = x0 | L.pair_bit;
      if (solo && L.solo == 1) x0 = x1;
    } else {
      x0 = item_chunk(L, 2ull * item) | L.hi_vals;
      x1 = 2ull * item + 1 < L.nact ? (item_chunk(L, 2ull * item + 1) | L.hi_vals) : 0ull;
    }
  };
  unsigned long long c0, c1;
  chunks_of(c0, c1);
  bool has1 = L.pair || 2ull * item + 1 < L.nact;
  // stage 1: both directory entries (warp 0 and warp 1), unless prefetched
  if (!have_entries) {
    if (threadIdx.x < 32u) {
      const uint4* src = reinterpret_cast<const uint4*>(dir_entry(P, c0));
      for (uint32_t i = threadIdx.x; i < dw4; i += 32u) reinterpret_cast<uint4*>(ent0)[i] = src[i];
    } else if (threadIdx.x < 64u && has1) {
      const uint4* src = reinterpret_cast<const uint4*>(dir_entry(P, c1));
      for (uint32_t i = threadIdx.x - 32u; i < dw4; i += 32u) reinterpret_cast<uint4*>(ent1)[i] = src[i];
    }
    __syncthreads();
  }
  // the next item's entries (asynchronously, into the other set); no other CTA writes
  // them, and this item touches only its own chunks
  unsigned long long nc0 = 0, nc1 = 0;
  bool nhas1 = false;
  if (PREF && nx != ~0ull) {
    if (L.pair) {
      nc0 = item_chunk(L, nx) | L.hi_vals;
      nc1 = nc0 | L.pair_bit;
      nhas1 = true;
    } else {
      nc0 = item_chunk(L, 2ull * nx) | L.hi_vals;
      nhas1 = 2ull * nx + 1 < L.nact;
      nc1 = nhas1 ? (item_chunk(L, 2ull * nx + 1) | L.hi_vals) : 0ull;
    }
    if (threadIdx.x < 32u) {
      const uint4* src = reinterpret_cast<const uint4*>(dir_entry(P, nc0));
      for (uint32_t i = threadIdx.x; i < dw4; i += 32u) cp_async16(reinterpret_cast<uint4*>(m.ent[st.cur ^ 1][0]) + i, src + i);
    } else if (threadIdx.x < 64u && nhas1) {
      const uint4* src = reinterpret_cast<const uint4*>(dir_entry(P, nc1));
      for (uint32_t i = threadIdx.x - 32u; i < dw4; i += 32u)
        cp_async16(reinterpret_cast<uint4*>(m.ent[st.cur ^ 1][1]) + i, src + i);
    }
    cp_async_commit();
    st.next_item = nx;
  }
  uint32_t np0 = ent0[1], np1 = has1 ? ent1[1] : 0u;
  uint32_t b0 = ent0[0], b1 = has1 ? ent1[0] : 0u;
  if (b0 > cap || b1 > cap || np0 > max_pages(kc) || np1 > max_pages(kc) || (np0 == 0u && b0 > inline_cap(kc)) ||
      (np1 == 0u && b1 > inline_cap(kc)) || (b0 & 15u) || (b1 & 15u)) {
    if (threadIdx.x == 0) atomicOr(&ctl->err, (unsigned)E_CORRUPT);
    return false;
  }
  // An all-zero chunk maps to an all-zero chunk under any gate (signed zeros are
  // stored as +0), and its image does not depend on the bound: skip it.
  const bool z0 = np0 == 0 && b0 == 16u && ent0[4] == 0u;
  const bool z1 = !has1 || (np1 == 0 && b1 == 16u && ent1[4] == 0u);
  if (z0 && z1) {
    if (threadIdx.x == 0) st.acc->rd += b0 + b1;
    QC_PHASE(5);
    return true;
  }
  // Two constant chunks (ZERO or CONST images, held inline) under a cross-chunk gate
  // with no in-chunk controls: every pair sees the same inputs, so one pair gives
  // both output chunks, which are constant again.
  if (L.pair && L.lo_mask == 0u && inline_cap(kc) >= 32u && np0 == 0u && np1 == 0u &&
      (z0 || (ent0[4] & 0xffu) == M_CONST) && (z1 || (ent1[4] & 0xffu) == M_CONST)) {
    if (threadIdx.x == 0) {
      st.acc->rd += b0 + b1;
      double2 a = make_double2(0.0, 0.0), b = make_double2(0.0, 0.0);
      if (!z0) a = make_double2(__longlong_as_double(((const long long*)(ent0 + 8))[0]),
                                __longlong_as_double(((const long long*)(ent0 + 8))[1]));
      if (!z1) b = make_double2(__longlong_as_double(((const long long*)(ent1 + 8))[0]),
                                __longlong_as_double(((const long long*)(ent1 + 8))[1]));
      apply_pair(L.g, a, b);
      uint32_t h0[8], h1[8];
      const uint32_t n0 = const_image((uint64_t)__double_as_longlong(a.x), (uint64_t)__double_as_longlong(a.y), S, h0);
      const uint32_t n1 = const_image((uint64_t)__double_as_longlong(b.x), (uint64_t)__double_as_longlong(b.y), S, h1);
      if (n0 == 0u || n1 == 0u) {
        atomicOr(&ctl->err, (unsigned)E_NONFINITE);
      } else {
        uint32_t* w0 = dir_entry(P, c0);
        uint32_t* w1 = dir_entry(P, c1);
        for (int k = 0; k < 8; ++k) {
          w0[4 + k] = h0[k];
          w1[4 + k] = h1[k];
        }
        w0[0] = n0;
        w1[0] = n1;
        w0[2] = w1[2] = L.modes;
        st.acc->dE += (long long)n0 + (long long)n1 - (long long)b0 - (long long)b1;
        auto wide = [](uint32_t h) { return ((h >> 8) & 0xffu) == 64u ? 1ll : 0ll; };
        st.acc->dn64 += wide(h0[0]) + wide(h1[0]) - (z0 ? 0ll : wide(ent0[4])) - (z1 ? 0ll : wide(ent1[4]));
        st.acc->wr += n0 + n1;
      }
    }
    QC_PHASE(5);
    return true;
  }
  // chunk modes: the mode set, or Solution C's set plus the trials the selector granted
  uint32_t md0 = L.modes, md1 = L.modes;
  if (L.sel_dec) {
    md0 = sel_modes(L.sel_dec[2ull * item]);
    md1 = has1 ? sel_modes(L.sel_dec[2ull * item + 1ull]) : kDefaultModes;
  }
  // A diagonal gate between chunks whose other row is an exact copy (T, CZ, a controlled
  // phase): the copy's image stays, if it is what the encoder would write, and only the
  // other chunk is decoded and encoded: half the item's codec work.
  if (L.solo >= 0 && !L.bc && !L.trace) {
    uint32_t hdr;
    solo = entry_stands(P, L.solo ? ent0 : ent1, S, L.solo ? md0 : md1, hdr);
  }
  if (solo) {
    const uint32_t mdc = L.solo ? md0 : md1;  // the copy would have run these trials
    if (threadIdx.x == 0) {
      if ((mdc >> M_SPLIT) & 1u) atomicAdd(&ctl->split_trials, 1ull);
      if ((mdc >> M_PALETTE) & 1u) atomicAdd(&ctl->palette_trials, 1ull);
    }
    if (L.solo) {
      ent0 = ent1;
      np0 = np1;
      b0 = b1;
      md0 = md1;
    }
    has1 = false;
    np1 = b1 = 0u;
    if (L.solo ? z1 : z0) {  // zeros stay zeros; their trials are counted as above
      if (threadIdx.x == 0) {
        st.acc->rd += b0;
        if ((md0 >> M_SPLIT) & 1u) atomicAdd(&ctl->split_trials, 1ull);
        if ((md0 >> M_PALETTE) & 1u) atomicAdd(&ctl->palette_trials, 1ull);
      }
      QC_PHASE(5);
      return true;
    }
  }
  if (threadIdx.x == 0) st.acc->rd += b0 + b1;
  // stage 2: both images in one pass (inline ones from the entry copies); page data is
  // copied asynchronously, so every copy of the thread is in flight at once
  {
    const uint32_t u0 = b0 >> 4, u1 = b1 >> 4;
    constexpr uint32_t upp = kPage / 16;
    for (uint32_t u = threadIdx.x; u < u0 + u1; u += kThreads) {
      const bool second = u >= u0;
      const uint32_t uu = second ? u - u0 : u;
      const uint32_t* ent = second ? ent1 : ent0;
      uint4* dst = reinterpret_cast<uint4*>(second ? m.img1 : m.img0) + uu;
      if ((second ? np1 : np0) == 0u) *dst = reinterpret_cast<const uint4*>(ent + 4)[uu];
      else cp_async16(dst, reinterpret_cast<const uint4*>(P.pages + (unsigned long long)ent[4 + uu / upp] * kPage) + (uu % upp));
    }
    cp_async_commit();
    cp_async_wait_all();
  }
  __syncthreads();
  if (threadIdx.x < 32u) free_pages_warp(P, st.cc, ent0 + 4, np0, ent1 + 4, has1 ? np1 : 0u);
  QC_PHASE(0);
  // the input images coded at 64 bits (thread 0), for the controller's count
  const long long old64 = threadIdx.x == 0 ? (long long)(m.img0[1] == 64u) + (long long)(has1 && m.img1[1] == 64u) : 0ll;
  // the next item's pages into L2: warp 0 for its first chunk, warp 1 for its second
  // (each warp waits only for the entry copies it issued itself)
  auto prefetch_next = [&]() {
    if (PREF && st.next_item != ~0ull && threadIdx.x < 64u && (threadIdx.x < 32u || nhas1) &&
        !(solo && (int)(threadIdx.x >> 5) != L.solo)) {
      cp_async_wait_all();
      __syncwarp();
      const uint32_t* e = m.ent[st.cur ^ 1][threadIdx.x >> 5];
      const uint32_t q = min(e[1], max_pages(kc));
      for (uint32_t k = threadIdx.x & 31u; k < q; k += 32u) {
        const uint32_t pid = e[4 + k];
        if (pid < P.npages) prefetch_l2_page(P.pages + (unsigned long long)pid * kPage);
      }
    }
  };
  // Section 3.4: an earlier item of this gate with the same two input blocks left its
  // outputs in the block cache (confirmed byte by byte); otherwise claim the line
  bool bc_hit = false, bc_claim = false;
  uint32_t n0 = 0, n1 = 1;
  if (L.bc && bc_on && has1) {
    const unsigned long long key = bc_key(m.img0, b0, m.img1, b1, *m.s);
    if (threadIdx.x == 0) st.acc->key = key;
    BcLine* line = reinterpret_cast<BcLine*>(L.bc + (key % (unsigned long long)kBcLines) * bc_line_bytes(cap));
    uint8_t* ldat = reinterpret_cast<uint8_t*>(line) + kBcHead;
    if (threadIdx.x == 0) {
      const unsigned long long t = atomicAdd(&line->tag, 0ull);
      int flag = 0;
      if (t == ((serial << 2) | 2ull)) {
        __threadfence();
        if (__ldcg(&line->key) == key && __ldcg(&line->len[0]) == b0 && __ldcg(&line->len[1]) == b1) flag = 1;
      } else if ((t >> 2) != serial && atomicCAS(&line->tag, t, (serial << 2) | 1ull) == t) {
        flag = 2;
      }
      m.s->bc_flag = flag;
      atomicAdd(&ctl->bc_gate_lookups, 1ull);
    }
    __syncthreads();
    const int flag = m.s->bc_flag;
    const uint4* lin = reinterpret_cast<const uint4*>(ldat);
    if (flag == 1) {
      const uint32_t u0 = b0 >> 4, u1 = b1 >> 4, c16 = cap >> 4;
      bool eq = true;
      for (uint32_t u = threadIdx.x; u < u0 + u1; u += kThreads) {
        const uint4 a = u < u0 ? reinterpret_cast<const uint4*>(m.img0)[u] : reinterpret_cast<const uint4*>(m.img1)[u - u0];
        const uint4 b = __ldcg(lin + (u < u0 ? u : c16 + (u - u0)));
        eq &= a.x == b.x && a.y == b.y && a.z == b.z && a.w == b.w;
      }
      if (__syncthreads_and(eq)) {
        n0 = __ldcg(&line->len[2]);
        n1 = __ldcg(&line->len[3]);
        const uint32_t v0 = n0 >> 4, v1 = n1 >> 4;
        for (uint32_t u = threadIdx.x; u < v0 + v1; u += kThreads) {
          if (u < v0) reinterpret_cast<uint4*>(m.img0)[u] = __ldcg(lin + 2u * c16 + u);
          else reinterpret_cast<uint4*>(m.img1)[u - v0] = __ldcg(lin + 3u * c16 + (u - v0));
        }
        __syncthreads();
        bc_hit = true;
        if (threadIdx.x == 0) atomicAdd(&ctl->bc_gate_hits, 1ull);
      }
    } else if (flag == 2) {
      const uint32_t u0 = b0 >> 4, u1 = b1 >> 4, c16 = cap >> 4;
      uint4* lout = reinterpret_cast<uint4*>(ldat);
      for (uint32_t u = threadIdx.x; u < u0 + u1; u += kThreads) {
        if (u < u0) lout[u] = reinterpret_cast<const uint4*>(m.img0)[u];
        else lout[c16 + (u - u0)] = reinterpret_cast<const uint4*>(m.img1)[u - u0];
      }
      bc_claim = true;
    }
  }
  if (bc_hit) {
    prefetch_next();
  } else {
  // two STREAM images of 32-bit width (the common case once the run is lossy) decode
  // together, sharing barriers; anything else chunk by chunk
  const bool paired = has1 && kThreads * VPT == 2u * A;
  bool ok0, ok1;
  if (paired && stream32_image(m.img0, b0, kc) && stream32_image(m.img1, b1, kc)) {
    ok0 = ok1 = decode_stream32_pair<VPT>(m.img0, m.img1, 2u * A, m.tile0, m.tile1, *m.s, st.pp);
  } else {
    ok0 = decode_block<VPT>(m.img0, b0, kc, m.tile0, *m.s, st.pp);
    ok1 = has1 ? decode_block<VPT>(m.img1, b1, kc, m.tile1, *m.s, st.pp) : true;
  }
  prefetch_next();
  QC_PHASE(1);
  if (!ok0 || !ok1) {
    if (threadIdx.x == 0) atomicOr(&ctl->err, (unsigned)E_CORRUPT);
    return false;
  }
  // apply the gate to every amplitude pair whose in-chunk control bits match
  double2* t0 = reinterpret_cast<double2*>(m.tile0);
  double2* t1 = reinterpret_cast<double2*>(m.tile1);
  if (solo) {
    const double2 z = make_double2(0.0, 0.0);  // the other amplitude has a zero coefficient
    for (uint32_t i = threadIdx.x; i < A; i += kThreads) {
      if ((i & L.lo_mask) != L.lo_vals) continue;
      const uint32_t pi = tile_amp(i);
      t0[pi] = L.solo ? apply_rows23(L.g, z, t0[pi]) : apply_rows01(L.g, t0[pi], z);
    }
  } else if (L.pair) {
    for (uint32_t i = threadIdx.x; i < A; i += kThreads) {
      if ((i & L.lo_mask) != L.lo_vals) continue;
      const uint32_t pi = tile_amp(i);
      double2 a = t0[pi], b = t1[pi];
      apply_pair(L.g, a, b);
      t0[pi] = a;
      t1[pi] = b;
    }
  } else {
    const uint32_t tb = 1u << L.target, lowm = tb - 1u;
    const uint32_t tot = has1 ? A : A / 2u;  // pairs over both tiles
    for (uint32_t q = threadIdx.x; q < tot; q += kThreads) {
      const uint32_t p = q & (A / 2u - 1u);
      double2* tt = (q < A / 2u) ? t0 : t1;
      const uint32_t i0 = ((p & ~lowm) << 1) | (p & lowm);
      if ((i0 & L.lo_mask) != L.lo_vals) continue;
      const uint32_t p0 = tile_amp(i0), p1 = tile_amp(i0 | tb);
      double2 a = tt[p0], b = tt[p1];
      apply_pair(L.g, a, b);
      tt[p0] = a;
      tt[p1] = b;
    }
  }
  __syncthreads();
  QC_PHASE(2);
  SelCtx sel;
  sel.gfeat = L.gfeat;
  sel.S_gate = S;
  sel.trace = L.trace;
  sel.trace_n = L.trace_n;
  sel.trace_cap = L.trace_cap;
  sel.split_trials = &ctl->split_trials;
  sel.palette_trials = &ctl->palette_trials;
  {
    const uint4 h = reinterpret_cast<const uint4*>(m.img0)[0];  // the pre-gate image header (still staged)
    sel.prev_hdr[0] = h.x; sel.prev_hdr[1] = h.y; sel.prev_hdr[2] = h.z; sel.prev_hdr[3] = h.w;
    sel.prev_len = b0;
  }
  // both chunks in one pass when neither needs a SPLIT or PALETTE trial, a training
  // record or 64-bit widths; otherwise (or if a chunk holds a subnormal) chunk by chunk
  const bool enc_paired = paired && S <= 32u && !L.trace && ((md0 | md1) >> M_SPLIT) == 0u &&
                          encode_pair32<VPT>(m.tile0, m.tile1, kc, S, md0, m.img0, m.img1, cap, *m.s, st.pp,
                                             &ctl->err, n0, n1);
  if (!enc_paired) {
    n0 = encode_block<VPT>(m.tile0, kc, S, -1, md0, m.img0, cap, *m.s, st.pp, &ctl->err, &sel);
    if (has1) {
      const uint4 h = reinterpret_cast<const uint4*>(m.img1)[0];
      sel.prev_hdr[0] = h.x; sel.prev_hdr[1] = h.y; sel.prev_hdr[2] = h.z; sel.prev_hdr[3] = h.w;
      sel.prev_len = b1;
      n1 = encode_block<VPT>(m.tile1, kc, S, -1, md1, m.img1, cap, *m.s, st.pp, &ctl->err, &sel);
    }
  }
  QC_PHASE(3);
  if (threadIdx.x == 0 && S <= 32u) {
    if (enc_paired || solo) ++st.acc->fast;
    else ++st.acc->rest;
  }
  // the error word for the next item's check (the load completes while this one ends)
  if (threadIdx.x == 0) st.err = *(volatile unsigned int*)&ctl->err;
  // a claimed cache line receives the outputs and is published for the rest of the gate
  if (bc_claim && n0 != 0u && n1 != 0u) {
    const unsigned long long key = st.acc->key;
    BcLine* line = reinterpret_cast<BcLine*>(L.bc + (key % (unsigned long long)kBcLines) * bc_line_bytes(cap));
    uint8_t* ldat = reinterpret_cast<uint8_t*>(line) + kBcHead;
    const uint32_t v0 = n0 >> 4, v1 = n1 >> 4, c16 = cap >> 4;
    uint4* lout = reinterpret_cast<uint4*>(ldat);
    for (uint32_t u = threadIdx.x; u < v0 + v1; u += kThreads) {
      if (u < v0) lout[2u * c16 + u] = reinterpret_cast<const uint4*>(m.img0)[u];
      else lout[3u * c16 + (u - v0)] = reinterpret_cast<const uint4*>(m.img1)[u - v0];
    }
    if (threadIdx.x == 0) {
      line->key = key;
      line->len[0] = b0;
      line->len[1] = b1;
      line->len[2] = n0;
      line->len[3] = n1;
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) atomicExch(&line->tag, (serial << 2) | 2ull);
  }
  }
  if (n0 == 0u || n1 == 0u) return false;
  fence_to_bulk();  // every thread's image writes, before the barrier below, for the bulk page stores
  if (threadIdx.x < 32u) {
    const uint32_t q0 = pages_for(n0, kc), q1 = has1 ? pages_for(n1, kc) : 0u;
    const bool ok = alloc_pages_warp(P, st.cc, ent0 + 4, q0, ent1 + 4, q1);
    if (threadIdx.x == 0) {
      m.np[0] = q0;
      m.np[1] = q1;
      if (!ok) atomicOr(&ctl->err, (unsigned)E_OOM);
      m.oom[0] = !ok;
    }
  }
  __syncthreads();
  if (m.oom[0]) return false;
  {
    unsigned long long x0, x1;
    chunks_of(x0, x1);
    commit_images(P, x0, m.img0, n0, ent0 + 4, m.np[0], has1, x1, m.img1, n1, ent1 + 4, m.np[1], md0, md1);
  }
  if (threadIdx.x == 0) {
    const uint32_t i0 = ent0[0], i1 = has1 ? ent1[0] : 0u;  // the old image lengths (entry copies)
    st.acc->dE += (long long)n0 - (long long)i0 + (has1 ? (long long)n1 - (long long)i1 : 0ll);
    st.acc->dn64 += (long long)(m.img0[1] == 64u) + (long long)(has1 && m.img1[1] == 64u) - old64;
    st.acc->wr += n0 + (has1 ? n1 : 0u);
  }
  __syncthreads();
  QC_PHASE(4);

  return true;
#undef QC_PHASE
}

// X between chunks (a cross-chunk target, both rows exact copies, no control inside a
// chunk): every amplitude of one chunk takes its partner's place in the other, so two
// images that stand as the encoder would write them are exchanged by exchanging their
// directory entries; any other item is left to the general path.  One warp; false: nothing
// changed.  `coded` counts the chunk encodings a trial count would have seen (none for two
// constant chunks held inline).
__device__ __forceinline__ bool swap_item(const GateLaunch& L, unsigned long long item, uint32_t S,
                                          unsigned long long& coded) {
  const Pool& P = L.P;
  const uint32_t lane = threadIdx.x & 31u, dw4 = P.dir_words / 4u;
  const unsigned long long c0 = item_chunk(L, item) | L.hi_vals;
  uint32_t* const e0 = dir_entry(P, c0);
  uint32_t* const e1 = dir_entry(P, c0 | L.pair_bit);
  uint32_t h0, h1;
  const bool s0 = entry_stands(P, e0, S, L.modes, h0), s1 = entry_stands(P, e1, S, L.modes, h1);
  if (!s0 || !s1) return false;
  if ((h0 & 0xffu) > M_CONST || (h1 & 0xffu) > M_CONST || (e0[1] | e1[1]) != 0u) coded += 2ull;
  __syncwarp();  // every lane has read what the exchange overwrites
  for (uint32_t i = lane; i < dw4; i += 32u) {
    const uint4 a = reinterpret_cast<const uint4*>(e0)[i], b = reinterpret_cast<const uint4*>(e1)[i];
    reinterpret_cast<uint4*>(e0)[i] = b;
    reinterpret_cast<uint4*>(e1)[i] = a;
  }
  __syncwarp();
  return true;
}
__device__ __forceinline__ void count_swap_trials(const GateLaunch& L, DevCtl* ctl, unsigned long long coded) {
  if (coded && ((L.modes >> M_SPLIT) & 1u)) atomicAdd(&ctl->split_trials, coded);
  if (coded && ((L.modes >> M_PALETTE) & 1u)) atomicAdd(&ctl->palette_trials, coded);
}

// After a gate: free pages back to the stack, then the controller bookkeeping.
// grid_ctas: the CTAs of the gate's general-kernel launch (no other CTA's cache holds
// pages).  Called by one block of 1024 threads.
__device__ __forceinline__ void post_body(const Pool& P, const CtlParams& cp, int grid_ctas) {
  DevCtl* ctl = P.ctl;
  __shared__ unsigned long long s_top;
  __shared__ int s_skip;
  if (threadIdx.x == 0) {
    // after a device error (the pool ran dry, a corrupt image ...) the handle is
    // finished: no bookkeeping, and never a stack index from a top below 0
    const long long top = *(volatile long long*)&ctl->top;
    s_skip = *(volatile unsigned int*)&ctl->err != 0u || top < 0;
    s_top = s_skip ? 0ull : (unsigned long long)top;
  }
  __syncthreads();
  if (s_skip) return;
  // The page caches of the launch's CTAs, back to the stack: a warp reads the counts of 32
  // CTAs with one load, takes the stack slots of them all with one atomic and visits only
  // those that hold ids.  Bound by a few dependent L2 latencies.  (Testing every one of the 128 slots
  // of every CTA the chip holds, one atomic per 32 slots, took 24 us a gate whatever the
  // gate's size; this saves 16 us of them on a state of 8 chunk pairs, 11 us at 456 CTAs.)
  const uint32_t lane = threadIdx.x & 31u, below = (1u << lane) - 1u, wid = threadIdx.x >> 5;
  const int warps = (int)(blockDim.x >> 5);
  for (int b0 = 0; b0 < grid_ctas; b0 += 32 * warps) {  // CTA b0 + wid + warps * lane is this lane's
    const int b = b0 + (int)wid + warps * (int)lane;
    const uint32_t mine = b < grid_ctas ? min(P.cache_n[b], (uint32_t)kCacheCap) : 0u;
    uint32_t todo = __ballot_sync(0xffffffffu, mine != 0u);
    uint32_t sum = mine;  // the warp's ids take consecutive slots, in lane order
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const uint32_t u = __shfl_up_sync(0xffffffffu, sum, d);
      if (lane >= (uint32_t)d) sum += u;
    }
    unsigned long long base = 0;
    if (lane == 31 && sum) base = atomicAdd(&s_top, (unsigned long long)sum);
    base = __shfl_sync(0xffffffffu, base, 31);
    while (todo) {  // two CTAs at a time: eight loads in flight per lane
      uint32_t id[2][kCacheCap / 32], n[2];
      unsigned long long at[2];
#pragma unroll
      for (int w = 0; w < 2; ++w) {
        const int src = todo ? __ffs((int)todo) - 1 : 0;
        const uint32_t have = todo ? 1u : 0u;
        todo &= todo - 1u;
        n[w] = have * __shfl_sync(0xffffffffu, mine, src);
        at[w] = base + __shfl_sync(0xffffffffu, sum - mine, src);
        const uint32_t* ids = P.cache + (size_t)(b0 + (int)wid + warps * src) * kCacheCap;
#pragma unroll
        for (int k = 0; k < kCacheCap / 32; ++k) id[w][k] = 32u * k + lane < n[w] ? ids[32u * k + lane] : 0u;
      }
#pragma unroll
      for (int w = 0; w < 2; ++w)
#pragma unroll
        for (int k = 0; k < kCacheCap / 32; ++k)
          if (32u * k + lane < n[w]) {
            if (at[w] + 32u * k + lane < P.npages) P.stack[at[w] + 32u * k + lane] = id[w][k];
            else atomicOr(&ctl->err, (unsigned)E_CORRUPT);
          }
    }
    if (mine) P.cache_n[b] = 0;
  }
  const unsigned long long nf = ctl->nfreed;
  for (unsigned long long i = threadIdx.x; i < ((nf + 31ull) & ~31ull); i += blockDim.x) {
    const bool has = i < nf;
    const uint32_t m = __ballot_sync(0xffffffffu, has);
    unsigned long long base = 0;
    if (lane == 0 && m) base = atomicAdd(&s_top, (unsigned long long)__popc(m));
    base = __shfl_sync(0xffffffffu, base, 0);
    if (has) {
      const unsigned long long at = base + __popc(m & below);
      if (at < P.npages) P.stack[at] = P.freed[i];
      else atomicOr(&ctl->err, (unsigned)E_CORRUPT);
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    ctl->top = (long long)s_top;
    ctl->nfreed = 0;
    ctl->ndefer = 0;
    ctl->fast_all = 0u;
    const int lvl = next_level(cp, ctl->E, ctl->level, ctl->n64);
    const int S = level_bits(cp, lvl);
    if (lvl > 0 && ctl->switch_gate < 0) ctl->switch_gate = (long long)ctl->gates;
    if (S < 64) {
      ctl->lb_sum += cp.delta[lvl - 1];
      ctl->lb_prod *= (1.0 - cp.delta[lvl - 1]);
    }
    ctl->level = lvl;
    ctl->S_last = S;
    ctl->E += ctl->dE;
    ctl->dE = 0;
    ctl->n64 += ctl->dn64;
    ctl->dn64 = 0;
    if (ctl->E > ctl->Emax) ctl->Emax = ctl->E;
    ctl->gates += 1;
    // block cache: pause it after kBcZeroGates gates in a row with lookups and no hit
    // (Section 3.4 switches it off when the hit rate stays zero), probe again later
    const unsigned long long lk = ctl->bc_gate_lookups, hit = ctl->bc_gate_hits;
    ctl->bc_lookups += lk;
    ctl->bc_hits += hit;
    ctl->bc_gate_lookups = ctl->bc_gate_hits = 0;
    if (ctl->bc_off) {
      ctl->bc_off -= 1u;
    } else if (lk) {
      ctl->bc_zero_streak = hit ? 0u : ctl->bc_zero_streak + 1u;
      if (ctl->bc_zero_streak >= kBcZeroGates) {
        ctl->bc_off = kBcPause;
        ctl->bc_zero_streak = 0u;
      }
    }
    const unsigned long long in_use = P.npages - s_top - ctl->wc_pages;  // pages holding images
    if (in_use > ctl->peak_pages) ctl->peak_pages = in_use;
  }
}

template <typename K>
inline cudaError_t prep(K kernel, size_t smem) {
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
}

#define QC_VPT_DISPATCH(kc, ...)                          \
  switch (vpt_for(kc)) {                                  \
    case 1: { constexpr int V = 1; __VA_ARGS__; } break;  \
    case 2: { constexpr int V = 2; __VA_ARGS__; } break;  \
    case 4: { constexpr int V = 4; __VA_ARGS__; } break;  \
    case 8: { constexpr int V = 8; __VA_ARGS__; } break;  \
    case 16: { constexpr int V = 16; __VA_ARGS__; } break; \
    default: return cudaErrorInvalidValue;                \
  }

}  // namespace qc
