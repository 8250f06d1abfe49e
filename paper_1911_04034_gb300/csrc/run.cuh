// run.cuh -- whole circuits of small states in one launch (k_run).
#pragma once
#include "gate_item.cuh"

namespace qc {

// Small states: a gate's work is shorter than the launches that carry it (gate kernels and
// bookkeeping, 12 to 30 us a gate), so one launch runs a whole circuit.  Each CTA takes its
// share of a step's chunk pairs, the simulator's CTAs meet at a counter in device memory,
// and the last to arrive does the bookkeeping and releases the others.  Every CTA is
// resident (a cooperative launch) and every wait is bounded (E_TIMEOUT, site 4) by a number of
// polls that grows with the pairs a CTA may have to itself (see run_polls): in a batch one CTA
// may hold all the chunks of a circuit that are not zero and take seconds over 32 gates, while
// the others wait.  (Counting finished items and waiting anew while the count moves needs no
// such rule, but made every step a tenth of a microsecond longer: 14-qubit random circuit 1.86
// -> 1.88 ms.)  Page ids
// freed by a CTA's items stay with it between steps, up to job.keep of them (counted in
// wc_pages like the streaming kernel's); the rest goes to the freed list.
//
// A step is one gate while the error bound may still change (Section 3.7 needs every
// gate's byte count before the next).  Once it cannot, a step is a group of gates that
// leave every pair of chunks to itself: gates inside chunks, diagonal gates anywhere, and
// gates on one cross-chunk target.  Values are truncated and coded after each gate, for its
// byte count and pages, but decoded once and written once a group, and the CTAs meet once.
// Lossy random circuits, a streaming, a general and a bookkeeping launch per gate -> whole
// circuits: 12 qubits in 2^8-amplitude chunks 22.5 -> 5.3 us a gate, 17 in 2^9 32.6 -> 8.1, 18 in
// 2^10 44.3 -> 10.0, 19 in 2^11 71.4 -> 14.6 (one gate a step: 14.1, 17.5, 24.0, 28.2).

// What a step's gates changed, per gate (shared memory, thread 0 of a CTA writes).
struct RunSums {
  long long dE[kRunGroup], dn64[kRunGroup], dpages[kRunGroup];
};

// Asynchronous copy of gate record k (all threads).
__device__ __forceinline__ void run_fetch(const RunJob& job, int k, GateLaunch* dst) {
  const uint4* src = reinterpret_cast<const uint4*>(job.gates + k);
  for (uint32_t i = threadIdx.x; i < sizeof(GateLaunch) / 16u; i += kThreads)
    cp_async16(reinterpret_cast<uint4*>(dst) + i, src + i);
  cp_async_commit();
}

// The gates [k, k + G) on chunks c0 and c1 (has1: c1 exists).  rec[b] holds record k (if
// `reload`, it has to be fetched again), rec[b ^ 1] is free.  False: a device error is set.
template <int VPT>
__device__ __forceinline__ bool run_item(const Pool& P, GateLaunch* rec, int b, const RunJob& job, int k, int G,
                                         unsigned long long c0, unsigned long long c1, bool has1, uint32_t S,
                                         bool reload, const GateSmem& m, GateCta& st, RunSums& sums) {
  const int kc = P.kc;
  const uint32_t A = 1u << kc, cap = imgcap(kc), dw4 = P.dir_words / 4u;
  DevCtl* ctl = P.ctl;
  auto active = [&](const GateLaunch& L, unsigned long long c) {
    return (c & ~(L.free_mask | L.pair_bit)) == L.hi_vals;
  };
  bulk_wait_read();  // the previous item's page stores have read the image buffers
  if (__syncthreads_or(threadIdx.x == 0 && st.err != 0u)) return false;
  if (G == 1 && !active(rec[b], c0) && !(has1 && active(rec[b], c1))) return true;
  if (reload) run_fetch(job, k, rec + b);
  uint32_t* const ent0 = m.ent[0][0];
  uint32_t* const ent1 = m.ent[0][1];
  if (threadIdx.x < 32u) {
    const uint4* src = reinterpret_cast<const uint4*>(dir_entry(P, c0));
    for (uint32_t i = threadIdx.x; i < dw4; i += 32u) reinterpret_cast<uint4*>(ent0)[i] = src[i];
  } else if (threadIdx.x < 64u && has1) {
    const uint4* src = reinterpret_cast<const uint4*>(dir_entry(P, c1));
    for (uint32_t i = threadIdx.x - 32u; i < dw4; i += 32u) reinterpret_cast<uint4*>(ent1)[i] = src[i];
  }
  __syncthreads();
  const uint32_t np0 = ent0[1], np1 = has1 ? ent1[1] : 0u;
  uint32_t n0 = ent0[0], n1 = has1 ? ent1[0] : 0u;  // lengths of the images as they stand
  if (n0 > cap || n1 > cap || np0 > max_pages(kc) || np1 > max_pages(kc) || (np0 == 0u && n0 > inline_cap(kc)) ||
      (np1 == 0u && n1 > inline_cap(kc)) || (n0 & 15u) || (n1 & 15u)) {
    if (threadIdx.x == 0) atomicOr(&ctl->err, (unsigned)E_CORRUPT);
    return false;
  }
  // stands: the encoder would write the same image again; wide: coded at 64 bits; a chunk of
  // zeros stays one under any gate
  uint32_t h0 = 0u, h1 = 0u;
  bool std0 = entry_stands(P, ent0, S, kDefaultModes, h0), std1 = has1 && entry_stands(P, ent1, S, kDefaultModes, h1);
  if (np0 != 0u && ent0[4] < P.npages) h0 = *reinterpret_cast<const uint32_t*>(P.pages + (unsigned long long)ent0[4] * kPage);
  if (np1 != 0u && ent1[4] < P.npages) h1 = *reinterpret_cast<const uint32_t*>(P.pages + (unsigned long long)ent1[4] * kPage);
  bool z0 = np0 == 0u && n0 == 16u && ent0[4] == 0u, z1 = !has1 || (np1 == 0u && n1 == 16u && ent1[4] == 0u);
  bool wide0 = !z0 && ((h0 >> 8) & 0xffu) == 64u, wide1 = !z1 && ((h1 >> 8) & 0xffu) == 64u;
  if (z0 && z1) {
    if (threadIdx.x == 0) st.acc->rd += n0 + n1;
    return true;
  }
  bool dec0 = false, dec1 = false, dirty0 = false, dirty1 = false;
  bool img0 = false, img1 = false;  // the image buffer holds the whole image of the tile's values
  double2* const t0 = reinterpret_cast<double2*>(m.tile0);
  double2* const t1 = reinterpret_cast<double2*>(m.tile1);
  // one turn per gate, which codes its result for the byte counts alone unless it is the
  // last, and one more for the images still to be written
  for (int g = 0; g <= G; ++g) {
    const bool write = g >= G - 1;
    bool on0, on1, both = false;  // the chunks this turn rewrites
    uint32_t r0 = 0u, r1 = 0u;
    if (g == G) {
      on0 = dirty0 && !img0;
      on1 = dirty1 && !img1;
      if (!on0 && !on1) break;
    } else {
      cp_async_wait_all();
      __syncthreads();  // record g has arrived; the previous gate is done with its record
      const GateLaunch& L = rec[(b + g) & 1];
      if (g + 1 < G) run_fetch(job, k + g + 1, rec + ((b + g + 1) & 1));
      on0 = active(L, c0);
      on1 = has1 && active(L, c1);
      r0 = L.pair && (c0 & L.pair_bit) != 0ull ? 1u : 0u;
      r1 = L.pair && (c1 & L.pair_bit) != 0ull ? 1u : 0u;
      both = L.pair && !L.diag;  // c1 is c0's partner
      if (both) {
        if (!on0 || (z0 && z1)) continue;
      } else {
        // a row that is an exact copy leaves an image that stands; zeros stay zeros
        on0 = on0 && !z0 && !(L.pair && ((L.copy >> r0) & 1u) && std0);
        on1 = on1 && !z1 && !(L.pair && ((L.copy >> r1) & 1u) && std1);
        if (!on0 && !on1) continue;
      }
    }
    const GateLaunch& L = rec[(b + g) & 1];  // (read only for g < G)
    // two constant chunks under a single cross-chunk gate (see gate_item)
    if (G == 1 && g == 0 && L.pair && L.lo_mask == 0u && inline_cap(kc) >= 32u && np0 == 0u && np1 == 0u &&
        (z0 || (ent0[4] & 0xffu) == M_CONST) && (z1 || (ent1[4] & 0xffu) == M_CONST)) {
      if (threadIdx.x == 0) {
        st.acc->rd += n0 + n1;
        double2 x = make_double2(0.0, 0.0), y = make_double2(0.0, 0.0);
        if (!z0) x = make_double2(__longlong_as_double(((const long long*)(ent0 + 8))[0]),
                                  __longlong_as_double(((const long long*)(ent0 + 8))[1]));
        if (!z1) y = make_double2(__longlong_as_double(((const long long*)(ent1 + 8))[0]),
                                  __longlong_as_double(((const long long*)(ent1 + 8))[1]));
        apply_pair(L.g, x, y);
        uint32_t w0[8], w1[8];
        const uint32_t l0 = const_image((uint64_t)__double_as_longlong(x.x), (uint64_t)__double_as_longlong(x.y), S, w0);
        const uint32_t l1 = const_image((uint64_t)__double_as_longlong(y.x), (uint64_t)__double_as_longlong(y.y), S, w1);
        if (l0 == 0u || l1 == 0u) {
          atomicOr(&ctl->err, (unsigned)E_NONFINITE);
        } else {
          uint32_t* d0 = dir_entry(P, c0);
          uint32_t* d1 = dir_entry(P, c1);
          for (int q = 0; q < 8; ++q) {
            d0[4 + q] = w0[q];
            d1[4 + q] = w1[q];
          }
          d0[0] = l0;
          d1[0] = l1;
          d0[2] = d1[2] = kDefaultModes;
          sums.dE[0] += (long long)l0 + (long long)l1 - (long long)n0 - (long long)n1;
          sums.dn64[0] += (((w0[0] >> 8) & 0xffu) == 64u) + (((w1[0] >> 8) & 0xffu) == 64u) - (long long)wide0 - (long long)wide1;
          st.acc->wr += l0 + l1;
        }
      }
      return true;
    }
    // decode what is needed for the first time
    const bool need0 = on0 && !dec0, need1 = on1 && !dec1;
    if (need0 || need1) {
      const uint32_t u0 = need0 ? n0 >> 4 : 0u, u1 = need1 ? n1 >> 4 : 0u;
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
      __syncthreads();
      bool ok = true;
      if (need0 && need1 && kThreads * VPT == 2u * A && stream32_image(m.img0, n0, kc) && stream32_image(m.img1, n1, kc)) {
        ok = decode_stream32_pair<VPT>(m.img0, m.img1, 2u * A, m.tile0, m.tile1, *m.s, st.pp);
      } else {
        for (int w = 0; w < 2; ++w)
          if (w ? need1 : need0)
            ok = decode_block<VPT>(w ? m.img1 : m.img0, w ? n1 : n0, kc, w ? m.tile1 : m.tile0, *m.s, st.pp) && ok;
      }
      if (!ok) {
        if (threadIdx.x == 0) atomicOr(&ctl->err, (unsigned)E_CORRUPT);
        return false;
      }
      if (threadIdx.x == 0) st.acc->rd += (need0 ? n0 : 0u) + (need1 ? n1 : 0u);
      dec0 |= need0;
      dec1 |= need1;
    }
    // the gate on every amplitude pair whose in-chunk control bits match
    if (g < G && both) {
      for (uint32_t i = threadIdx.x; i < A; i += kThreads) {
        if ((i & L.lo_mask) != L.lo_vals) continue;
        const uint32_t pi = tile_amp(i);
        double2 x = t0[pi], y = t1[pi];
        if (!L.pow2 || !pow2_pair(L.sgn, L.sk, x, y)) apply_pair(L.g, x, y);
        t0[pi] = x;
        t1[pi] = y;
      }
    } else if (g < G && L.pair) {
      const double2 z = make_double2(0.0, 0.0);  // the other amplitude has a zero coefficient
      for (uint32_t q = threadIdx.x; q < 2u * A; q += kThreads) {
        const uint32_t i = q & (A - 1u);
        const bool second = q >= A;
        if (!(second ? on1 : on0) || (i & L.lo_mask) != L.lo_vals) continue;
        double2* const t = (second ? t1 : t0) + tile_amp(i);
        *t = (second ? r1 : r0) ? apply_rows23(L.g, z, *t) : apply_rows01(L.g, *t, z);
      }
    } else if (g < G) {
      const uint32_t tb = 1u << L.target, lowm = tb - 1u;
      for (uint32_t q = threadIdx.x; q < A; q += kThreads) {  // pairs over both tiles
        const uint32_t p = q & (A / 2u - 1u);
        const bool second = q >= A / 2u;
        const uint32_t i0 = ((p & ~lowm) << 1) | (p & lowm);
        if (!(second ? on1 : on0) || (i0 & L.lo_mask) != L.lo_vals) continue;
        double2* const t = second ? t1 : t0;
        const uint32_t p0 = tile_amp(i0), p1 = tile_amp(i0 | tb);
        double2 x = t[p0], y = t[p1];
        if (!L.pow2 || !pow2_pair(L.sgn, L.sk, x, y)) apply_pair(L.g, x, y);
        t[p0] = x;
        t[p1] = y;
      }
    }
    __syncthreads();
    // truncation and coding: the gate's byte counts (and, in the end, the new images)
    uint32_t l0 = n0, l1 = n1;
    const bool paired = on0 && on1 && kThreads * VPT == 2u * A && S <= 32u &&
                        encode_pair32<VPT>(m.tile0, m.tile1, kc, S, kDefaultModes, m.img0, m.img1, cap, *m.s, st.pp,
                                           &ctl->err, l0, l1, write);
    if (!paired) {
      for (int w = 0; w < 2; ++w)
        if (w ? on1 : on0) {
          const uint32_t l = encode_block<VPT>(w ? m.tile1 : m.tile0, kc, S, -1, kDefaultModes, w ? m.img1 : m.img0, cap,
                                               *m.s, st.pp, &ctl->err, nullptr, write);
          if (w) l1 = l;
          else l0 = l;
        }
    }
    __syncthreads();
    if (l0 == 0u || l1 == 0u) {
      if (has1 || l0 == 0u) return false;
      l1 = 0u;
    }
    const uint32_t g0 = on0 ? *reinterpret_cast<const uint32_t*>(m.img0) : 0u;
    const uint32_t g1 = on1 ? *reinterpret_cast<const uint32_t*>(m.img1) : 0u;
    if (threadIdx.x == 0 && g < G) {
      long long pages = 0, n64 = 0;
      if (on0) pages += (long long)pages_for(l0, kc) - (long long)pages_for(n0, kc);
      if (on1) pages += (long long)pages_for(l1, kc) - (long long)pages_for(n1, kc);
      if (on0) n64 += (((g0 >> 8) & 0xffu) == 64u) - (long long)wide0;
      if (on1) n64 += (((g1 >> 8) & 0xffu) == 64u) - (long long)wide1;
      sums.dE[g] += (long long)l0 - (long long)n0 + (long long)l1 - (long long)n1;
      sums.dn64[g] += n64;
      sums.dpages[g] += pages;
      if (S <= 32u) {
        if ((!on0 || (g0 & 0xffu) == M_STREAM) && (!on1 || (g1 & 0xffu) == M_STREAM)) ++st.acc->fast;
        else ++st.acc->rest;
      }
    }
    if (on0) {
      n0 = l0;
      z0 = (g0 & 0xffu) == M_ZERO;
      wide0 = ((g0 >> 8) & 0xffu) == 64u;
      std0 = z0 || ((g0 >> 8) & 0xffu) == S;
      dirty0 = true;
      img0 = write;
    }
    if (on1) {
      n1 = l1;
      z1 = (g1 & 0xffu) == M_ZERO;
      wide1 = ((g1 >> 8) & 0xffu) == 64u;
      std1 = z1 || ((g1 >> 8) & 0xffu) == S;
      dirty1 = true;
      img1 = write;
    }
  }
  if (!dirty0 && !dirty1) return true;
  fence_to_bulk();  // every thread's image writes, before the barrier below, for the bulk page stores
  if (threadIdx.x < 32u) {
    free_pages_warp(P, st.cc, ent0 + 4, dirty0 ? np0 : 0u, ent1 + 4, dirty1 ? np1 : 0u);
    const uint32_t q0 = dirty0 ? pages_for(n0, kc) : 0u, q1 = dirty1 ? pages_for(n1, kc) : 0u;
    const bool ok = alloc_pages_warp(P, st.cc, ent0 + 4, q0, ent1 + 4, q1);
    if (threadIdx.x == 0) {
      m.np[0] = q0;
      m.np[1] = q1;
      if (!ok) atomicOr(&ctl->err, (unsigned)E_OOM);
      m.oom[0] = !ok;
      st.acc->wr += (dirty0 ? n0 : 0u) + (dirty1 ? n1 : 0u);
    }
  }
  __syncthreads();
  if (m.oom[0]) return false;
  if (dirty0) commit_images(P, c0, m.img0, n0, ent0 + 4, m.np[0], dirty1, c1, m.img1, n1, ent1 + 4, m.np[1],
                            kDefaultModes, kDefaultModes);
  else commit_images(P, c1, m.img1, n1, ent1 + 4, m.np[1], false, 0ull, nullptr, 0u, nullptr, 0u, kDefaultModes, 0u);
  __syncthreads();
  return true;
}

// Bookkeeping of a step of G gates (one block; every CTA of the simulator has arrived).
__device__ __forceinline__ void run_book(const Pool& P, const CtlParams& cp, int G) {
  DevCtl* ctl = P.ctl;
  __shared__ unsigned long long s_top, s_nf;
  __shared__ int s_skip;
  if (threadIdx.x == 0) {
    const long long top = *(volatile long long*)&ctl->top;
    s_skip = *(volatile unsigned int*)&ctl->err != 0u || top < 0;  // see post_body
    s_top = s_skip ? 0ull : (unsigned long long)top;
    s_nf = ctl->nfreed;  // read here alone: thread 0 clears it below while other warps still copy
  }
  __syncthreads();
  if (s_skip) return;
  const unsigned long long nf = s_nf;
  const unsigned long long top = s_top;
  for (unsigned long long i = threadIdx.x; i < nf; i += blockDim.x) {
    if (top + i < P.npages) P.stack[top + i] = P.freed[i];
    else atomicOr(&ctl->err, (unsigned)E_CORRUPT);
  }
  // the gates in order: thread 0, the sums in registers
  if (threadIdx.x == 0) {
    ctl->top = (long long)(top + nf);
    ctl->nfreed = 0;
    ctl->ndefer = 0;
    unsigned long long E = ctl->E, Emax = ctl->Emax, gates = ctl->gates;
    long long n64 = ctl->n64, sw = ctl->switch_gate;
    double lb_sum = ctl->lb_sum, lb_prod = ctl->lb_prod;
    int lvl = ctl->level;
    long long later = 0;  // pages the gates after the current one add
    for (int g = 1; g < G; ++g) later += ctl->run_dpages[g];
    const unsigned long long end_use = P.npages - (top + nf) - ctl->wc_pages;
    unsigned long long peak = ctl->peak_pages;
    for (int g = 0; g < G; ++g) {
      lvl = next_level(cp, E, lvl, n64);
      if (lvl > 0 && sw < 0) sw = (long long)gates;
      if (level_bits(cp, lvl) < 64) {
        lb_sum += cp.delta[lvl - 1];
        lb_prod *= 1.0 - cp.delta[lvl - 1];
      }
      E += (unsigned long long)ctl->run_dE[g];
      n64 += ctl->run_dn64[g];
      if (E > Emax) Emax = E;
      const unsigned long long use = end_use - (unsigned long long)later;  // pages holding images after this gate
      if (use > peak) peak = use;
      if (g + 1 < G) later -= ctl->run_dpages[g + 1];
      ctl->run_dE[g] = ctl->run_dn64[g] = ctl->run_dpages[g] = 0;
      ++gates;
    }
    ctl->E = E;
    ctl->Emax = Emax;
    ctl->gates = gates;
    ctl->n64 = n64;
    ctl->switch_gate = sw;
    ctl->lb_sum = lb_sum;
    ctl->lb_prod = lb_prod;
    ctl->level = lvl;
    ctl->S_last = level_bits(cp, lvl);
    ctl->peak_pages = peak;
  }
}

// CTAS: resident CTAs an SM its registers are sized for.  2 (128 registers) runs an item
// sooner, 3 (80) more of them: a circuit by itself takes 2 where its items fit (12-qubit
// Grover 14.1 -> 13.3 ms, 14-qubit random circuit 2.06 -> 1.90, 18-qubit QFT 3.29 -> 2.67,
// 23 qubits lossless 6.4 -> 5.7), a batch 3 (16 circuits 38.8 ms, 46.5 at 2).
template <int VPT, int CTAS>
__global__ void __launch_bounds__(kThreads, VPT >= 16 ? 1 : CTAS)
    k_run(const RunJob* __restrict__ jobs, int njobs) {
  extern __shared__ __align__(16) uint8_t smem[];
  __shared__ __align__(16) GateLaunch s_rec[2];
  __shared__ Pool s_P;
  __shared__ RunSums s_sums;
  __shared__ int s_oom, s_swapped, s_last, s_late;
  __shared__ uint32_t s_np[2];
  __shared__ uint32_t s_cache[kCacheCap];
  __shared__ uint32_t s_cache_n;
  __shared__ CtaAcc s_acc;
  static_assert(sizeof(GateLaunch) % 16 == 0, "gate records are copied in 16-byte units");
  static_assert(sizeof(RunSums) == 3u * 8u * kRunGroup && 3 * kRunGroup <= kThreads - 32, "a thread per sum beside warp 0");
  int lo = 0, hi = njobs - 1;  // the job of this CTA
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (jobs[mid].first <= (int)blockIdx.x) lo = mid;
    else hi = mid - 1;
  }
  const RunJob job = jobs[lo];
  const int rank = (int)blockIdx.x - job.first;
  const uint32_t lane = threadIdx.x & 31u;
  run_fetch(job, 0, s_rec);
  cp_async_wait_all();
  if (threadIdx.x == 0) {
    s_cache_n = 0u;
    s_acc.fast = s_acc.rest = s_acc.rd = s_acc.wr = 0ull;
  }
  __syncthreads();
  if (threadIdx.x == 0) s_P = s_rec[0].P;
  __syncthreads();
  const Pool& P = s_P;
  const unsigned long long nchunks = s_rec[0].ctl.nchunks;
  const GateSmem m = gate_smem(smem, P.kc, P.dir_words, nullptr, &s_oom, s_np);
  DevCtl* const ctl = P.ctl;
  GateCta st;
  st.cc.ids = s_cache;
  st.cc.n = &s_cache_n;
  st.acc = &s_acc;
  st.pp = 0;
  uint32_t counted = 0u;  // thread 0: cached ids counted in wc_pages
  uint32_t steps = 0u;
  int b = 0;  // the record buffer of the step's first gate
  for (int k = 0; k < job.ngates;) {
    cp_async_wait_all();
    if (threadIdx.x < 3 * kRunGroup) reinterpret_cast<long long*>(&s_sums)[threadIdx.x] = 0;
    st.err = threadIdx.x == 0 ? *(volatile unsigned int*)&ctl->err : 0u;
    __syncthreads();
    const GateLaunch& L = s_rec[b];
    const uint32_t S = gate_bits(L);
    // (every CTA reads the same level: it changes only while they meet)
    const bool settled = L.ctl.nlevels == 0 || *(volatile int*)&ctl->level >= L.ctl.nlevels;
    const int G = job.list ? job.ngates : (settled ? L.group : 1);
    const bool swap = L.swap != 0 && !job.list;
    unsigned long long bit = G > 1 ? L.group_bit : L.pair_bit;
    if (!bit) bit = 1ull;
    const unsigned long long low = bit - 1ull, items = job.list ? *(volatile unsigned long long*)&ctl->ndefer : (nchunks > 1ull ? nchunks / 2ull : 1ull);
    const unsigned long long swaps = L.items;
    if (swap) {  // X between chunks: a warp per pair, the others by the general way below
      for (unsigned long long item = rank; item < swaps; item += (unsigned)job.ctas) {
        if (threadIdx.x < 32u) {
          unsigned long long coded = 0;
          const bool failed = __shfl_sync(0xffffffffu, st.err, 0) != 0u;
          const bool done = !failed && swap_item(L, item, S, coded);
          if (lane == 0) {
            s_swapped = done;
            if (done && S <= 32u) ++s_acc.fast;
          }
        }
        __syncthreads();
        const bool done = s_swapped != 0;
        __syncthreads();  // the flag is read before the next item sets it
        if (done) continue;
        const unsigned long long c0 = item_chunk(L, item) | L.hi_vals;
        if (!run_item<VPT>(P, s_rec, b, job, k, 1, c0, c0 | L.pair_bit, true, S, false, m, st, s_sums)) break;
      }
    } else {
      bool reload = false;
      for (unsigned long long it = rank; it < items; it += (unsigned)job.ctas) {
        const unsigned long long item = job.list ? job.list[it] : it;
        const unsigned long long c0 = ((item & ~low) << 1) | (item & low);
        if (!run_item<VPT>(P, s_rec, b, job, k, G, c0, c0 | bit, nchunks > 1ull, S, reload, m, st, s_sums)) break;
        reload = G > 2;  // the first record's buffer has held others
      }
    }
    cp_async_wait_all();
    bulk_wait_all();  // this thread's page stores have reached memory
    asm volatile("fence.proxy.async;" ::: "memory");
    __syncthreads();
    const bool end = k + G >= job.ngates;
    if (!end) run_fetch(job, k + G, s_rec + (b ^ 1));
    if (threadIdx.x < 32u) {
      // cached ids beyond what may stay (at the end: all) to the freed list
      const uint32_t n = s_cache_n, keep = end ? 0u : min(n, job.keep);
      unsigned long long base = 0;
      if (lane == 0 && n > keep) base = atomicAdd(&ctl->nfreed, (unsigned long long)(n - keep));
      base = __shfl_sync(0xffffffffu, base, 0);
      for (uint32_t q = keep + lane; q < n; q += 32u) {
        const unsigned long long at = base + (q - keep);
        if (at < P.npages) P.freed[at] = s_cache[q];
        else atomicOr(&ctl->err, (unsigned)E_CORRUPT);
      }
      __syncwarp();
      if (lane == 0) {
        s_cache_n = keep;
        if (keep != counted) atomicAdd(&ctl->wc_pages, (unsigned long long)((long long)keep - (long long)counted));
        counted = keep;
        if (end) {
          if (s_acc.rd) atomicAdd(&ctl->bytes_in, s_acc.rd);
          if (s_acc.wr) atomicAdd(&ctl->bytes_out, s_acc.wr);
          if (s_acc.fast) atomicAdd(&ctl->fast_items, s_acc.fast);
          if (s_acc.rest) atomicAdd(&ctl->fast_deferred, s_acc.rest);
        }
      }
      __syncwarp();
    } else if (threadIdx.x >= kThreads - 3 * kRunGroup) {
      const uint32_t q = threadIdx.x - (kThreads - 3 * kRunGroup);
      const long long v = reinterpret_cast<const long long*>(&s_sums)[q];
      if (v) atomicAdd(reinterpret_cast<unsigned long long*>(ctl->run_dE) + q, (unsigned long long)v);  // dE, dn64, dpages in a row
    }
    __syncthreads();
    // the simulator's CTAs meet; the last one books the step's gates
    ++steps;
    if (threadIdx.x == 0) {
      __threadfence();
      s_last = atomicAdd(&ctl->run_arrived, 1u) + 1u == (uint32_t)job.ctas * steps;
      __threadfence();
    }
    __syncthreads();
    if (s_last) {
      run_book(P, s_rec[b].ctl, G);
      __syncthreads();
      if (threadIdx.x == 0) {
        __threadfence();
        if (end) ctl->run_arrived = 0u;  // nobody waits after the last step
        atomicExch(&ctl->run_gate, end ? 0u : steps);
      }
      __syncthreads();
    } else if (!end) {
      if (threadIdx.x == 0) {
        // (once a wait has given up, here or in an earlier launch, the arrivals do not add up)
        const uint32_t limit = (st.err & (unsigned)E_TIMEOUT) ? 0u : job.polls;
        uint32_t it = 0;
        while (*(volatile unsigned int*)&ctl->run_gate != steps) {
          if (++it > limit) {
            atomicOr(&ctl->err, (unsigned)E_TIMEOUT);
            atomicExch(&ctl->timeout_site, 4u);
            break;
          }
        }
        s_late = it > limit;
        __threadfence();
      }
      __syncthreads();
      if (s_late) {
        cp_async_wait_all();
        return;
      }
    }
    k += G;
    b ^= 1;
  }
}

template <int CTAS>
static int run_occupancy(int kc) {
  int n = 0;
  cudaError_t e = cudaErrorInvalidValue;
  const size_t smem = gate_smem_bytes(kc);
  auto ask = [&](auto kernel) {
    e = prep(kernel, smem);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kernel, kThreads, smem);
  };
  switch (vpt_for(kc)) {
    case 1: ask(k_run<1, CTAS>); break;
    case 2: ask(k_run<2, CTAS>); break;
    case 4: ask(k_run<4, CTAS>); break;
    case 8: ask(k_run<8, CTAS>); break;
    case 16: if constexpr (CTAS == 3) ask(k_run<16, CTAS>); break;
  }
  return e != cudaSuccess || n < 1 ? 0 : n;
}

template <int CTAS>
static cudaError_t run_launch(const RunJob* jobs, int njobs, int kc, int grid, cudaStream_t st) {
  const size_t smem = gate_smem_bytes(kc);
  void* args[] = {(void*)&jobs, (void*)&njobs};
  auto go = [&](auto kernel) {
    const cudaError_t e = prep(kernel, smem);
    return e != cudaSuccess
               ? e
               : cudaLaunchCooperativeKernel((const void*)kernel, dim3((unsigned)grid), dim3(kThreads), args, smem, st);
  };
  switch (vpt_for(kc)) {
    case 1: return go(k_run<1, CTAS>);
    case 2: return go(k_run<2, CTAS>);
    case 4: return go(k_run<4, CTAS>);
    case 8: return go(k_run<8, CTAS>);
    case 16: if constexpr (CTAS == 3) return go(k_run<16, CTAS>);
  }
  return cudaErrorInvalidValue;
}

}  // namespace qc
