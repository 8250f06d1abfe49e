// group.cu -- several gates per pass over a large lossy state.
//
// Once the error bound is settled (Section 3.7: it never tightens), consecutive gates that
// leave every pair of chunks to itself -- gates inside chunks, diagonal gates anywhere, gates
// on one cross-chunk target -- need the state decoded and written only once.  A pair of warps
// takes a pair of chunks, decodes both into shared memory (high words: S <= 32), applies the
// gates in order, truncating after each (Section 4.2) and counting the bytes and pages its
// images would take, then encodes the last values.  A pair of chunks that is not STREAM at S
// on the way in, or would not be after one of the gates, is left as it was and listed for
// k_run, which takes it through the same gates and books them.
//
// Bound: instructions, about a third as many per value for a gate in the middle of a group
// (load, gate, truncation, length of the codes) as for one by itself.
// 2^10-amplitude chunks, 1e-4: a 30-qubit random-circuit layer 517 -> 434 ms, a 26-qubit
// QAOA round 104 -> 71.5 ms; 21 qubits in 2^9, two layers 3.16 -> 1.76 ms.
#include "stream.cuh"

namespace qc {

constexpr int kGroupWarps = 4;  // two pairs; 20 warps an SM with 2^10-amplitude chunks (43 KB a CTA)
constexpr int kGroupPairs = kGroupWarps / 2;

// Per warp: its chunk's high words, two windows (the first also the output window), input
// and output page ids, its page cache.
__host__ __device__ __forceinline__ uint32_t group_warp_bytes(int kc) {
  return 4u * (2u << kc) + 2u * kFastWin + 8u * fast_pg_words(kc) + 4u * kWarpCache + 16u;
}

// The lane's 8 values of pass p: two 16-byte units 512 bytes apart (no bank conflicts).
__device__ __forceinline__ void vals_load(const uint32_t* vals, uint32_t p, uint32_t v[8]) {
  const uint4* q = reinterpret_cast<const uint4*>(vals) + 64u * p + (threadIdx.x & 31u);
  const uint4 a = q[0], b = q[32];
  v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w; v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
}
__device__ __forceinline__ void vals_store(uint32_t* vals, uint32_t p, const uint32_t v[8]) {
  uint4* q = reinterpret_cast<uint4*>(vals) + 64u * p + (threadIdx.x & 31u);
  q[0] = make_uint4(v[0], v[1], v[2], v[3]);
  q[32] = make_uint4(v[4], v[5], v[6], v[7]);
}
// Word of value 0 and of value 5 of a lane's pass (the period filter's samples).
__device__ __forceinline__ const uint32_t* val0(const uint32_t* vals, uint32_t p) {
  return vals + 256u * p + 4u * (threadIdx.x & 31u);
}
__device__ __forceinline__ const uint32_t* val5(const uint32_t* vals, uint32_t p) {
  return vals + 256u * p + 128u + 4u * (threadIdx.x & 31u) + 1u;
}

// signed_rows / signed_pair need every input at least 2^-959 or zero.
__device__ __forceinline__ bool too_small(uint32_t h) { return ((h & 0x7fffffffu) - 1u) < ((64u << 20) - 1u); }

// A gate that is not diagonal on this warp's chunk; kind 4 (the pair's chunks a and b): this
// warp's half of the amplitudes, both rows.
template <int ARITH>
__device__ __forceinline__ void group_apply(const GroupGate& g, uint32_t* mine, uint32_t* ca, uint32_t* cb, uint32_t side,
                                            uint32_t NP, uint32_t mh, bool& spec) {
  const uint32_t lane = threadIdx.x & 31u;
  auto pair_of = [&](uint32_t* a, uint32_t pa, uint32_t* b, uint32_t pb) {
    uint32_t x[8], y[8];
    vals_load(a, pa, x);
    vals_load(b, pb, y);
    if constexpr (ARITH == 4) {
#pragma unroll
      for (int k = 0; k < 8; ++k) spec |= too_small(x[k]) | too_small(y[k]);
    }
#pragma unroll
    for (int k = 0; k < 4; ++k)
      fast_pair<ARITH>(g, 128u * pa + 4u * lane + (uint32_t)k, x[2 * k], x[2 * k + 1], y[2 * k], y[2 * k + 1], mh, spec);
    vals_store(a, pa, x);
    vals_store(b, pb, y);
  };
  if (g.kind == 4) {
    const uint32_t lo = NP > 1u ? side * (NP / 2u) : side, hi = NP > 1u ? lo + NP / 2u : 1u;
    for (uint32_t p = lo; p < hi; ++p) pair_of(ca, p, cb, p);
  } else if (g.kind == 2) {
    const uint32_t d = 1u << (g.target - 7);
    for (uint32_t q = 0; q < NP / 2u; ++q) {
      const uint32_t p = ((q & ~(d - 1u)) << 1) | (q & (d - 1u));
      pair_of(mine, p, mine, p + d);
    }
  } else {
    for (uint32_t p = 0; p < NP; ++p) {
      uint32_t v[8];
      vals_load(mine, p, v);
      if constexpr (ARITH == 4) {
#pragma unroll
        for (int k = 0; k < 8; ++k) spec |= too_small(v[k]);
      }
      const uint32_t i = 128u * p + 4u * lane;
      if (g.kind == 0) {
        if (g.target == 0) {
          fast_pair<ARITH>(g, i, v[0], v[1], v[2], v[3], mh, spec);
          fast_pair<ARITH>(g, i + 2u, v[4], v[5], v[6], v[7], mh, spec);
        } else {
          fast_pair<ARITH>(g, i, v[0], v[1], v[4], v[5], mh, spec);
          fast_pair<ARITH>(g, i + 1u, v[2], v[3], v[6], v[7], mh, spec);
        }
      } else {  // partner in lane ^ 2^(t-2): this lane forms its own row
        const uint32_t row = (lane >> (g.target - 2)) & 1u;
        uint32_t w[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) w[k] = __shfl_xor_sync(0xffffffffu, v[k], 1u << (g.target - 2));
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          uint32_t outr = v[2 * k], outi = v[2 * k + 1];
          if ((((i + (uint32_t)k) & ~(1u << g.target)) & g.lo_mask) == g.lo_vals) {
            const uint32_t ar = row ? w[2 * k] : v[2 * k], ai = row ? w[2 * k + 1] : v[2 * k + 1];
            const uint32_t br = row ? v[2 * k] : w[2 * k], bi = row ? v[2 * k + 1] : w[2 * k + 1];
            if constexpr (ARITH == 4) {
              signed_rows(g, row, ar, ai, br, bi, mh, outr, outi, spec);
            } else if constexpr (ARITH == 2) {
              row_op(g, row, w[2 * k], w[2 * k + 1], mh, outr, outi, spec);
            } else {
              const double2 a = make_double2(hi_as_double(ar), hi_as_double(ai));
              const double2 b = make_double2(hi_as_double(br), hi_as_double(bi));
              const double2 o = ARITH == 0 ? dense_rows(g.cf + 8u * row, a, b) : real_rows(g.cf + 8u * row, a, b);
              outr = fast_trunc(o.x, mh, spec);
              outi = fast_trunc(o.y, mh, spec);
            }
          }
          v[2 * k] = outr;
          v[2 * k + 1] = outi;
        }
      }
      vals_store(mine, p, v);
    }
  }
}

// A diagonal gate on this warp's chunk: row by the chunk (pair_bit) or by the amplitude.
__device__ __forceinline__ void group_diag(const GroupGate& g, uint32_t* mine, uint32_t chunk_row, uint32_t NP, uint32_t mh,
                                           bool& spec) {
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t tb = g.pair_bit ? 0u : 1u << g.target;
  for (uint32_t p = 0; p < NP; ++p) {
    const uint32_t i = 128u * p + 4u * lane;
    // a pass whose index bits miss the controls, or whose row is a copy, stays
    if (((128u * p) & g.lo_mask & ~127u) != (g.lo_vals & ~127u)) continue;
    if (tb >= 128u && ((g.copy >> ((128u * p & tb) ? 1u : 0u)) & 1u)) continue;
    uint32_t v[8];
    vals_load(mine, p, v);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const uint32_t a = i + (uint32_t)k, row = tb ? ((a & tb) ? 1u : 0u) : chunk_row;
      if (((a & ~tb) & g.lo_mask) == g.lo_vals) {
        uint32_t x, y;
        row_op(g, row, v[2 * k], v[2 * k + 1], mh, x, y, spec);
        v[2 * k] = x;
        v[2 * k + 1] = y;
      }
    }
    vals_store(mine, p, v);
  }
}

// Residual bits of the chunk's values, and whether its image is surely STREAM (fast_item's
// filters: not constant, not zero, no period).  All lanes get both.
__device__ __forceinline__ bool group_size(const uint32_t* vals, uint32_t NP, uint32_t S, uint32_t& bits) {
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t refr = vals[0], refi = vals[1];
  uint32_t sum = 0u, prv = 0u, nzor = 0u;
  bool cst = true, halves = true;
  for (uint32_t p = 0; p < NP; ++p) {
    uint32_t v[8];
    vals_load(vals, p, v);
    uint32_t pr = __shfl_up_sync(0xffffffffu, v[7], 1);
    if (lane == 0) pr = prv;
    prv = __shfl_sync(0xffffffffu, v[7], 31);
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const uint32_t x = v[k] ^ (k ? v[k - 1] : pr);
      sum += rlen(S, min((uint32_t)__clz((int)x), 24u) & 0x18u);
      nzor |= v[k];
      cst &= v[k] == ((k & 1) ? refi : refr);
    }
    if (NP == 1u) {
      const uint32_t a = __shfl_xor_sync(0xffffffffu, v[0], 16), b = __shfl_xor_sync(0xffffffffu, v[5], 16);
      halves &= (a == v[0]) & (b == v[5]);
    } else if (p >= NP / 2u) {
      halves &= *val0(vals, p - NP / 2u) == v[0] && *val5(vals, p - NP / 2u) == v[5];
    }
  }
  bits = __reduce_add_sync(0xffffffffu, sum);
  const bool c = __all_sync(0xffffffffu, cst), z = __any_sync(0xffffffffu, nzor != 0u), h = __all_sync(0xffffffffu, halves);
  return !c && z && !h;
}

__global__ void __launch_bounds__(32 * kGroupWarps, 5) k_group(const __grid_constant__ GroupLaunch L) {
  extern __shared__ __align__(16) uint8_t smem[];
  __shared__ uint32_t s_slots[kGroupPairs][4];
  __shared__ uint32_t s_seq[kGroupPairs][2];
  const Pool& P = L.P;
  const int kc = P.kc;
  const uint32_t lane = threadIdx.x & 31u, wid = threadIdx.x >> 5, pr = wid >> 1, side = wid & 1u;
  if (threadIdx.x < 2u * kGroupPairs) s_seq[threadIdx.x >> 1][threadIdx.x & 1u] = 0u;
  __syncthreads();
  DevCtl* ctl = P.ctl;
  const uint32_t N = 2u << kc, cb = N >> 2, NP = N >> 8, S = L.S, mh = (uint32_t)(trunc_mask(S) >> 32);
  const uint32_t per = group_warp_bytes(kc);
  uint32_t* const vals = reinterpret_cast<uint32_t*>(smem + (size_t)wid * per);
  uint32_t* const peer = reinterpret_cast<uint32_t*>(smem + (size_t)(wid ^ 1u) * per);
  uint32_t* const win0 = vals + N;
  uint32_t* const win1 = win0 + kFastWin / 4u;
  uint32_t* const ipg = win1 + kFastWin / 4u;
  uint32_t* const opg = ipg + fast_pg_words(kc);
  WarpPages wp;
  wp.ids = opg + fast_pg_words(kc);
  wp.n = wp.ids + kWarpCache;
  const size_t gw = (size_t)blockIdx.x * kGroupWarps + wid;
  const uint32_t n_start = P.wcache_n[gw];
  for (uint32_t q = lane; q < n_start; q += 32u) wp.ids[q] = P.wcache[gw * kWarpCache + q];
  if (lane == 0) *wp.n = n_start;
  __syncwarp();
  uint32_t phase = 0;
  volatile uint32_t* seq = s_seq[pr];
  long long dE = 0;             // lane g: change of E by gate g
  int dpages = 0;               // ... and of the pages holding images
  unsigned long long rd = 0, wr = 0, done = 0, deferred = 0;
  const unsigned long long low = L.bit - 1ull, pairs = (unsigned long long)gridDim.x * kGroupPairs;
  for (unsigned long long item = (unsigned long long)blockIdx.x * kGroupPairs + pr; item < L.items; item += pairs) {
    const unsigned long long ch = (((item & ~low) << 1) | (item & low)) | (side ? L.bit : 0ull);
    // the gates that rewrite this chunk (bit g), and whether one leaves it by a copy row
    uint32_t mine = 0u;
    bool copied = false;
    for (int g = 0; g < L.ngates; ++g) {
      const GroupGate& q = L.g[g];
      if ((ch & q.fixed) != q.hi_vals) continue;
      if (q.kind == 3 && q.pair_bit && ((q.copy >> ((ch & q.pair_bit) ? 1u : 0u)) & 1u)) copied = true;
      else mine |= 1u << g;
    }
    uint32_t ib = 0u, inp = 0u, bits_in = 0u;
    bool ok = true;
    if (mine) {
      const uint32_t* e = dir_entry(P, ch);
      const uint2 h = *reinterpret_cast<const uint2*>(e);
      ib = h.x;
      inp = h.y;
      ok = inp >= 1u && ib <= fast_max_image(kc) && inp == (ib + kPage - 1u) / kPage;
      if (ok) {
        bool good = true;
        for (uint32_t k = lane; k < inp; k += 32u) {
          const uint32_t pid = e[4 + k];
          ipg[k] = pid;
          good &= pid < P.npages;
        }
        ok = __all_sync(0xffffffffu, good);
        __syncwarp();
      }
      if (ok) {
        const uint4 hd = *reinterpret_cast<const uint4*>(P.pages + (unsigned long long)ipg[0] * kPage);
        bits_in = hd.w;
        ok = stream32_header(hd, ib, kc) && ((hd.x >> 8) & 0xffu) == S;
      }
    } else if (copied) {
      ok = image_stands(P, ch, S, kDefaultModes);
    }
    unsigned int err = 0;
    if (lane == 0) err = *(volatile unsigned int*)&ctl->err;
    err = __shfl_sync(0xffffffffu, err, 0);
    {
      const uint32_t me = (ok ? 1u : 0u) | (err ? 2u : 0u);
      const uint32_t other = pair_agree(s_slots[pr], seq, phase, side, me, ctl, 5u);
      if ((me | other) & 2u) break;
      if (!((me & other) & 1u)) {
        if (side == 0 && lane == 0) {
          L.defer[atomicAdd(&ctl->ndefer, 1ull)] = (uint32_t)item;
          ++deferred;
        }
        continue;
      }
    }
    bool corrupt = false, lost = false, keep = true, spec = false;
    if (mine)
      corrupt = !stream_decode(PagedImage{P.pages, ipg}, kc, S, bits_in, ib, win0, win1,
                               [&](uint32_t p, const uint32_t v[8]) { vals_store(vals, p, v); });
    __syncwarp();
    uint32_t size = ib;  // lane g: the image's bytes after gate g
    const int last = mine ? 31 - __clz((int)mine) : -1;
    for (int g = 0; g <= last; ++g) {
      if (!((mine >> g) & 1u)) continue;
      const GroupGate& q = L.g[g];
      const bool cross = q.kind == 4;  // both warps come here or neither
      if (cross) {
        ++phase;
        if (!lost) lost = !pair_sync(seq, side, phase, ctl, 6u);
      }
      if (q.kind == 3) {
        group_diag(q, vals, (ch & q.pair_bit) ? 1u : 0u, NP, mh, spec);
      } else {
        uint32_t* const ca = side ? peer : vals;
        uint32_t* const cbv = side ? vals : peer;
        switch (q.arith) {
          case 0: group_apply<0>(q, vals, ca, cbv, side, NP, mh, spec); break;
          case 2: group_apply<2>(q, vals, ca, cbv, side, NP, mh, spec); break;
          case 3: group_apply<3>(q, vals, ca, cbv, side, NP, mh, spec); break;
          default: group_apply<4>(q, vals, ca, cbv, side, NP, mh, spec); break;
        }
      }
      if (cross) {
        ++phase;
        if (!lost) lost = !pair_sync(seq, side, phase, ctl, 7u);
      }
      __syncwarp();
      if (g < last) {  // the last one's bytes come from the encoder
        uint32_t bits;
        keep &= group_size(vals, NP, S, bits);
        if ((int)lane >= g) size = 16u + cb + resid_bytes(bits);
      }
    }
    // the new image: codes, residuals through the output window, finished blocks to pages
    uint32_t onp = 0u, ooff = 0u;
    bool oom = false;
    if (mine) {
      uint32_t* const owin = win0;
      uint4* const w4 = reinterpret_cast<uint4*>(owin);
      for (uint32_t k = lane; k < kWinBlocks; k += 32u) w4[k] = make_uint4(0u, 0u, 0u, 0u);
      oom = !wp_grow(P, wp, opg, onp, (16u + cb + kPage - 1u) / kPage);
      __syncwarp();
      const uint32_t refr = vals[0], refi = vals[1];
      uint32_t prv = 0u, nzor = 0u;
      bool cst = true, halves = true;
      for (uint32_t p = 0; p < NP; ++p) {
        uint32_t v[8];
        vals_load(vals, p, v);
        uint32_t before = __shfl_up_sync(0xffffffffu, v[7], 1);
        if (lane == 0) before = prv;
        prv = __shfl_sync(0xffffffffu, v[7], 31);
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          nzor |= v[k];
          cst &= v[k] == ((k & 1) ? refi : refr);
        }
        if (NP == 1u) {
          const uint32_t a = __shfl_xor_sync(0xffffffffu, v[0], 16), b = __shfl_xor_sync(0xffffffffu, v[5], 16);
          halves &= (a == v[0]) & (b == v[5]);
        } else if (p >= NP / 2u) {
          halves &= *val0(vals, p - NP / 2u) == v[0] && *val5(vals, p - NP / 2u) == v[5];
        }
        uint32_t osum, otot;
        const uint32_t ocw = fast_codes(v, before, S, osum);
        const uint32_t ob = ooff >> 7;
        fast_pack(owin, 4u * ob, ooff + warp_excl(osum, otot), v, ocw, S);
        const uint32_t pairw = ocw | (__shfl_down_sync(0xffffffffu, ocw, 1) << 16);
        if ((lane & 1u) == 0u && !oom) {
          const uint32_t b = 16u + 64u * p + 2u * lane;
          *reinterpret_cast<uint32_t*>(P.pages + (unsigned long long)opg[b >> 9] * kPage + (b & (kPage - 1u))) = pairw;
        }
        ooff += otot;
        __syncwarp();
        const bool end = p + 1u == NP;
        const uint32_t endb = end ? (ooff + 127u) >> 7 : ooff >> 7, nb = endb - ob;
        if (!oom) oom = !wp_grow(P, wp, opg, onp, (16u + cb + 16u * endb + kPage - 1u) / kPage);
        if (!oom)
          for (uint32_t k = lane; k < nb; k += 32u) {
            const uint32_t b = 16u + cb + 16u * (ob + k);
            reinterpret_cast<uint4*>(P.pages + (unsigned long long)opg[b >> 9] * kPage + (b & (kPage - 1u)))[0] = w4[k];
          }
        if (!end) {
          uint4 carry = make_uint4(0u, 0u, 0u, 0u);
          if (lane == 0) carry = w4[nb];
          __syncwarp();
          for (uint32_t k = lane; k <= nb; k += 32u) w4[k] = k == 0u ? carry : make_uint4(0u, 0u, 0u, 0u);
          __syncwarp();
        }
      }
      const bool c = __all_sync(0xffffffffu, cst), z = __any_sync(0xffffffffu, nzor != 0u), hh = __all_sync(0xffffffffu, halves);
      const bool any_spec = __any_sync(0xffffffffu, spec);
      keep = keep && !c && z && !hh && !any_spec;
      if ((int)lane >= last) size = 16u + cb + resid_bytes(ooff);
    }
    if (corrupt && lane == 0) atomicOr(&ctl->err, (unsigned)E_CORRUPT);
    const uint32_t me = (keep ? 1u : 0u) | ((corrupt || oom || lost) ? 2u : 0u);
    const uint32_t other = lost ? 2u : pair_agree(s_slots[pr], seq, phase, side, me, ctl, 8u);
    if (((me | other) & 2u) || !((me & other) & 1u)) {
      if (mine) wp_free(P, wp, opg, onp);
      if ((me | other) & 2u) break;
      if (side == 0 && lane == 0) {
        L.defer[atomicAdd(&ctl->ndefer, 1ull)] = (uint32_t)item;
        ++deferred;
      }
      continue;
    }
    if (mine) {
      const uint32_t plen = cb + resid_bytes(ooff), bytes = 16u + plen;
      if (lane == 0)
        reinterpret_cast<uint4*>(P.pages + (unsigned long long)opg[0] * kPage)[0] = make_uint4(M_STREAM | (S << 8), plen, N, ooff);
      uint32_t* e = dir_entry(P, ch);
      for (uint32_t k = lane; k < onp; k += 32u) e[4 + k] = opg[k];
      uint32_t prev = __shfl_up_sync(0xffffffffu, size, 1);
      if (lane == 0) prev = ib;
      dE += (long long)size - (long long)prev;
      dpages += (int)((size + kPage - 1u) / kPage) - (int)((prev + kPage - 1u) / kPage);
      if (lane == 0) {
        *reinterpret_cast<uint4*>(e) = make_uint4(bytes, onp, kDefaultModes, 0u);
        rd += ib;
        wr += bytes;
      }
      wp_free(P, wp, ipg, inp);
    }
    if (side == 0) ++done;
    __syncwarp();
  }
  cp_async_wait_all();
  __syncwarp();
  {
    const uint32_t n = *wp.n;
    for (uint32_t q = lane; q < n; q += 32u) P.wcache[gw * kWarpCache + q] = wp.ids[q];
    if (lane == 0) {
      P.wcache_n[gw] = n;
      if (n != n_start) atomicAdd(&ctl->wc_pages, (unsigned long long)((long long)n - (long long)n_start));
    }
  }
  if (dE) atomicAdd(reinterpret_cast<unsigned long long*>(&ctl->run_dE[lane]), (unsigned long long)dE);
  if (dpages) atomicAdd(reinterpret_cast<unsigned long long*>(&ctl->run_dpages[lane]), (unsigned long long)(long long)dpages);
  if (lane == 0) {
    if (rd) atomicAdd(&ctl->bytes_in, rd);
    if (wr) atomicAdd(&ctl->bytes_out, wr);
    if (done) atomicAdd(&ctl->fast_items, done);
    if (deferred) atomicAdd(&ctl->fast_deferred, deferred);
  }
}

int group_ctas_per_sm(int kc) {
  int n = 0;
  const size_t smem = (size_t)kGroupWarps * group_warp_bytes(kc);
  if (cudaFuncSetAttribute(k_group, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_group, 32 * kGroupWarps, smem) != cudaSuccess)
    return 0;
  return n;
}
int group_warps() { return kGroupWarps; }

cudaError_t launch_group(const GroupLaunch& L, int grid, cudaStream_t st) {
  const size_t smem = (size_t)kGroupWarps * group_warp_bytes(L.P.kc);
  const cudaError_t e = cudaFuncSetAttribute(k_group, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  const unsigned long long want = (L.items + kGroupPairs - 1ull) / kGroupPairs;
  k_group<<<(unsigned)(want < (unsigned long long)grid ? want : (unsigned long long)grid), 32 * kGroupWarps, smem, st>>>(L);
  return cudaGetLastError();
}

}  // namespace qc
