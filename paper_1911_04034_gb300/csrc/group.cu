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
// Gate by gate -> by groups, 2^10-amplitude chunks, 1e-4: a 30-qubit random-circuit layer 490
// -> 348 ms, a 26-qubit QAOA round 96 -> 65 ms; 21 qubits in 2^9, two layers 2.95 -> 1.56 ms.
#include "stream.cuh"

namespace qc {

constexpr int kGroupWarps = 4;  // two pairs; 20 warps an SM with 2^10-amplitude chunks (43 KB a CTA)
constexpr int kGroupPairs = kGroupWarps / 2;
static_assert(kRunGroup <= 32, "a lane and a mask bit per gate of a group");

// Per warp: its chunk's high words, what is known of each pass of it (see group_note), two
// windows (the first also the output window), input and output page ids, its page cache.
constexpr uint32_t kGroupPasses = 16;  // of a chunk, at most
__host__ __device__ __forceinline__ uint32_t group_warp_bytes(int kc) {
  return 4u * (2u << kc) + 4u * kGroupPasses + 2u * kFastWin + 8u * fast_pg_words(kc) + 4u * kWarpCache + 16u;
}

// A chunk's values stand in order; a lane takes amplitude 32 j + lane of a pass (128
// amplitudes), so that one loop body serves every target and an instruction cache holds the
// whole kernel (unrolled over a lane's 8 consecutive values, with a body per kind of target,
// it was 228 KB and waited for instructions more than for anything else).
__device__ __forceinline__ uint2* amps(uint32_t* vals, uint32_t p) { return reinterpret_cast<uint2*>(vals) + 128u * p; }
__device__ __forceinline__ const uint2* amps(const uint32_t* vals, uint32_t p) {
  return reinterpret_cast<const uint2*>(vals) + 128u * p;
}
__device__ __forceinline__ uint32_t code_bits(uint32_t x, uint32_t S) { return rest_bits(code_rest(x), S); }

// The passes of a chunk whose index bits satisfy a gate's controls (bit p), for a diagonal
// gate on an in-chunk target those not on an exact copy's row: the others stay.
__device__ __forceinline__ uint32_t group_passes(const GroupGate& g, uint32_t NP) {
  const uint32_t hm = g.lo_mask >> 7, hv = g.lo_vals >> 7, lane = threadIdx.x & 31u;
  bool on = lane < NP && (lane & hm) == hv;
  if (g.kind == 3 && !g.pair_bit && g.target >= 7) on = on && !((g.copy >> ((lane >> (g.target - 7)) & 1u)) & 1u);
  return __ballot_sync(0xffffffffu, on);
}

// Notes what the byte count needs to know of the passes in `mask`: the residual bits of all
// but a pass's first value (whose predecessor lies in the pass before), and in the top bit
// whether some lane's amplitudes differ (the chunk is then neither constant nor zero).
// Passes a gate leaves keep their notes.
__device__ __forceinline__ void group_note(const uint32_t* vals, uint32_t* notes, uint32_t mask, uint32_t S) {
  const uint32_t lane = threadIdx.x & 31u;
#pragma unroll 1
  while (mask) {
    const uint32_t p = (uint32_t)__ffs((int)mask) - 1u;
    mask &= mask - 1u;
    const uint2* a = amps(vals, p) + lane;
    uint2 v[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) v[j] = a[32 * j];
    uint32_t sum = 0u, carry = 0u, varies = 0u;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      uint32_t before = __shfl_up_sync(0xffffffffu, v[j].y, 1);
      if (lane == 0) before = carry;
      carry = __shfl_sync(0xffffffffu, v[j].y, 31);
      if (j > 0 || lane > 0) sum += code_bits(v[j].x ^ before, S);
      sum += code_bits(v[j].y ^ v[j].x, S);
      varies |= (v[j].x ^ v[0].x) | (v[j].y ^ v[0].y);
    }
    const uint32_t bits = __reduce_add_sync(0xffffffffu, sum);
    const bool any = __any_sync(0xffffffffu, varies != 0u);
    if (lane == 0) notes[p] = bits | (any ? 0x80000000u : 0u);
  }
  __syncwarp();
}

// signed_pair needs every input at least 2^-959 or zero.
__device__ __forceinline__ bool too_small(uint32_t h) { return ((h & 0x7fffffffu) - 1u) < ((64u << 20) - 1u); }

// The pairs of one pass (in-chunk target below 7: A = B, 64 pairs) or of two (A and B hold the
// pairs' first and second amplitudes, 128 pairs); i0: in-chunk index of A's first amplitude.
template <int ARITH>
__device__ __forceinline__ void group_pairs(const GroupGate& g, uint2* A, uint2* B, uint32_t i0, bool inner, uint32_t mh,
                                            bool& spec) {
  const uint32_t lane = threadIdx.x & 31u, tb = inner ? 1u << g.target : 0u, low = tb - 1u;
#pragma unroll 1
  for (uint32_t q = lane; q < (inner ? 64u : 128u); q += 32u) {
    const uint32_t ia = inner ? ((q & ~low) << 1) | (q & low) : q, ib = ia | tb;
    if (((i0 + ia) & g.lo_mask) != g.lo_vals) continue;
    uint2 a = A[ia], b = B[ib];
    if constexpr (ARITH == 4) spec |= too_small(a.x) | too_small(a.y) | too_small(b.x) | too_small(b.y);
    fast_pair<ARITH>(g, i0 + ia, a.x, a.y, b.x, b.y, mh, spec);
    A[ia] = a;
    B[ib] = b;
  }
}
// A gate that is not diagonal on the passes `mask` of this warp's chunk; a cross-chunk gate
// (chunks ca and cb): this warp's half of them, both rows.
template <int ARITH>
__device__ __forceinline__ void group_apply(const GroupGate& g, uint32_t* mine, uint32_t* ca, uint32_t* cb, uint32_t side,
                                            uint32_t NP, uint32_t mask, uint32_t mh, bool& spec) {
  const bool inner = g.kind < 2;
  uint32_t todo = mask, d = 0u;
  if (g.kind == 4) {
    const uint32_t half = NP > 1u ? (1u << (NP / 2u)) - 1u : 1u;
    todo &= side ? ~half : half;
  } else if (g.kind == 2) {
    d = 1u << (g.target - 7);
  }
#pragma unroll 1
  while (todo) {
    const uint32_t p = (uint32_t)__ffs((int)todo) - 1u;
    todo &= todo - 1u;
    if (p & d) continue;  // the second pass of a pair of passes
    group_pairs<ARITH>(g, amps(g.kind == 4 ? ca : mine, p), amps(g.kind == 4 ? cb : mine, p + d), 128u * p, inner, mh, spec);
  }
}

// A diagonal gate on the passes `mask` of this warp's chunk: row by the chunk (a cross-chunk
// target) or by the amplitude.
__device__ __forceinline__ void group_diag(const GroupGate& g, uint32_t* mine, uint32_t chunk_row, uint32_t mask, uint32_t mh,
                                           bool& spec) {
  const uint32_t lane = threadIdx.x & 31u, tb = g.pair_bit ? 0u : 1u << g.target;
#pragma unroll 1
  while (mask) {
    const uint32_t p = (uint32_t)__ffs((int)mask) - 1u;
    mask &= mask - 1u;
    uint2* a = amps(mine, p);
#pragma unroll 1
    for (uint32_t q = lane; q < 128u; q += 32u) {
      const uint32_t i = 128u * p + q, row = tb ? ((i & tb) ? 1u : 0u) : chunk_row;
      if (((i & ~tb) & g.lo_mask) != g.lo_vals || ((g.copy >> row) & 1u)) continue;
      uint2 v = a[q], o;
      row_op(g, row, v.x, v.y, mh, o.x, o.y, spec);
      a[q] = o;
    }
  }
}

// Whether some amplitude of the chunk differs from its first (a chunk of zeros: no), and
// whether some amplitude differs from the one half a chunk on (a period: none does).
__device__ __forceinline__ bool group_differs(const uint32_t* vals, uint32_t NP) {
  const uint32_t lane = threadIdx.x & 31u;
  bool any = false;
#pragma unroll 1
  for (uint32_t q = 0; q < 4u * NP && !any; ++q) {
    const uint2 v = amps(vals, 0u)[32u * q + lane];
    any = __any_sync(0xffffffffu, v.x != vals[0] || v.y != vals[1]);
  }
  return any;
}
__device__ __forceinline__ bool group_moves(const uint32_t* vals, uint32_t NP) {
  const uint32_t lane = threadIdx.x & 31u;
  bool any = false;
#pragma unroll 1
  for (uint32_t q = 0; q < 2u * NP && !any; ++q) {
    const uint2 v = amps(vals, 0u)[32u * q + lane], w = amps(vals, 0u)[32u * (q + 2u * NP) + lane];
    any = __any_sync(0xffffffffu, v.x != w.x || v.y != w.y);
  }
  return any;
}

// Residual bits of the chunk's values from its notes, and whether its image is surely STREAM
// (fast_item's filters: not constant, not zero, no period).  All lanes get both.
__device__ __forceinline__ bool group_size(const uint32_t* vals, const uint32_t* notes, uint32_t NP, uint32_t S,
                                           uint32_t& bits) {
  const uint32_t lane = threadIdx.x & 31u;
  uint32_t mine = 0u, varies = 0u;
  if (lane < NP) {
    const uint32_t x = vals[256u * lane] ^ (lane ? vals[256u * lane - 1u] : 0u);  // a pass's first value and the one before
    mine = (notes[lane] & 0x7fffffffu) + code_bits(x, S);
    varies = notes[lane] >> 31;
  }
  bits = __reduce_add_sync(0xffffffffu, mine);
  // (lanes that vary: not constant, not zero)
  return (__any_sync(0xffffffffu, varies != 0u) || group_differs(vals, NP)) && group_moves(vals, NP);
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
  uint32_t* const notes = vals + N;
  uint32_t* const win0 = notes + kGroupPasses;
  uint32_t* const win1 = win0 + kFastWin / 4u;
  uint32_t* const ipg = win1 + kFastWin / 4u;
  uint32_t* const opg = ipg + fast_pg_words(kc);
  WarpPages wp;
  wp.ids = opg + fast_pg_words(kc);
  wp.n = wp.ids + kWarpCache;
  const size_t gw = (size_t)blockIdx.x * kGroupWarps + wid;
  const uint32_t n_start = P.wcache_n[gw];
#pragma unroll 1
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
#pragma unroll 1
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
#pragma unroll 1
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
                               [&](uint32_t p, const uint32_t v[8], uint32_t, uint32_t) {
                                 uint4* q = reinterpret_cast<uint4*>(vals + 256u * p) + 2u * lane;
                                 q[0] = make_uint4(v[0], v[1], v[2], v[3]);
                                 q[1] = make_uint4(v[4], v[5], v[6], v[7]);
                               });
    __syncwarp();
    uint32_t size = ib;  // lane g: the image's bytes after gate g
    const int last = mine ? 31 - __clz((int)mine) : -1;
    // the byte count after a gate in the middle needs a note of every pass
    if (mine & (mine - 1u)) group_note(vals, notes, (1u << NP) - 1u, S);
    for (int g = 0; g <= last; ++g) {
      if (!((mine >> g) & 1u)) continue;
      const GroupGate& q = L.g[g];
      const bool cross = q.kind == 4;  // both warps come here or neither
      if (cross) {
        ++phase;
        if (!lost) lost = !pair_sync(seq, side, phase, ctl, 6u);
      }
      const uint32_t passes = group_passes(q, NP);
      if (q.kind == 3) {
        group_diag(q, vals, (ch & q.pair_bit) ? 1u : 0u, passes, mh, spec);
      } else {
        uint32_t* const ca = side ? peer : vals;
        uint32_t* const cbv = side ? vals : peer;
        switch (q.arith) {
          case 0: group_apply<0>(q, vals, ca, cbv, side, NP, passes, mh, spec); break;
          case 2: group_apply<2>(q, vals, ca, cbv, side, NP, passes, mh, spec); break;
          case 3: group_apply<3>(q, vals, ca, cbv, side, NP, passes, mh, spec); break;
          case 5: group_apply<5>(q, vals, ca, cbv, side, NP, passes, mh, spec); break;
          default: group_apply<4>(q, vals, ca, cbv, side, NP, passes, mh, spec); break;
        }
      }
      if (cross) {
        ++phase;
        if (!lost) lost = !pair_sync(seq, side, phase, ctl, 7u);
      }
      __syncwarp();
      if (g < last) {  // the last one's bytes come from the encoder
        uint32_t bits;
        group_note(vals, notes, passes, S);
        keep &= group_size(vals, notes, NP, S, bits);
        if ((int)lane >= g) size = 16u + cb + resid_bytes(bits);
      }
    }
    // the new image: codes, residuals through the output window, finished blocks to pages
    uint32_t onp = 0u, ooff = 0u;
    bool oom = false;
    if (mine) {
      uint32_t* const owin = win0;
      uint4* const w4 = reinterpret_cast<uint4*>(owin);
#pragma unroll 1
      for (uint32_t k = lane; k < kWinBlocks; k += 32u) w4[k] = make_uint4(0u, 0u, 0u, 0u);
      oom = !wp_grow(P, wp, opg, onp, (16u + cb + kPage - 1u) / kPage);
      __syncwarp();
      uint32_t prv = 0u;
#pragma unroll 1
      for (uint32_t p = 0; p < NP; ++p) {
        const uint4* q8 = reinterpret_cast<const uint4*>(vals + 256u * p) + 2u * lane;
        const uint4 va = q8[0], vb = q8[1];
        const uint32_t v[8] = {va.x, va.y, va.z, va.w, vb.x, vb.y, vb.z, vb.w};
        uint32_t before = __shfl_up_sync(0xffffffffu, v[7], 1);
        if (lane == 0) before = prv;
        prv = __shfl_sync(0xffffffffu, v[7], 31);
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
#pragma unroll 1
          for (uint32_t k = lane; k < nb; k += 32u) {
            const uint32_t b = 16u + cb + 16u * (ob + k);
            reinterpret_cast<uint4*>(P.pages + (unsigned long long)opg[b >> 9] * kPage + (b & (kPage - 1u)))[0] = w4[k];
          }
        if (!end) {
          uint4 carry = make_uint4(0u, 0u, 0u, 0u);
          if (lane == 0) carry = w4[nb];
          __syncwarp();
#pragma unroll 1
          for (uint32_t k = lane; k <= nb; k += 32u) w4[k] = k == 0u ? carry : make_uint4(0u, 0u, 0u, 0u);
          __syncwarp();
        }
      }
      keep = keep && group_differs(vals, NP) && group_moves(vals, NP) && !__any_sync(0xffffffffu, spec);
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
#pragma unroll 1
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
#pragma unroll 1
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
