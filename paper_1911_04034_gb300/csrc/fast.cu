// fast.cu -- the streaming form of the fused gate kernel (sm_103a).
//
// The general kernel (k_gate) gives a work item of two chunks to a whole CTA: decode
// into shared-memory tiles, apply, encode, each step a CTA-wide pass with barriers.
// For the case that dominates a lossy run -- both input chunks coded as STREAM at a
// width S <= 32 and the output again a STREAM image at the gate's S <= 32 -- this
// kernel gives a work item to a pair of warps instead, one chunk each; a warp walks its
// chunk in passes of 256 values (8 per lane) and keeps every value in registers from
// the decoder through the gate arithmetic to the encoder (a cross-chunk gate swaps the
// partner values of each pass with the other warp through shared memory):
//
//   per pass: codes -> residual lengths -> warp scan of the offsets ->
//             explicit parts from the staged input window -> warp scan of the
//             leading bytes (Section 4.2, Solution C decoding) -> the 2x2 unitary on
//             the amplitude pairs (Section 3.1, Eq. matrix1/matrix2) -> truncation to
//             S bits (Eq. sigbits) -> XOR leading-byte codes -> warp scan of the output
//             offsets -> packing into the output window -> finished 16-byte blocks out
//             to freshly allocated pages.
//
// An in-chunk target t >= 7 puts the partner 2^(t-7) passes on: those passes are held in
// shared memory (kind 4; the general kernel took them before: 26-qubit QAOA layer, its
// share of the general kernel fell from 13.1 ms to under 1).  A cross-chunk diagonal gate
// with a row that is an exact copy (T, CZ, a controlled phase) gives a warp an item to
// itself and rewrites one chunk of it (kind 5): a pair of warps would leave one idle
// (30 qubits with kind 4: 591.8 -> 516.8 ms a layer; 21 qubits 121 -> 66 us a gate).
//
// Scans are warp shuffles and every carry between passes (stream offsets, the
// predecessor's leading bytes, the encoder's predecessor) stays in registers, so the
// kernel has no CTA-wide barrier; the warps of an SM overlap their FP64 arithmetic
// with each other's integer codec work.  Input windows are double-buffered with
// cp.async (the next pass's window is in flight while the current one is decoded).
//
// Anything else goes to the general kernel unchanged: an item whose input images are
// not STREAM at S <= 32, whose output chunk would not be a STREAM image (all-zero,
// constant, possibly periodic -- Section 4.2's period rule needs the whole chunk; a
// chunk whose sampled values all equal their partners half a chunk away is left to
// the general kernel, which runs the full test -- or holding a subnormal or non-finite
// value), or one whose chunk the learned selector granted a SPLIT / PALETTE trial, is
// appended to a device list before any of its state changes, and k_gate runs the list
// right after this kernel.  Both kernels write the bytes the oracle writes.
#include "stream.cuh"

namespace qc {

constexpr int kFastWarps = 8;   // four pairs: the two warps of a pair share a work item, one chunk each
constexpr int kFastPairs = kFastWarps / 2;
constexpr int kFastThreads = 32 * kFastWarps;
#ifndef QC_FAST_MIN_CTAS
#define QC_FAST_MIN_CTAS 3
#endif
constexpr size_t kSmSharedBytes = 227u * 1024u;

// Passes held in a warp's exchange area: two for the partner warp (cross-chunk pairs);
// for an in-chunk target t >= 7 the 2^(t-7) passes between an amplitude and its partner.
__host__ __device__ __forceinline__ uint32_t fast_held(int kind, int target) {
  return kind == 4 && target > 8 ? 1u << (target - 7) : 2u;
}
// Per warp (one chunk): two input windows, one output window, the input and the output
// page ids, the exchange area (1 KB a pass), its page cache, one sample per lane of each
// pass of the chunk's first half.
__host__ __device__ __forceinline__ uint32_t fast_warp_bytes(int kc, uint32_t held) {
  return 3u * kFastWin + 8u * fast_pg_words(kc) + held * 1024u + 4u * kWarpCache + 16u + (1u << (kc - 1));
}

// Shared-memory buffers of one warp (its chunk of the pair's item).
struct FastWarp {
  uint32_t* iwin0;
  uint32_t* iwin1;
  uint32_t* owin;
  uint32_t* ipg;
  uint32_t* opg;
  uint32_t* xch;  // [held passes][256]: decoded high words for the partner warp, or held for the partner pass
  uint32_t* half;  // [passes / 2][32]: one sample per lane of each first-half pass
};

__device__ __forceinline__ FastWarp fast_warp(uint8_t* base, int kc, uint32_t held) {
  FastWarp f;
  f.iwin0 = reinterpret_cast<uint32_t*>(base);
  f.iwin1 = f.iwin0 + kFastWin / 4u;
  f.owin = f.iwin1 + kFastWin / 4u;
  f.ipg = f.owin + kFastWin / 4u;
  f.opg = f.ipg + fast_pg_words(kc);
  f.xch = f.opg + fast_pg_words(kc);
  f.half = f.xch + 256u * held + kWarpCache + 4u;
  return f;
}

// One work item: this warp's chunk (side 0 or 1 of the pair; kind 5: the warp alone, side =
// the row that is not a copy).  Returns 0 when both chunks were committed, 1 when the pair left the item to the general kernel (nothing
// of the state changed), 2 when the pair stops (a device error is set).
// Per-phase SM cycles of a warp when profiling (lane 0 counts): 0 staging (directory
// entries, headers, the partners' agreement, waits for input windows), 1 decoding, 2 the
// gate (with the exchange between the partners), 3 encoding, 4 committing (finished
// blocks, header, codes, directory entry, pages).
struct FastPhases {
  long long* t;  // shared memory: the five sums, then the last clock
  bool on;
  __device__ __forceinline__ void mark(int k) {
    if (on) {
      const long long now = clock64();
      t[k] += now - t[5];
      t[5] = now;
    }
  }
};

template <int KIND, int ARITH>
__device__ __forceinline__ int fast_item(const GateLaunch& L, unsigned long long item, uint32_t S, const FastWarp& fw,
                                         const uint32_t* xpeer, const WarpPages& wp, uint32_t side,
                                         volatile uint32_t* seq, uint32_t* slots, uint32_t& phase, long long& dE,
                                         unsigned long long& rd, unsigned long long& wr, FastPhases& ph) {
  const Pool& P = L.P;
  const int kc = P.kc;
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t N = 2u << kc, cb = N >> 2, NP = N >> 8;
  // this warp's chunk; an in-chunk gate with an odd number of chunks has a last item of one
  const bool whole = L.pair || 2ull * item + 1ull < L.nact;
  unsigned long long ch = 0;
  if (whole) ch = L.pair ? ((item_chunk(L, item) | L.hi_vals) | (side ? L.pair_bit : 0ull))
                         : (item_chunk(L, 2ull * item + side) | L.hi_vals);
  // directory entry and header: a STREAM image at S <= 32, granted no selector trial
  uint32_t ib = 0, inp = 0, Sin = 0, bits_in = 0;
  bool ok = whole && (!L.sel_dec || L.sel_dec[2ull * item + side] == 0u);
  if constexpr (KIND == 5) {
    // the other chunk of the item: an exact copy of itself, whose image stays if it is what
    // the encoder would write (its reading overlaps with this chunk's)
    if (L.sel_dec) ok = ok && L.sel_dec[2ull * item + (side ^ 1u)] == 0u;
    ok = ok && image_stands(P, ch ^ L.pair_bit, S, kDefaultModes);
  }
  if (ok) {
    const uint32_t* e = dir_entry(P, ch);
    const uint2 h = *reinterpret_cast<const uint2*>(e);
    ib = h.x;
    inp = h.y;
    ok = inp >= 1u && ib >= 16u + cb && ib <= fast_max_image(kc) && (ib & 15u) == 0u && inp == (ib + kPage - 1u) / kPage;
    if (ok) {
      bool good = true;
      for (uint32_t k = lane; k < inp; k += 32u) {
        const uint32_t pid = e[4 + k];
        fw.ipg[k] = pid;
        good &= pid < P.npages;
      }
      ok = __all_sync(0xffffffffu, good);
      __syncwarp();
    }
    if (ok) {
      const uint4 hd = *reinterpret_cast<const uint4*>(P.pages + (unsigned long long)fw.ipg[0] * kPage);
      const uint32_t mode = hd.x & 0xffu, lp = (hd.x >> 16) & 0xffu, fl = hd.x >> 24;
      Sin = (hd.x >> 8) & 0xffu;
      bits_in = hd.w;
      ok = mode == M_STREAM && fl == 0u && lp == 0u && Sin >= 13u && Sin <= 32u && hd.y + 16u == ib && hd.z == N &&
           cb + resid_bytes(hd.w) == hd.y;
    }
  }
  unsigned int err = 0;
  if (lane == 0) err = *(volatile unsigned int*)&P.ctl->err;
  err = __shfl_sync(0xffffffffu, err, 0);
  if constexpr (KIND == 5) {  // the warp has the item to itself
    if (err) return 2;
    if (!ok) return 1;
  } else {
    const uint32_t mine = (ok ? 1u : 0u) | (err ? 2u : 0u);
    const uint32_t other = pair_agree(slots, seq, phase, side, mine, P.ctl, 1u);
    if ((mine | other) & 2u) return 2;
    if (!((mine & other) & 1u)) return 1;
  }
  const uint32_t nbs = (ib - 16u - cb) >> 4;
  const PagedImage src{P.pages, fw.ipg};
  // the code word of this lane's values in pass p (image byte 16 + 64 p + 4 (lane / 2))
  auto code_word_at = [&](uint32_t p) -> uint32_t {
    return *reinterpret_cast<const uint32_t*>(src.at(16u + 64u * p + 4u * (lane >> 1)));
  };
  uint32_t cw_next = code_word_at(0u);
  // the first pass's window; output window cleared; the output pages of header and codes
  fast_issue_window(src, fw.iwin0, cb, 0u, nbs);
  cp_async_commit();
  for (uint32_t k = lane; k < kWinBlocks; k += 32u) reinterpret_cast<uint4*>(fw.owin)[k] = make_uint4(0u, 0u, 0u, 0u);
  uint32_t onp = 0u;
  bool oom = !wp_grow(P, wp, fw.opg, onp, (16u + cb + kPage - 1u) / kPage);
  __syncwarp();
  ph.mark(0);
  const uint32_t mh = (uint32_t)(trunc_mask(S) >> 32), mhin = (uint32_t)(trunc_mask(Sin) >> 32);
  uint32_t ioff = 0u, ooff = 0u, lead = 0u, prv = 0u, refr = 0u, refi = 0u, nzor = 0u;
  bool spec = false, cst = true, halves = true, lost = false;
  // KIND 4: an amplitude's partner lies `dist` passes on.  In each group of 2 dist passes,
  // dist steps decode and hold the first half, dist steps decode the second half, form
  // both outputs, encode the first half's and hold the second's, dist steps encode those.
  const uint32_t dist = KIND == 4 ? 1u << (L.target - 7) : 0u;
  uint32_t step = 0u, pdec = 0u, penc = 0u;  // the step in its group, passes decoded and encoded
  while (penc < NP) {
    uint32_t v[8];
    if (KIND != 4 || step < 2u * dist) {
    const uint32_t p = pdec;
    uint32_t* const win = (p & 1u) ? fw.iwin1 : fw.iwin0;
    uint32_t* const wnext = (p & 1u) ? fw.iwin0 : fw.iwin1;
    // residual lengths of this lane's 8 values, their offsets in the pass
    const uint32_t cw = (cw_next >> (16u * (lane & 1u))) & 0xffffu;
    if (p + 1u < NP) cw_next = code_word_at(p + 1u);  // in flight while this pass runs
    uint32_t tot;
    const uint32_t ps = ioff;
    const uint32_t o = ps + warp_excl(rsum8(cw, Sin), tot);
    ioff += tot;
    // the next pass's window is in flight while this pass runs
    if (p + 1u < NP) fast_issue_window(src, wnext, cb, ioff >> 7, nbs);
    cp_async_commit();
    ph.mark(1);
    cp_async_wait_group<1>();
    __syncwarp();
    ph.mark(0);
    // explicit parts, leading bytes from the predecessors
    {
      const uint32_t W = fast_extract(win, 4u * (ps >> 7), o, cw, Sin, mhin, v);
      uint32_t after;
      const uint32_t Pl = lead_scan_warp(W, lead, after);
      lead = after;
      fast_rebuild(v, cw, Pl);
    }
    if constexpr (ARITH == 4) {
      // signed_rows needs every input at least 2^-959 (or zero): each warp checks its own
      // values, and the pair's agreement defers the item if either chunk has one below
#pragma unroll
      for (int k = 0; k < 8; ++k) spec |= ((v[k] & 0x7fffffffu) - 1u) < ((64u << 20) - 1u);  // nonzero, exponent < 64
    }
    ph.mark(1);
    ++pdec;
    }
    if constexpr (KIND == 4) {
      const uint32_t at = step++;
      if (step == 3u * dist) step = 0u;
      uint4* const hold = reinterpret_cast<uint4*>(fw.xch) + 64u * (at & (dist - 1u));
      const uint4 h0 = hold[lane], h1 = hold[32u + lane];
      if (at >= dist) {
        uint32_t a[8] = {h0.x, h0.y, h0.z, h0.w, h1.x, h1.y, h1.z, h1.w};
        if (at < 2u * dist) {
#pragma unroll
          for (int k = 0; k < 4; ++k)
            fast_pair<ARITH>(L, 128u * penc + 4u * lane + (uint32_t)k, a[2 * k], a[2 * k + 1], v[2 * k], v[2 * k + 1], mh, spec);
        }
        if (at < 2u * dist) {
          hold[lane] = make_uint4(v[0], v[1], v[2], v[3]);
          hold[32u + lane] = make_uint4(v[4], v[5], v[6], v[7]);
        }
#pragma unroll
        for (int k = 0; k < 8; ++k) v[k] = a[k];
      } else {
        hold[lane] = make_uint4(v[0], v[1], v[2], v[3]);
        hold[32u + lane] = make_uint4(v[4], v[5], v[6], v[7]);
        continue;
      }
    }
    const uint32_t p = penc++;
    // the gate on every amplitude pair whose in-chunk control bits match; results
    // truncated to S bits in place
    const uint32_t ibase = 128u * p + 4u * lane;  // the lane's first amplitude in the chunk
    uint32_t w[8];                                // the partner amplitudes' high words (kinds 0 and 2)
    if constexpr (KIND == 0 && ARITH != 1) {
      // the partner warp holds the other amplitude of every pair, at the same position
      // (a diagonal gate needs only the amplitude itself)
      uint32_t* xs = fw.xch + 256u * (p & 1u);
      reinterpret_cast<uint4*>(xs)[lane] = make_uint4(v[0], v[1], v[2], v[3]);
      reinterpret_cast<uint4*>(xs)[32u + lane] = make_uint4(v[4], v[5], v[6], v[7]);
      ++phase;
      if (!lost) lost = !pair_sync(seq, side, phase, P.ctl, 2u);
      const uint32_t* xo = xpeer + 256u * (p & 1u);
      const uint4 w0 = reinterpret_cast<const uint4*>(xo)[lane], w1 = reinterpret_cast<const uint4*>(xo)[32u + lane];
      w[0] = w0.x; w[1] = w0.y; w[2] = w0.z; w[3] = w0.w; w[4] = w1.x; w[5] = w1.y; w[6] = w1.z; w[7] = w1.w;
    } else if constexpr (KIND == 2) {
      // partner amplitude i ^ 2^t (2 <= t <= 6): the same slot of lane ^ 2^(t-2)
#pragma unroll
      for (int k = 0; k < 8; ++k) w[k] = __shfl_xor_sync(0xffffffffu, v[k], 1u << (L.target - 2));
    }
    if constexpr (KIND == 1) {
      // partner in the lane: amplitudes k and k ^ 2^t, t = 0 or 1
      if (L.target == 0) {
        fast_pair<ARITH>(L, ibase, v[0], v[1], v[2], v[3], mh, spec);
        fast_pair<ARITH>(L, ibase + 2u, v[4], v[5], v[6], v[7], mh, spec);
      } else {
        fast_pair<ARITH>(L, ibase, v[0], v[1], v[4], v[5], mh, spec);
        fast_pair<ARITH>(L, ibase + 1u, v[2], v[3], v[6], v[7], mh, spec);
      }
    } else if constexpr (KIND != 4) {
      // which row pair this lane's amplitudes take: the pair's second amplitude (b) takes
      // rows 2-3 (kinds 0 and 5: the chunk with the target bit; kind 2: lanes with bit t - 2
      // set; kind 3 per amplitude, bit t)
      const uint32_t lane_row = KIND == 0 || KIND == 5 ? side : (KIND == 2 ? ((lane >> (L.target - 2)) & 1u) : 0u);
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const uint32_t i = ibase + (uint32_t)k;
        const uint32_t row = KIND == 3 ? ((i >> L.target) & 1u) : lane_row;
        const uint32_t i0 = i & ~(1u << (KIND == 0 || KIND == 5 ? 31u : (uint32_t)L.target));
        uint32_t outr = v[2 * k] & mh, outi = v[2 * k + 1] & mh;  // unchanged amplitude, truncated
        if ((i0 & L.lo_mask) == L.lo_vals) {
          if constexpr (ARITH == 4) {
            const uint32_t ar = row ? w[2 * k] : v[2 * k], ai = row ? w[2 * k + 1] : v[2 * k + 1];
            const uint32_t br = row ? v[2 * k] : w[2 * k], bi = row ? v[2 * k + 1] : w[2 * k + 1];
            signed_rows(L, row, ar, ai, br, bi, mh, outr, outi, spec);
          } else if constexpr (ARITH == 0 || ARITH == 3 || ARITH == 5) {
            // a = the pair's first amplitude, b = its second
            const uint32_t ar = row ? w[2 * k] : v[2 * k], ai = row ? w[2 * k + 1] : v[2 * k + 1];
            const uint32_t br = row ? v[2 * k] : w[2 * k], bi = row ? v[2 * k + 1] : w[2 * k + 1];
            const double2 a = make_double2(hi_as_double(ar), hi_as_double(ai));
            const double2 b = make_double2(hi_as_double(br), hi_as_double(bi));
            const double2 out = form_rows<ARITH>(L.cf, row, a, b);
            outr = fast_trunc(out.x, mh, spec);
            outi = fast_trunc(out.y, mh, spec);
          } else if constexpr (ARITH == 1) {
            row_op(L, row, v[2 * k], v[2 * k + 1], mh, outr, outi, spec);
          } else {
            row_op(L, row, w[2 * k], w[2 * k + 1], mh, outr, outi, spec);
          }
        }
        v[2 * k] = outr;
        v[2 * k + 1] = outi;
      }
    }
    ph.mark(2);
    // encoder: constant-chunk and period filters, codes, output offsets
    if (p == 0u) {
      refr = __shfl_sync(0xffffffffu, v[0], 0);
      refi = __shfl_sync(0xffffffffu, v[1], 0);
    }
    uint32_t pr = __shfl_up_sync(0xffffffffu, v[7], 1);
    if (lane == 0) pr = prv;
    prv = __shfl_sync(0xffffffffu, v[7], 31);
    {
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        nzor |= v[k];
        cst &= v[k] == ((k & 1) ? refi : refr);
      }
      // period filter: a chunk with a period below its length equals itself shifted by
      // half a chunk; two values per lane are compared with their partners
      if (NP == 1u) {  // both halves in this pass: lanes 0-15 and 16-31 (every lane shuffles)
        const uint32_t a = __shfl_xor_sync(0xffffffffu, v[0], 16);
        const uint32_t b = __shfl_xor_sync(0xffffffffu, v[5], 16);
        halves &= (a == v[0]) & (b == v[5]);
      } else if (p < NP / 2u) {
        fw.half[32u * p + lane] = v[0] ^ __funnelshift_l(v[5], v[5], 13);
      } else {
        halves &= fw.half[32u * (p - NP / 2u) + lane] == (v[0] ^ __funnelshift_l(v[5], v[5], 13));
      }
    }
    uint32_t osum, otot;
    const uint32_t ocw = fast_codes(v, pr, S, osum);
    const uint32_t ob = ooff >> 7;
    fast_pack(fw.owin, 4u * ob, ooff + warp_excl(osum, otot), v, ocw, S);
    // codes: two lanes fill one 32-bit word
    const uint32_t pairw = ocw | (__shfl_down_sync(0xffffffffu, ocw, 1) << 16);
    if ((lane & 1u) == 0u && !oom) {  // image byte 16 + 64 p + 2 lane
      const uint32_t b = 16u + 64u * p + 2u * lane;
      *reinterpret_cast<uint32_t*>(P.pages + (unsigned long long)fw.opg[b >> 9] * kPage + (b & (kPage - 1u))) = pairw;
    }
    ooff += otot;
    __syncwarp();
    ph.mark(3);
    // finished blocks to the pages (the last pass also its unfinished one, zero-padded)
    const bool last = p + 1u == NP;
    const uint32_t endb = last ? (ooff + 127u) >> 7 : ooff >> 7;
    const uint32_t nb = endb - ob;
    if (!oom) oom = !wp_grow(P, wp, fw.opg, onp, (16u + cb + 16u * endb + kPage - 1u) / kPage);
    const uint4* w4 = reinterpret_cast<const uint4*>(fw.owin);
    if (!oom)
      for (uint32_t k = lane; k < nb; k += 32u) {
        const uint32_t b = 16u + cb + 16u * (ob + k);
        reinterpret_cast<uint4*>(P.pages + (unsigned long long)fw.opg[b >> 9] * kPage + (b & (kPage - 1u)))[0] = w4[k];
      }
    if (!last) {
      uint4 carry = make_uint4(0u, 0u, 0u, 0u);
      if (lane == 0) carry = w4[nb];
      __syncwarp();
      // the unfinished block becomes block 0 of the next pass's window
      uint4* z = reinterpret_cast<uint4*>(fw.owin);
      for (uint32_t k = lane; k <= nb; k += 32u) z[k] = k == 0u ? carry : make_uint4(0u, 0u, 0u, 0u);
      __syncwarp();
    }
    ph.mark(4);
  }
  // every input bit consumed exactly (else the image is corrupt); this chunk a STREAM
  // image unless it is constant or possibly periodic, or holds special values
  const bool corrupt = ioff != bits_in;
  // (every lane takes every vote: a warp-wide primitive must never sit behind a branch)
  const bool any_spec = __any_sync(0xffffffffu, spec), all_cst = __all_sync(0xffffffffu, cst);
  const bool any_nz = __any_sync(0xffffffffu, nzor != 0u), all_halves = __all_sync(0xffffffffu, halves);
  const bool keep = !any_spec && !all_cst && any_nz && !all_halves;
  if (corrupt && lane == 0) atomicOr(&P.ctl->err, (unsigned)E_CORRUPT);
  const uint32_t mine = (keep ? 1u : 0u) | ((corrupt || oom || lost) ? 2u : 0u);
  const uint32_t other = KIND == 5 ? mine : (lost ? 2u : pair_agree(slots, seq, phase, side, mine, P.ctl, 3u));
  if (((mine | other) & 2u) || !((mine & other) & 1u)) {
    wp_free(P, wp, fw.opg, onp);
    cp_async_wait_all();
    __syncwarp();
    return ((mine | other) & 2u) ? 2 : 1;
  }
  // the header, then the directory entry; the old pages freed
  const uint32_t plen = cb + resid_bytes(ooff), bytes = 16u + plen;
  if (lane == 0)
    reinterpret_cast<uint4*>(P.pages + (unsigned long long)fw.opg[0] * kPage)[0] = make_uint4(M_STREAM | (S << 8), plen, N, ooff);
  uint32_t* e = dir_entry(P, ch);
  for (uint32_t k = lane; k < onp; k += 32u) e[4 + k] = fw.opg[k];
  if (lane == 0) {
    *reinterpret_cast<uint4*>(e) = make_uint4(bytes, onp, kDefaultModes, 0u);
    dE += (long long)bytes - (long long)ib;
    rd += ib;
    wr += bytes;
  }
  wp_free(P, wp, fw.ipg, inp);
  ph.mark(4);
  return 0;
}

template <int KIND, int ARITH>
__global__ void __launch_bounds__(kFastThreads, QC_FAST_MIN_CTAS) k_gate_fast(const __grid_constant__ GateLaunch L) {
  extern __shared__ __align__(16) uint8_t smem[];
  __shared__ uint32_t s_slots[kFastPairs][4];
  __shared__ uint32_t s_seq[kFastPairs][2];
  const int kc = L.P.kc;
  const uint32_t lane = threadIdx.x & 31u, wid = threadIdx.x >> 5;
  const uint32_t pr = wid >> 1, side = KIND == 5 ? (uint32_t)L.solo : wid & 1u;
  if (threadIdx.x < 2u * kFastPairs) s_seq[threadIdx.x >> 1][threadIdx.x & 1u] = 0u;
  __syncthreads();  // the only CTA-wide barrier: every sequence number starts at 0
  DevCtl* ctl = L.P.ctl;
  const uint32_t S = gate_bits(L);
  if (S > 32u) {  // lossless or wide values: the general kernel takes the whole gate
    if (blockIdx.x == 0 && threadIdx.x == 0) ctl->fast_all = 1u;
    return;
  }
  const uint32_t held = fast_held(KIND, L.target);
  uint8_t* wb = smem + (size_t)wid * fast_warp_bytes(kc, held);
  const FastWarp fw = fast_warp(wb, kc, held);
  const uint32_t* xpeer = fast_warp(smem + (size_t)(wid ^ 1u) * fast_warp_bytes(kc, held), kc, held).xch;
  // the warp's page cache, kept in global memory between launches
  WarpPages wp;
  wp.ids = fw.xch + 256u * held;
  wp.n = wp.ids + kWarpCache;
  const size_t gw = (size_t)blockIdx.x * kFastWarps + wid;
  const uint32_t n_start = L.P.wcache_n[gw];
  {
    const uint32_t n = n_start;
    for (uint32_t q = lane; q < n; q += 32u) wp.ids[q] = L.P.wcache[gw * kWarpCache + q];
    if (lane == 0) *wp.n = n;
    __syncwarp();
  }
  uint32_t phase = 0;
  __shared__ long long s_ph[kFastWarps][6];
  FastPhases ph;
  ph.t = s_ph[wid];
  ph.on = L.prof && lane == 0;
  if (ph.on) {
    for (int k = 0; k < 5; ++k) ph.t[k] = 0;
    ph.t[5] = clock64();
  }
  long long dE = 0;
  unsigned long long rd = 0, wr = 0, done = 0, deferred = 0;
  constexpr bool solo = KIND == 5;  // an item per warp instead of per pair of warps
  const unsigned long long pairs = (unsigned long long)gridDim.x * (solo ? kFastWarps : kFastPairs);
  for (unsigned long long item = (unsigned long long)blockIdx.x * (solo ? kFastWarps : kFastPairs) + (solo ? wid : pr);
       item < L.items; item += pairs) {
    const int r = fast_item<KIND, ARITH>(L, item, S, fw, xpeer, wp, side, s_seq[pr], s_slots[pr], phase, dE, rd, wr, ph);
    if (r == 2) break;
    if (r == 1) {
      if ((solo || side == 0) && lane == 0) {
        const unsigned long long k = atomicAdd(&ctl->ndefer, 1ull);
        L.defer[k] = (uint32_t)item;
        ++deferred;
      }
    } else if (solo || side == 0) {
      ++done;
    }
  }
  cp_async_wait_all();
  __syncwarp();
  // the warp's cached pages stay with it for the next launch
  {
    const uint32_t n = *wp.n;
    for (uint32_t q = lane; q < n; q += 32u) L.P.wcache[gw * kWarpCache + q] = wp.ids[q];
    if (lane == 0) {
      L.P.wcache_n[gw] = n;
      if (n != n_start) atomicAdd(&ctl->wc_pages, (unsigned long long)((long long)n - (long long)n_start));
    }
  }
  if (lane == 0) {
    if (dE) atomicAdd(&ctl->dE, (unsigned long long)dE);
    if (rd) atomicAdd(&ctl->bytes_in, rd);
    if (wr) atomicAdd(&ctl->bytes_out, wr);
    if (done) atomicAdd(&ctl->fast_items, done);
    if (deferred) atomicAdd(&ctl->fast_deferred, deferred);
    if (ph.on)
      for (int k = 0; k < 5; ++k)
        if (ph.t[k]) atomicAdd(&ctl->phase_cycles[k], (unsigned long long)ph.t[k]);
  }
}

// ------------------------------------------------------------- launchers -- //
template <typename K>
static cudaError_t prep_fast(K kernel, size_t smem) {
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
}

static size_t fast_smem_bytes(int kc, uint32_t held) { return (size_t)kFastWarps * fast_warp_bytes(kc, held); }
int fast_warps() { return kFastWarps; }
int fast_items(int kind) { return kind == 5 ? kFastWarps : kFastPairs; }
int fast_warp_cache() { return (int)kWarpCache; }

int fast_ctas_per_sm(int kc) {
  int n = 0;
  const size_t smem = fast_smem_bytes(kc, 2u);
  prep_fast(k_gate_fast<0, 0>, smem);
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_gate_fast<0, 0>, kFastThreads, smem) != cudaSuccess || n < 1)
    n = 1;
  return n;
}

template <int KIND, int ARITH>
static cudaError_t launch_fast_as(const GateLaunch& L, int grid, size_t smem, cudaStream_t st) {
  const cudaError_t e = prep_fast(k_gate_fast<KIND, ARITH>, smem);
  if (e != cudaSuccess) return e;
  k_gate_fast<KIND, ARITH><<<grid, kFastThreads, smem, st>>>(L);
  return cudaGetLastError();
}

// Kinds and arithmetic forms that occur: cross-chunk pairs of any gate class, in-chunk
// partners of dense, real, RX-like, power-of-two or anti-diagonal gates, in-chunk diagonal gates,
// cross-chunk diagonal gates with a row that is an exact copy.
cudaError_t launch_gate_fast(const GateLaunch& L, int grid, cudaStream_t st) {
  const uint32_t held = fast_held(L.fast_kind, L.target);
  const size_t smem = fast_smem_bytes(L.P.kc, held);
  // held passes take shared memory: no more CTAs than fit at once
  if (held > 2u) grid = min(grid, num_sms() * max(1, (int)(kSmSharedBytes / (smem + 2048u))));
  switch (L.fast_kind * 8 + L.arith) {
    case 0: return launch_fast_as<0, 0>(L, grid, smem, st);
    case 1: return launch_fast_as<0, 1>(L, grid, smem, st);
    case 2: return launch_fast_as<0, 2>(L, grid, smem, st);
    case 3: return launch_fast_as<0, 3>(L, grid, smem, st);
    case 4: return launch_fast_as<0, 4>(L, grid, smem, st);
    case 5: return launch_fast_as<0, 5>(L, grid, smem, st);
    case 8: return launch_fast_as<1, 0>(L, grid, smem, st);
    case 10: return launch_fast_as<1, 2>(L, grid, smem, st);
    case 11: return launch_fast_as<1, 3>(L, grid, smem, st);
    case 12: return launch_fast_as<1, 4>(L, grid, smem, st);
    case 13: return launch_fast_as<1, 5>(L, grid, smem, st);
    case 16: return launch_fast_as<2, 0>(L, grid, smem, st);
    case 18: return launch_fast_as<2, 2>(L, grid, smem, st);
    case 19: return launch_fast_as<2, 3>(L, grid, smem, st);
    case 20: return launch_fast_as<2, 4>(L, grid, smem, st);
    case 21: return launch_fast_as<2, 5>(L, grid, smem, st);
    case 25: return launch_fast_as<3, 1>(L, grid, smem, st);
    case 32: return launch_fast_as<4, 0>(L, grid, smem, st);
    case 34: return launch_fast_as<4, 2>(L, grid, smem, st);
    case 35: return launch_fast_as<4, 3>(L, grid, smem, st);
    case 36: return launch_fast_as<4, 4>(L, grid, smem, st);
    case 37: return launch_fast_as<4, 5>(L, grid, smem, st);
    case 41: return launch_fast_as<5, 1>(L, grid, smem, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace qc
