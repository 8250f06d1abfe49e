// stream.cuh -- STREAM images at S <= 32 bits, one warp a chunk, 256 values a pass (8 per
// lane): what the streaming gate kernels (fast.cu, group.cu) and the readout and codec
// kernels (stream_io.cu) share.
#pragma once
#include "gate_common.cuh"

namespace qc {

constexpr uint32_t kFastWin = 1056;   // bytes of a pass window: 1024 bytes of stream at most, plus alignment and read slack
constexpr uint32_t kWinBlocks = kFastWin / 16;
__host__ __device__ __forceinline__ uint32_t fast_pg_words(int kc) { return (max_pages(kc) + 3u) & ~3u; }
// Largest STREAM image of a chunk at S <= 32 bits.
__host__ __device__ __forceinline__ uint32_t fast_max_image(int kc) {
  return 16u + code_bytes(2u << kc) + resid_bytes(32u * (2u << kc));
}

// Bit position (within a lane's 16-bit code field) of the 2-bit code of the lane's
// value k: four codes per byte, the first in the top bits, bytes in memory order.
__host__ __device__ constexpr uint32_t code_shift(int k) { return 8u * (uint32_t)(k >> 2) + 6u - 2u * (uint32_t)(k & 3); }
// 8 * (code of value k) from the lane's code field.
template <int k>
__device__ __forceinline__ uint32_t code8(uint32_t cw) {
  constexpr uint32_t s = code_shift(k);
  if constexpr (s >= 3) return (cw >> (s - 3)) & 0x18u;
  else return (cw << (3 - s)) & 0x18u;
}
__device__ __forceinline__ uint32_t code8_at(uint32_t cw, int k) {
  switch (k) {
    case 0: return code8<0>(cw);
    case 1: return code8<1>(cw);
    case 2: return code8<2>(cw);
    case 3: return code8<3>(cw);
    case 4: return code8<4>(cw);
    case 5: return code8<5>(cw);
    case 6: return code8<6>(cw);
    default: return code8<7>(cw);
  }
}
__device__ __forceinline__ uint32_t rlen(uint32_t S, uint32_t c8) { return S > c8 ? S - c8 : 0u; }

// Sum of the residual lengths max(S - 8c, 0) of the 8 codes of a lane's 16-bit field.
__device__ __forceinline__ uint32_t rsum8(uint32_t cw, uint32_t S) {
  const uint32_t lo = cw & 0x5555u, hi = (cw >> 1) & 0x5555u;
  const uint32_t n1 = __popc(lo & ~hi), n2 = __popc(hi & ~lo), n3 = __popc(lo & hi);
  return (8u - n1 - n2 - n3) * S + n1 * rlen(S, 8u) + n2 * rlen(S, 16u) + n3 * rlen(S, 24u);
}

// Exclusive warp scan (plus the warp total, to all lanes).
__device__ __forceinline__ uint32_t warp_excl(uint32_t v, uint32_t& total) {
  const uint32_t lane = threadIdx.x & 31u;
  uint32_t inc = v;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const uint32_t u = __shfl_up_sync(0xffffffffu, inc, d);
    if (lane >= (uint32_t)d) inc += u;
  }
  total = __shfl_sync(0xffffffffu, inc, 31);
  return inc - v;
}

// The leading-byte run of a lane, packed: bits 8..31 the bytes its values set, bits 0..1
// the smallest code among them (3: none set).  Composition (earlier A, later B): B's
// explicit bytes replace A's; the smallest code is the smaller of the two.
__device__ __forceinline__ uint32_t lead_compose(uint32_t A, uint32_t B) {
  const uint32_t mb = B & 3u;
  const uint32_t ex = 0xFFFFFF00u & (0xFFFFFFFFu >> (8u * mb));
  return (A & ~ex & 0xFFFFFF00u) | (B & 0xFFFFFF00u) | min(A & 3u, mb);
}
// Exclusive warp scan of lead runs after `carry` (the top bytes of the value before the
// warp's first): returns the top bytes of the lane's predecessor; `after` receives (on
// all lanes) the top bytes of the warp's last value.
__device__ __forceinline__ uint32_t lead_scan_warp(uint32_t W, uint32_t carry, uint32_t& after) {
  const uint32_t lane = threadIdx.x & 31u;
  if (__all_sync(0xffffffffu, (W & 3u) == 0u)) {
    // every lane has a value with code 0 (all three leading bytes explicit): a lane's
    // predecessor's leading bytes are the previous lane's run alone
    uint32_t exc = __shfl_up_sync(0xffffffffu, W, 1);
    if (lane == 0) exc = carry;
    after = __shfl_sync(0xffffffffu, W, 31) & 0xFFFFFF00u;
    return exc & 0xFFFFFF00u;
  }
  uint32_t inc = W;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const uint32_t u = __shfl_up_sync(0xffffffffu, inc, d);
    if (lane >= (uint32_t)d) inc = lead_compose(u, inc);
  }
  uint32_t exc = __shfl_up_sync(0xffffffffu, inc, 1);
  if (lane == 0) exc = 3u;  // empty run
  const uint32_t last = __shfl_sync(0xffffffffu, inc, 31);
  const uint32_t cw = (carry & 0xFFFFFF00u) | 3u;
  after = lead_compose(cw, last) & 0xFFFFFF00u;
  return lead_compose(cw, exc) & 0xFFFFFF00u;
}

// Where a warp reads an image from: pool pages listed in shared memory, or one buffer.
struct PagedImage {
  const uint8_t* pages;
  const uint32_t* ids;
  __device__ __forceinline__ const uint8_t* at(uint32_t b) const {
    return pages + (unsigned long long)ids[b >> 9] * kPage + (b & (kPage - 1u));
  }
};
struct FlatImage {
  const uint8_t* base;
  __device__ __forceinline__ const uint8_t* at(uint32_t b) const { return base + b; }
};

// Stages stream blocks [wb, wb + kWinBlocks) of the input image (only those inside its
// nbs stream blocks) into a window with cp.async.  16-byte block k of the stream is
// image byte 16 + cb + 16k.
template <class Image>
__device__ __forceinline__ void fast_issue_window(const Image& img, uint32_t* win, uint32_t cb, uint32_t wb, uint32_t nbs) {
  const uint32_t lane = threadIdx.x & 31u;
#pragma unroll
  for (uint32_t k = lane; k < kWinBlocks; k += 32u) {
    const uint32_t blk = wb + k;
    if (blk < nbs) cp_async16(win + 4u * k, img.at(16u + cb + 16u * blk));
  }
}

__device__ __forceinline__ double hi_as_double(uint32_t h) { return __longlong_as_double((long long)((uint64_t)h << 32)); }

// The truncated high word of a result (S <= 32: the low word is always cut); a signed
// zero becomes +0.  `spec` is set for a subnormal or non-finite result: a chunk holding
// one is coded at 64 bits or is an error, which the general kernel handles.
__device__ __forceinline__ uint32_t fast_trunc(double v, uint32_t mh, bool& spec) {
  const uint64_t u = (uint64_t)__double_as_longlong(v);
  const uint32_t hi = (uint32_t)(u >> 32), ahi = hi & 0x7fffffffu;
  const bool zero = (ahi | (uint32_t)u) == 0u;
  spec |= (ahi - 0x00100000u) >= 0x7fe00000u && !zero;
  return zero ? 0u : (hi & mh);
}

// The explicit parts of a lane's 8 values from the input window (stream unit q at
// win[(q ^ 1) - w4]), starting at stream bit o; e[k] receives bits [8c, S) of value k's
// high word; returns the lane's lead run (see lead_compose).
__device__ __forceinline__ uint32_t fast_extract(const uint32_t* win, uint32_t w4, uint32_t o, uint32_t cw,
                                                 uint32_t S, uint32_t mh, uint32_t e[8]) {
  uint32_t W = 3u;
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const uint32_t c8 = code8_at(cw, k);
    const uint32_t q = o >> 5;
    const uint32_t x = __funnelshift_l(win[((q + 1u) ^ 1u) - w4], win[(q ^ 1u) - w4], o);
    e[k] = (x >> c8) & mh;
    o += rlen(S, c8);
    const uint32_t ex = 0xFFFFFF00u & (0xFFFFFFFFu >> c8);
    W = (W & ~ex & 0xFFFFFF00u) | (e[k] & ex) | min(W & 3u, c8 >> 3);
  }
  return W;
}

// Rebuilds the high words from the explicit parts: value k takes its copied leading
// bytes from its predecessor (P: the top bytes of the lane's predecessor).
__device__ __forceinline__ void fast_rebuild(uint32_t e[8], uint32_t cw, uint32_t P) {
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    P = e[k] | (P & ~(0xFFFFFFFFu >> code8_at(cw, k)));
    e[k] = P;
  }
}

// 24 - 8 (code) of a value whose XOR with its predecessor is x: with f the index of the
// highest set bit of x | 1, 8 times the leading identical bytes, at most 3, is 24 - (f & 24).
__device__ __forceinline__ uint32_t code_rest(uint32_t x) {
  uint32_t f;
  asm("bfind.u32 %0, %1;" : "=r"(f) : "r"(x | 1u));
  return f & 0x18u;
}
// Its residual bits max(S - 8 code, 0).
__device__ __forceinline__ uint32_t rest_bits(uint32_t rest, uint32_t S) {
  return (uint32_t)max((int)(S + rest) - 24, 0);
}

// Codes of a lane's 8 truncated values (predecessor of the first: pr), as the lane's
// 16-bit code field; `sum` receives their residual-length sum.
__device__ __forceinline__ uint32_t fast_codes(const uint32_t t[8], uint32_t pr, uint32_t S, uint32_t& sum) {
  uint32_t inv = 0u, s = 0u;  // inv: 3 - code, the codes' bits inverted
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const uint32_t r = code_rest(t[k] ^ (k ? t[k - 1] : pr));
    s += rest_bits(r, S);
    inv |= (r >> 3) << code_shift(k);
  }
  sum = s;
  return ~inv & 0xffffu;
}

// Packs the residuals of a lane's 8 values (high words t, codes in the lane's code
// field cw) at stream bit o of a cleared window whose block 0 is stream block w4 / 4
// (stream unit q is win[(q ^ 1) - w4]).  The first unit the lane touches and its last,
// unfinished one may be shared with the neighbouring lanes: atomicOr; units in
// between are stored.
__device__ __forceinline__ void fast_pack(uint32_t* win, uint32_t w4, uint32_t o, const uint32_t t[8], uint32_t cw,
                                          uint32_t S) {
  uint32_t q = o >> 5, fill = o & 31u, cur = 0u;
  bool first = true;
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const uint32_t c8 = code8_at(cw, k);
    const uint32_t r = rlen(S, c8);
    const uint32_t f = t[k] << c8;  // the residual in the top r bits, zeros below
    cur |= f >> fill;
    const uint32_t nf = fill + r;
    if (nf >= 32u) {
      if (first) atomicOr(&win[(q ^ 1u) - w4], cur);
      else win[(q ^ 1u) - w4] = cur;
      first = false;
      ++q;
      cur = __funnelshift_r(0u, f, fill);
      fill = nf - 32u;
    } else {
      fill = nf;
    }
  }
  if (fill > 0u && cur) atomicOr(&win[(q ^ 1u) - w4], cur);
}

// Decodes a STREAM image of ib bytes (header checked: width S, `bits` residual bits) pass by
// pass: f(p, v, tot, cw) receives the high words of the lane's 8 values of pass p, the
// pass's residual bits and the lane's code field.  win: two windows of kFastWin bytes.  False if the residual lengths disagree with the header.
template <class Image, class F>
__device__ __forceinline__ bool stream_decode(const Image& img, int kc, uint32_t S, uint32_t bits, uint32_t ib,
                                              uint32_t* win0, uint32_t* win1, const F& f) {
  const uint32_t lane = threadIdx.x & 31u, N = 2u << kc, cb = N >> 2, NP = N >> 8, nbs = (ib - 16u - cb) >> 4;
  const uint32_t mh = (uint32_t)(trunc_mask(S) >> 32);
  auto codes = [&](uint32_t p) { return *reinterpret_cast<const uint32_t*>(img.at(16u + 64u * p + 4u * (lane >> 1))); };
  uint32_t cw_next = codes(0u), off = 0u, lead = 0u;
  fast_issue_window(img, win0, cb, 0u, nbs);
  cp_async_commit();
#pragma unroll 1
  for (uint32_t p = 0; p < NP; ++p) {
    uint32_t* const win = (p & 1u) ? win1 : win0;
    const uint32_t cw = (cw_next >> (16u * (lane & 1u))) & 0xffffu;
    if (p + 1u < NP) cw_next = codes(p + 1u);
    uint32_t tot;
    const uint32_t ps = off, o = ps + warp_excl(rsum8(cw, S), tot);
    off += tot;
    if (p + 1u < NP) fast_issue_window(img, (p & 1u) ? win0 : win1, cb, off >> 7, nbs);
    cp_async_commit();
    cp_async_wait_group<1>();
    __syncwarp();
    uint32_t v[8], after;
    const uint32_t W = fast_extract(win, 4u * (ps >> 7), o, cw, S, mh, v);
    const uint32_t before = lead_scan_warp(W, lead, after);
    lead = after;
    fast_rebuild(v, cw, before);
    f(p, v, tot, cw);
    __syncwarp();  // every lane is done with the window the next pass refills
  }
  return off == bits;
}

// True if image header hd (length ib) is a STREAM image at S <= 32 bits of a chunk of 2^kc.
__device__ __forceinline__ bool stream32_header(const uint4& hd, uint32_t ib, int kc) {
  const uint32_t N = 2u << kc, cb = N >> 2, S = (hd.x >> 8) & 0xffu;
  return ib >= 16u + cb && ib <= fast_max_image(kc) && (ib & 15u) == 0u && (hd.x & 0xffu) == M_STREAM &&
         (hd.x >> 16) == 0u && S >= 13u && S <= 32u && hd.y + 16u == ib && hd.z == N && cb + resid_bytes(hd.w) == hd.y;
}

// ------------------------------------------- gate kernels: pages, pairs -- //
constexpr uint32_t kWarpCache = 64;   // page ids a warp keeps between its items

// A warp's own page cache in shared memory: ids[0, *n).
struct WarpPages {
  uint32_t* ids;
  uint32_t* n;
};

// All lanes: at least `want` (<= 32) ids in the cache, refilled from the global stack
// half a cache (P.wkeep / 2) at a time.  False (E_OOM set, the stack top restored) if the stack is dry.
__device__ __forceinline__ bool wp_reserve(const Pool& P, const WarpPages& wp, uint32_t want) {
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t n = *wp.n;
  if (n >= want) return true;
  const uint32_t take = max(want - n, P.wkeep / 2u);  // at most 32
  long long old = 0;
  if (lane == 0)
    old = (long long)atomicAdd(reinterpret_cast<unsigned long long*>(&P.ctl->top), (unsigned long long)(-(long long)take));
  old = __shfl_sync(0xffffffffu, old, 0);
  if (old - (long long)take < 0) {  // the stack is dry: give the reservation back (top never stays below 0)
    if (lane == 0) {
      atomicAdd(reinterpret_cast<unsigned long long*>(&P.ctl->top), (unsigned long long)take);
      atomicOr(&P.ctl->err, (unsigned)E_OOM);
    }
    return false;
  }
  if (lane < take) wp.ids[n + lane] = P.stack[old - 1 - (long long)lane];
  __syncwarp();
  if (lane == 0) *wp.n = n + take;
  __syncwarp();
  return true;
}

// All lanes: pushes ids[0, cnt) into the cache; what does not fit goes to the global
// freed list (merged into the stack after the gate).
__device__ __forceinline__ void wp_free(const Pool& P, const WarpPages& wp, const uint32_t* ids, uint32_t cnt) {
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t n = *wp.n, room = P.wkeep > n ? P.wkeep - n : 0u;
  unsigned long long base = 0;
  if (cnt > room) {
    if (lane == 0) base = atomicAdd(&P.ctl->nfreed, (unsigned long long)(cnt - room));
    base = __shfl_sync(0xffffffffu, base, 0);
  }
#pragma unroll 1
  for (uint32_t q = lane; q < cnt; q += 32u) {
    const uint32_t id = ids[q];
    if (q < room) {
      wp.ids[n + q] = id;
    } else {
      const unsigned long long at = base + (q - room);
      if (at < P.npages) P.freed[at] = id;  // the list holds every page at most once
      else atomicOr(&P.ctl->err, (unsigned)E_CORRUPT);
    }
  }
  __syncwarp();
  if (lane == 0) *wp.n = n + min(cnt, room);
  __syncwarp();
}

// All lanes: the output page list grows to `need` pages.
__device__ __forceinline__ bool wp_grow(const Pool& P, const WarpPages& wp, uint32_t* opg, uint32_t& onp,
                                        uint32_t need) {
  while (onp < need) {
    const uint32_t k = min(need - onp, 32u);
    if (!wp_reserve(P, wp, k)) return false;
    const uint32_t lane = threadIdx.x & 31u;
    const uint32_t n = *wp.n;
    if (lane < k) opg[onp + lane] = wp.ids[n - 1u - lane];
    __syncwarp();
    if (lane == 0) *wp.n = n - k;
    __syncwarp();
    onp += k;
  }
  return true;
}

// The two warps of a pair meet through a sequence number per warp in shared memory:
// each raises its own to `phase` (after its earlier shared-memory writes) and waits
// until the partner's has reached it.  The wait is bounded: after kSpinLimit polls it
// sets E_TIMEOUT (and the site) and returns false, so no protocol error can hang the
// kernel.
constexpr uint32_t kSpinLimit = 1u << 22;
__device__ __forceinline__ bool pair_sync(volatile uint32_t* seq, uint32_t side, uint32_t phase, DevCtl* ctl,
                                          uint32_t site) {
  __syncwarp();
  bool ok = true;
  if ((threadIdx.x & 31u) == 0) {
    __threadfence_block();
    seq[side] = phase;
    uint32_t it = 0;
    while ((int)(seq[side ^ 1u] - phase) < 0) {
      if (++it > kSpinLimit) {
        ok = false;
        atomicOr(&ctl->err, (unsigned)E_TIMEOUT);
        atomicExch(&ctl->timeout_site, site);
        break;
      }
    }
    __threadfence_block();
  }
  ok = __shfl_sync(0xffffffffu, ok ? 1u : 0u, 0) != 0u;
  __syncwarp();  // orders lane 0's acquire before the other lanes' reads
  return ok;
}

// The two warps of a pair agree on a flag word: each publishes its own, then both read
// both.  Slots alternate, so a slot is rewritten only after the partner has passed the
// next meeting, i.e. after it read the slot.  A failed wait reads as an error (bit 1).
__device__ __forceinline__ uint32_t pair_agree(uint32_t* slots, volatile uint32_t* seq, uint32_t& phase,
                                               uint32_t side, uint32_t mine, DevCtl* ctl, uint32_t site) {
  volatile uint32_t* s = slots + 2u * (phase & 1u);
  if ((threadIdx.x & 31u) == 0) s[side] = mine;
  ++phase;
  if (!pair_sync(seq, side, phase, ctl, site)) return 2u;
  return s[side ^ 1u];
}

// ------------------------------------------------ gate kernels: arithmetic -- //
// (L: GateLaunch or GroupGate, which name these fields alike.)
// One output amplitude of a dense-class gate: row pair (r, r + 1) of Eq. matrix1 /
// matrix2 over every coefficient (cf: that row pair's eight, from GateLaunch.cf), in
// the order of the kept-term sums; zero coefficients add exact zeros.
__device__ __forceinline__ double2 dense_rows(const double* cf, double2 a, double2 b) {
  return make_double2(__fma_rn(cf[3], b.y, __fma_rn(cf[2], b.x, __fma_rn(cf[1], a.y, __dmul_rn(cf[0], a.x)))),
                      __fma_rn(cf[7], b.x, __fma_rn(cf[6], b.y, __fma_rn(cf[5], a.x, __dmul_rn(cf[4], a.y)))));
}

// The same output for a real matrix (every imaginary coefficient zero): the chains
// above with their zero terms left out -- each dropped term adds an exact zero -- so
// the products of the real parts alone, in the same order (cf[0] = cf[4] = the row's
// first real coefficient, cf[2] = cf[6] its second).
__device__ __forceinline__ double2 real_rows(const double* cf, double2 a, double2 b) {
  return make_double2(__fma_rn(cf[2], b.x, __dmul_rn(cf[0], a.x)), __fma_rn(cf[2], b.y, __dmul_rn(cf[0], a.y)));
}

// The same output for a matrix with a real diagonal and imaginary off-diagonal entries (RX):
// the two products of each chain that are left, in their order (row 0: cf[0], cf[3] and cf[4],
// cf[7]; row 1: cf[1], cf[2] and cf[5], cf[6]).
__device__ __forceinline__ double2 rx_rows(const double* cf, uint32_t row, double2 a, double2 b) {
  const double ax = row ? a.y : a.x, ay = row ? a.x : a.y, bx = row ? b.x : b.y, by = row ? b.y : b.x;
  return make_double2(__fma_rn(cf[3u - row], bx, __dmul_rn(cf[row], ax)), __fma_rn(cf[7u - row], by, __dmul_rn(cf[4u + row], ay)));
}
// Row pair `row` of the dense (0), real (3) or RX (5) form; cf: all sixteen coefficients.
template <int ARITH>
__device__ __forceinline__ double2 form_rows(const double* cf, uint32_t row, double2 a, double2 b) {
  return ARITH == 0 ? dense_rows(cf + 8u * row, a, b)
                    : (ARITH == 3 ? real_rows(cf + 8u * row, a, b) : rx_rows(cf + 8u * row, row, a, b));
}

// The same output for a gate whose coefficient parts are all +-2^k, none zero (sqrt(X),
// sqrt(Y)): every product of the chains above is exact, so each chain equals 2^k times
// the chain of the signed inputs in the same order (scaling by a power of two commutes
// with rounding while no partial sum leaves the normal range): three additions per
// output part, then the scale added to the exponent field.  The inputs are checked
// once per pass (an item holding a value below 2^-959 goes to the general kernel), and
// then no partial sum leaves the normal range: inputs of at least 2^-959 truncated to at
// most 20 mantissa bits are multiples of 2^-979, so a nonzero sum is at least that, and
// 2^k <= 1.  Only an overflow to infinity is left to catch.  Bit q of L.sgn is the sign
// of coefficient cf[q].
template <class Gate>
__device__ __forceinline__ void signed_rows(const Gate& L, uint32_t r, uint32_t ar, uint32_t ai, uint32_t br,
                                            uint32_t bi, uint32_t mh, uint32_t& outr, uint32_t& outi, bool& spec) {
  const uint32_t sg = L.sgn >> (8u * r);
  auto t = [&](int q, uint32_t h) { return hi_as_double(h ^ ((sg >> q) << 31)); };
  const double re = __dadd_rn(__dadd_rn(__dadd_rn(t(0, ar), t(1, ai)), t(2, br)), t(3, bi));
  const double im = __dadd_rn(__dadd_rn(__dadd_rn(t(4, ai), t(5, ar)), t(6, bi)), t(7, br));
  auto scaled = [&](double y) -> uint32_t {
    const uint64_t u = (uint64_t)__double_as_longlong(y);
    const uint32_t hi = (uint32_t)(u >> 32);
    if ((hi & 0x7fffffffu) == 0u && (uint32_t)u == 0u) return 0u;
    spec |= (hi & 0x7ff00000u) == 0x7ff00000u;
    return (hi + ((uint32_t)L.sk << 20)) & mh;
  };
  outr = scaled(re);
  outi = scaled(im);
}

// Row r of a diagonal (x = the amplitude itself) or anti-diagonal (x = its partner)
// gate on x, given as high words: a complex product in the order of the kept-term sums,
// or an exact copy / negation done on the high words (no FP64); results truncated.
template <class Gate>
__device__ __forceinline__ void row_op(const Gate& L, uint32_t r, uint32_t xr, uint32_t xi, uint32_t mh,
                                       uint32_t& outr, uint32_t& outi, bool& spec) {
  const int op = L.rop[r];
  if (op == 0) {
    const double ur = L.du[2u * r], ui = L.du[2u * r + 1u];
    const double x = hi_as_double(xr), y = hi_as_double(xi);
    outr = fast_trunc(__fma_rn(-ui, y, __dmul_rn(ur, x)), mh, spec);
    outi = fast_trunc(__fma_rn(ui, x, __dmul_rn(ur, y)), mh, spec);
  } else if (op == 1) {
    outr = xr & mh;
    outi = xi & mh;
  } else {
    outr = xr ? ((xr ^ 0x80000000u) & mh) : 0u;
    outi = xi ? ((xi ^ 0x80000000u) & mh) : 0u;
  }
}

// Both outputs of an ARITH 4 pair held by one lane.  The first sums of the four chains of
// signed_rows are +-(ar + ai) and +-(ar - ai): two additions serve all four, 10 FP64
// additions instead of 12 (a zero sum's sign may differ; a zero is stored as +0).
template <class Gate>
__device__ __forceinline__ void signed_pair(const Gate& L, uint32_t ar, uint32_t ai, uint32_t br, uint32_t bi,
                                            uint32_t mh, uint32_t o[4], bool& spec) {
  const uint32_t sg = L.sgn;
  const double sum = __dadd_rn(hi_as_double(ar), hi_as_double(ai)), dif = __dsub_rn(hi_as_double(ar), hi_as_double(ai));
  auto first = [&](int q, bool im) {
    const uint32_t sx = (sg >> (im ? q + 1 : q)) << 31, sy = (sg >> (im ? q : q + 1)) << 31;  // signs of ar, ai
    const double m = sx == sy ? sum : dif;
    return __hiloint2double((int)((uint32_t)__double2hiint(m) ^ sx), __double2loint(m));
  };
  auto t = [&](int q, uint32_t h) { return hi_as_double(h ^ ((sg >> q) << 31)); };
  auto scaled = [&](double y) -> uint32_t {
    const uint32_t hi = (uint32_t)__double2hiint(y);
    if (((hi << 1) | (uint32_t)__double2loint(y)) == 0u) return 0u;
    spec |= (hi & 0x7ff00000u) == 0x7ff00000u;
    return (hi + ((uint32_t)L.sk << 20)) & mh;
  };
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    o[2 * r] = scaled(__dadd_rn(__dadd_rn(first(8 * r, false), t(8 * r + 2, br)), t(8 * r + 3, bi)));
    o[2 * r + 1] = scaled(__dadd_rn(__dadd_rn(first(8 * r + 4, true), t(8 * r + 6, bi)), t(8 * r + 7, br)));
  }
}

// A pair of amplitudes (a, b) held by the same lane, a at in-chunk index i: both outputs in
// place, truncated.
template <int ARITH, class Gate>
__device__ __forceinline__ void fast_pair(const Gate& L, uint32_t i, uint32_t& ar, uint32_t& ai, uint32_t& br,
                                          uint32_t& bi, uint32_t mh, bool& spec) {
  uint32_t o[4] = {ar & mh, ai & mh, br & mh, bi & mh};
  if ((i & L.lo_mask) == L.lo_vals) {
    if constexpr (ARITH == 4) {
      signed_pair(L, ar, ai, br, bi, mh, o, spec);
    } else if constexpr (ARITH == 0 || ARITH == 3 || ARITH == 5) {
      const double2 a = make_double2(hi_as_double(ar), hi_as_double(ai)), b = make_double2(hi_as_double(br), hi_as_double(bi));
      const double2 x = form_rows<ARITH>(L.cf, 0u, a, b), y = form_rows<ARITH>(L.cf, 1u, a, b);
      o[0] = fast_trunc(x.x, mh, spec);
      o[1] = fast_trunc(x.y, mh, spec);
      o[2] = fast_trunc(y.x, mh, spec);
      o[3] = fast_trunc(y.y, mh, spec);
    } else {  // anti-diagonal: a' from b, b' from a
      row_op(L, 0u, br, bi, mh, o[0], o[1], spec);
      row_op(L, 1u, ar, ai, mh, o[2], o[3], spec);
    }
  }
  ar = o[0];
  ai = o[1];
  br = o[2];
  bi = o[3];
}

}  // namespace qc
