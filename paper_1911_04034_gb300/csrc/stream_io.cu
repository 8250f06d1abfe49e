// stream_io.cu -- reading the state (amplitude ranges, chunk norms, inner products) and the
// codec entry points on many chunks: a warp per chunk for STREAM images at S <= 32 bits, a
// CTA per chunk for every other image.
#include "gate_item.cuh"
#include "stream.cuh"

namespace qc {

enum { kReadRange, kReadNorm, kReadDot, kReadCodec };
struct ReadArgs {
  Pool P;
  unsigned long long cfirst, nchunks;   // chunks read: [cfirst, cfirst + nchunks)
  unsigned long long first_amp, count;  // kReadRange: the amplitudes wanted
  const double* ref;                    // kReadDot: chunk cfirst's part first
  double* out;
  const uint8_t* in;                    // kReadCodec: images, stride bytes apart, and their lengths
  unsigned long long stride;
  const uint32_t* lens;
  unsigned int* err;
  uint32_t per;                         // chunks a CTA takes at once: kWarps (a warp each first) or 1 (block path only)
};
constexpr uint32_t kReadStage = 1024u;  // a pass's high words
__host__ __device__ __forceinline__ uint32_t read_warp_bytes(int kc) {
  return 2u * kFastWin + 4u * fast_pg_words(kc) + kReadStage;
}
static size_t read_smem_bytes(int kc) {
  const size_t a = codec_smem_bytes(kc), b = (size_t)kWarps * read_warp_bytes(kc);
  return a > b ? a : b;
}

// A warp reads chunk number cl of the call.  False: left to the block path (nothing is lost
// by what was written already: it writes everything again).
template <int MODE>
__device__ __forceinline__ bool read_warp(const ReadArgs& R, unsigned long long cl, uint8_t* smem) {
  const Pool& P = R.P;
  const int kc = P.kc;
  const uint32_t lane = threadIdx.x & 31u;
  uint32_t* const win0 = reinterpret_cast<uint32_t*>(smem);
  uint32_t* const win1 = win0 + kFastWin / 4u;
  uint32_t* const stage = win1 + kFastWin / 4u;
  uint32_t* const ids = stage + kReadStage / 4u;
  const unsigned long long c = R.cfirst + cl;
  uint32_t ib;
  uint4 hd;
  if constexpr (MODE == kReadCodec) {
    ib = R.lens[cl];
    if (ib < 16u || ib > fast_max_image(kc) || (ib & 15u)) return false;
    hd = *reinterpret_cast<const uint4*>(R.in + cl * R.stride);
  } else {
    const uint32_t* e = dir_entry(P, c);
    const uint2 h = *reinterpret_cast<const uint2*>(e);
    ib = h.x;
    if (h.y == 0u || ib > fast_max_image(kc) || h.y != (ib + kPage - 1u) / kPage) return false;
    bool good = true;
    for (uint32_t k = lane; k < h.y; k += 32u) {
      const uint32_t pid = e[4 + k];
      ids[k] = pid;
      good &= pid < P.npages;
    }
    if (!__all_sync(0xffffffffu, good)) return false;
    __syncwarp();
    hd = *reinterpret_cast<const uint4*>(P.pages + (unsigned long long)ids[0] * kPage);
  }
  if (!stream32_header(hd, ib, kc)) return false;
  const uint32_t S = (hd.x >> 8) & 0xffu;
  const bool vec = (reinterpret_cast<uintptr_t>(MODE == kReadDot ? R.ref : R.out) & 15u) == 0u;
  double x = 0.0, y = 0.0, z = 0.0;
  double2 r[4];  // kReadDot: the reference amplitudes of the coming pass
  auto fetch = [&](uint32_t p) {
    const double* s = R.ref + 2ull * ((cl << kc) + 128u * p + 4u * lane);
#pragma unroll
    for (int k = 0; k < 4; ++k)
      r[k] = vec ? reinterpret_cast<const double2*>(s)[k] : make_double2(s[2 * k], s[2 * k + 1]);
  };
  if constexpr (MODE == kReadDot) fetch(0u);
  auto pass = [&](uint32_t p, const uint32_t v[8], uint32_t, uint32_t) {
    if constexpr (MODE == kReadRange || MODE == kReadCodec) {
      // through shared memory: a warp's stores then cover whole lines
      reinterpret_cast<uint4*>(stage)[2u * lane] = make_uint4(v[0], v[1], v[2], v[3]);
      reinterpret_cast<uint4*>(stage)[2u * lane + 1u] = make_uint4(v[4], v[5], v[6], v[7]);
      __syncwarp();
#pragma unroll
      for (uint32_t j = 0; j < 4u; ++j) {
        const uint2 q = reinterpret_cast<const uint2*>(stage)[32u * j + lane];
        unsigned long long a = (c << kc) + 128u * p + 32u * j + lane;
        if (MODE == kReadRange && (a < R.first_amp || a - R.first_amp >= R.count)) continue;
        if (MODE == kReadRange) a -= R.first_amp;
        uint32_t* d = reinterpret_cast<uint32_t*>(R.out + 2ull * a);
        if (vec) {
          *reinterpret_cast<uint4*>(d) = make_uint4(0u, q.x, 0u, q.y);
        } else {
          *reinterpret_cast<uint2*>(d) = make_uint2(0u, q.x);
          *reinterpret_cast<uint2*>(d + 2) = make_uint2(0u, q.y);
        }
      }
    } else {
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const double pr = hi_as_double(v[2 * k]), pi = hi_as_double(v[2 * k + 1]);
        z = __fma_rn(pr, pr, __fma_rn(pi, pi, z));
        if (MODE == kReadDot) {
          x = __fma_rn(r[k].x, pr, __fma_rn(r[k].y, pi, x));
          y = __fma_rn(r[k].x, pi, __fma_rn(-r[k].y, pr, y));
        }
      }
      if (MODE == kReadDot && p + 1u < (2u << kc) / 256u) fetch(p + 1u);
    }
  };
  bool ok;
  if constexpr (MODE == kReadCodec) ok = stream_decode(FlatImage{R.in + cl * R.stride}, kc, S, hd.w, ib, win0, win1, pass);
  else ok = stream_decode(PagedImage{P.pages, ids}, kc, S, hd.w, ib, win0, win1, pass);
  cp_async_wait_all();
  __syncwarp();
  if (!ok) return false;
  if constexpr (MODE == kReadNorm || MODE == kReadDot) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      z += __shfl_xor_sync(0xffffffffu, z, o);
      if (MODE == kReadDot) {
        x += __shfl_xor_sync(0xffffffffu, x, o);
        y += __shfl_xor_sync(0xffffffffu, y, o);
      }
    }
    if (lane == 0) {
      if (MODE == kReadDot) {
        R.out[3 * cl] = x;
        R.out[3 * cl + 1] = y;
        R.out[3 * cl + 2] = z;
      } else {
        R.out[cl] = z;
      }
    }
  }
  return true;
}

// The whole CTA reads chunk number cl.  False: a corrupt entry (error set).
template <int VPT, int MODE>
__device__ __forceinline__ bool read_block(const ReadArgs& R, unsigned long long cl, uint8_t* smem, int& pp, double* red) {
  const Pool& P = R.P;
  const int kc = P.kc;
  const uint32_t A = 1u << kc, N = 2u << kc, cap = MODE == kReadCodec ? codedcap(kc) : imgcap(kc);
  uint64_t* tile = reinterpret_cast<uint64_t*>(smem);
  uint8_t* img = reinterpret_cast<uint8_t*>(tile + tile_words(kc));
  uint32_t* pages = reinterpret_cast<uint32_t*>(img + codedcap(kc));
  ScanSmem& s = *reinterpret_cast<ScanSmem*>(pages + pagelist_words(kc));
  const unsigned long long c = R.cfirst + cl;
  uint32_t len;
  if constexpr (MODE == kReadCodec) {
    len = R.lens[cl];
    const bool fits = len <= cap && (len & 15u) == 0u && len >= 16u;
    if (fits) {
      const uint4* src = reinterpret_cast<const uint4*>(R.in + cl * R.stride);
      for (uint32_t u = threadIdx.x; u < len / 16u; u += kThreads) reinterpret_cast<uint4*>(img)[u] = src[u];
    } else {
      if (threadIdx.x == 0) reinterpret_cast<uint32_t*>(img)[0] = 0xffu;  // fails the header checks
      len = 16u;
    }
    __syncthreads();
  } else {
    const uint32_t* e = dir_entry(P, c);
    len = e[0];
    if (len > cap || e[1] > max_pages(kc)) {
      if (threadIdx.x == 0) atomicOr(R.err, (unsigned)E_CORRUPT);
      return false;
    }
    load_image_block(P, c, img, pages, cap);
  }
  if (!decode_block<VPT>(img, len, kc, tile, s, pp) && threadIdx.x == 0) atomicOr(R.err, (unsigned)E_CORRUPT);
  if constexpr (MODE == kReadCodec) {
    unsigned long long* dst = reinterpret_cast<unsigned long long*>(R.out) + cl * N;
    for (uint32_t j = threadIdx.x; j < N; j += kThreads) dst[j] = tile[tile_val(j)];
  } else if constexpr (MODE == kReadRange) {
    unsigned long long* dst = reinterpret_cast<unsigned long long*>(R.out);
    for (uint32_t i = threadIdx.x; i < A; i += kThreads) {
      const unsigned long long a = (c << kc) + i;
      if (a >= R.first_amp && a < R.first_amp + R.count) {
        dst[2 * (a - R.first_amp)] = tile[tile_val(2 * i)];
        dst[2 * (a - R.first_amp) + 1] = tile[tile_val(2 * i + 1)];
      }
    }
  } else {
    const double* v = reinterpret_cast<const double*>(tile);
    double x = 0.0, y = 0.0, z = 0.0;
    for (uint32_t i = threadIdx.x; i < A; i += kThreads) {
      const double pr = v[tile_val(2 * i)], pi = v[tile_val(2 * i + 1)];
      z = __fma_rn(pr, pr, __fma_rn(pi, pi, z));
      if (MODE == kReadDot) {
        const double rr = R.ref[(cl << kc) * 2 + 2 * i], ri = R.ref[(cl << kc) * 2 + 2 * i + 1];
        x = __fma_rn(rr, pr, __fma_rn(ri, pi, x));
        y = __fma_rn(rr, pi, __fma_rn(-ri, pr, y));
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      z += __shfl_xor_sync(0xffffffffu, z, o);
      if (MODE == kReadDot) {
        x += __shfl_xor_sync(0xffffffffu, x, o);
        y += __shfl_xor_sync(0xffffffffu, y, o);
      }
    }
    const uint32_t w = threadIdx.x >> 5;
    if ((threadIdx.x & 31u) == 0u) {
      red[w] = x;
      red[kWarps + w] = y;
      red[2 * kWarps + w] = z;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      x = y = z = 0.0;
      for (int k = 0; k < kWarps; ++k) {
        x += red[k];
        y += red[kWarps + k];
        z += red[2 * kWarps + k];
      }
      if (MODE == kReadDot) {
        R.out[3 * cl] = x;
        R.out[3 * cl + 1] = y;
        R.out[3 * cl + 2] = z;
      } else {
        R.out[cl] = z;
      }
    }
  }
  __syncthreads();
  return true;
}

// Bound: the decoder's instructions, with the output (16 B an amplitude) or the reference
// next.  A warp walks its chunk with the values in registers: no tile in shared memory, no
// barrier per scan, sums reduced once per chunk.  2^26 amplitudes at 1e-4:
// decoding 405 -> 270 us (codec), norms 891 -> 320 us, inner products 1735 -> 760 us (FP64: six
// multiply-adds an amplitude), a third of them as amplitudes 377 -> 201 us, against a CTA per chunk.
template <int VPT, int MODE>
__global__ void __launch_bounds__(kThreads, VPT >= 16 ? 1 : 3) k_read(const __grid_constant__ ReadArgs R) {
  extern __shared__ __align__(16) uint8_t smem[];
  __shared__ uint32_t s_done[kWarps];
  __shared__ double s_red[3 * kWarps];
  int pp = 0;
  const uint32_t wid = threadIdx.x >> 5;
  for (unsigned long long c0 = (unsigned long long)blockIdx.x * R.per; c0 < R.nchunks;
       c0 += (unsigned long long)gridDim.x * R.per) {
    if (R.per > 1u) {
      const bool done = c0 + wid < R.nchunks && read_warp<MODE>(R, c0 + wid, smem + (size_t)wid * read_warp_bytes(R.P.kc));
      if ((threadIdx.x & 31u) == 0u) s_done[wid] = done;
      __syncthreads();
    }
    for (uint32_t k = 0; k < R.per && c0 + k < R.nchunks; ++k)
      if (R.per == 1u || !s_done[k])
        if (!read_block<VPT, MODE>(R, c0 + k, smem, pp, s_red)) return;
    __syncthreads();  // flags and shared memory are free again
  }
}

// Encodes dense chunks at S <= 32 bits: a warp per chunk, the image built in shared memory
// and written once it is known to be a STREAM image (see fast_item's filters); any other
// chunk gets length 0, is counted in *todo and left to k_codec_encode.  pad: the rest of
// every image's slot is cleared too.
// 2^26 Gaussian amplitudes at 1e-4 in 2^10-amplitude chunks: 857 us (a CTA per chunk, slots
// cleared before it in another 274) -> 396 us with the clearing.
__global__ void __launch_bounds__(kThreads, 3)
    k_stream_encode(const double* in, unsigned long long nchunks, int kc, uint32_t S, uint8_t* out,
                    unsigned long long stride, uint32_t* lens, unsigned int* todo, int pad) {
  extern __shared__ __align__(16) uint8_t smem[];
  const uint32_t lane = threadIdx.x & 31u, wid = threadIdx.x >> 5, warps = blockDim.x >> 5;
  const uint32_t N = 2u << kc, cb = N >> 2, NP = N >> 8, mh = (uint32_t)(trunc_mask(S) >> 32);
  const uint32_t image = fast_max_image(kc);
  uint8_t* const img = smem + (size_t)wid * (image + (1u << (kc - 1)));
  uint32_t* const half = reinterpret_cast<uint32_t*>(img + image);
  uint32_t* const stream = reinterpret_cast<uint32_t*>(img + 16u + cb);
  for (unsigned long long c = (unsigned long long)blockIdx.x * warps + wid; c < nchunks;
       c += (unsigned long long)gridDim.x * warps) {
    const double2* src = reinterpret_cast<const double2*>(in + c * N) + 4u * lane;
    double2 a[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) a[k] = __ldcs(src + k);
    for (uint32_t u = lane; u < image / 16u; u += 32u) reinterpret_cast<uint4*>(img)[u] = make_uint4(0u, 0u, 0u, 0u);
    __syncwarp();
    uint32_t off = 0u, prv = 0u, refr = 0u, refi = 0u, nzor = 0u;
    bool spec = false, cst = true, halves = true, give_up = false;
    for (uint32_t p = 0; p < NP; ++p) {
      uint32_t v[8];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        v[2 * k] = fast_trunc(a[k].x, mh, spec);
        v[2 * k + 1] = fast_trunc(a[k].y, mh, spec);
      }
      if (p + 1u < NP) {
#pragma unroll
        for (int k = 0; k < 4; ++k) a[k] = __ldcs(src + 128u * (p + 1u) + k);
      }
      if (p == 0u) {
        refr = __shfl_sync(0xffffffffu, v[0], 0);
        refi = __shfl_sync(0xffffffffu, v[1], 0);
      }
      uint32_t pr = __shfl_up_sync(0xffffffffu, v[7], 1);
      if (lane == 0) pr = prv;
      prv = __shfl_sync(0xffffffffu, v[7], 31);
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        nzor |= v[k];
        cst &= v[k] == ((k & 1) ? refi : refr);
      }
      if (NP == 1u) {
        const uint32_t x = __shfl_xor_sync(0xffffffffu, v[0], 16), y = __shfl_xor_sync(0xffffffffu, v[5], 16);
        halves &= (x == v[0]) & (y == v[5]);
      } else if (p < NP / 2u) {
        half[32u * p + lane] = v[0] ^ __funnelshift_l(v[5], v[5], 13);
      } else {
        halves &= half[32u * (p - NP / 2u) + lane] == (v[0] ^ __funnelshift_l(v[5], v[5], 13));
      }
      // a first pass of one repeated amplitude or of special values is not a dense chunk
      if (p == 0u && (__all_sync(0xffffffffu, cst) || __any_sync(0xffffffffu, spec))) {
        give_up = true;
        break;
      }
      uint32_t sum, tot;
      const uint32_t cw = fast_codes(v, pr, S, sum);
      fast_pack(stream, 0u, off + warp_excl(sum, tot), v, cw, S);
      *reinterpret_cast<uint16_t*>(img + 16u + 64u * p + 2u * lane) = (uint16_t)cw;
      off += tot;
      __syncwarp();
    }
    const bool any_spec = __any_sync(0xffffffffu, spec), all_cst = __all_sync(0xffffffffu, cst);
    const bool any_nz = __any_sync(0xffffffffu, nzor != 0u), all_halves = __all_sync(0xffffffffu, halves);
    uint4* const dst = reinterpret_cast<uint4*>(out + c * stride);
    uint32_t len = 0u;
    if (!give_up && !any_spec && !all_cst && any_nz && !all_halves) {
      const uint32_t plen = cb + resid_bytes(off);
      len = 16u + plen;
      if (lane == 0) *reinterpret_cast<uint4*>(img) = make_uint4(M_STREAM | (S << 8), plen, N, off);
      __syncwarp();
      for (uint32_t u = lane; u < len / 16u; u += 32u) dst[u] = reinterpret_cast<const uint4*>(img)[u];
      if (pad)
        for (unsigned long long u = len / 16u + lane; u < stride / 16u; u += 32u) dst[u] = make_uint4(0u, 0u, 0u, 0u);
    }
    if (lane == 0) {
      lens[c] = len;
      if (!len) atomicAdd(todo, 1u);
    }
    __syncwarp();  // the image is read before the next chunk clears it
  }
}

// ------------------------------------------------------------- launchers -- //
template <int MODE>
static cudaError_t launch_read(ReadArgs& R, cudaStream_t st) {
  const int kc = R.P.kc;
  const size_t smem = read_smem_bytes(kc);
  const unsigned long long sms = (unsigned long long)num_sms();
  // A warp per chunk from about 2000 chunks on; fewer decode sooner by a CTA each (measurement
  // in 2^9-amplitude chunks: 512 of them 68 us by CTAs, 81 by warps; 2048, 81 and 78).
  R.per = kc >= kFastMinKC && R.nchunks >= 12ull * sms ? (uint32_t)kWarps : 1u;
  const unsigned long long want = (R.nchunks + R.per - 1ull) / R.per, grid = want < 8ull * sms ? want : 8ull * sms;
  QC_VPT_DISPATCH(kc, {
    const cudaError_t e = prep(k_read<V, MODE>, smem);
    if (e != cudaSuccess) return e;
    k_read<V, MODE><<<(unsigned)grid, kThreads, smem, st>>>(R);
  });
  return cudaGetLastError();
}

cudaError_t launch_codec_decode(const uint8_t* in, unsigned long long stride, const uint32_t* lens,
                                unsigned long long nchunks, int kc, double* out, unsigned int* err, cudaStream_t st) {
  ReadArgs R{};
  R.P.kc = kc;
  R.nchunks = nchunks;
  R.in = in;
  R.stride = stride;
  R.lens = lens;
  R.out = out;
  R.err = err;
  return launch_read<kReadCodec>(R, st);
}

cudaError_t launch_decode_range(const Pool& P, unsigned long long first_amp, unsigned long long count, double* out,
                                cudaStream_t st) {
  if (count == 0) return cudaSuccess;
  ReadArgs R{};
  R.P = P;
  R.cfirst = first_amp >> P.kc;
  R.nchunks = ((first_amp + count - 1ull) >> P.kc) - R.cfirst + 1ull;
  R.first_amp = first_amp;
  R.count = count;
  R.out = out;
  R.err = &P.ctl->err;
  return launch_read<kReadRange>(R, st);
}

cudaError_t launch_chunk_norms(const Pool& P, unsigned long long cfirst, unsigned long long nchunks, double* out,
                               cudaStream_t st) {
  ReadArgs R{};
  R.P = P;
  R.cfirst = cfirst;
  R.nchunks = nchunks;
  R.out = out;
  R.err = &P.ctl->err;
  return launch_read<kReadNorm>(R, st);
}

cudaError_t launch_chunk_dots(const Pool& P, unsigned long long cfirst, unsigned long long nchunks, const double* ref,
                              double* out, cudaStream_t st) {
  ReadArgs R{};
  R.P = P;
  R.cfirst = cfirst;
  R.nchunks = nchunks;
  R.ref = ref;
  R.out = out;
  R.err = &P.ctl->err;
  return launch_read<kReadDot>(R, st);
}

cudaError_t launch_stream_encode(const double* in, unsigned long long nchunks, int kc, uint32_t S, uint8_t* out,
                                 unsigned long long stride, uint32_t* lens, unsigned int* todo, bool pad,
                                 cudaStream_t st) {
  const int warps = kc >= 11 ? 4 : kWarps;  // at 2^11 amplitudes four images fill the shared memory eight take below
  const size_t smem = (size_t)warps * (fast_max_image(kc) + (1u << (kc - 1)));
  const cudaError_t e = prep(k_stream_encode, smem);
  if (e != cudaSuccess) return e;
  const unsigned long long want = (nchunks + warps - 1ull) / warps, most = 3ull * num_sms();
  k_stream_encode<<<(unsigned)(want < most ? want : most), 32 * warps, smem, st>>>(in, nchunks, kc, S, out, stride,
                                                                                 lens, todo, pad ? 1 : 0);
  return cudaGetLastError();
}

}  // namespace qc
