// kernels.cu -- CUDA kernels of libqcsim (sm_103a).
//
// k_gate   the fused persistent kernel of the hot path: for each work item (two
//          chunks) it stages the compressed images in shared memory, decodes them,
//          applies the gate to every amplitude pair (Section 3.1, Eq. matrix1/2) and
//          re-encodes them with the hybrid codec (Section 4.2, Solution C) under the
//          bound chosen by the controller (Section 3.7), then commits the new images
//          to the page pool.  Decoded amplitudes never leave shared memory.
// k_post   after each gate: returns freed pages to the stack, adds the gate's byte
//          change to E, and records the controller's level and fidelity bounds.
// others   image exchange, initialisation, the general codec encoder, checkpoints.
#include "launch.h"
#include "gate_item.cuh"

namespace qc {

int vpt_for(int kc) {
  const int N = 2 << kc;
  return N <= kThreads ? 1 : N / kThreads;
}
size_t gate_smem_bytes(int kc) {
  return 2 * size_t(tile_words(kc)) * 8 + 2 * size_t(imgbuf(kc)) + 4 * size_t(dir_stride(kc)) +
         round16(sizeof(ScanSmem));
}
size_t codec_smem_bytes(int kc) {
  return size_t(tile_words(kc)) * 8 + size_t(codedcap(kc)) + 4 * size_t(pagelist_words(kc)) + round16(sizeof(ScanSmem));
}

template <int VPT>
__global__ void __launch_bounds__(kThreads, VPT >= 16 ? 1 : QC_GATE_MIN_CTAS) k_gate(const __grid_constant__ GateLaunch L) {
  extern __shared__ __align__(16) uint8_t smem[];
  __shared__ long long s_ph[7];
  __shared__ int s_oom;
  __shared__ uint32_t s_np[2];
  __shared__ uint32_t s_cache[kCacheCap];
  __shared__ uint32_t s_cache_n;
  __shared__ CtaAcc s_acc;
  const GateSmem m = gate_smem(smem, L.P.kc, L.P.dir_words, s_ph, &s_oom, s_np);
  GateCta st;
  st.cc.ids = s_cache;
  st.cc.n = &s_cache_n;
  st.acc = &s_acc;
  cta_begin(L.P, st, L.prof, s_ph);
  const uint32_t S = gate_bits(L);
  const unsigned long long serial = L.P.ctl->gates + 1ull;
  const bool bc_on = L.bc != nullptr && L.P.ctl->bc_off == 0u;
  // all items of the gate, or (list) those the streaming kernel left to this one
  const bool listed = L.list && !L.P.ctl->fast_all;
  const unsigned long long count = listed ? L.P.ctl->ndefer : L.items;
  for (unsigned long long k = blockIdx.x; k < count; k += gridDim.x) {
    const unsigned long long nk = k + gridDim.x;
    const unsigned long long item = listed ? (unsigned long long)L.defer[k] : k;
    const unsigned long long nx = nk < count ? (listed ? (unsigned long long)L.defer[nk] : nk) : ~0ull;
    if (!gate_item<VPT, true>(L, item, nx, S, serial, bc_on, m, st)) break;
  }
  cp_async_wait_all();  // no copy may still target shared memory at exit
  bulk_wait_all();      // nor read from it
  cta_end(L, st, s_ph);
}

// Many simulators in one launch: job j is one gate of one simulator, and its work
// items are the global items [begin_j, begin_{j+1}).  All simulators share chunk_log2.
template <int VPT>
__global__ void __launch_bounds__(kThreads, VPT >= 16 ? 1 : QC_GATE_MIN_CTAS)
    k_gate_batch(const BatchJob* __restrict__ jobs, int njobs, unsigned long long total) {
  extern __shared__ __align__(16) uint8_t smem[];
  __shared__ long long s_ph[7];
  __shared__ int s_oom;
  __shared__ uint32_t s_np[2];
  __shared__ uint32_t s_cache[kCacheCap];
  __shared__ uint32_t s_cache_n;
  __shared__ CtaAcc s_acc;
  const GateSmem m = gate_smem(smem, jobs[0].L.P.kc, jobs[0].L.P.dir_words, s_ph, &s_oom, s_np);
  GateCta st;
  st.cc.ids = s_cache;
  st.cc.n = &s_cache_n;
  st.acc = &s_acc;
  int cur = -1;
  uint32_t S = 64;
  unsigned long long serial = 0;
  bool bc_on = false;
  for (unsigned long long g = blockIdx.x; g < total; g += gridDim.x) {
    int lo = 0, hi = njobs - 1;  // last job whose first item is <= g
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (jobs[mid].begin <= g) lo = mid;
      else hi = mid - 1;
    }
    if (lo != cur) {
      if (cur >= 0) cta_end(jobs[cur].L, st, s_ph);
      cur = lo;
      __syncthreads();  // the previous job's items are done with the shared parameters
      cta_begin(jobs[cur].L.P, st, jobs[cur].L.prof, s_ph);
      S = gate_bits(jobs[cur].L);
      serial = jobs[cur].L.P.ctl->gates + 1ull;
      bc_on = jobs[cur].L.bc != nullptr && jobs[cur].L.P.ctl->bc_off == 0u;
    }
    gate_item<VPT, false>(jobs[cur].L, g - jobs[cur].begin, ~0ull, S, serial, bc_on, m, st);
  }
  bulk_wait_all();  // no bulk page store may still read shared memory at exit
  if (cur >= 0) cta_end(jobs[cur].L, st, s_ph);
}

// swap_item over a gate's items, a warp per item, the others to the deferred list; bound by
// directory traffic.  18 qubits, 2^10-amplitude chunks: 22 us a
// gate decoded and encoded by the streaming kernel, 3.1 us exchanged.
__global__ void __launch_bounds__(256) k_swap(const __grid_constant__ GateLaunch L) {
  DevCtl* ctl = L.P.ctl;
  if (*(volatile unsigned int*)&ctl->err != 0u) return;
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t S = gate_bits(L);
  const unsigned long long warps = (unsigned long long)gridDim.x * (blockDim.x >> 5);
  unsigned long long done = 0, left = 0, coded = 0;
  for (unsigned long long item = (unsigned long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); item < L.items;
       item += warps) {
    if (swap_item(L, item, S, coded)) {
      ++done;
    } else {
      if (lane == 0) L.defer[atomicAdd(&ctl->ndefer, 1ull)] = (uint32_t)item;
      ++left;
    }
  }
  if (lane == 0) {
    if (S <= 32u) {
      if (done) atomicAdd(&ctl->fast_items, done);
      if (left) atomicAdd(&ctl->fast_deferred, left);
    }
    count_swap_trials(L, ctl, coded);
  }
}

__global__ void __launch_bounds__(1024) k_post(const Pool P, const CtlParams cp, int grid_ctas) {
  post_body(P, cp, grid_ctas);
}

// One block per job of a batched launch.
__global__ void __launch_bounds__(1024) k_post_batch(const BatchJob* __restrict__ jobs, int grid_ctas) {
  const BatchJob& j = jobs[blockIdx.x];
  post_body(j.L.P, j.L.ctl, grid_ctas);
}

// ------------------------------------------------------------ initialise -- //
__global__ void k_pool_init(const Pool P, unsigned long long nchunks) {
  const unsigned long long stride = (unsigned long long)gridDim.x * blockDim.x;
  for (unsigned long long i = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; i < P.npages; i += stride)
    P.stack[i] = (uint32_t)i;
  // every chunk starts as a ZERO image held inline: header only, all fields 0
  for (unsigned long long c = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; c < nchunks; c += stride) {
    uint32_t* e = dir_entry(P, c);
    e[0] = 16u;
    e[1] = 0u;
    e[2] = kAllModes;  // a ZERO image under any mode set
    e[3] = 0u;
    e[4] = e[5] = e[6] = e[7] = 0u;
  }
}

// Chunk 0 holds amplitude 1 at index 0 (the state |0...0>), encoded losslessly.
template <int VPT>
__global__ void __launch_bounds__(kThreads) k_init_chunk0(const Pool P, unsigned long long nchunks) {
  extern __shared__ __align__(16) uint8_t smem[];
  const int kc = P.kc;
  const uint32_t N = 2u << kc, cap = codedcap(kc);
  uint64_t* tile = reinterpret_cast<uint64_t*>(smem);
  uint8_t* img = reinterpret_cast<uint8_t*>(tile + tile_words(kc));
  uint32_t* pages = reinterpret_cast<uint32_t*>(img + cap);
  ScanSmem& s = *reinterpret_cast<ScanSmem*>(pages + pagelist_words(kc));
  __shared__ uint32_t s_np;
  __shared__ int s_ok;
  for (uint32_t j = threadIdx.x; j < N; j += kThreads) tile[tile_val(j)] = j == 0 ? 0x3FF0000000000000ull : 0ull;
  __syncthreads();
  int pp = 0;
  const uint32_t n0 = encode_block<VPT>(tile, kc, 64u, -1, kDefaultModes, img, imgcap(kc), s, pp, &P.ctl->err);
  __shared__ uint32_t s_cache_n;
  if (threadIdx.x < 32u) {
    const uint32_t q0 = pages_for(n0, kc);
    if (threadIdx.x == 0) s_cache_n = 0u;
    __syncwarp();
    CtaCache cc;
    cc.ids = nullptr;  // empty cache: every page comes from the stack
    cc.n = &s_cache_n;
    const bool ok = n0 != 0u && alloc_pages_warp(P, cc, pages, q0, nullptr, 0u);
    if (threadIdx.x == 0) {
      s_np = q0;
      s_ok = ok;
      if (!ok) atomicOr(&P.ctl->err, (unsigned)E_OOM);
    }
  }
  __syncthreads();
  if (!s_ok) return;
  store_image_block(P, 0ull, img, n0, pages, s_np);
  if (threadIdx.x == 0) dir_entry(P, 0ull)[2] = kDefaultModes;
  if (threadIdx.x == 0) {
    P.ctl->E = 16ull * (nchunks - 1ull) + n0;
    P.ctl->Emax = P.ctl->E;
    P.ctl->n64 = ((reinterpret_cast<const uint32_t*>(img)[0] >> 8) & 0xffu) == 64u ? 1 : 0;
    P.ctl->peak_pages = P.npages - (unsigned long long)P.ctl->top;
  }
}

// -------------------------------------------------------- codec entries -- //
template <int VPT>
__global__ void __launch_bounds__(kThreads)
    k_codec_encode(const double* in, unsigned long long nchunks, int kc, uint32_t S, int force, uint32_t modes,
                   uint8_t* out, unsigned long long stride, uint32_t* lens, unsigned int* err,
                   const unsigned int* todo, int pad) {
  if (todo && *todo == 0u) return;  // only the chunks of length 0 (k_stream_encode), of which there are none
  extern __shared__ __align__(16) uint8_t smem[];
  const uint32_t N = 2u << kc, cap = codedcap(kc);
  uint64_t* tile = reinterpret_cast<uint64_t*>(smem);
  uint8_t* img = reinterpret_cast<uint8_t*>(tile + tile_words(kc));
  uint32_t* pages = reinterpret_cast<uint32_t*>(img + cap);
  ScanSmem& s = *reinterpret_cast<ScanSmem*>(pages + pagelist_words(kc));
  int pp = 0;
  for (unsigned long long c = blockIdx.x; c < nchunks; c += gridDim.x) {
    if (todo && lens[c] != 0u) continue;
    const unsigned long long* src = reinterpret_cast<const unsigned long long*>(in) + c * N;
    for (uint32_t j = threadIdx.x; j < N; j += kThreads) tile[tile_val(j)] = src[j];
    __syncthreads();
    const uint32_t n = encode_block<VPT>(tile, kc, S, force, modes, img, cap, s, pp, err);
    uint4* dst = reinterpret_cast<uint4*>(out + c * stride);
    const uint4* sv = reinterpret_cast<const uint4*>(img);
    for (uint32_t u = threadIdx.x; u < n / 16u; u += kThreads) dst[u] = sv[u];
    if (pad)
      for (unsigned long long u = n / 16u + threadIdx.x; u < stride / 16u; u += kThreads) dst[u] = make_uint4(0u, 0u, 0u, 0u);
    if (threadIdx.x == 0) lens[c] = n;
    __syncthreads();
  }
}

// --------------------------------------------------------------- readout -- //
// Chunks per mode (counts[8]) and, if wide is not null, the images whose header says
// S = 64 (added to *wide).
__global__ void k_mode_counts(const Pool P, unsigned long long nchunks, unsigned long long* counts,
                              unsigned long long* wide) {
  __shared__ unsigned long long sc[9];
  if (threadIdx.x < 9) sc[threadIdx.x] = 0;
  __syncthreads();
  const unsigned long long stride = (unsigned long long)gridDim.x * blockDim.x;
  for (unsigned long long c = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; c < nchunks; c += stride) {
    const uint32_t* e = dir_entry(P, c);
    uint32_t h = e[4];
    if (e[1] != 0u) h = *reinterpret_cast<const uint32_t*>(P.pages + (unsigned long long)e[4] * kPage);
    atomicAdd(&sc[h & 7u], 1ull);
    if (((h >> 8) & 0xffu) == 64u) atomicAdd(&sc[8], 1ull);
  }
  __syncthreads();
  if (threadIdx.x < 8 && sc[threadIdx.x]) atomicAdd(&counts[threadIdx.x], sc[threadIdx.x]);
  if (threadIdx.x == 8 && wide && sc[8]) atomicAdd(wide, sc[8]);
}

__global__ void k_copy_image(const Pool P, unsigned long long chunk, uint8_t* out) {
  const uint32_t* e = dir_entry(P, chunk);
  const uint32_t b = e[0], np = e[1];
  if (b > max_image_bytes(P.kc) || np > max_pages(P.kc)) return;
  for (uint32_t u = threadIdx.x; u < b / 16u; u += blockDim.x) {
    uint4 v;
    if (np == 0) v = reinterpret_cast<const uint4*>(e + 4)[u];
    else v = reinterpret_cast<const uint4*>(P.pages + (unsigned long long)e[4 + u / (kPage / 16)] * kPage)[u % (kPage / 16)];
    reinterpret_cast<uint4*>(out)[u] = v;
  }
}

// ------------------------------------------------------ uncompressed path -- //
__global__ void k_sv_init(double2* psi, unsigned long long amps) {
  const unsigned long long stride = (unsigned long long)gridDim.x * blockDim.x;
  for (unsigned long long i = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; i < amps; i += stride)
    psi[i] = make_double2(i == 0 ? 1.0 : 0.0, 0.0);
}

// ----------------------------------------------------------- checkpoint -- //
// Section 3.5: the compressed state is saved as its chunk images and restored by
// rebuilding the directory and the page arena around them.

// Image length of every chunk (directory entry word 0).
__global__ void k_ck_lengths(const Pool P, unsigned long long nchunks, uint32_t* len) {
  const unsigned long long stride = (unsigned long long)gridDim.x * blockDim.x;
  for (unsigned long long c = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; c < nchunks; c += stride)
    len[c] = dir_entry(P, c)[0];
}

// Copies every chunk's image to out + off[c] (one warp per chunk; off multiples of 16).
__global__ void k_ck_gather(const Pool P, unsigned long long nchunks, const unsigned long long* off, uint8_t* out) {
  const unsigned long long warps = (unsigned long long)gridDim.x * (blockDim.x / 32u);
  const uint32_t lane = threadIdx.x & 31u;
  constexpr uint32_t upp = kPage / 16;
  for (unsigned long long c = blockIdx.x * (unsigned long long)(blockDim.x / 32u) + threadIdx.x / 32u; c < nchunks;
       c += warps) {
    const uint32_t* e = dir_entry(P, c);
    const uint32_t units = e[0] >> 4, np = e[1];
    uint4* dst = reinterpret_cast<uint4*>(out + off[c]);
    for (uint32_t u = lane; u < units; u += 32u)
      dst[u] = np == 0u ? reinterpret_cast<const uint4*>(e + 4)[u]
                        : reinterpret_cast<const uint4*>(P.pages + (unsigned long long)e[4 + u / upp] * kPage)[u % upp];
  }
}

// Writes chunk c's image from in + off[c] (len[c] bytes) back: inline in the directory
// entry when it fits, else into pages pbase[c], pbase[c] + 1, ...
__global__ void k_ck_scatter(const Pool P, unsigned long long nchunks, const unsigned long long* off,
                             const unsigned long long* pbase, const uint32_t* len, const uint8_t* in) {
  const unsigned long long warps = (unsigned long long)gridDim.x * (blockDim.x / 32u);
  const uint32_t lane = threadIdx.x & 31u;
  constexpr uint32_t upp = kPage / 16;
  for (unsigned long long c = blockIdx.x * (unsigned long long)(blockDim.x / 32u) + threadIdx.x / 32u; c < nchunks;
       c += warps) {
    uint32_t* e = dir_entry(P, c);
    const uint32_t bytes = len[c], units = bytes >> 4, np = pages_for(bytes, P.kc);
    const uint4* src = reinterpret_cast<const uint4*>(in + off[c]);
    for (uint32_t u = lane; u < units; u += 32u) {
      if (np == 0u) reinterpret_cast<uint4*>(e + 4)[u] = src[u];
      else reinterpret_cast<uint4*>(P.pages + (pbase[c] + u / upp) * kPage)[u % upp] = src[u];
    }
    if (np) for (uint32_t k = lane; k < np; k += 32u) e[4 + k] = (uint32_t)(pbase[c] + k);
    if (lane == 0) {
      e[0] = bytes;
      e[1] = np;
      e[2] = e[3] = 0u;
    }
  }
}

// After a restore pages [0, used) hold images: the free stack lists the others.
__global__ void k_ck_stack(const Pool P, unsigned long long used) {
  const unsigned long long stride = (unsigned long long)gridDim.x * blockDim.x;
  for (unsigned long long i = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; used + i < P.npages; i += stride)
    P.stack[i] = (uint32_t)(used + i);
}

// ------------------------------------------------------------- launchers -- //
int num_sms() {
  static int sms = 0;
  if (!sms) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (sms <= 0) sms = 1;
  }
  return sms;
}

int gate_ctas_per_sm(int kc) {
  int n = 0;
  const size_t smem = gate_smem_bytes(kc);
  cudaError_t e = cudaSuccess;
  switch (vpt_for(kc)) {
    case 1: prep(k_gate<1>, smem); e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_gate<1>, kThreads, smem); break;
    case 2: prep(k_gate<2>, smem); e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_gate<2>, kThreads, smem); break;
    case 4: prep(k_gate<4>, smem); e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_gate<4>, kThreads, smem); break;
    case 8: prep(k_gate<8>, smem); e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_gate<8>, kThreads, smem); break;
    case 16: prep(k_gate<16>, smem); e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_gate<16>, kThreads, smem); break;
  }
  if (e != cudaSuccess || n < 1) n = 1;
  return n;
}

cudaError_t launch_gate(const GateLaunch& L, int grid, cudaStream_t st) {
  const size_t smem = gate_smem_bytes(L.P.kc);
  QC_VPT_DISPATCH(L.P.kc, {
    cudaError_t e = prep(k_gate<V>, smem);
    if (e != cudaSuccess) return e;
    k_gate<V><<<grid, kThreads, smem, st>>>(L);
  });
  return cudaGetLastError();
}

cudaError_t launch_swap(const GateLaunch& L, cudaStream_t st) {
  const unsigned long long want = (L.items + 7ull) / 8ull, most = (unsigned long long)num_sms() * 8ull;
  k_swap<<<(unsigned)(want < most ? want : most), 256, 0, st>>>(L);
  return cudaGetLastError();
}

cudaError_t launch_post(const Pool& P, const CtlParams& cp, int grid_ctas, cudaStream_t st) {
  k_post<<<1, 1024, 0, st>>>(P, cp, grid_ctas);
  return cudaGetLastError();
}

cudaError_t launch_gate_batch(const BatchJob* jobs, int njobs, unsigned long long total, int kc, int grid,
                              cudaStream_t st) {
  const size_t smem = gate_smem_bytes(kc);
  QC_VPT_DISPATCH(kc, {
    cudaError_t e = prep(k_gate_batch<V>, smem);
    if (e != cudaSuccess) return e;
    k_gate_batch<V><<<grid, kThreads, smem, st>>>(jobs, njobs, total);
  });
  return cudaGetLastError();
}

cudaError_t launch_post_batch(const BatchJob* jobs, int njobs, int grid_ctas, cudaStream_t st) {
  k_post_batch<<<njobs, 1024, 0, st>>>(jobs, grid_ctas);
  return cudaGetLastError();
}

cudaError_t launch_pool_init(const Pool& P, unsigned long long nchunks, cudaStream_t st) {
  k_pool_init<<<num_sms() * 4, 256, 0, st>>>(P, nchunks);
  return cudaGetLastError();
}

cudaError_t launch_init_chunk0(const Pool& P, unsigned long long nchunks, cudaStream_t st) {
  const size_t smem = codec_smem_bytes(P.kc);
  QC_VPT_DISPATCH(P.kc, {
    cudaError_t e = prep(k_init_chunk0<V>, smem);
    if (e != cudaSuccess) return e;
    k_init_chunk0<V><<<1, kThreads, smem, st>>>(P, nchunks);
  });
  return cudaGetLastError();
}

cudaError_t launch_codec_encode(const double* in, unsigned long long nchunks, int kc, uint32_t S, int force,
                                uint8_t* out, unsigned long long stride, uint32_t* lens, unsigned int* err,
                                cudaStream_t st) {
  return launch_codec_encode(in, nchunks, kc, S, force, kDefaultModes, out, stride, lens, err, nullptr, false, st);
}

cudaError_t launch_codec_encode(const double* in, unsigned long long nchunks, int kc, uint32_t S, int force,
                                uint32_t modes, uint8_t* out, unsigned long long stride, uint32_t* lens,
                                unsigned int* err, unsigned int* todo, bool pad, cudaStream_t st) {
  const size_t smem = codec_smem_bytes(kc);
  const unsigned long long sms = (unsigned long long)num_sms(), g = nchunks < sms * 8 ? nchunks : sms * 8;
  // Solution C's modes at S <= 32 on enough chunks: a warp per chunk first, then the general
  // encoder on the chunks it left.  (With fewer chunks a CTA each is sooner done.)
  const bool warp = todo && force < 0 && modes == kDefaultModes && S <= 32u && kc >= kFastMinKC &&
                    nchunks >= 12ull * sms && (reinterpret_cast<uintptr_t>(in) & 15u) == 0u;
  if (warp) {
    const cudaError_t e = launch_stream_encode(in, nchunks, kc, S, out, stride, lens, todo, pad, st);
    if (e != cudaSuccess) return e;
  }
  QC_VPT_DISPATCH(kc, {
    cudaError_t e = prep(k_codec_encode<V>, smem);
    if (e != cudaSuccess) return e;
    k_codec_encode<V><<<(unsigned)g, kThreads, smem, st>>>(in, nchunks, kc, S, force, modes, out, stride, lens, err,
                                                          warp ? todo : nullptr, pad ? 1 : 0);
  });
  return cudaGetLastError();
}

cudaError_t launch_mode_counts(const Pool& P, unsigned long long nchunks, unsigned long long* counts,
                               unsigned long long* wide, cudaStream_t st) {
  const unsigned long long blocks = (nchunks + 255ull) / 256ull;
  const unsigned g = (unsigned)(blocks < (unsigned long long)num_sms() * 8 ? blocks : (unsigned long long)num_sms() * 8);
  k_mode_counts<<<g, 256, 0, st>>>(P, nchunks, counts, wide);
  return cudaGetLastError();
}

cudaError_t launch_copy_image(const Pool& P, unsigned long long chunk, uint8_t* out, cudaStream_t st) {
  k_copy_image<<<1, 256, 0, st>>>(P, chunk, out);
  return cudaGetLastError();
}

cudaError_t launch_sv_init(double* psi, unsigned long long amps, cudaStream_t st) {
  k_sv_init<<<num_sms() * 8, 256, 0, st>>>(reinterpret_cast<double2*>(psi), amps);
  return cudaGetLastError();
}

cudaError_t launch_checkpoint_lengths(const Pool& P, unsigned long long nchunks, uint32_t* len, cudaStream_t st) {
  const unsigned long long g = (nchunks + 255) / 256;
  k_ck_lengths<<<(unsigned)(g < 65535ull ? g : 65535ull), 256, 0, st>>>(P, nchunks, len);
  return cudaGetLastError();
}
cudaError_t launch_checkpoint_gather(const Pool& P, unsigned long long nchunks, const unsigned long long* off,
                                     uint8_t* out, cudaStream_t st) {
  k_ck_gather<<<num_sms() * 8, 256, 0, st>>>(P, nchunks, off, out);
  return cudaGetLastError();
}
cudaError_t launch_checkpoint_scatter(const Pool& P, unsigned long long nchunks, const unsigned long long* off,
                                      const unsigned long long* pbase, const uint32_t* len, const uint8_t* in,
                                      unsigned long long used, cudaStream_t st) {
  k_ck_scatter<<<num_sms() * 8, 256, 0, st>>>(P, nchunks, off, pbase, len, in);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  k_ck_stack<<<num_sms() * 8, 256, 0, st>>>(P, used);
  return cudaGetLastError();
}

}  // namespace qc
