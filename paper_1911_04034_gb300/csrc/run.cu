// run.cu -- whole circuits of small states in one launch (k_run).
#include "gate_item.cuh"

namespace qc {

// Small states: a gate's work is shorter than the launches that carry it (gate kernels and
// bookkeeping, 12 to 30 us a gate), so one launch runs a whole circuit.  Each CTA takes its
// share of a gate's items (gate_item), the simulator's CTAs meet at a counter in device
// memory, and the last to arrive does the bookkeeping (post_body) and releases the others.
// Every CTA is resident (a cooperative launch) and every wait is bounded (E_TIMEOUT, site
// 4).  Page ids freed by a CTA's items stay with it between gates, up to job.keep of them
// (counted in wc_pages like the streaming kernel's); the rest goes to the freed list.
// Against a streaming, a general and a bookkeeping launch per gate (lossy random circuit):
// 12 qubits in 2^8-amplitude chunks 23.1 -> 14.1 us a gate, 17 in 2^9 31.1 -> 17.3, 18 in
// 2^10 45.5 -> 24.0, 19 in 2^11 118 -> 28.
constexpr uint32_t kRunSpins = 1u << 22;

template <int VPT>
__global__ void __launch_bounds__(kThreads, VPT >= 16 ? 1 : QC_GATE_MIN_CTAS)
    k_run(const RunJob* __restrict__ jobs, int njobs) {
  extern __shared__ __align__(16) uint8_t smem[];
  __shared__ __align__(16) GateLaunch s_L[2];
  __shared__ long long s_ph[7];
  __shared__ int s_oom, s_swapped, s_last, s_late;
  __shared__ uint32_t s_np[2];
  __shared__ uint32_t s_cache[kCacheCap];
  __shared__ uint32_t s_cache_n;
  __shared__ CtaAcc s_acc;
  int lo = 0, hi = njobs - 1;  // the job of this CTA
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (jobs[mid].first <= (int)blockIdx.x) lo = mid;
    else hi = mid - 1;
  }
  const RunJob job = jobs[lo];
  const int rank = (int)blockIdx.x - job.first;
  const uint32_t lane = threadIdx.x & 31u;
  constexpr uint32_t lw = sizeof(GateLaunch) / 16u;
  static_assert(sizeof(GateLaunch) % 16 == 0, "gate records are copied in 16-byte units");
  auto fetch = [&](int k) {  // gate k's record, asynchronously
    const uint4* src = reinterpret_cast<const uint4*>(job.gates + k);
    for (uint32_t i = threadIdx.x; i < lw; i += kThreads) cp_async16(reinterpret_cast<uint4*>(&s_L[k & 1]) + i, src + i);
    cp_async_commit();
  };
  fetch(0);
  cp_async_wait_all();
  if (threadIdx.x == 0) {
    s_cache_n = 0u;
    s_acc.fast = s_acc.rest = 0ull;
  }
  __syncthreads();
  const GateSmem m = gate_smem(smem, s_L[0].P.kc, s_L[0].P.dir_words, s_ph, &s_oom, s_np);
  DevCtl* const ctl = s_L[0].P.ctl;
  GateCta st;
  st.cc.ids = s_cache;
  st.cc.n = &s_cache_n;
  st.acc = &s_acc;
  uint32_t counted = 0u;  // thread 0: cached ids counted in wc_pages
  for (int k = 0; k < job.ngates; ++k) {
    const GateLaunch& L = s_L[k & 1];
    if (k + 1 < job.ngates) fetch(k + 1);
    if (threadIdx.x == 0) s_acc.dE = s_acc.dn64 = 0;
    if (threadIdx.x == 0) s_acc.rd = s_acc.wr = 0ull;
    st.err = threadIdx.x == 0 ? *(volatile unsigned int*)&ctl->err : 0u;
    st.pp = 0;
    st.cur = 0;
    st.next_item = ~0ull;
    const uint32_t S = gate_bits(L);
    for (unsigned long long item = rank; item < L.items; item += (unsigned)job.ctas) {
      if (L.swap) {
        if (threadIdx.x < 32u) {
          unsigned long long coded = 0;
          const bool failed = __shfl_sync(0xffffffffu, st.err, 0) != 0u;
          const bool done = !failed && swap_item(L, item, S, coded);
          if (lane == 0) {
            s_swapped = done;
            if (done && S <= 32u) ++s_acc.fast;
            count_swap_trials(L, ctl, coded);
          }
        }
        __syncthreads();
        const bool done = s_swapped != 0;
        __syncthreads();  // the flag is read before the next item sets it
        if (done) continue;
      }
      const unsigned long long nx = item + (unsigned)job.ctas;
      if (!gate_item<VPT, true>(L, item, nx < L.items && !L.swap ? nx : ~0ull, S, 0ull, false, m, st)) break;
    }
    cp_async_wait_all();
    bulk_wait_all();  // this thread's page stores have reached memory
    asm volatile("fence.proxy.async;" ::: "memory");
    __syncthreads();
    if (threadIdx.x < 32u) {
      // cached ids beyond what may stay (after the last gate: all) to the freed list
      const Pool& P = L.P;
      const uint32_t n = s_cache_n, keep = k + 1 < job.ngates ? min(n, job.keep) : 0u;
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
        if (s_acc.dE) atomicAdd(&ctl->dE, (unsigned long long)s_acc.dE);
        if (s_acc.dn64) atomicAdd(reinterpret_cast<unsigned long long*>(&ctl->dn64), (unsigned long long)s_acc.dn64);
        if (s_acc.rd) atomicAdd(&ctl->bytes_in, s_acc.rd);
        if (s_acc.wr) atomicAdd(&ctl->bytes_out, s_acc.wr);
        if (k + 1 == job.ngates) {
          if (s_acc.fast) atomicAdd(&ctl->fast_items, s_acc.fast);
          if (s_acc.rest) atomicAdd(&ctl->fast_deferred, s_acc.rest);
        }
      }
      __syncwarp();
    }
    __syncthreads();
    // the simulator's CTAs meet; the last one books the gate
    const uint32_t last_of = (uint32_t)job.ctas * (uint32_t)(k + 1);
    if (threadIdx.x == 0) {
      __threadfence();
      s_last = atomicAdd(&ctl->run_arrived, 1u) + 1u == last_of;
      __threadfence();
    }
    __syncthreads();
    if (s_last) {
      post_body(L.P, L.ctl, 0);
      __syncthreads();
      if (threadIdx.x == 0) {
        __threadfence();
        const bool end = k + 1 == job.ngates;  // nobody waits after the last gate
        if (end) ctl->run_arrived = 0u;
        atomicExch(&ctl->run_gate, end ? 0u : (uint32_t)(k + 1));
      }
      __syncthreads();
    } else if (k + 1 < job.ngates) {
      if (threadIdx.x == 0) {
        uint32_t it = 0;
        while (*(volatile unsigned int*)&ctl->run_gate != (uint32_t)(k + 1)) {
          if (++it > kRunSpins) {
            atomicOr(&ctl->err, (unsigned)E_TIMEOUT);
            atomicExch(&ctl->timeout_site, 4u);
            break;
          }
        }
        s_late = it > kRunSpins;
        __threadfence();
      }
      __syncthreads();
      if (s_late) return;  // no copy in flight: all were waited for above
    }
  }
}

int run_ctas_per_sm(int kc) {
  int n = 0;
  const size_t smem = gate_smem_bytes(kc);
  cudaError_t e = cudaSuccess;
  switch (vpt_for(kc)) {
    case 1: prep(k_run<1>, smem); e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_run<1>, kThreads, smem); break;
    case 2: prep(k_run<2>, smem); e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_run<2>, kThreads, smem); break;
    case 4: prep(k_run<4>, smem); e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_run<4>, kThreads, smem); break;
    case 8: prep(k_run<8>, smem); e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_run<8>, kThreads, smem); break;
    case 16: prep(k_run<16>, smem); e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_run<16>, kThreads, smem); break;
  }
  return e != cudaSuccess || n < 1 ? 0 : n;
}

cudaError_t launch_run(const RunJob* jobs, int njobs, int kc, int grid, cudaStream_t st) {
  const size_t smem = gate_smem_bytes(kc);
  void* args[] = {(void*)&jobs, (void*)&njobs};
  cudaError_t e = cudaSuccess;
  QC_VPT_DISPATCH(kc, {
    e = prep(k_run<V>, smem);
    if (e == cudaSuccess)
      e = cudaLaunchCooperativeKernel((const void*)k_run<V>, dim3((unsigned)grid), dim3(kThreads), args, smem, st);
  });
  return e;
}

}  // namespace qc
