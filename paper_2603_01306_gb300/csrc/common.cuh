// Device helpers for sm_103a: mbarriers, 1-D bulk (TMA) copies, cluster
// distributed shared memory, and bounded waits.  Every wait in this library is
// bounded: it gives up after `limit_ns` of %globaltimer, records an error code
// in a global status word and lets the caller unwind.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace relax {

enum : int { ST_OK = 0, ST_TIMEOUT = 5, ST_NUMERIC = 6 };

__device__ __forceinline__ uint64_t globaltimer_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// ---------------------------------------------------------------- mbarrier
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}
__device__ __forceinline__ void fence_mbar_init_cluster() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
               "r"(bytes)
               : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      " selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
// Bounded wait on an mbarrier phase.  Returns false (and records ST_TIMEOUT in
// *status) when the phase has not completed within limit_ns.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, uint64_t limit_ns,
                                          int* status) {
  if (mbar_try_wait(bar, parity)) return true;
  const uint64_t t0 = globaltimer_ns();
  for (uint32_t it = 1;; ++it) {
    if (mbar_try_wait(bar, parity)) return true;
    if ((it & 63u) == 0u && globaltimer_ns() - t0 > limit_ns) {
      atomicCAS(status, ST_OK, ST_TIMEOUT);
      return false;
    }
  }
}

// ------------------------------------------------------------ bulk copies
__device__ __forceinline__ uint64_t policy_evict_first() {
  uint64_t p;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
  return p;
}

// ------------------------------------------------------------------ cluster
// shared::cluster address of `local` in CTA `rank` of this cluster
__device__ __forceinline__ uint32_t mapa(const void* local, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem_u32(local)), "r"(rank));
  return r;
}
__device__ __forceinline__ void st_cluster(uint32_t addr, float v) {
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory");
}
__device__ __forceinline__ void st_cluster(uint32_t addr, double v) {
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(addr), "d"(v) : "memory");
}

__device__ __forceinline__ unsigned long long ld_cluster_u64(uint32_t addr) {
  unsigned long long v;
  asm volatile("ld.shared::cluster.u64 %0, [%1];" : "=l"(v) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ double ld_cluster_f64(uint32_t addr) {
  double v;
  asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(addr) : "memory");
  return v;
}

// consumer-only named barrier (id 1), `nthreads` a multiple of 32
__device__ __forceinline__ void named_sync(uint32_t id, uint32_t nthreads) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(nthreads) : "memory");
}

// ------------------------------------------------------------- grid barrier
// Sense-free barrier for a co-resident grid: a monotone arrival counter.
// Barrier number b completes when the counter reaches (b+1)*nblocks.  The
// caller keeps b in a register (all blocks execute the same barrier sequence).
// Bounded: returns false after limit_ns and records ST_TIMEOUT.
__device__ __forceinline__ bool grid_barrier(unsigned long long* counter, unsigned long long target,
                                             uint64_t limit_ns, int* status) {
  __syncthreads();
  __shared__ int ok_sh;
  if (threadIdx.x == 0) {
    // release at GPU scope: the block's writes before the __syncthreads are
    // visible to every block that acquires the counter's final value
    asm volatile("red.release.gpu.global.add.u64 [%0], 1;" ::"l"(counter) : "memory");
    int ok = 1;
    unsigned long long v;
    asm volatile("ld.acquire.gpu.u64 %0, [%1];" : "=l"(v) : "l"(counter) : "memory");
    if (v < target) {
      const uint64_t t0 = globaltimer_ns();
      for (uint32_t it = 1;; ++it) {
        asm volatile("ld.acquire.gpu.u64 %0, [%1];" : "=l"(v) : "l"(counter) : "memory");
        if (v >= target) break;
        if ((it & 15u) == 0u) {
          if (globaltimer_ns() - t0 > limit_ns) {
            atomicCAS(status, ST_OK, ST_TIMEOUT);
            ok = 0;
            break;
          }
          __nanosleep(64);
        }
      }
    }
    ok_sh = ok;
  }
  __syncthreads();
  return ok_sh != 0;
}

// Stream-ordered scratch from the library's own memory pool of the current
// device (pool.cu); returned with cudaFreeAsync.
cudaError_t pool_alloc(void** p, size_t bytes, cudaStream_t st);
void pool_trim();   // gives what the current device's pool holds unused back to the driver
// At least `bytes` of dynamic shared memory for the kernel on the current device
// (attr.cu); never lowered, safe from several threads.
cudaError_t raise_smem(const void* kernel, size_t bytes);

// ------------------------------------------------------------ misc helpers
template <typename T>
__device__ __forceinline__ T warp_sum(T v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

__device__ __forceinline__ uint32_t key_of(float x) { return __float_as_uint(x); }
__device__ __forceinline__ uint64_t key_of(double x) {
  return static_cast<uint64_t>(__double_as_longlong(x));
}
__device__ __forceinline__ float from_key(uint32_t k, float) { return __uint_as_float(k); }
__device__ __forceinline__ double from_key(uint64_t k, double) {
  return __longlong_as_double(static_cast<long long>(k));
}

template <typename T> struct KeyOf;
template <> struct KeyOf<float> { using type = uint32_t; static constexpr uint32_t kInf = 0x7F800000u; };
template <> struct KeyOf<double> {
  using type = uint64_t;
  static constexpr uint64_t kInf = 0x7FF0000000000000ull;
};

}  // namespace relax
