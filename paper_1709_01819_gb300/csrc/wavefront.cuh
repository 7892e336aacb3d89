// wavefront.cuh -- device helpers of the kernels that march over dependent cells:
// asynchronous copies and progress flags between the warps of a block.
#pragma once

#include <cuda_runtime.h>

namespace idg {

// cp.async helpers: asynchronous global -> shared copies used to prefetch
// the next hyperplanes of a wavefront while the current one is computed
__device__ __forceinline__ unsigned smem_addr(const void *p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void cp_async16(void *s, const void *g)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(smem_addr(s)), "l"(g) : "memory");
}
__device__ __forceinline__ void cp_async8(void *s, const void *g)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(smem_addr(s)), "l"(g) : "memory");
}
__device__ __forceinline__ void cp_async4(void *s, const void *g)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(smem_addr(s)), "l"(g) : "memory");
}
template <int B> __device__ __forceinline__ void cp_async_b(void *s, const void *g);
template <> __device__ __forceinline__ void cp_async_b<4>(void *s, const void *g) { cp_async4(s, g); }
template <> __device__ __forceinline__ void cp_async_b<8>(void *s, const void *g) { cp_async8(s, g); }
template <> __device__ __forceinline__ void cp_async_b<16>(void *s, const void *g) { cp_async16(s, g); }
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory"); }

// 1 / x, correctly rounded: in float32 one Newton step on the approximation,
// which gives __frcp_rn(x) for every normal x with a normal reciprocal (x is a
// sum of areas and rates, far from the ends of the range, where this one
// flushes); __frcp_rn's own checks for those ends took 7% of a 64 x 64
// iteration
__device__ __forceinline__ float rcp_nr(float x)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return fmaf(r, fmaf(-x, r, 1.0f), r);
}
__device__ __forceinline__ double rcp_nr(double x) { return __drcp_rn(x); }

// Wavefronts over lines of cells (k_macro_lines, k_sweep_lines, k_adj_lines): the
// warps of a block run kSweepBlock steps between two looks at their neighbours'
// progress.
constexpr int kSweepBlock = 4;

// progress flags between the warps of one block
__device__ __forceinline__ void flag_store(int *f, int v)
{
    asm volatile("st.release.cta.shared.b32 [%0], %1;" ::"r"(smem_addr(f)), "r"(v) : "memory");
}
__device__ __forceinline__ int flag_load(const int *f)
{
    int v;
    asm volatile("ld.acquire.cta.shared.b32 %0, [%1];" : "=r"(v) : "r"(smem_addr(f)) : "memory");
    return v;
}
// waits until *f >= need (seen: what the last poll found).  The warps of a block
// run at the same time, so the wait ends; should it not within limit more polls
// than the first, the status word takes IDG_ERR_TIMEOUT (over anything else it
// holds) and the sweep goes on without waiting, on whatever the ring holds.
__device__ __forceinline__ void flag_wait(const int *f, int need, int &seen, int *status, int limit)
{
    for (int n = 0; seen < need; ++n) {
        seen = flag_load(f);
        if (seen < need && n >= limit) {
            *status = 6;
            seen = 0x7fffffff;
        }
    }
}

}  // namespace idg
