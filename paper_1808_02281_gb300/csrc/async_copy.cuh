// Asynchronous 16-byte copies from global to shared memory, past L1, counted
// in groups by the thread that starts them.  A thread that reads only what it
// copied itself needs no barrier.
#pragma once

namespace lqcd {

namespace {

__device__ __forceinline__ void copy_async(float4 *dst, const float4 *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void copies_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
// All but the LEFT last groups have arrived.
template <int LEFT> __device__ __forceinline__ void copies_wait()
{
    asm volatile("cp.async.wait_group %0;" ::"n"(LEFT) : "memory");
}

} // namespace

} // namespace lqcd
