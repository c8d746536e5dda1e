// A kernel of a caller that lets its programmatic dependents start at once and then goes on for a while before it does its
// work: two copies of bytes, one to what the call behind it reads and one from what that call writes.
#include <cstdint>
#include <cuda_runtime.h>

__device__ __forceinline__ uint64_t now_ns()
{
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__global__ void early_trigger_copy(uint8_t* in_dst, const uint8_t* in_src, long long in_bytes, uint8_t* out_dst, const uint8_t* out_src, long long out_bytes, long long wait_ns)
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const uint64_t end = now_ns() + (uint64_t)wait_ns;
    for (int i = 0; i < 4000000 && now_ns() < end; ++i) __nanosleep(1000);      // (ends whatever the timer does)
    const long long first = blockIdx.x * (long long)blockDim.x + threadIdx.x, step = gridDim.x * (long long)blockDim.x;
    for (long long i = first; i < in_bytes; i += step) in_dst[i] = in_src[i];
    for (long long i = first; i < out_bytes; i += step) out_dst[i] = out_src[i];
}

extern "C" int early_trigger_copy_launch(void* in_dst, const void* in_src, long long in_bytes, void* out_dst, const void* out_src, long long out_bytes,
                                         long long wait_ns, void* stream)
{
    early_trigger_copy<<<64, 256, 0, static_cast<cudaStream_t>(stream)>>>(static_cast<uint8_t*>(in_dst), static_cast<const uint8_t*>(in_src), in_bytes,
                                                                         static_cast<uint8_t*>(out_dst), static_cast<const uint8_t*>(out_src), out_bytes, wait_ns);
    return static_cast<int>(cudaGetLastError());
}
