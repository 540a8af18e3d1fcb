// Values exchanged between the blocks of one cooperative launch as 64-bit words: 32 bits of the value and a
// 32-bit tag that tells which turn it belongs to.  A word is written and read whole, so a reader that finds
// the tag it waits for has the value; no flag, fence or barrier orders the two.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace vga {

__device__ __forceinline__ unsigned long long ld_word(const unsigned long long *p) {
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(__cvta_generic_to_global(p)) : "memory");
    return v;
}

__device__ __forceinline__ void st_word_raw(unsigned long long *p, unsigned long long w) {
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(__cvta_generic_to_global(p)), "l"(w) : "memory");
}

__device__ __forceinline__ void st_word(unsigned long long *p, float v, uint32_t tag) {
    st_word_raw(p, ((unsigned long long)tag << 32) | __float_as_uint(v));
}

}  // namespace vga
