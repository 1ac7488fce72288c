// Tensor-core helpers of the digit sweeps (sweep_dg.cuh, sweep_d4.cuh): shared-memory addresses, the
// operand descriptor and a bounded barrier wait.
#pragma once

constexpr long long TC_WAIT_TRIES = 1ll << 24;

__device__ __forceinline__ uint32_t tc_s32(const void *p) { return static_cast<uint32_t>(__cvta_generic_to_shared(p)); }

// shared-memory matrix descriptor: K-major, 128-byte swizzle, 8-row groups 1 KB apart
__device__ __forceinline__ uint64_t tc_desc(uint32_t saddr) {
    uint64_t d = 0;
    d |= (uint64_t)((saddr >> 4) & 0x3FFFu);
    d |= (uint64_t)1u << 16;
    d |= (uint64_t)(1024u >> 4) << 32;
    d |= (uint64_t)1u << 46;
    d |= (uint64_t)2u << 61;
    return d;
}

__device__ __forceinline__ bool tc_wait(uint64_t *bar, unsigned parity, long long tries) {
    const uint32_t a = tc_s32(bar);
    for (long long i = 0; i < tries; ++i) {
        uint32_t done;
        asm volatile(
            "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(done)
            : "r"(a), "r"(parity)
            : "memory");
        if (done) return true;
    }
    return false;
}
