// chunk_pipe.cuh -- bounded mbarrier waits, and the staging of bead arrays in
// shared memory chunk by chunk by asynchronous bulk copies.
#pragma once

#include "hpf_internal.cuh"

namespace hpf {

constexpr unsigned kWaitLimit = 1u << 22;          // polls of an mbarrier before giving up
constexpr unsigned long long kWaitNs = 200000000ull;  // or 0.2 s, whichever comes first

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ unsigned long long global_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Returns false if the barrier did not complete within kWaitLimit polls or
// kWaitNs nanoseconds (a tensor copy completes within microseconds).
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity) {
    const unsigned long long t0 = global_ns();
    for (unsigned it = 0; it < kWaitLimit; ++it) {
        uint32_t done;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(done)
            : "r"(bar), "r"(parity)
            : "memory");
        if (done) return true;
        if ((it & 63) == 63 && global_ns() - t0 > kWaitNs) return false;
    }
    return false;
}

// A CTA walks a run of chunks of kC consecutive beads, one bead per thread, with kChunkHalo more staged on both sides for the chain neighbours.
// The bead arrays are streamed by one bulk copy per array and chunk
// (cp.async.bulk, completion on the stage's mbarrier), kChunkStages chunks
// deep, so that a thread's only exposed latency is the field gather: with
// plain loads a bead's state, its neighbours and its field corners are three
// dependent trips to memory per thread.  The arrays leave room for the copies
// in front of their first and behind their last element (kBeadPad and
// bead_stride), so every copy starts on a 16-byte boundary and none needs a
// bounds check.
constexpr int kChunkHalo = 4;
constexpr int kChunkStages = 3;
static_assert(kChunkHalo <= kBeadPad && kChunkHalo * 4 % 16 == 0, "copies start at the halo");

template <int kArrays, int kC>
struct ChunkPipe {
    static constexpr int kSpan = kC + 2 * kChunkHalo;
    float (*stage)[kArrays][kSpan];  // [kChunkStages]
    uint32_t bar;                    // shared address of the stages' mbarriers
    int first, count;                // this CTA's chunks

    static constexpr size_t bytes() { return sizeof(float) * kChunkStages * kArrays * kSpan; }

    __device__ __forceinline__ void begin(float* smem, unsigned long long* bars, int n) {
        stage = reinterpret_cast<float(*)[kArrays][kSpan]>(smem);
        bar = smem_u32(bars);
        const long long chunks = (n + kC - 1) / kC;
        first = (int)(chunks * blockIdx.x / gridDim.x);
        count = (int)(chunks * (blockIdx.x + 1) / gridDim.x) - first;
        if (threadIdx.x == 0) {
            for (int k = 0; k < kChunkStages; ++k)
                asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar + 8 * k) : "memory");
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        }
    }

    // Copies of the CTA's chunk i into its stage; lane k of one warp issues array k.
    __device__ __forceinline__ void issue(int i, const void* src) {
        constexpr uint32_t kBytes = sizeof(float) * kSpan;
        static_assert(kBytes % 16 == 0, "bulk copies move multiples of 16 bytes");
        const int lane = threadIdx.x & 31, s = i % kChunkStages;
        const uint32_t b = bar + 8 * s;
        if (lane == 0)
            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(b),
                         "r"(kBytes * kArrays)
                         : "memory");
        __syncwarp();
        if (lane < kArrays)
            asm volatile(
                "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, "
                "[%3];" ::"r"(smem_u32(&stage[s][lane][0])),
                "l"(reinterpret_cast<const float*>(src) + (long long)(first + i) * kC - kChunkHalo),
                "r"(kBytes), "r"(b)
                : "memory");
    }

    // First bead of chunk i.
    __device__ __forceinline__ int bead0(int i) const { return (first + i) * kC; }
    __device__ __forceinline__ bool wait(int i) const {
        return mbar_wait(bar + 8 * (i % kChunkStages), (i / kChunkStages) & 1);
    }

    // After a wait gave up at chunk i: the copies issued from it on land (bounded).
    __device__ __forceinline__ void drain(int i) const {
        for (int k = i; k < i + kChunkStages && k < count; ++k) wait(k);
    }
};

}  // namespace hpf
