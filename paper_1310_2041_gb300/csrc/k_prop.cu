// k_prop.cu -- the learned density propagator: a 3-D periodic conv net
// (4 -> 16 -> 16 -> 2 channels, 3x3x3 kernels, SiLU) on BF16 tensor cores.
//
// Forward convolutions (k_conv_sweep): persistent, warp-specialised kernels
// that sweep columns of the mesh along z -- TMA loads of padded activation
// planes, tcgen05 MMAs with tensor-memory accumulators in a ring of output
// planes, an epilogue that gathers the x offsets from neighbouring lanes.
// Activations between the forward layers live in a periodically padded
// layout [2][Mz + 2][PY][PX][8] (channel halves planar); the first layer's
// four input channels enter as an x-im2col, so its three x offsets share one
// K = 16 step.  Training keeps the plain channels-last layout [V][16] for the
// back-propagated gradients: the data-gradient convolutions run on a tiled
// tcgen05 kernel (k_conv_tc), the weight gradient reduces over voxels with
// warp-level MMAs (ldmatrix.trans operands), accumulating in registers over
// many tiles before writing one partial block per CTA.
#include <cuda_bf16.h>
#include <math.h>
#include <string.h>

#include <chrono>
#include <string>

#include "hpf_internal.cuh"

namespace hpf {

constexpr int kPC = 16;                      // padded channels
constexpr int kTX = 8, kTY = 8, kTZ = 8;     // tile of the weight gradients
constexpr int kBX = kTX + 2, kBY = kTY + 2, kBZ = kTZ + 2;
constexpr int kBoxVox = kBX * kBY * kBZ;     // 1000 (32 000 bytes)
constexpr int kTileVox = kTX * kTY * kTZ;    // 512
constexpr int kOffsets = 27;
// channels of the three layers: 4 -> 16 -> 16 -> 2
__host__ __device__ constexpr int layer_in(int l) { return l == 0 ? 4 : 16; }
__host__ __device__ constexpr int layer_out(int l) { return l == 2 ? 2 : 16; }

struct PropGeom {
    int mx, my, mz, V;
    int tiles_x, tiles_y, tiles_z, tiles;
};

__device__ __forceinline__ int pwrap(int i, int m) {
    i %= m;
    return i < 0 ? i + m : i;
}

__device__ __forceinline__ uint32_t saddr(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}

__device__ __forceinline__ void mma_bf16(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2,
                                         uint32_t a3, uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, "
        "{%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

__device__ __forceinline__ void tile_origin(const PropGeom& g, int t, int& x0, int& y0, int& z0) {
    x0 = (t % g.tiles_x) * kTX;
    y0 = ((t / g.tiles_x) % g.tiles_y) * kTY;
    z0 = (t / (g.tiles_x * g.tiles_y)) * kTZ;
}

// ------------------------------------------------------------------ tcgen05 data gradients
//
// The data-gradient convolutions of training (a convolution of the back-
// propagated gradient with flipped, transposed weights, no bias), multiplied by
// the SiLU derivative of the layer below in the epilogue, on the
// fifth-generation tensor cores.  A CTA (one warpgroup) works on tiles of
// 8 x 16 x 2 voxels of the plain channels-last layout [V][16]; a
// z-plane of a tile is 128 voxels = the 128 rows of one MMA (eight
// x-consecutive voxels per 8-row core-matrix group, one group per y row).
// The periodic 10 x 18 x 4 input box sits in shared memory as two planes of
// 8-channel halves (16 bytes per voxel): the canonical K-major layout without
// swizzle, so the box shifted by any in-plane offset (dy, dx) is a matrix
// descriptor that starts at the shifted voxel (K halves one plane apart,
// 8-row groups one box row apart).
//
// Each input plane z (box planes -1 .. 2 of the tile) feeds the output planes
// z + 1, z and z - 1 through the kernel offsets dz = -1, 0, +1 (an output
// voxel n sums W[d] in(n + d)).  So the weights of one in-plane offset are
// stacked for the three dz values as N = 3 x 16 columns, and the accumulators
// of the output planes sit in tensor memory in reverse order, 16 columns
// each: the planes an input plane feeds are then consecutive columns,
// and one tcgen05.mma (M 128, K 16, BF16 in, FP32 accumulate) per input
// plane and in-plane offset updates them all (N = 32 inside the tile, 16 at its
// first and last input planes).  That is 4 x 9 MMAs per tile instead of 27 x 2
// of width 16, and an MMA reads its A operand once for two output planes.  The accumulators are cleared by tcgen05.st
// before the tile's MMAs, which then all accumulate.
//
// One thread issues the MMAs and commits them to an mbarrier; all eight warps
// then read the accumulators back (tcgen05.ld) for the FP32 stores.  Waits are
// bounded (kTcWaitLimit polls);
// a wait that gives up sets kFlagTimeout and the CTA stops after releasing
// its tensor memory.
// Two z-planes a tile: six CTAs fit an SM (37 KB each), and 70^3 voxels, 1575
// tiles, take 1.7 rounds of them; with four planes (48 KB, four CTAs, 810 tiles)
// the second of two rounds was one third full.  A training step at 70^3: 168.1 us at
// four planes, 162.5 at two, 175.6 at six (three CTAs).  A launch takes 20.2 us: 60 %
// of its issue slots go to filling boxes and to the epilogue, the tensor pipe is 13 %
// busy.
constexpr int kTcX = 8, kTcY = 16, kTcZ = 2;
constexpr int kTcPerSM = 6;
constexpr int kTcBX = kTcX + 2, kTcBY = kTcY + 2, kTcBZ = kTcZ + 2;
constexpr int kTcPlane = kTcBX * kTcBY;   // box voxels per z-plane
constexpr int kTcBox = kTcPlane * kTcBZ;  // voxels per channel half
constexpr int kTcInPlane = 9;             // in-plane offsets (dy, dx)
constexpr int kTcRows16 = 48;             // B rows per in-plane offset: (dz, co)
constexpr int kTcCols = 16 * kTcZ;        // accumulator columns per set (a power of two from 32)
constexpr unsigned kTcWaitLimit = 1u << 22;
constexpr int kTcThreads = 256;          // two warps per tensor-memory lane quarter
constexpr int kTcWCopies = 8;            // replicas of each packed weight image (spread L2 reads)
// shared memory of a CTA with kBuf box buffers (and kBuf accumulator sets)
constexpr size_t tc_smem_bytes(int kBuf) {
    return sizeof(uint4) * ((size_t)kBuf * 2 * kTcBox + 2 * kTcInPlane * kTcRows16) + 64;
}

// The weight images of the data-gradient convolutions, [copy][half][in-plane
// offset][B row]: 0 the second layer's, 1 the last layer's.
constexpr int kTcImages = 2;
constexpr int kTcImageWords = 2 * kTcInPlane * kTcRows16;  // uint4 per copy
__host__ __device__ constexpr int tc_image_offset(int k) {  // uint4, all copies
    return k * kTcWCopies * kTcImageWords;
}

// Shared-memory matrix descriptor: start address, leading and stride byte
// offsets (all in 16-byte units), descriptor version 1, no swizzle.
__device__ __forceinline__ uint64_t umma_smem_desc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
    return (uint64_t)((addr >> 4) & 0x3FFFu) | ((uint64_t)((lbo >> 4) & 0x3FFFu) << 16) |
           ((uint64_t)((sbo >> 4) & 0x3FFFu) << 32) | ((uint64_t)1 << 46);
}

// Instruction descriptor of kind::f16: FP32 accumulator, BF16 A and B, both
// K-major, N >> 3 at bit 17, M >> 4 at bit 24.
__host__ __device__ constexpr uint32_t umma_idesc_bf16(int M, int N) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) |
           ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ bool tc_wait(uint32_t bar, uint32_t parity) {
    for (unsigned it = 0; it < kTcWaitLimit; ++it) {
        uint32_t done;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(done)
            : "r"(bar), "r"(parity)
            : "memory");
        if (done) return true;
    }
    return false;
}

__device__ __forceinline__ void tc_origin(const PropGeom& g, int t, int& x0, int& y0, int& z0) {
    const int tx = (g.mx + kTcX - 1) / kTcX, ty = (g.my + kTcY - 1) / kTcY;
    x0 = (t % tx) * kTcX;
    y0 = ((t / tx) % ty) * kTcY;
    z0 = (t / (tx * ty)) * kTcZ;
}

// Box of the tile at (x0, y0, z0) into the buffer at shared address box_s:
// 16-byte asynchronous copies of channel halves, [half][voxel].
// i in [-1, m + box extent]: one period at most when m spans the box extent
// (near), the general remainder otherwise.
__device__ __forceinline__ int tc_wrap(int i, int m, bool near) {
    if (near) return i < 0 ? i + m : (i >= m ? i - m : i);
    return pwrap(i, m);
}

// A thread's share of the box copies: elements e = tid + kTcThreads k of the
// [half][voxel] order, their box coordinates and shared-memory offsets, the
// same for every tile.
constexpr int kTcSlots = (kTcBox * 2 + kTcThreads - 1) / kTcThreads;

struct TcSlots {
    int c[kTcSlots];       // bx | by << 8 | bz << 16 | half << 24, or -1
    uint32_t s[kTcSlots];  // byte offset in a box buffer
};

__device__ __forceinline__ void tc_slots(TcSlots& sl) {
#pragma unroll
    for (int k = 0; k < kTcSlots; ++k) {
        const int e = threadIdx.x + kTcThreads * k;
        const int half = e / kTcBox, v = e % kTcBox;
        const int bx = v % kTcBX, by = (v / kTcBX) % kTcBY, bz = v / kTcPlane;
        sl.c[k] = e < kTcBox * 2 ? (bx | (by << 8) | (bz << 16) | (half << 24)) : -1;
        sl.s[k] = (uint32_t)sizeof(uint4) * (uint32_t)(half * kTcBox + v);
    }
}

__device__ __forceinline__ void tc_load_box(const __nv_bfloat16* __restrict__ in,
                                            const PropGeom& g, int x0, int y0, int z0,
                                            uint32_t box_s, const TcSlots& sl, bool near) {
#pragma unroll
    for (int k = 0; k < kTcSlots; ++k) {
        const int c = sl.c[k];
        if (c < 0) continue;
        const int gx = tc_wrap(x0 - 1 + (c & 0xff), g.mx, near);
        const int gy = tc_wrap(y0 - 1 + ((c >> 8) & 0xff), g.my, near);
        const int gz = tc_wrap(z0 - 1 + ((c >> 16) & 0xff), g.mz, near);
        const int gv = (gz * g.my + gy) * g.mx + gx;
        cp_async16(box_s + sl.s[k], in + ((size_t)(c >> 24) * g.V + gv) * 8);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
}

__device__ __forceinline__ void tc_zero_cols16(uint32_t taddr) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %1, %1, %1, %1, %1, %1, %1, %1, %1, "
        "%1, %1, %1, %1, %1, %1};" ::"r"(taddr),
        "r"(0u)
        : "memory");
}

// g SiLU'(z), to be rounded to BF16, by the hardware's exponential and
// reciprocal (a training step at 70^3 161.2 us, with expf and a full division
// 164.3).  Ten networks on meshes of 16^3 to 80 x 73 x 79: the gradient's error against
// 64 bits (2.2e-3 to 7.2e-3 of its norm, the BF16 operands') is the same with either to
// 5e-6 of itself.
__device__ __forceinline__ float silu_backward(float g, float z) {
    const float s = __fdividef(1.0f, 1.0f + __expf(-z));
    return g * s * (1.0f + z * (1.0f - s));
}

// Epilogue of one output plane: the warp's 32 accumulator rows (lanes 32w ..)
// from columns col .. col + 15, voxel (x0 + row % 8, y0 + row / 8, z): the
// gradient of the layer input through the SiLU of the layer below (its FP32
// pre-activations z_in [V][16]), in BF16 for the next tensor-core passes
// (planar channel halves [2][V][8]).
// Multiplying here instead of in an elementwise pass keeps the FP32 gradient
// out of memory (44 MB written and read back per layer at 70^3).
__device__ __forceinline__ void tc_epilogue(uint32_t tcol, const PropGeom& g, int x0, int y0,
                                            int z, const float* __restrict__ z_in,
                                            __nv_bfloat16* __restrict__ gz_out) {
    const int lane = threadIdx.x & 31, w = (threadIdx.x >> 5) & 3;  // lane quarter
    const uint32_t taddr = tcol + ((uint32_t)(32 * w) << 16);
    const int row = 32 * w + lane;
    const int X = x0 + (row & 7), Y = y0 + (row >> 3);
    const bool valid = X < g.mx && Y < g.my && z < g.mz;
    const size_t gv = ((size_t)z * g.my + Y) * g.mx + X;
    float4 zz[4];
#pragma unroll
    for (int q = 0; q < 4; ++q)
        zz[q] = valid ? __ldg(reinterpret_cast<const float4*>(z_in + gv * kPC) + q)
                      : make_float4(0.f, 0.f, 0.f, 0.f);
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, "
        "%10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),
          "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
    if (!valid) return;
    uint4* o = reinterpret_cast<uint4*>(gz_out) + gv;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        __nv_bfloat162 v[4];
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const float4 zq = zz[2 * h + q];
            const uint32_t* a = r + 8 * h + 4 * q;
            v[2 * q] = __floats2bfloat162_rn(silu_backward(__uint_as_float(a[0]), zq.x),
                                             silu_backward(__uint_as_float(a[1]), zq.y));
            v[2 * q + 1] = __floats2bfloat162_rn(silu_backward(__uint_as_float(a[2]), zq.z),
                                                 silu_backward(__uint_as_float(a[3]), zq.w));
        }
        o[(size_t)h * g.V] = *reinterpret_cast<uint4*>(v);
    }
}

// Wp: a packed weight image (k_pack_images) of the data-gradient weights
// [27][16 out][16 in], offset index 9 dz_index + in-plane offset (dy, dx);
// K = 16 input channels of the planar layout [2][V][8].
template <int kBuf>
__global__ void __launch_bounds__(kTcThreads, kBuf == 1 ? kTcPerSM : 1)
    k_conv_tc(const __nv_bfloat16* __restrict__ in, const uint4* __restrict__ Wp,
              const float* __restrict__ z_in, __nv_bfloat16* __restrict__ gz_out, PropGeom g,
              int n_tiles, int* __restrict__ flag) {
    constexpr int kRows = kTcRows16, kIP = kTcInPlane;
    extern __shared__ __align__(128) uint4 tc_smem[];
    uint4* boxp = tc_smem;                    // [buffer][channel half][kTcBox]
    uint4* wp = tc_smem + kBuf * 2 * kTcBox;  // [channel half][in-plane offset][kRows]
    unsigned long long* bar =
        reinterpret_cast<unsigned long long*>(wp + 2 * kTcInPlane * kTcRows16);
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bar + 3);
    const int tid = threadIdx.x, w = tid >> 5;
    if (w == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         saddr(tmem_slot)),
                     "r"(kBuf * kTcCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(saddr(&bar[0])) : "memory");
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(saddr(&bar[1])) : "memory");
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(saddr(&bar[2])) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    griddep_wait();
    griddep_launch_dependents();
    // B, pre-packed in its shared-memory layout (k_pack_images): one bulk
    // copy from one of kTcWCopies replicas of the image in global memory
    constexpr uint32_t kWBytes = (uint32_t)sizeof(uint4) * 2 * kIP * kRows;
    if (tid == 0) {
        const uint4* src = Wp + (size_t)(blockIdx.x % kTcWCopies) * (kWBytes / sizeof(uint4));
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(
                         saddr(&bar[2])),
                     "r"(kWBytes)
                     : "memory");
        asm volatile(
            "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, "
            "[%3];" ::"r"(saddr(wp)),
            "l"(src), "r"(kWBytes), "r"(saddr(&bar[2]))
            : "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *tmem_slot;
    const uint32_t lbo_a = sizeof(uint4) * kTcBox, sbo_a = sizeof(uint4) * kTcBX;
    const uint32_t lbo_b = sizeof(uint4) * kIP * kRows, sbo_b = sizeof(uint4) * 8;
    const uint32_t box0 = saddr(boxp), wp0 = saddr(wp);
    const bool near = g.mx >= kTcBY && g.my >= kTcBY && g.mz >= kTcBY;
    TcSlots sl;
    tc_slots(sl);
    uint32_t phase[2] = {0u, 0u};
    int px0 = 0, py0 = 0, pz0 = 0;  // origin of the previous tile
    int i = 0;
    bool failed = false;
    bool w_ok = true;  // the weights arrived (thread 0)
    // the box of a tile is loaded one iteration ahead, into the buffer that the
    // MMAs of the tile before the previous one have finished reading
    int t = blockIdx.x;
    if (t < n_tiles) {
        int x0, y0, z0;
        tc_origin(g, t, x0, y0, z0);
        tc_load_box(in, g, x0, y0, z0, box0, sl, near);
    }
    for (; t < n_tiles; t += gridDim.x, ++i) {
        if (kBuf == 1 && i > 0) break;  // one tile per CTA (the grid covers the tiles)
        const int b = kBuf == 1 ? 0 : (i & 1);
        int x0, y0, z0;
        tc_origin(g, t, x0, y0, z0);
        if (i > 0) {
            // the MMAs of the previous tile: done before its box buffer is refilled
            // and before its epilogue
            const bool ok = tc_wait(saddr(&bar[b ^ 1]), phase[b ^ 1]);
            if (__syncthreads_or(!ok)) {  // every thread takes the same branch
                if (tid == 0) atomicOr(flag, kFlagTimeout);
                failed = true;
                break;
            }
            phase[b ^ 1] ^= 1u;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        }
        const int tn = t + (int)gridDim.x;
        if (kBuf > 1 && tn < n_tiles) {
            int xn, yn, zn;
            tc_origin(g, tn, xn, yn, zn);
            tc_load_box(in, g, xn, yn, zn,
                        box0 + (uint32_t)(sizeof(uint4) * 2 * kTcBox) * (b ^ 1), sl, near);
            asm volatile("cp.async.wait_group 1;" ::: "memory");
        } else {
            asm volatile("cp.async.wait_group 0;" ::: "memory");
        }
        const uint32_t boxb = box0 + (uint32_t)(sizeof(uint4) * 2 * kTcBox) * b;
        // accumulator set b was last read by the epilogue of tile i - 2
        const uint32_t accb = tmem + (uint32_t)(kTcCols * b);
#pragma unroll
        for (int c = 0; c < kTcCols / 2; c += 16)
            tc_zero_cols16(accb + (w >> 2) * (kTcCols / 2) + c + ((uint32_t)(32 * (w & 3)) << 16));
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncthreads();
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        if (tid == 0 && i == 0) {
            // the bulk copy of the weights (issued in the prologue)
            w_ok = tc_wait(saddr(&bar[2]), 0u);
            if (!w_ok) atomicOr(flag, kFlagTimeout);
        }
        if (tid == 0 && w_ok) {
            // descriptors: the start-address field is the low 14 bits (16-byte
            // units); offsets inside shared memory are added to it directly
            const uint64_t a0 = umma_smem_desc(boxb, lbo_a, sbo_a);
            const uint64_t b0 = umma_smem_desc(wp0, lbo_b, sbo_b);
#pragma unroll
            for (int z = -1; z <= kTcZ; ++z) {
                const int pf = z + 1 < kTcZ - 1 ? z + 1 : kTcZ - 1;  // first plane fed
                const int pl = z - 1 > 0 ? z - 1 : 0;                 // last plane fed
                const int N = 16 * (pf - pl + 1);
                const uint32_t idesc = umma_idesc_bf16(128, N);
                const uint32_t d = accb + (uint32_t)(16 * (kTcZ - 1 - pf));
                const int row0 = 16 * (z - pf + 1);  // B row of the first plane's dz
#pragma unroll
                for (int o9 = 0; o9 < kIP; ++o9) {
                    const int dy = o9 / 3 - 1, dx = o9 % 3 - 1;
                    const int v0 = ((z + 1) * kTcBY + (1 + dy)) * kTcBX + (1 + dx);
                    const uint64_t ad = a0 + (uint64_t)v0;
                    const uint64_t bd = b0 + (uint64_t)(o9 * kRows + row0);
                    asm volatile(
                        "{\n\t.reg .pred p;\n\t"
                        "setp.ne.u32 p, 1, 0;\n\t"
                        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d),
                        "l"(ad), "l"(bd), "r"(idesc)
                        : "memory");
                }
            }
        }
        if (tid == 0)
            asm volatile(
                "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                    saddr(&bar[b]))
                : "memory");
        if (i > 0) {
            // epilogue of the previous tile while this one is on the tensor cores
            const uint32_t accp = tmem + (uint32_t)(kTcCols * (b ^ 1));
#pragma unroll 1
            for (int p = (kTcZ / 2) * (w >> 2); p < (kTcZ / 2) * (w >> 2) + kTcZ / 2; ++p)
                tc_epilogue(accp + (uint32_t)(16 * (kTcZ - 1 - p)), g, px0, py0, pz0 + p, z_in,
                            gz_out);
        }
        px0 = x0;
        py0 = y0;
        pz0 = z0;
    }
    if (!failed && i > 0) {
        const int pb = (i - 1) & 1;
        const bool ok = tc_wait(saddr(&bar[pb]), phase[pb]);
        if (__syncthreads_or(!ok)) {
            if (tid == 0) atomicOr(flag, kFlagTimeout);
            failed = true;
        } else {
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t accp = tmem + (uint32_t)(kTcCols * pb);
#pragma unroll 1
            for (int p = (kTcZ / 2) * (w >> 2); p < (kTcZ / 2) * (w >> 2) + kTcZ / 2; ++p)
                tc_epilogue(accp + (uint32_t)(16 * (kTcZ - 1 - p)), g, px0, py0, pz0 + p, z_in,
                            gz_out);
        }
    }
    if (failed) {
        // MMAs of the last tiles may still be in flight: one more bounded wait on
        // each accumulator set before the tensor memory is released
        tc_wait(saddr(&bar[0]), phase[0]);
        if (kBuf > 1) tc_wait(saddr(&bar[1]), phase[1]);
    }
    if (tid == 0 && (!w_ok || i == 0)) tc_wait(saddr(&bar[2]), 0u);  // the weights' bulk copy
    asm volatile("cp.async.wait_all;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (w == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                     "r"(kBuf * kTcCols)
                     : "memory");
}

int conv_tc_tiles(const PropGeom& g) {
    return ((g.mx + kTcX - 1) / kTcX) * ((g.my + kTcY - 1) / kTcY) * ((g.mz + kTcZ - 1) / kTcZ);
}

// One tile per CTA, single-buffered (37 KB of shared memory and 32
// tensor-memory columns per CTA, six CTAs per SM overlap one another's box
// loads, MMAs and epilogues); the attribute is set once per device.
void conv_tc_setup() {
    static std::once_flag once[64];
    once_per_device(once, [] {
        cudaFuncSetAttribute(k_conv_tc<1>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)tc_smem_bytes(1));
        cudaGetLastError();
    });
}

// Data-gradient convolution of in [2][V][8] with weight image k of tcw, through
// the SiLU at pre-activations z_in [V][16], into gz_out [2][V][8] (not in).
void launch_conv_tc(const __nv_bfloat16* in, const uint4* tcw, int k, const float* z_in,
                    __nv_bfloat16* gz_out, const PropGeom& g, int* flag, cudaStream_t s) {
    conv_tc_setup();
    const int n = conv_tc_tiles(g);
    launch_pdl(k_conv_tc<1>, dim3(n), dim3(kTcThreads), tc_smem_bytes(1), s, in,
               tcw + tc_image_offset(k), z_in, gz_out, g, n, flag);
}

// ------------------------------------------------------------------ z-sweep convolution
//
// The forward convolutions: persistent and warp-specialised.  The mesh is cut
// into columns of 14 x 8 output voxels (x, y) through the whole z extent; the
// output planes of all columns, in column-major order (column, z), are split
// evenly over the CTAs (one per SM), and a CTA sweeps its share plane by plane.
//
// Activations live in a periodically padded layout [2][Mz + 2][PY][PX][8] BF16
// (channel halves planar; one halo voxel on each side in x, y and z holding
// the opposite face; PX >= Mx + 2, PY >= My + 2), so the 16 x 10 voxel boxes
// of two consecutive input planes -- the column's 14 x 8 voxels with their x
// and y neighbours -- are one TMA box of twenty 256-byte rows per channel half
// (x and channel form the innermost dimension of the tensor map).  A stage
// holds two input planes.  In shared memory a plane's box is the canonical
// K-major layout without swizzle (8 channels = 16 bytes per voxel, core
// matrices of 8 x-consecutive voxels, the channel halves 5120 bytes apart),
// and its 128 voxels from box row dy + 1 on are the A operand
// (M = 128: 8 rows of 16) of the in-plane offset dy, a descriptor into the
// same box for every dy.
//
// For each dy, N stacks the weights of the three dz and, in the 16 -> 16
// layer, of the three dx as well.  An output voxel n sums W[d] in(n + d):
// input plane zi feeds output planes zi + 1, zi, zi - 1 (dz = -1, 0, +1), and
// the dx block of the product at box voxel u belongs to the output voxel
// u - dx, which the epilogue gathers from the neighbouring tensor-memory lanes
// with warp shuffles (a 16-voxel box row keeps x - 1 and x + 1 of each of its
// 14 interior voxels in the same warp).  So an input plane costs three MMAs
// (one per dy) of N up to 3 x 48 = 144 that read the box three times, not
// nine.  The first layer's x-im2col input (K index (dx + 1) 4 + ci) needs no
// dx block (N up to 48); the two-channel last layer keeps 16 columns per
// plane, 6 of them used (zero weight rows behind).
//
// Output planes accumulate in a ring of kSwRing tensor-memory slots in
// reverse column order, so the planes an input plane feeds are adjacent
// columns except where the ring wraps (the MMA is split there).  A slot
// starts at the bias (dx = 0 block) or zero and every MMA accumulates; the
// epilogue reads a finished plane, resets its slot and hands it back before
// its own arithmetic and stores.
//
// Warp 0: TMA producer (a ring of kSwStages two-plane stages); warp 1: owner
// of the tensor memory and MMA issuer; warps 2..9: epilogue, two per
// tensor-memory lane quarter, each with one channel half (8 channels).  Every wait is bounded; one that gives up raises
// kFlagTimeout and a shared abort word that ends every role's loop, after
// which the CTA waits (bounded) for its copies and MMAs in flight and
// releases its tensor memory.
constexpr int kSwOX = 14;                                // output voxels of a column along x
constexpr int kSwBX = 16, kSwY = 8, kSwBY = 10;          // box: x with halo, output rows, rows
constexpr uint32_t kSwPlaneBytes = 16u * kSwBX * kSwBY;  // one channel half of a plane box
constexpr uint32_t kSwHalfBytes = 2u * kSwPlaneBytes;    // one channel half of a stage
constexpr uint32_t kSwStageBytes = 2u * kSwHalfBytes;    // two input planes
constexpr int kSwStages = 9;
constexpr int kSwRingMax = 10;
constexpr int kSwEpiWarps = 8;                           // two per tensor-memory lane quarter
constexpr int kSwThreads = 32 * (2 + kSwEpiWarps);
constexpr int kSwPerSM = 2;                              // CTAs (sweeps) per SM
constexpr size_t kSwSmemFloor = 80 * 1024;               // at most two CTAs per SM

// layer kL: 0 first (x-im2col input), 1 second (16 -> 16), 2 last (16 -> 2)
__host__ __device__ constexpr int sw_cols(int L) { return L == 1 ? 48 : 16; }  // per plane
__host__ __device__ constexpr int sw_rows(int L) { return 3 * sw_cols(L); }    // B rows per dy
__host__ __device__ constexpr int sw_image_words(int L) { return 2 * 3 * sw_rows(L); }
__host__ __device__ constexpr int sw_image_offset(int L) {
    return L == 0 ? 0 : sw_image_offset(L - 1) + kTcWCopies * sw_image_words(L - 1);
}
// accumulator slots: 5 x 48 or 10 x 16 columns, 256 allocated (two CTAs per SM)
__host__ __device__ constexpr int sw_ring(int L) { return L == 1 ? 5 : 10; }
__host__ __device__ constexpr uint32_t sw_tmem_cols(int L) { return 256u; }
constexpr int kSwBars = 2 * kSwStages + kSwRingMax + 2;  // full, empty, acc full, weights, done
constexpr size_t sw_smem_bytes(int L) {
    return (size_t)1024 + (size_t)kSwStages * kSwStageBytes + 16 * (size_t)sw_image_words(L) +
                   8 * (size_t)kSwBars + 64 <
                   kSwSmemFloor
               ? kSwSmemFloor
               : (size_t)1024 + (size_t)kSwStages * kSwStageBytes +
                     16 * (size_t)sw_image_words(L) + 8 * (size_t)kSwBars + 64;
}

struct SweepArgs {
    const uint4* w;            // packed weight image of the layer (kTcWCopies replicas)
    const float* bias;         // [16]
    float* z_out;              // hidden: pre-activations [V][16] FP32 (optional)
    __nv_bfloat16* act_out;    // hidden: SiLU output, padded layout [2][Mz + 2][PY][PX][8]
    float* f_out;              // last: [V][2] FP32 (optional)
    float* y_out;              // last: planar [2][V], times inv_scale (optional)
    float inv_scale;
    int* flag;
    int mx, my, mz, px, py;    // mesh and padded pitches
    int ncx, total;            // columns along x; output planes of all columns
    int withhold;              // self-test: no finished plane is signalled, so the
                               // epilogue's waits give up (hpf_prop_selftest_timeout)
};

__device__ __forceinline__ bool mbar_test(uint32_t bar, uint32_t parity) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(bar), "r"(parity)
        : "memory");
    return done != 0;
}

// A wait gives up after kTcWaitLimit polls or kSwWaitNs of wall time,
// whichever comes first (work that arrives at all arrives within
// microseconds); the clock is read every 64 polls.
constexpr unsigned long long kSwWaitNs = 200000000ull;

__device__ __forceinline__ unsigned long long sw_now() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ bool sw_late(unsigned it, unsigned long long t0) {
    return (it & 63u) == 63u && sw_now() - t0 > kSwWaitNs;
}

// Bounded wait that also gives up when another role has aborted.
__device__ __forceinline__ bool sw_wait(uint32_t bar, uint32_t parity, volatile int* abort_w,
                                        int* flag) {
    if (mbar_test(bar, parity)) return true;  // without a look at the clock
    const unsigned long long t0 = sw_now();
    for (unsigned it = 0; it < kTcWaitLimit && !sw_late(it, t0); ++it) {
        if (mbar_test(bar, parity)) return true;
        if (*abort_w) return false;
    }
    *abort_w = 1;
    atomicOr(flag, kFlagTimeout);
    return false;
}

// Each epilogue warp counts the accumulator slots it has released (a release
// add after its tensor-memory reads and resets); a slot is free once every
// warp's count has passed it (acquire loads before the MMAs that reuse it).
// One count per warp: the warps drift apart by a few planes, and a sum could
// pass a plane that a slow warp has not read yet.
__device__ __forceinline__ void count_release(uint32_t addr) {
    asm volatile("red.release.cta.shared::cta.add.u32 [%0], 1;" ::"r"(addr) : "memory");
}

__device__ __forceinline__ uint32_t count_acquire(uint32_t addr) {
    uint32_t v;
    asm volatile("ld.acquire.cta.shared::cta.u32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
    return v;
}

__device__ __forceinline__ bool mbar_test_now(uint32_t bar, uint32_t parity) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(bar), "r"(parity)
        : "memory");
    return done != 0;
}

__device__ __forceinline__ void count_publish(uint32_t addr, uint32_t v) {
    asm volatile("st.release.cta.shared::cta.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}

__device__ __forceinline__ bool sw_wait_count(uint32_t addr, uint32_t target, uint32_t& known,
                                              volatile int* abort_w, int* flag) {
    if (known >= target) return true;
    const unsigned long long t0 = sw_now();
    for (unsigned it = 0; it < kTcWaitLimit && !sw_late(it, t0); ++it) {
        if (it) __nanosleep(32);
        known = count_acquire(addr);
        if (known >= target) return true;
        if (*abort_w) return false;
    }
    *abort_w = 1;
    atomicOr(flag, kFlagTimeout);
    return false;
}

// known: the smallest count seen so far (counts only grow), so that a target
// it already covers needs no loads.
__device__ __forceinline__ bool sw_wait_released(uint32_t addr, uint32_t target, uint32_t& known,
                                                 volatile int* abort_w, int* flag) {
    if (known >= target) return true;
    const unsigned long long t0 = sw_now();
    for (unsigned it = 0; it < kTcWaitLimit && !sw_late(it, t0); ++it) {
        if (it) __nanosleep(32);  // a poll leaves the issue slots to the working warps
        uint32_t m = count_acquire(addr);
#pragma unroll
        for (int w = 1; w < kSwEpiWarps; ++w) {
            const uint32_t c = count_acquire(addr + 4u * w);
            m = c < m ? c : m;
        }
        known = m;
        if (m >= target) return true;
        if (*abort_w) return false;
    }
    *abort_w = 1;
    atomicOr(flag, kFlagTimeout);
    return false;
}

__device__ __forceinline__ void umma_commit(uint32_t bar) {
    asm volatile(
        "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
        : "memory");
}

__device__ __forceinline__ void umma_bf16(uint32_t d, uint64_t ad, uint64_t bd, uint32_t idesc) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.u32 p, 1, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d),
        "l"(ad), "l"(bd), "r"(idesc)
        : "memory");
}

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float* v) {
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, "
        "%10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),
          "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
#pragma unroll
    for (int c = 0; c < 16; ++c) v[c] = __uint_as_float(r[c]);
}

__device__ __forceinline__ void tmem_st16(uint32_t taddr, const float* v) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, "
        "%10, %11, %12, %13, %14, %15, %16};" ::"r"(taddr),
        "r"(__float_as_uint(v[0])), "r"(__float_as_uint(v[1])), "r"(__float_as_uint(v[2])),
        "r"(__float_as_uint(v[3])), "r"(__float_as_uint(v[4])), "r"(__float_as_uint(v[5])),
        "r"(__float_as_uint(v[6])), "r"(__float_as_uint(v[7])), "r"(__float_as_uint(v[8])),
        "r"(__float_as_uint(v[9])), "r"(__float_as_uint(v[10])), "r"(__float_as_uint(v[11])),
        "r"(__float_as_uint(v[12])), "r"(__float_as_uint(v[13])), "r"(__float_as_uint(v[14])),
        "r"(__float_as_uint(v[15]))
        : "memory");
}

__device__ __forceinline__ void tmem_ld8(uint32_t taddr, float* v) {
    uint32_t r[8];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7])
        : "r"(taddr));
#pragma unroll
    for (int c = 0; c < 8; ++c) v[c] = __uint_as_float(r[c]);
}

__device__ __forceinline__ void tmem_st8(uint32_t taddr, const float* v) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"r"(taddr),
        "r"(__float_as_uint(v[0])), "r"(__float_as_uint(v[1])), "r"(__float_as_uint(v[2])),
        "r"(__float_as_uint(v[3])), "r"(__float_as_uint(v[4])), "r"(__float_as_uint(v[5])),
        "r"(__float_as_uint(v[6])), "r"(__float_as_uint(v[7]))
        : "memory");
}

// Initial value of a slot, the columns of this warp's channel half g: the
// bias in the dx = 0 block (channels 8g .. 8g + 7 of the first layer, columns
// 16 + 8g .. of the second), zero elsewhere; the last layer's 16 columns
// (bias in columns 2 and 3) belong to the g = 0 warps.
template <int kL>
__device__ __forceinline__ void sw_reset_slot(uint32_t taddr, int g, const float (&binit)[16]) {
    float zero[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) zero[c] = 0.f;
    if (kL == 1) {
        tmem_st8(taddr + 8 * g, zero);
        tmem_st8(taddr + 16 + 8 * g, binit);
        tmem_st8(taddr + 32 + 8 * g, zero);
    } else if (kL == 0) {
        tmem_st8(taddr + 8 * g, binit);
    } else if (g == 0) {
        tmem_st16(taddr, binit);
    }
}

// u / (1 + e^-u) from the hardware's 2^x and reciprocal (flushing subnormals,
// which keeps their range handling out of the epilogue's inner loop).
__device__ __forceinline__ float silu(float u) {
    float e, r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e) : "f"(u * -1.44269504088896341f));
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(1.0f + e));
    return u * r;
}

// Where an epilogue lane stores its channel half (8 BF16 channels, 16 bytes)
// of a voxel in the padded layout: the voxel itself and, when it lies on a
// face, its periodic copies in the halo (up to eight places at a corner).  All
// but the plane is the same for a whole run of planes, so it is worked out
// once per run: the words from a plane's start, and the steps to the copies
// beyond the x and y faces (0: none).
struct HalfStore {
    uint4* base;       // channel half, voxel (X, Y) of padded plane 0
    int plane;         // words per padded plane
    int dx, dy;
    bool faces;        // some lane of the warp stores copies in x or y
    __device__ __forceinline__ void begin(const SweepArgs& a, int X, int Y, int h, bool valid) {
        plane = a.py * a.px;
        base = reinterpret_cast<uint4*>(a.act_out) + (size_t)h * (a.mz + 2) * plane +
               (Y + 1) * a.px + X + 1;
        dx = !valid ? 0 : (X == 0 ? a.mx : (X == a.mx - 1 ? -a.mx : 0));
        dy = !valid ? 0 : (Y == 0 ? a.my * a.px : (Y == a.my - 1 ? -a.my * a.px : 0));
        faces = __any_sync(0xffffffffu, (dx | dy) != 0);
    }
    __device__ __forceinline__ void put(uint4* p, uint4 v) const {
        *p = v;
        if (faces) {
            if (dx) p[dx] = v;
            if (dy) p[dy] = v;
            if (dx && dy) p[dx + dy] = v;
        }
    }
    __device__ __forceinline__ void operator()(const SweepArgs& a, int Z, uint4 v) const {
        put(base + (size_t)(Z + 1) * plane, v);
        if (Z == 0) put(base + (size_t)(a.mz + 1) * plane, v);
        if (Z == a.mz - 1) put(base, v);
    }
};

// The output planes [q0, q1) of this CTA in the order q = column Mz + z.
__device__ __forceinline__ void sw_share(const SweepArgs& a, long long& q0, long long& q1) {
    q0 = (long long)a.total * blockIdx.x / gridDim.x;
    q1 = (long long)a.total * (blockIdx.x + 1) / gridDim.x;
}

// The run of output planes [zs, ze) of one column starting at q.
__device__ __forceinline__ void sw_chunk(const SweepArgs& a, long long q, long long q1, int& x0,
                                         int& y0, int& zs, int& ze) {
    const int col = (int)(q / a.mz);
    zs = (int)(q % a.mz);
    const long long left = q1 - q;
    ze = zs + (int)(left < (long long)(a.mz - zs) ? left : (long long)(a.mz - zs));
    x0 = (col % a.ncx) * kSwOX;
    y0 = (col / a.ncx) * kSwY;
}

// The stages of a CTA in order: each run of input planes zs - 1 .. ze of a
// column, two planes per stage (an odd run ends with a padding plane that no
// MMA reads).  zi: the stage's first input plane.
struct SwStages {
    long long q, q1;
    int x0, y0, zs, ze, zi;
    __device__ __forceinline__ void begin(const SweepArgs& a, long long q0, long long q1_) {
        q = q0;
        q1 = q1_;
        if (q < q1) {
            sw_chunk(a, q, q1, x0, y0, zs, ze);
            zi = zs - 1;
        }
    }
    __device__ __forceinline__ void next(const SweepArgs& a) {
        zi += 2;
        if (zi > ze) {
            q += ze - zs;
            if (q < q1) {
                sw_chunk(a, q, q1, x0, y0, zs, ze);
                zi = zs - 1;
            }
        }
    }
};

template <int kL>
__global__ void __launch_bounds__(kSwThreads, kSwPerSM)
    k_conv_sweep(const __grid_constant__ CUtensorMap tmap, const SweepArgs a) {
    constexpr int C = sw_cols(kL), RW = sw_rows(kL), kSwRing = sw_ring(kL);
    constexpr uint32_t kWBytes = 16u * sw_image_words(kL);
    extern __shared__ __align__(1024) uint8_t sw_raw[];
    const uint32_t raw_s = saddr(sw_raw);
    const uint32_t stage_s = (raw_s + 1023u) & ~1023u;  // TMA boxes, 1024-byte aligned
    uint8_t* base = sw_raw + (stage_s - raw_s);
    const uint32_t w_s = stage_s + kSwStages * kSwStageBytes;
    unsigned long long* bars =
        reinterpret_cast<unsigned long long*>(base + kSwStages * kSwStageBytes + kWBytes);
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + kSwBars);
    volatile int* abort_w = reinterpret_cast<volatile int*>(tmem_slot + 1);
    uint32_t* released = tmem_slot + 2;  // [kSwEpiWarps] slot releases per epilogue warp
    uint32_t* loaded = released + kSwEpiWarps;  // input planes landed in shared memory
    const uint32_t rel_s = saddr(released), loaded_s = saddr(loaded);
    const uint32_t bar0 = saddr(bars);
    // barrier k at bar0 + 8 k: full [0, S), empty [S, 2S), acc full [2S, 2S + R),
    // weights, done
    const uint32_t full_b = bar0, empty_b = bar0 + 8 * kSwStages;
    const uint32_t accf_b = bar0 + 16 * kSwStages;
    const uint32_t w_b = accf_b + 8 * kSwRingMax, done_b = w_b + 8;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    // the next layer may be scheduled now: its CTAs take an SM as ours leave it
    // and run their prologue while this grid finishes
    griddep_launch_dependents();
    if (tid == 0) {
        for (int k = 0; k < kSwBars; ++k)
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar0 + 8 * k) : "memory");
        *abort_w = 0;
        for (int w = 0; w < kSwEpiWarps; ++w) released[w] = 0;
        *loaded = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         saddr(tmem_slot)),
                     "r"(sw_tmem_cols(kL))
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *tmem_slot;
    const int eg = (warp - 2) >> 2;  // an epilogue warp's channel half
    float binit[16];
#pragma unroll
    for (int c = 0; c < 16; ++c) binit[c] = 0.f;
    if (warp >= 2) {
        if (kL == 2) {
            binit[2] = a.bias[0];
            binit[3] = a.bias[1];
        } else {
#pragma unroll
            for (int c = 0; c < 8; ++c) binit[c] = a.bias[8 * eg + c];
        }
    }
    const uint32_t lane_off = (uint32_t)(32 * (warp & 3)) << 16;
    if (warp >= 2) {
#pragma unroll 1
        for (int s = 0; s < kSwRing; ++s)
            sw_reset_slot<kL>(tmem + (uint32_t)((kSwRing - 1 - s) * C) + lane_off, eg, binit);
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    long long q0, q1;
    sw_share(a, q0, q1);
    int n_stages = 0;  // every run of input planes zs - 1 .. ze, padded to an even count
    for (long long q = q0; q < q1;) {
        int x0, y0, zs, ze;
        sw_chunk(a, q, q1, x0, y0, zs, ze);
        n_stages += (ze - zs + 3) / 2;
        q += ze - zs;
    }

    if (warp == 0 && lane == 0) {
        // ---------------------------------------------------------------- producer
        const uint4* src = a.w + (size_t)(blockIdx.x % kTcWCopies) * sw_image_words(kL);
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(w_b),
                     "r"(kWBytes)
                     : "memory");
        asm volatile(
            "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, "
            "[%3];" ::"r"(w_s),
            "l"(src), "r"(kWBytes), "r"(w_b)
            : "memory");
        griddep_wait();  // the activations are the previous layer's output
        // Stages run up to kSwStages ahead (a stage is reused once the MMAs that
        // read it are done); between issues the producer watches the copies
        // land, in order, and publishes their count, so that the MMA thread
        // polls one word instead of a barrier per stage.
        SwStages in;
        in.begin(a, q0, q1);
        int si = 0, pub = 0;
        unsigned idle = 0;
        unsigned long long idle_t0 = 0;
        while (si < n_stages || pub < si) {
            bool progress = false;
            const int st = si % kSwStages;
            if (si < n_stages && mbar_test_now(empty_b + 8 * st, ((si / kSwStages) & 1) ^ 1)) {
                const uint32_t dst = stage_s + st * kSwStageBytes, fb = full_b + 8 * st;
                asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(fb),
                             "r"(kSwStageBytes)
                             : "memory");
                // planes zi, zi + 1 at padded z = zi + 1 (0 .. Mz + 1): one box per
                // channel half; x0 8 elements = 16 x0 bytes keeps the copy aligned
#pragma unroll
                for (int h = 0; h < 2; ++h)
                    asm volatile(
                        "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::"
                        "bytes [%0], [%1, {%2, %3, %4, %5}], [%6];" ::"r"(dst + h * kSwHalfBytes),
                        "l"(reinterpret_cast<uint64_t>(&tmap)), "r"(8 * in.x0), "r"(in.y0),
                        "r"(in.zi + 1), "r"(h), "r"(fb)
                        : "memory");
                in.next(a);
                ++si;
                progress = true;
            }
            if (pub < si &&
                mbar_test_now(full_b + 8 * (pub % kSwStages), (pub / kSwStages) & 1)) {
                ++pub;
                count_publish(loaded_s, (uint32_t)pub);
                progress = true;
            }
            if (progress) {
                idle = 0;
            } else if (*abort_w) {
                break;
            } else {
                if (idle == 0) idle_t0 = sw_now();
                if (++idle >= kTcWaitLimit || sw_late(idle, idle_t0)) {
                    *abort_w = 1;
                    atomicOr(a.flag, kFlagTimeout);
                    break;
                }
                __nanosleep(64);  // nothing to issue or publish yet
            }
        }
        // every copy issued lands before the CTA ends (the last phase of each
        // stage is the one to wait for)
        const int used = si < kSwStages ? si : kSwStages;
        const unsigned long long t0 = sw_now();
        for (int st = 0; st < used; ++st) {
            const int j = si - 1 - ((si - 1 - st) % kSwStages);
            for (unsigned k = 0; k < kTcWaitLimit && !sw_late(k, t0) &&
                                 !mbar_test(full_b + 8 * st, (j / kSwStages) & 1);
                 ++k) {
            }
        }
        for (unsigned k = 0; k < kTcWaitLimit && !sw_late(k, t0) && !mbar_test(w_b, 0); ++k) {
        }
    } else if (warp == 1 && lane == 0) {
        // ---------------------------------------------------------------- MMA issuer
        // A single thread: descriptors are formed once and offset per MMA (the
        // start-address field, in 16-byte units, is the low bits).
        griddep_wait();
        bool ok = sw_wait(w_b, 0, abort_w, a.flag);
        const uint64_t adesc0 = umma_smem_desc(stage_s, kSwHalfBytes, 128u);
        const uint64_t bdesc0 = umma_smem_desc(w_s, 16u * 3 * RW, 128u);
        const uint32_t idesc0 = umma_idesc_bf16(128, 0);
        SwStages in;
        in.begin(a, q0, q1);
        int kb = 0;       // ring index of the run's first plane
        int s_first = 0;  // its slot
        uint32_t known_loaded = 0, known_released = 0;
        for (int si = 0; si < n_stages && ok; ++si) {
            if (!sw_wait_count(loaded_s, (uint32_t)(si + 1), known_loaded, abort_w, a.flag)) {
                ok = false;
                break;
            }
            const int st = si % kSwStages;
            const int zs = in.zs, ze = in.ze;
            if (in.zi == zs - 1) s_first = kb % kSwRing;
#pragma unroll 1
            for (int pl = 0; pl < 2; ++pl) {
                const int zi = in.zi + pl;
                if (zi > ze) break;  // the padding plane of an odd run
                const int hi = zi + 1 < ze - 1 ? zi + 1 : ze - 1;
                const int lo = zi - 1 > zs ? zi - 1 : zs;
                const int khi = kb + hi - zs;
                if (zi + 1 < ze && khi >= kSwRing) {
                    // plane khi is first fed now: its slot was released with plane khi - R
                    if (!sw_wait_released(rel_s, (uint32_t)(khi - kSwRing + 1), known_released,
                                          abort_w, a.flag)) {
                        ok = false;
                        break;
                    }
                }
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                int slot = s_first + (hi - zs);
                while (slot >= kSwRing) slot -= kSwRing;
                const uint64_t a_pl =
                    adesc0 + (uint64_t)((st * kSwStageBytes + pl * kSwPlaneBytes) >> 4);
                int dzi = zi - hi + 1;
                for (int left = hi - lo + 1; left > 0;) {
                    const int n = left < slot + 1 ? left : slot + 1;  // adjacent columns
                    const uint32_t d = tmem + (uint32_t)((kSwRing - 1 - slot) * C);
                    const uint32_t idesc = idesc0 + ((uint32_t)(n * C) >> 3 << 17);
                    const uint64_t b_run = bdesc0 + (uint64_t)(dzi * C);
#pragma unroll
                    for (int dyi = 0; dyi < 3; ++dyi)
                        umma_bf16(d, a_pl + (uint64_t)(16 * dyi), b_run + (uint64_t)(dyi * RW),
                                  idesc);
                    left -= n;
                    dzi += n;
                    slot = kSwRing - 1;
                }
                if (zi - 1 >= zs && !a.withhold) {  // plane zi - 1 has all its inputs
                    int s1 = s_first + (zi - 1 - zs);
                    while (s1 >= kSwRing) s1 -= kSwRing;
                    umma_commit(accf_b + 8 * s1);
                }
            }
            if (!ok) break;
            umma_commit(empty_b + 8 * st);  // the stage is read once these MMAs are done
            if (in.zi + 2 > ze) kb += ze - zs;  // the run's last stage
            in.next(a);
        }
        umma_commit(done_b);
        const unsigned long long t0 = sw_now();
        for (unsigned k = 0; k < kTcWaitLimit && !sw_late(k, t0) && !mbar_test(done_b, 0); ++k) {
        }
    } else if (warp >= 2) {
        // ---------------------------------------------------------------- epilogue
        griddep_wait();  // before the first store
        const int r = 32 * (warp & 3) + lane, bx = r & 15, by = r >> 4;
        int k = 0;
        bool ok = true;
        for (long long q = q0; q < q1 && ok;) {
            int x0, y0, zs, ze;
            sw_chunk(a, q, q1, x0, y0, zs, ze);
            const int X = x0 - 1 + bx, Y = y0 + by;
            const bool valid = bx >= 1 && bx <= kSwOX && X < a.mx && Y < a.my;
            HalfStore store;
            if (kL != 2) store.begin(a, X, Y, eg, valid);
            for (int zo = zs; zo < ze; ++zo, ++k) {
                const int slot = k % kSwRing;
                int got = 1;
                if (lane == 0) got = sw_wait(accf_b + 8 * slot, (k / kSwRing) & 1, abort_w, a.flag);
                got = __shfl_sync(0xffffffffu, got, 0);
                if (!got) {
                    ok = false;
                    break;
                }
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t taddr = tmem + (uint32_t)((kSwRing - 1 - slot) * C) + lane_off;
                // this warp's columns: per dx block (second layer) its 8 channels
                float v[24];
                if (kL == 1) {
#pragma unroll
                    for (int b = 0; b < 3; ++b) tmem_ld8(taddr + 16 * b + 8 * eg, v + 8 * b);
                } else if (kL == 0 || eg == 0) {
                    tmem_ld8(taddr + (kL == 0 ? 8 * eg : 0), v);
                }
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                sw_reset_slot<kL>(taddr, eg, binit);
                asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                __syncwarp();
                if (lane == 0) count_release(rel_s + 4u * (warp - 2));
                const size_t gv = ((size_t)zo * a.my + Y) * a.mx + X;
                if (kL == 2) {
                    if (eg != 0) continue;
                    float o[2];
#pragma unroll
                    for (int c = 0; c < 2; ++c)
                        o[c] = __shfl_up_sync(0xffffffffu, v[c], 1) + v[2 + c] +
                               __shfl_down_sync(0xffffffffu, v[4 + c], 1);
                    if (valid) {
                        if (a.f_out)
                            *reinterpret_cast<float2*>(a.f_out + 2 * gv) = make_float2(o[0], o[1]);
                        if (a.y_out) {
                            const size_t V = (size_t)a.mx * a.my * a.mz;
                            a.y_out[gv] = o[0] * a.inv_scale;
                            a.y_out[V + gv] = o[1] * a.inv_scale;
                        }
                    }
                } else {
                    float o[8];
                    if (kL == 1) {
#pragma unroll
                        for (int c = 0; c < 8; ++c)
                            o[c] = __shfl_up_sync(0xffffffffu, v[c], 1) + v[8 + c] +
                                   __shfl_down_sync(0xffffffffu, v[16 + c], 1);
                    } else {
#pragma unroll
                        for (int c = 0; c < 8; ++c) o[c] = v[c];
                    }
                    if (valid) {
                        if (a.z_out) {
                            float4* zo4 = reinterpret_cast<float4*>(a.z_out + gv * kPC + 8 * eg);
                            zo4[0] = make_float4(o[0], o[1], o[2], o[3]);
                            zo4[1] = make_float4(o[4], o[5], o[6], o[7]);
                        }
                        __nv_bfloat162 h[4];
#pragma unroll
                        for (int c = 0; c < 4; ++c) {
                            h[c] = __floats2bfloat162_rn(silu(o[2 * c]), silu(o[2 * c + 1]));
                        }
                        store(a, zo, *reinterpret_cast<uint4*>(h));
                    }
                }
            }
            q += ze - zs;
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 1) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                     "r"(sw_tmem_cols(kL))
                     : "memory");
    }
}

template <int kL>
void sweep_attr() {
    cudaFuncSetAttribute(k_conv_sweep<kL>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)sw_smem_bytes(kL));
}

void conv_sweep_setup() {
    static std::once_flag once[64];
    once_per_device(once, [] {
        sweep_attr<0>();
        sweep_attr<1>();
        sweep_attr<2>();
        cudaGetLastError();
    });
}

// The padded-activation geometry of a mesh: pitches PX, PY (at least one box).
void sweep_pitches(const PropGeom& g, int& px, int& py) {
    px = g.mx + 2 > kSwBX ? g.mx + 2 : kSwBX;
    py = g.my + 2 > kSwBY ? g.my + 2 : kSwBY;
}

// Tensor map of a padded activation buffer [2 halves][Mz + 2][PY][PX][8] with
// x and channel folded into one innermost dimension of 8 PX elements, so that
// a box row (16 voxels x 8 channels, 256 bytes) is one contiguous TMA row; the
// box is one channel half of the 16 x 10 voxel boxes of two planes.
bool make_act_tensor_map(CUtensorMap* map, __nv_bfloat16* act, const PropGeom& g) {
    int px, py;
    sweep_pitches(g, px, py);
    const cuuint64_t pz = (cuuint64_t)g.mz + 2;
    const cuuint64_t dims[4] = {8ull * px, (cuuint64_t)py, pz, 2};
    const cuuint64_t strides[3] = {16ull * px, 16ull * px * py, 16ull * px * py * pz};
    const cuuint32_t box[4] = {8 * kSwBX, (cuuint32_t)kSwBY, 2, 1};
    return encode_tiled_map(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, act, dims, strides, box);
}

// The weight gradients' boxes: a tile with one neighbour on every side of the
// padded activations (both channel halves), and a tile of the gradients.
bool make_wgrad_tensor_maps(CUtensorMap* in, CUtensorMap* gzm, __nv_bfloat16* act,
                            __nv_bfloat16* gz, const PropGeom& g) {
    int px, py;
    sweep_pitches(g, px, py);
    const cuuint64_t pz = (cuuint64_t)g.mz + 2;
    const cuuint64_t dims[4] = {8ull * px, (cuuint64_t)py, pz, 2};
    const cuuint64_t strides[3] = {16ull * px, 16ull * px * py, 16ull * px * py * pz};
    const cuuint32_t box[4] = {8 * kBX, kBY, kBZ, 2};
    const cuuint64_t mx = g.mx, my = g.my, mz = g.mz;
    const cuuint64_t gdims[4] = {8 * mx, my, mz, 2};
    const cuuint64_t gstrides[3] = {16 * mx, 16 * mx * my, 16 * mx * my * mz};
    const cuuint32_t gbox[4] = {8 * kTX, kTY, kTZ, 2};
    return encode_tiled_map(in, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, act, dims, strides, box) &&
           encode_tiled_map(gzm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, gz, gdims, gstrides, gbox);
}

template <int kL>
void launch_conv_sweep(const CUtensorMap& tmap, const SweepArgs& a, int ctas, cudaStream_t s) {
    conv_sweep_setup();
    const int grid = a.total < ctas ? a.total : ctas;
    // programmatic launch: the prologue overlaps the previous layer's tail;
    // every role waits for the previous grid before touching its output
    if (grid > 0) launch_pdl(k_conv_sweep<kL>, grid, kSwThreads, sw_smem_bytes(kL), s, tmap, a);
}

// dW[o][ci][co] = sum_n in(n + d_o)[ci] gz(n)[co]: a voxel reduction on the
// tensor cores (warp-level MMAs, A = in^T and B = gz by ldmatrix.trans).  A
// persistent CTA walks tiles of 8^3 voxels grid-stride and writes its register
// sums to its own slice part[blockIdx.x] (every entry that is read, once);
// k_sum_grads adds the slices in a fixed order, so the gradient is
// deterministic.  Index arithmetic bound the form with cp.async copies of a
// periodic box and swizzled rows (ALU pipe 46 % busy, tensor pipe 18 %, 33 us
// a layer at 70^3): here one thread issues two TMA boxes per tile -- the
// padded activations hold their periodic halo, and boxes past the mesh arrive
// as zeros -- into one of two stages, the other being multiplied.  Both
// operands sit in shared memory as planar channel halves, 16 bytes per voxel,
// so the eight x-consecutive voxels of an ldmatrix phase are 128 contiguous
// bytes (no bank conflict, no swizzle) and every address is a per-lane base
// plus a constant.  A k-step's gradient fragment is loaded once for all of a
// warp's offsets.  Layers 2, 1, 0 take 20.6, 21.9 and 14.0 us, the tensor pipe 31, 59
// and 28 % busy, the L1 data pipe 56, 57 and 44 %: at 16 warps an SM an MMA waits for
// its ldmatrix in 12, 8 and 4 cycles an instruction.  Layer kL: 1, 2 (27 offsets): warp w owns offsets w, w + 8,
// w + 16 and, w < 3, w + 24; the two-channel last layer (2) multiplies only
// the first eight output channels.  0: the x-im2col input carries the three dx
// as channels (dx + 1) 4 + ci, so nine offsets (dz, dy) do: warp w owns offset
// w, and all warps share the ninth, each over its z-plane.  The bias gradient,
// the sum of gz itself, comes from the same stages in FP32, into the slice's
// last 16 entries.
constexpr int kGradEntries = kOffsets * kPC * kPC + kPC;  // a slice: weights, then biases
constexpr uint32_t kWgBoxHalf = 16u * kBoxVox, kWgBoxBytes = 2u * kWgBoxHalf;
constexpr uint32_t kWgTileHalf = 16u * kTileVox, kWgTileBytes = 2u * kWgTileHalf;
constexpr uint32_t kWgBoxPitch = (kWgBoxBytes + 127u) & ~127u;  // TMA targets: 128-byte aligned
constexpr uint32_t kWgStage = kWgBoxPitch + kWgTileBytes;
constexpr size_t kWgSmem = 2 * (size_t)kWgStage + 128 + 64;

template <int kOff>
__device__ __forceinline__ void ldsm_x4_t(uint32_t addr, uint32_t (&r)[4]) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4 + %5];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr), "n"(kOff));
}

// k-step kKs (16 voxels: two y rows) of the offsets at lane bases a[0 .. n).
template <int kKs, int kN, bool kHalf>
__device__ __forceinline__ void wgrad_step(const uint32_t (&a)[4], uint32_t b, bool last,
                                           float (&acc)[4][2][4]) {
    // two y rows further in the box per k-step, a z-plane every fourth
    constexpr int kStep = 16 * ((kKs >> 2) * kBY * kBX + (kKs & 3) * 2 * kBX);
    uint32_t gb[4];
    ldsm_x4_t<256 * kKs>(b, gb);
#pragma unroll
    for (int s = 0; s < kN; ++s) {
        if (s == 3 && !last) break;
        uint32_t ga[4];
        ldsm_x4_t<kStep>(a[s], ga);
        mma_bf16(acc[s][0], ga[0], ga[1], ga[2], ga[3], gb[0], gb[1]);
        if (!kHalf) mma_bf16(acc[s][1], ga[0], ga[1], ga[2], ga[3], gb[2], gb[3]);
    }
}

template <int kL, int kKs = 0>
__device__ __forceinline__ void wgrad_tile(const uint32_t (&a)[4], uint32_t b, bool last,
                                           float (&acc)[4][2][4]) {
    if constexpr (kKs < kTileVox / 16) {
        wgrad_step<kKs, kL == 0 ? 1 : 4, kL == 2>(a, b, last, acc);
        wgrad_tile<kL, kKs + 1>(a, b, last, acc);
    }
}

template <int kL>
__global__ void __launch_bounds__(256, 2)
    k_conv_wgrad(const __grid_constant__ CUtensorMap in, const __grid_constant__ CUtensorMap gz,
                 float* __restrict__ part, const PropGeom g, int* __restrict__ flag) {
    extern __shared__ uint8_t wg_raw[];
    __shared__ __align__(8) unsigned long long bars[2];
    const uint32_t stage_s = (saddr(wg_raw) + 127u) & ~127u;
    const uint8_t* base = wg_raw + (stage_s - saddr(wg_raw));
    const uint32_t bar = saddr(bars);
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar) : "memory");
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar + 8) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    griddep_wait();
    griddep_launch_dependents();
    const int mine = (g.tiles - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x;
    // tile i of this CTA into stage i & 1: the voxels with one neighbour on every
    // side (padded coordinates start at 0) and their gradients
    auto issue = [&](int i) {
        int x0, y0, z0;
        tile_origin(g, (int)blockIdx.x + i * (int)gridDim.x, x0, y0, z0);
        const uint32_t st = stage_s + (i & 1) * kWgStage, fb = bar + 8 * (i & 1);
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(fb),
                     "r"(kWgBoxBytes + kWgTileBytes)
                     : "memory");
        asm volatile(
            "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
            " [%0], [%1, {%2, %3, %4, %5}], [%6];" ::"r"(st),
            "l"(reinterpret_cast<uint64_t>(&in)), "r"(8 * x0), "r"(y0), "r"(z0), "r"(0), "r"(fb)
            : "memory");
        asm volatile(
            "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
            " [%0], [%1, {%2, %3, %4, %5}], [%6];" ::"r"(st + kWgBoxPitch),
            "l"(reinterpret_cast<uint64_t>(&gz)), "r"(8 * x0), "r"(y0), "r"(z0), "r"(0), "r"(fb)
            : "memory");
    };
    if (tid == 0) {
        for (int i = 0; i < 2 && i < mine; ++i) issue(i);
    }
    __syncthreads();  // the barriers are initialised
    float acc[4][2][4];
#pragma unroll
    for (int s = 0; s < 4; ++s)
#pragma unroll
        for (int j = 0; j < 2; ++j)
#pragma unroll
            for (int c = 0; c < 4; ++c) acc[s][j][c] = 0.f;
    float bsum[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) bsum[c] = 0.f;
    // A: lane -> voxel (lane & 7) + 8 (lane >= 16), channel half ((lane >> 3) & 1), so that
    // a0 = ci 0-7 / vox 0-7, a1 = ci 8-15 / vox 0-7, a2 = ci 0-7 / vox 8-15,
    // a3 = ci 8-15 / vox 8-15.  B: lane -> voxel (lane & 7) + 8 ((lane >> 3) & 1), co half
    // (lane >> 4): b0 = vox 0-7 / co 0-7, b1 = vox 8-15 / co 0-7, b2, b3 the same of co 8-15
    auto box_at = [&](int o) {  // the lane's A row at kernel offset o of the first k-step
        const int dz = o / 9, dy = (o / 3) % 3, dx = o % 3;
        return ((lane >> 3) & 1) * kWgBoxHalf +
               16u * (uint32_t)((dz * kBY + dy + (lane >> 4)) * kBX + dx + (lane & 7));
    };
    const bool last = w + 24 < kOffsets;
    uint32_t off[4];
#pragma unroll
    for (int s = 0; s < 4; ++s) {
        const int o = w + 8 * s;
        off[s] = kL == 0 ? box_at(3 * (s == 0 ? w : 8) + 1) : box_at(o < kOffsets ? o : w);
    }
    const uint32_t b_off = (lane >> 4) * kWgTileHalf +
                           16u * (uint32_t)((lane & 7) + (((lane >> 3) & 1) << 3));
    bool failed = false;
    int i = 0;
    for (; i < mine; ++i) {
        const bool ok = tc_wait(bar + 8 * (i & 1), (i >> 1) & 1);
        if (ok) {
            const uint32_t st = stage_s + (i & 1) * kWgStage;
            const uint32_t a[4] = {st + off[0], st + off[1], st + off[2], st + off[3]};
            const uint32_t b = st + kWgBoxPitch + b_off;
            wgrad_tile<kL>(a, b, last, acc);
            if (kL == 0) {  // the ninth offset over z-plane w: k-steps 4 w .. 4 w + 3
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    uint32_t ga[4], gb[4];
                    ldsm_x4_t<0>(b + 256u * (4 * w + q), gb);
                    ldsm_x4_t<0>(a[1] + 16u * (w * kBY * kBX + 2 * q * kBX), ga);
                    mma_bf16(acc[1][0], ga[0], ga[1], ga[2], ga[3], gb[0], gb[1]);
                    mma_bf16(acc[1][1], ga[0], ga[1], ga[2], ga[3], gb[2], gb[3]);
                }
            }
            const uint4* gt = reinterpret_cast<const uint4*>(base + (i & 1) * kWgStage + kWgBoxPitch) +
                              (tid >> 7) * kTileVox + (tid & 127);
#pragma unroll
            for (int j = 0; j < kTileVox / 128; ++j) {
                const uint4 v = gt[128 * j];
                const uint32_t u[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    bsum[2 * c] += __uint_as_float(u[c] << 16);
                    bsum[2 * c + 1] += __uint_as_float(u[c] & 0xffff0000u);
                }
            }
        }
        if (__syncthreads_or(!ok)) {  // every thread is done with the stage
            failed = true;
            break;
        }
        if (tid == 0 && i + 2 < mine) issue(i + 2);
    }
    if (failed) {
        // report; the copies issued for this and the next tile land (bounded) before the CTA ends
        if (tid == 0) {
            atomicOr(flag, kFlagTimeout);
            for (int k = i; k < i + 2 && k < mine; ++k) tc_wait(bar + 8 * (k & 1), (k >> 1) & 1);
        }
        return;
    }
    float* out = part + (size_t)blockIdx.x * kGradEntries;
    const int gq = lane >> 2, q = lane & 3;
    auto entry = [&](int c, int j) { return (gq + 8 * (c >> 1)) * kPC + 8 * j + 2 * q + (c & 1); };
#pragma unroll
    for (int s = 0; s < (kL == 0 ? 1 : 4); ++s) {
        const int o = w + 8 * s;
        if (o >= kOffsets) break;
#pragma unroll
        for (int j = 0; j < (kL == 2 ? 1 : 2); ++j)
#pragma unroll
            for (int c = 0; c < 4; ++c) out[o * kPC * kPC + entry(c, j)] = acc[s][j][c];
    }
    // across the warps, through the stages: the first layer's ninth offset, the biases
    float* sums = reinterpret_cast<float*>(const_cast<uint8_t*>(base));
    float* rows = sums + 8 * kPC * kPC;
    if (kL == 0) {
#pragma unroll
        for (int j = 0; j < 2; ++j)
#pragma unroll
            for (int c = 0; c < 4; ++c) sums[w * kPC * kPC + entry(c, j)] = acc[1][j][c];
    }
#pragma unroll
    for (int c = 0; c < 8; ++c) {
#pragma unroll
        for (int m = 1; m < 32; m <<= 1) bsum[c] += __shfl_xor_sync(0xffffffffu, bsum[c], m);
        if (lane == 0) rows[w * 8 + c] = bsum[c];
    }
    __syncthreads();
    if (kL == 0) {
        float t = sums[tid];
#pragma unroll
        for (int k = 1; k < 8; ++k) t += sums[k * kPC * kPC + tid];
        out[8 * kPC * kPC + tid] = t;
    }
    if (tid < kPC) {  // warps 0-3 hold the first channel half, 4-7 the second
        const float* r = rows + (tid >> 3) * 32 + (tid & 7);
        out[kOffsets * kPC * kPC + tid] = (r[0] + r[8]) + (r[16] + r[24]);
    }
}

template <int kL>
void launch_conv_wgrad(const CUtensorMap& in, const CUtensorMap& gz, float* part,
                       const PropGeom& g, int blocks, int* flag, cudaStream_t s) {
    static std::once_flag once[64];
    once_per_device(once, [] {
        cudaFuncSetAttribute(k_conv_wgrad<kL>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)kWgSmem);
    });
    launch_pdl(k_conv_wgrad<kL>, dim3(blocks), dim3(256), kWgSmem, s, in, gz, part, g, flag);
}

// ------------------------------------------------------------------ elementwise

// The network's input channels from x = (phi_A, phi_B at t - K, phi_A, phi_B
// at t), planar FP32: the scaled changes scale * (phi(t) - phi(t - K)) and the
// current phi(t) per species, formed in FP32 before the BF16 rounding (a
// one-step change of about 1e-2 is far below the BF16 spacing of phi ~ 0.5),
// zero-padded to 16.
//
// out_x: the same four channels as the x-im2col input of the first layer's
// tensor-core convolution, K index (dx + 1) * 4 + ci holding channel ci of
// voxel (x + dx, y, z) (periodic in x) for dx = -1, 0, 1, zeros from 12 on.
__device__ __forceinline__ void input_features(const float* __restrict__ x, int V, int v,
                                               float scale, float (&f)[4]) {
    const float a0 = x[v], b0 = x[(size_t)V + v];
    const float a1 = x[(size_t)2 * V + v], b1 = x[(size_t)3 * V + v];
    f[0] = scale * (a1 - a0);
    f[1] = scale * (b1 - b0);
    f[2] = a1;
    f[3] = b1;
}

// One thread per voxel of the padded array [Mz + 2][My + 2][Mx + 2] (grid y:
// the padded plane; halo
// included, each halo voxel a copy of the opposite face): out_x in the padded
// layout of the forward convolutions [2][Mz + 2][py][px][8]; with phi_next
// (training, for the loss) diff: the change phi_next - phi(t) [V][2].
__global__ void k_pack_input(const float* __restrict__ x, PropGeom g, int px, int py, float scale,
                             __nv_bfloat16* __restrict__ out_x, const float* __restrict__ phi_next,
                             float2* __restrict__ diff) {
    // the first convolution (a programmatic launch) may start its prologue now;
    // it waits for this grid before reading what it writes
    griddep_launch_dependents();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;  // voxel of the padded plane hz
    const int wx = g.mx + 2, wy = g.my + 2, wz = g.mz + 2;
    if (i >= wx * wy) return;
    const int hy = i / wx, hx = i - hy * wx, hz = blockIdx.y;
    const int xi = hx == 0 ? g.mx - 1 : (hx == g.mx + 1 ? 0 : hx - 1);
    const int yi = hy == 0 ? g.my - 1 : (hy == g.my + 1 ? 0 : hy - 1);
    const int z = hz == 0 ? g.mz - 1 : (hz == g.mz + 1 ? 0 : hz - 1);
    const int row = (z * g.my + yi) * g.mx;
    const int xm = xi == 0 ? g.mx - 1 : xi - 1, xp = xi == g.mx - 1 ? 0 : xi + 1;
    float f[3][4];
    input_features(x, g.V, row + xm, scale, f[0]);
    input_features(x, g.V, row + xi, scale, f[1]);
    input_features(x, g.V, row + xp, scale, f[2]);
    __nv_bfloat16 cols[kPC];
#pragma unroll
    for (int c = 0; c < kPC; ++c) cols[c] = __float2bfloat16_rn(c < 12 ? f[c >> 2][c & 3] : 0.f);
    uint4* ox = reinterpret_cast<uint4*>(out_x) + ((size_t)hz * py + hy) * px + hx;
    ox[0] = reinterpret_cast<uint4*>(cols)[0];
    ox[(size_t)wz * py * px] = reinterpret_cast<uint4*>(cols)[1];
    if (phi_next && hx >= 1 && hx <= g.mx && hy >= 1 && hy <= g.my && hz >= 1 && hz <= g.mz) {
        const int v = row + xi;
        diff[v] = make_float2(__fsub_rn(phi_next[v], f[1][2]),
                              __fsub_rn(phi_next[(size_t)g.V + v], f[1][3]));
    }
}

// One autoregressive step on the planar input x [4][V] = (phi(t - 1), phi(t))
// with the predicted change dphi [2][V]: x becomes (phi(t), phi(t) + dphi).
__global__ void k_rollout_shift(float* __restrict__ x, const float* __restrict__ dphi, int V) {
    const int v = blockIdx.x * blockDim.x + threadIdx.x;
    if (v >= V) return;
#pragma unroll
    for (int c = 0; c < 2; ++c) {
        const float cur = x[(size_t)(2 + c) * V + v];
        x[(size_t)c * V + v] = cur;
        x[(size_t)(2 + c) * V + v] = cur + dphi[(size_t)c * V + v];
    }
}

// Mean squared error of the network output y against scale * diff, diff =
// phi_next - phi_cur ([V][2] each), and its gradient 2 (y - target) / (2V) in
// BF16 (the first channel half of a planar buffer, whose second half stays
// zero); the loss in FP64 per thread, one partial per block.
constexpr int kLossBlocks = 608;

__global__ void __launch_bounds__(256) k_loss(const float2* __restrict__ y,
                                              const float2* __restrict__ diff, int V, float scale,
                                              __nv_bfloat16* __restrict__ gy,
                                              double* __restrict__ loss_part) {
    griddep_wait();
    griddep_launch_dependents();
    __shared__ double sh[8];
    double l = 0.0;
    for (int v = blockIdx.x * blockDim.x + threadIdx.x; v < V; v += gridDim.x * blockDim.x) {
        const float2 yv = y[v], dv = diff[v];
        const float a = fmaf(-scale, dv.x, yv.x), b = fmaf(-scale, dv.y, yv.y);
        l += (double)a * a;
        l += (double)b * b;
        const __nv_bfloat162 g2 = __floats2bfloat162_rn(a / (float)V, b / (float)V);
        reinterpret_cast<uint4*>(gy)[v] =
            make_uint4(*reinterpret_cast<const uint32_t*>(&g2), 0u, 0u, 0u);
    }
    for (int o = 16; o > 0; o >>= 1) l += __shfl_down_sync(0xffffffffu, l, o);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = l;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int k = 0; k < (int)(blockDim.x >> 5); ++k) s += sh[k];
        loss_part[blockIdx.x] = s / (2.0 * (double)V);
    }
}

// First packed parameter of layer l.
__host__ __device__ constexpr int param_offset(int l) {
    return l == 0 ? 0 : param_offset(l - 1) + kOffsets * layer_in(l - 1) * layer_out(l - 1) +
                            layer_out(l - 1);
}

// Adam (Kingma & Ba, 2015) on the FP32 master parameters.
struct AdamArgs {
    float *p, *m, *v;  // p null: no update
    float lr, c1, c2;  // c1, c2: the bias corrections 1 - b^t
};

__device__ __forceinline__ void adam_update(const AdamArgs& a, int i, float g) {
    constexpr float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
    const float mi = b1 * a.m[i] + (1.f - b1) * g;
    const float vi = b2 * a.v[i] + (1.f - b2) * g * g;
    a.m[i] = mi;
    a.v[i] = vi;
    a.p[i] -= a.lr * (mi / a.c1) / (sqrtf(vi / a.c2) + eps);
}

__global__ void k_adam(const AdamArgs a, const float* __restrict__ g, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) adam_update(a, i, g[i]);
}

// The weight gradients' slices added up: block (x, layer) takes 32 consecutive
// entries of that layer, sixteen threads per entry each adding every sixteenth
// slice (nb of them), then the sixteen sums in order -- a fixed order, with the
// loads of a thread in flight together instead of one thread walking all slices.
// The packed gradient goes to grads and, with adam.p, straight into the Adam
// update.  One more block adds the loss partials.
constexpr int kSumEntries = 32, kSumShare = 16;
constexpr int kSumBlocks = (kGradEntries + kSumEntries - 1) / kSumEntries;

__global__ void __launch_bounds__(kSumEntries * kSumShare) k_sum_grads(const float* __restrict__ part, int nb,
                                                   float* __restrict__ grads, const AdamArgs adam,
                                                   const double* __restrict__ loss_part, int nl,
                                                   double* __restrict__ loss) {
    griddep_wait();
    griddep_launch_dependents();
    const int tid = threadIdx.x, layer = blockIdx.y;
    if (blockIdx.x == kSumBlocks) {
        if (layer != 0) return;
        __shared__ double shd[kSumShare];
        double l = 0.0;
        for (int k = tid; k < nl; k += kSumEntries * kSumShare) l += loss_part[k];
        for (int o = 16; o > 0; o >>= 1) l += __shfl_down_sync(0xffffffffu, l, o);
        if ((tid & 31) == 0) shd[tid >> 5] = l;
        __syncthreads();
        if (tid == 0) {
            double t = 0.0;
            for (int k = 0; k < kSumShare; ++k) t += shd[k];
            *loss = t;
        }
        return;
    }
    __shared__ float sh[kSumShare][kSumEntries];
    const int e = blockIdx.x * kSumEntries + (tid & 31), slice = tid >> 5;
    // entry e: offset o, input channel ci, output channel co; the biases follow the
    // weights.  First layer: offset 3 dz index + dy index, channel (dx index) 4 + ci.
    const int ci_n = layer_in(layer), co_n = layer_out(layer);
    const bool bias = e >= kOffsets * kPC * kPC;
    int o = e / (kPC * kPC), ci = (e / kPC) % kPC;
    const int co = e % kPC;
    bool valid = e < kGradEntries && co < co_n && (bias || ci < ci_n);
    if (layer == 0 && !bias) {
        valid = o < 9 && ci < 12;
        o = 3 * o + (ci >> 2);
        ci &= 3;
    }
    float s = 0.f;
    if (valid) {
        const float* p = part + (size_t)layer * nb * kGradEntries + e;
#pragma unroll 10
        for (int b = slice; b < nb; b += kSumShare) s += p[(size_t)b * kGradEntries];
    }
    sh[slice][tid & 31] = s;
    __syncthreads();
    if (slice != 0 || !valid) return;
    s = sh[0][tid];
#pragma unroll
    for (int k = 1; k < kSumShare; ++k) s += sh[k][tid];
    const int j = (layer == 0 ? param_offset(0) : (layer == 1 ? param_offset(1) : param_offset(2))) +
                  (bias ? kOffsets * ci_n * co_n + co : (o * ci_n + ci) * co_n + co);
    grads[j] = s;
    if (adam.p) adam_update(adam, j, s);
}

// The tensor-core weight images and the padded biases from the FP32
// parameters, kTcWCopies replicas each, one thread per 16-byte word (eight
// channels of one row).  Forward images (k_conv_sweep), layer L:
// [half][dy index][row], row = dz index C + column, column = co (first layer,
// K index (dx + 1) 4 + ci of its x-im2col input, zeros from 12 on), dx index 16 + co
// (second), dx index 2 + co < 6 (last).  Data-gradient images (k_conv_tc),
// layer L = 1, 2: [half][in-plane offset][dz index 16 + input channel], the
// kernel offset flipped and the channels transposed.
constexpr int kSweepWords = sw_image_words(0) + sw_image_words(1) + sw_image_words(2);
constexpr int kPackWords = kSweepWords + kTcImages * kTcImageWords;

__global__ void k_pack_images(const float* __restrict__ params, uint4* __restrict__ sww,
                              uint4* __restrict__ tcw, float* __restrict__ bias) {
    griddep_wait();
    griddep_launch_dependents();
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < 3 * kPC) {
        const int L = t / kPC, c = t % kPC, co_n = layer_out(L);
        const float* Wl = params + (L == 0 ? param_offset(0) : (L == 1 ? param_offset(1) : param_offset(2)));
        bias[t] = c < co_n ? Wl[kOffsets * layer_in(L) * co_n + c] : 0.f;
    }
    if (t >= kPackWords) return;
    // which image, which word of it
    const bool fwd = t < kSweepWords;
    int L = 0, e = t;
    if (fwd) {
        while (e >= sw_image_words(L)) e -= sw_image_words(L++);
    } else {
        e -= kSweepWords;
        L = 1 + e / kTcImageWords;
        e %= kTcImageWords;
    }
    const int ci_n = layer_in(L), co_n = layer_out(L);
    const float* Wl = params + (L == 0 ? param_offset(0) : (L == 1 ? param_offset(1) : param_offset(2)));
    float v[8];
    uint4* out;
    int per;
    if (fwd) {
        const int C = sw_cols(L), RW = sw_rows(L);
        const int half = e / (3 * RW), dyi = (e / RW) % 3, row = e % RW;
        const int dzi = row / C, c = row % C;
        const int cols = L == 1 ? 16 : 2;  // columns per dx block
        const int co = L == 0 ? c : c % cols;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int k = 8 * half + j;
            const int dxi = L == 0 ? k >> 2 : c / cols, ci = L == 0 ? k & 3 : k;
            const bool on = dxi < 3 && ci < ci_n && co < co_n;
            v[j] = on ? Wl[((dzi * 9 + dyi * 3 + dxi) * ci_n + ci) * co_n + co] : 0.f;
        }
        out = sww + (L == 0 ? sw_image_offset(0) : (L == 1 ? sw_image_offset(1) : sw_image_offset(2))) + e;
        per = sw_image_words(L);
    } else {
        const int half = e / (kTcInPlane * kTcRows16), rest = e % (kTcInPlane * kTcRows16);
        const int o9 = rest / kTcRows16, n = rest % kTcRows16;
        const int o = (n / 16) * kTcInPlane + o9, ci = n % 16;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int co = 8 * half + j;
            const bool on = ci < ci_n && co < co_n;
            v[j] = on ? Wl[((kOffsets - 1 - o) * ci_n + ci) * co_n + co] : 0.f;
        }
        out = tcw + tc_image_offset(L - 1) + e;
        per = kTcImageWords;
    }
    __nv_bfloat162 h[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) h[j] = __floats2bfloat162_rn(v[2 * j], v[2 * j + 1]);
    const uint4 w = *reinterpret_cast<uint4*>(h);
#pragma unroll
    for (int k = 0; k < kTcWCopies; ++k) out[k * per] = w;
}

// ------------------------------------------------------------------ learned-step mesh kernels


// phi_K(n) = D_K(n) phi_c: the volume fractions of an int64 fixed-point mesh.
__global__ void k_mesh_to_phi(const unsigned long long* __restrict__ D, long long n, double phi_c,
                              float* __restrict__ phi) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) phi[i] = (float)((double)(long long)D[i] * phi_c);
}

// D_out = max(0, D_base + rint(dphi * frac / phi_c)): a predicted density in
// the mesh's fixed point (D_base == nullptr: from zero).  In place is allowed.
__global__ void k_mesh_predict(const unsigned long long* D_base, const float* __restrict__ dphi,
                               long long n, double frac_over_phi_c, unsigned long long* D_out) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const long long base = D_base ? (long long)D_base[i] : 0ll;
    long long d = base + __double2ll_rn((double)dphi[i] * frac_over_phi_c);
    D_out[i] = (unsigned long long)(d > 0 ? d : 0ll);
}

// One pass of the periodic binomial filter (1/4, 1/2, 1/4) along one axis of
// C channels of an FP32 [C][Mz][My][Mx] mesh: out(n) = (in(n - e) + 2 in(n) +
// in(n + e)) / 4 with the neighbours e along the axis (periodic).
__global__ void k_binomial_pass(const float* __restrict__ in, float* __restrict__ out, int mx,
                                int my, int mz, int C, int axis) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long n = (long long)C * mx * my * mz;
    if (i >= n) return;
    const int x = (int)(i % mx), y = (int)((i / mx) % my), z = (int)((i / ((long long)mx * my)) % mz);
    long long lo, hi;
    if (axis == 0) {
        lo = i - x + (x == 0 ? mx - 1 : x - 1);
        hi = i - x + (x == mx - 1 ? 0 : x + 1);
    } else if (axis == 1) {
        const long long r = (long long)mx;
        lo = i + (long long)((y == 0 ? my - 1 : y - 1) - y) * r;
        hi = i + (long long)((y == my - 1 ? 0 : y + 1) - y) * r;
    } else {
        const long long r = (long long)mx * my;
        lo = i + (long long)((z == 0 ? mz - 1 : z - 1) - z) * r;
        hi = i + (long long)((z == mz - 1 ? 0 : z + 1) - z) * r;
    }
    out[i] = 0.25f * (in[lo] + in[hi]) + 0.5f * in[i];
}

// passes x 3 axes of the binomial filter from in to out, ping-ponging between
// out and tmp (same size, distinct from out) so that the last pass writes out;
// in may equal out.
void launch_smooth_phi(const float* in, float* out, float* tmp, int mx, int my, int mz, int C,
                       int passes, cudaStream_t s) {
    const long long n = (long long)C * mx * my * mz;
    if (n <= 0) return;
    const unsigned blocks = (unsigned)((n + 255) / 256);
    const int total = 3 * (passes > 0 ? passes : 0);
    if (total == 0) {
        if (in != out) cudaMemcpyAsync(out, in, sizeof(float) * n, cudaMemcpyDeviceToDevice, s);
        return;
    }
    const float* src = in;
    for (int k = 0; k < total; ++k) {
        float* dst = ((total - 1 - k) % 2 == 0) ? out : tmp;
        if (dst == src) {  // only at the first pass, when in is the target buffer
            float* other = dst == out ? tmp : out;
            cudaMemcpyAsync(other, src, sizeof(float) * n, cudaMemcpyDeviceToDevice, s);
            src = other;
        }
        k_binomial_pass<<<blocks, 256, 0, s>>>(src, dst, mx, my, mz, C, k % 3);
        src = dst;
    }
}

void launch_mesh_to_phi(const unsigned long long* D, long long n, double phi_c, float* phi,
                        cudaStream_t s) {
    if (n > 0) k_mesh_to_phi<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(D, n, phi_c, phi);
}

void launch_mesh_predict(const unsigned long long* D_base, const float* dphi, long long n,
                         double frac_over_phi_c, unsigned long long* D_out, cudaStream_t s) {
    if (n > 0)
        k_mesh_predict<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(D_base, dphi, n,
                                                                   frac_over_phi_c, D_out);
}

// ------------------------------------------------------------------ host side

int prop_param_count() {
    int n = 0;
    for (int l = 0; l < 3; ++l) n += kOffsets * layer_in(l) * layer_out(l) + layer_out(l);
    return n;
}

}  // namespace hpf

using namespace hpf;

struct hpf_prop {
    cudaStream_t stream = nullptr;
    PropGeom g{};
    float scale = 1.f;  // change-channel scale (input times, output divided by)
    int np = 0;
    float* params = nullptr;  // FP32 master [np]
    float* grads = nullptr;
    float* adam_m = nullptr;
    float* adam_v = nullptr;
    int adam_t = 0;
    float* bias = nullptr;        // [3][16]
    float* wpart = nullptr;       // gradient slices [3][grid_wgrad][kGradEntries]
    double* lpart = nullptr;      // loss partials [kLossBlocks]
    // act[1], act[2]: the hidden activations in the padded layout
    // [2][Mz + 2][py][px][8]
    __nv_bfloat16* act[3] = {};
    // back-propagated gradients of the three layers' outputs, [2][V][8] (the
    // last layer's second half is zero)
    __nv_bfloat16* gz[3] = {};
    __nv_bfloat16* act_x = nullptr;  // the input as x-im2col, padded layout
    uint4* tcw = nullptr;            // packed weight images of the data-gradient convolutions
    uint4* sww = nullptr;            // packed weight images of the forward convolutions
    CUtensorMap tmap[3];             // act_x, act[1], act[2]
    CUtensorMap wmap[3];             // the same, for the weight gradients' boxes
    CUtensorMap gmap[3];             // gz
    int px = 0, py = 0;              // padded pitches
    int ctas = 1;                    // CTAs of the persistent convolutions (kSwPerSM per SM)
    float* z[2] = {};             // pre-activations of layers 1, 2 [V][16]
    float* fbuf = nullptr;        // FP32 output [V][2]
    float2* diff = nullptr;       // the change to learn [V][2]
    float* xin = nullptr;         // staging of the planar input [4][V]
    float* tin = nullptr;         // staging of the planar next densities [2][V]
    float* yout = nullptr;        // planar output [2][V]
    double* loss = nullptr;
    double* h_loss = nullptr;
    int* flag = nullptr;          // device status bits of the tensor-core waits
    int* h_flag = nullptr;        // pinned mirror
    int grid_wgrad = 0;
};

namespace {

hpf_status prop_copy_out(hpf_prop* p, void* dst, const void* src, size_t bytes) {
    if (!dst) return HPF_OK;
    if (cudaMemcpyAsync(dst, src, bytes, cudaMemcpyDefault, p->stream) != cudaSuccess) {
        cudaGetLastError();
        return HPF_ERR_CUDA;
    }
    cudaPointerAttributes a;
    const bool dev = cudaPointerGetAttributes(&a, dst) == cudaSuccess &&
                     (a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged);
    cudaGetLastError();
    if (!dev && cudaStreamSynchronize(p->stream) != cudaSuccess) return HPF_ERR_CUDA;
    return HPF_OK;
}

// The biases and the tensor-core weight images from the FP32 parameters.
void pack_all_weights(hpf_prop* p, cudaStream_t s) {
    launch_pdl(k_pack_images, dim3((kPackWords + 127) / 128), dim3(128), 0, s,
               (const float*)p->params, p->sww, p->tcw, p->bias);
}

SweepArgs sweep_args(const hpf_prop* p, int layer, int* flag) {
    SweepArgs a{};
    a.w = p->sww + sw_image_offset(layer);
    a.bias = p->bias + layer * kPC;
    a.inv_scale = 1.0f / p->scale;
    a.flag = flag;
    a.mx = p->g.mx;
    a.my = p->g.my;
    a.mz = p->g.mz;
    a.px = p->px;
    a.py = p->py;
    a.ncx = (p->g.mx + kSwOX - 1) / kSwOX;
    a.total = a.ncx * ((p->g.my + kSwY - 1) / kSwY) * p->g.mz;
    return a;
}

// Forward pass of planar input x [4][V] (device).  With phi_next (training):
// the pre-activations, the plain input and the change phi_next - x[2:4] are
// stored and the FP32 output goes to fbuf [V][2] for a backward pass (the
// first kernel alone reads x and phi_next); y_planar (optional): the
// predicted change [2][V] (the output divided by scale).
void prop_forward(hpf_prop* p, const float* x, const float* phi_next, cudaStream_t s, int* flag,
                  float* y_planar = nullptr) {
    const bool train = phi_next != nullptr;
    const int hp = (p->g.mx + 2) * (p->g.my + 2);  // padded voxels per plane
    k_pack_input<<<dim3((unsigned)((hp + 255) / 256), (unsigned)(p->g.mz + 2)), 256, 0, s>>>(
        x, p->g, p->px, p->py, p->scale, p->act_x, phi_next, p->diff);
    SweepArgs a = sweep_args(p, 0, flag);
    a.z_out = train ? p->z[0] : nullptr;
    a.act_out = p->act[1];
    launch_conv_sweep<0>(p->tmap[0], a, p->ctas, s);
    a = sweep_args(p, 1, flag);
    a.z_out = train ? p->z[1] : nullptr;
    a.act_out = p->act[2];
    launch_conv_sweep<1>(p->tmap[1], a, p->ctas, s);
    a = sweep_args(p, 2, flag);
    a.f_out = train ? p->fbuf : nullptr;
    a.y_out = y_planar;
    launch_conv_sweep<2>(p->tmap[2], a, p->ctas, s);
}

// Loss and packed gradients (p->grads, p->loss) after a training forward
// pass, and with adam.p the parameter update.
void prop_backward(hpf_prop* p, const AdamArgs& adam) {
    const int V = p->g.V, nb = p->grid_wgrad;
    const int lb = (V + 255) / 256 < kLossBlocks ? (V + 255) / 256 : kLossBlocks;
    cudaStream_t s = p->stream;
    const size_t slices = (size_t)nb * kGradEntries;
    // the last layer has no activation: its gz is dL/dy
    launch_pdl(k_loss, dim3(lb), dim3(256), 0, s, (const float2*)p->fbuf, (const float2*)p->diff, V,
               p->scale, p->gz[2], p->lpart);
    launch_conv_wgrad<2>(p->wmap[2], p->gmap[2], p->wpart + 2 * slices, p->g, nb, p->flag, s);
    launch_conv_tc(p->gz[2], p->tcw, 1, p->z[1], p->gz[1], p->g, p->flag, s);
    launch_conv_wgrad<1>(p->wmap[1], p->gmap[1], p->wpart + slices, p->g, nb, p->flag, s);
    launch_conv_tc(p->gz[1], p->tcw, 0, p->z[0], p->gz[0], p->g, p->flag, s);
    launch_conv_wgrad<0>(p->wmap[0], p->gmap[0], p->wpart, p->g, nb, p->flag, s);
    launch_pdl(k_sum_grads, dim3(kSumBlocks + 1, 3), dim3(kSumEntries * kSumShare), 0, s, (const float*)p->wpart, nb,
               p->grads, adam, (const double*)p->lpart, lb, p->loss);
}

// The next Adam step's arguments.
AdamArgs adam_args(hpf_prop* p, float lr) {
    p->adam_t += 1;
    return AdamArgs{p->params, p->adam_m, p->adam_v, lr,
                    (float)(1.0 - pow(0.9, (double)p->adam_t)),
                    (float)(1.0 - pow(0.999, (double)p->adam_t))};
}

// Planar inputs are staged into library buffers (host or device sources).
hpf_status prop_stage(hpf_prop* p, float* dst, const float* src, size_t n) {
    if (!src) return HPF_ERR_INVALID;
    if (cudaMemcpyAsync(dst, src, sizeof(float) * n, cudaMemcpyDefault, p->stream) != cudaSuccess) {
        cudaGetLastError();
        return HPF_ERR_CUDA;
    }
    return HPF_OK;
}

// The loss of the last backward pass (synchronises), with the status of the
// tensor-core waits: HPF_ERR_TIMEOUT once if a wait gave up.
hpf_status prop_read_loss(hpf_prop* p, double* loss) {
    if (!loss) return HPF_OK;
    if (cudaMemcpyAsync(p->h_loss, p->loss, sizeof(double), cudaMemcpyDeviceToHost, p->stream) !=
            cudaSuccess ||
        cudaMemcpyAsync(p->h_flag, p->flag, sizeof(int), cudaMemcpyDeviceToHost, p->stream) !=
            cudaSuccess ||
        cudaStreamSynchronize(p->stream) != cudaSuccess) {
        cudaGetLastError();
        return HPF_ERR_CUDA;
    }
    *loss = *p->h_loss;
    if (*p->h_flag & kFlagTimeout) {
        cudaMemsetAsync(p->flag, 0, sizeof(int), p->stream);
        return HPF_ERR_TIMEOUT;
    }
    return HPF_OK;
}

// Whether the kernels read n floats at src in place (*src stays) or from the
// staging buffer dst, filled here.
hpf_status prop_input(hpf_prop* p, float* dst, const float** src, size_t n) {
    const Placed at = placed(*src, sizeof(float) * n, true);
    if (at == Placed::kInPlace) return HPF_OK;
    if (at == Placed::kShort) return HPF_ERR_CUDA;
    const float* from = *src;
    *src = dst;
    return prop_stage(p, dst, from, n);
}

hpf_status prop_launched(hpf_prop* p) {
    (void)p;
    return cudaGetLastError() == cudaSuccess ? HPF_OK : HPF_ERR_CUDA;
}

// Status of the tensor-core waits of the work enqueued so far (synchronises):
// HPF_ERR_TIMEOUT once if a wait gave up.
hpf_status prop_flag_status(hpf_prop* p) {
    if (cudaMemcpyAsync(p->h_flag, p->flag, sizeof(int), cudaMemcpyDeviceToHost, p->stream) !=
            cudaSuccess ||
        cudaStreamSynchronize(p->stream) != cudaSuccess) {
        cudaGetLastError();
        return HPF_ERR_CUDA;
    }
    if (*p->h_flag & kFlagTimeout) {
        cudaMemsetAsync(p->flag, 0, sizeof(int), p->stream);
        return HPF_ERR_TIMEOUT;
    }
    return HPF_OK;
}

}  // namespace

namespace hpf {

bool prop_mesh_is(const hpf_prop* p, const MeshGeom& g) {
    return p && p->g.mx == g.mx && p->g.my == g.my && p->g.mz == g.mz;
}

void prop_predict(hpf_prop* p, const float* x, float* dphi, cudaStream_t s, int* flag) {
    prop_forward(p, x, nullptr, s, flag ? flag : p->flag, dphi);
}

}  // namespace hpf

extern "C" {

hpf_status hpf_prop_init(const int32_t mesh[3], void* stream, hpf_prop** out) {
    if (!out || !mesh) return HPF_ERR_INVALID;
    *out = nullptr;
    long long V = 1;
    for (int a = 0; a < 3; ++a) {
        if (mesh[a] < 2 || mesh[a] > 1024) return HPF_ERR_INVALID;
        V *= mesh[a];
    }
    if (V > (1ll << 26)) return HPF_ERR_INVALID;
    hpf_prop* p = new hpf_prop();
    p->stream = (cudaStream_t)stream;
    PropGeom& g = p->g;
    g.mx = mesh[0];
    g.my = mesh[1];
    g.mz = mesh[2];
    g.V = (int)V;
    g.tiles_x = (g.mx + kTX - 1) / kTX;
    g.tiles_y = (g.my + kTY - 1) / kTY;
    g.tiles_z = (g.mz + kTZ - 1) / kTZ;
    g.tiles = g.tiles_x * g.tiles_y * g.tiles_z;
    p->np = prop_param_count();
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaGetLastError();
    if (sms < 1) sms = 1;
    p->grid_wgrad = g.tiles < 2 * sms ? g.tiles : 2 * sms;
    p->ctas = kSwPerSM * sms;
    sweep_pitches(g, p->px, p->py);
    const size_t Vp = (size_t)(g.mz + 2) * p->py * p->px;  // padded voxels
    const size_t Vs = (size_t)g.V;
    cudaError_t e = cudaSuccess;
    e = e ? e : cudaMalloc(&p->params, sizeof(float) * p->np);
    e = e ? e : cudaMalloc(&p->grads, sizeof(float) * p->np);
    e = e ? e : cudaMalloc(&p->adam_m, sizeof(float) * p->np);
    e = e ? e : cudaMalloc(&p->adam_v, sizeof(float) * p->np);
    e = e ? e : cudaMalloc(&p->bias, sizeof(float) * 3 * kPC);
    e = e ? e : cudaMalloc(&p->wpart, sizeof(float) * 3 * (size_t)p->grid_wgrad * kGradEntries);
    e = e ? e : cudaMalloc(&p->lpart, sizeof(double) * kLossBlocks);
    for (int k = 1; k < 3; ++k) e = e ? e : cudaMalloc(&p->act[k], sizeof(__nv_bfloat16) * Vp * kPC);
    for (int k = 0; k < 3; ++k) e = e ? e : cudaMalloc(&p->gz[k], sizeof(__nv_bfloat16) * Vs * kPC);
    for (int k = 0; k < 2; ++k) e = e ? e : cudaMalloc(&p->z[k], sizeof(float) * Vs * kPC);
    e = e ? e : cudaMalloc(&p->fbuf, sizeof(float) * Vs * 2);
    e = e ? e : cudaMalloc(&p->diff, sizeof(float2) * Vs);
    e = e ? e : cudaMalloc(&p->xin, sizeof(float) * Vs * 4);
    e = e ? e : cudaMalloc(&p->tin, sizeof(float) * Vs * 2);
    e = e ? e : cudaMalloc(&p->yout, sizeof(float) * Vs * 2);
    e = e ? e : cudaMalloc(&p->loss, sizeof(double));
    e = e ? e : cudaMallocHost(&p->h_loss, sizeof(double));
    e = e ? e : cudaMalloc(&p->flag, sizeof(int));
    e = e ? e : cudaMalloc(&p->act_x, sizeof(__nv_bfloat16) * Vp * kPC);
    e = e ? e : cudaMalloc(&p->sww, sizeof(uint4) * sw_image_offset(3));
    e = e ? e : cudaMalloc(&p->tcw, sizeof(uint4) * tc_image_offset(kTcImages));
    e = e ? e : cudaMallocHost(&p->h_flag, sizeof(int));
    if (e == cudaSuccess) {
        // padded buffers: the pitch beyond the halo (meshes narrower than a box)
        // is read by the box copies and stays zero
        cudaMemsetAsync(p->act_x, 0, sizeof(__nv_bfloat16) * Vp * kPC, p->stream);
        cudaMemsetAsync(p->act[1], 0, sizeof(__nv_bfloat16) * Vp * kPC, p->stream);
        cudaMemsetAsync(p->act[2], 0, sizeof(__nv_bfloat16) * Vp * kPC, p->stream);
        cudaMemsetAsync(p->gz[2], 0, sizeof(__nv_bfloat16) * Vs * kPC, p->stream);
        if (!make_wgrad_tensor_maps(&p->wmap[0], &p->gmap[0], p->act_x, p->gz[0], g) ||
            !make_wgrad_tensor_maps(&p->wmap[1], &p->gmap[1], p->act[1], p->gz[1], g) ||
            !make_wgrad_tensor_maps(&p->wmap[2], &p->gmap[2], p->act[2], p->gz[2], g) ||
            !make_act_tensor_map(&p->tmap[0], p->act_x, g) ||
            !make_act_tensor_map(&p->tmap[1], p->act[1], g) ||
            !make_act_tensor_map(&p->tmap[2], p->act[2], g))
            e = cudaErrorNotSupported;
    }
    if (e == cudaSuccess) {
        cudaMemsetAsync(p->flag, 0, sizeof(int), p->stream);
        // zero weights until hpf_prop_set_weights: the network predicts no change
        cudaMemsetAsync(p->params, 0, sizeof(float) * p->np, p->stream);
        cudaMemsetAsync(p->adam_m, 0, sizeof(float) * p->np, p->stream);
        cudaMemsetAsync(p->adam_v, 0, sizeof(float) * p->np, p->stream);
        pack_all_weights(p, p->stream);
        e = cudaGetLastError();
        if (e == cudaSuccess) e = cudaStreamSynchronize(p->stream);
    }
    if (e != cudaSuccess) {
        cudaGetLastError();
        hpf_prop_destroy(p);
        return e == cudaErrorMemoryAllocation ? HPF_ERR_NOMEM : HPF_ERR_CUDA;
    }
    *out = p;
    return HPF_OK;
}

hpf_status hpf_prop_destroy(hpf_prop* p) {
    if (!p) return HPF_OK;
    cudaStreamSynchronize(p->stream);
    cudaFree(p->params);
    cudaFree(p->grads);
    cudaFree(p->adam_m);
    cudaFree(p->adam_v);
    cudaFree(p->bias);
    cudaFree(p->wpart);
    cudaFree(p->lpart);
    for (int k = 0; k < 3; ++k) {
        cudaFree(p->act[k]);
        cudaFree(p->gz[k]);
    }
    for (int k = 0; k < 2; ++k) cudaFree(p->z[k]);
    cudaFree(p->fbuf);
    cudaFree(p->diff);
    cudaFree(p->xin);
    cudaFree(p->tin);
    cudaFree(p->yout);
    cudaFree(p->loss);
    cudaFreeHost(p->h_loss);
    cudaFree(p->flag);
    cudaFreeHost(p->h_flag);
    cudaFree(p->act_x);
    cudaFree(p->tcw);
    cudaFree(p->sww);
    cudaGetLastError();
    delete p;
    return HPF_OK;
}

int32_t hpf_prop_param_count(void) { return prop_param_count(); }

hpf_status hpf_prop_set_weights(hpf_prop* p, const float* params) {
    if (!p || !params) return HPF_ERR_INVALID;
    hpf_status s = prop_stage(p, p->params, params, (size_t)p->np);
    if (s != HPF_OK) return s;
    cudaMemsetAsync(p->adam_m, 0, sizeof(float) * p->np, p->stream);
    cudaMemsetAsync(p->adam_v, 0, sizeof(float) * p->np, p->stream);
    p->adam_t = 0;
    pack_all_weights(p, p->stream);
    if (cudaGetLastError() != cudaSuccess || cudaStreamSynchronize(p->stream) != cudaSuccess)
        return HPF_ERR_CUDA;
    return HPF_OK;
}

hpf_status hpf_prop_get_weights(hpf_prop* p, float* params) {
    if (!p || !params) return HPF_ERR_INVALID;
    return prop_copy_out(p, params, p->params, sizeof(float) * p->np);
}

hpf_status hpf_prop_selftest_timeout(hpf_prop* p, double* seconds) {
    if (!p) return HPF_ERR_INVALID;
    if (cudaStreamSynchronize(p->stream) != cudaSuccess ||
        cudaMemsetAsync(p->flag, 0, sizeof(int), p->stream) != cudaSuccess) {
        cudaGetLastError();
        return HPF_ERR_CUDA;
    }
    // the first layer on the handle's current input, its finished planes never
    // signalled: every CTA's epilogue waits run out, the CTAs abort and release
    // their tensor memory
    SweepArgs a = sweep_args(p, 0, p->flag);
    a.act_out = p->act[1];
    a.withhold = 1;
    const auto t0 = std::chrono::steady_clock::now();
    launch_conv_sweep<0>(p->tmap[0], a, p->ctas, p->stream);
    hpf_status st = prop_launched(p);
    if (st == HPF_OK) st = prop_flag_status(p);  // synchronises; clears the flag it reports
    if (seconds)
        *seconds = std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
    return st;
}

hpf_status hpf_prop_set_ctas(hpf_prop* p, int32_t ctas) {
    if (!p || ctas < 0) return HPF_ERR_INVALID;
    if (ctas == 0) {
        int dev = 0, sms = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        cudaGetLastError();
        ctas = kSwPerSM * (sms > 0 ? sms : 1);
    }
    p->ctas = ctas;
    return HPF_OK;
}

hpf_status hpf_prop_set_scale(hpf_prop* p, float scale) {
    if (!p || !(scale > 0.f) || !(scale < 3.0e38f)) return HPF_ERR_INVALID;
    p->scale = scale;
    return HPF_OK;
}

hpf_status hpf_prop_get_scale(const hpf_prop* p, float* scale) {
    if (!p || !scale) return HPF_ERR_INVALID;
    *scale = p->scale;
    return HPF_OK;
}

hpf_status hpf_prop_forward(hpf_prop* p, const float* x, float* dphi) {
    if (!p || !dphi || !x) return HPF_ERR_INVALID;
    // device arrays of the current device are read and written in place (the
    // input is consumed by the first kernel, so x may even alias dphi); host
    // arrays go through the handle's staging buffers
    const size_t out_bytes = sizeof(float) * 2 * p->g.V;
    const Placed out = placed(dphi, out_bytes, true);
    if (out == Placed::kShort) return HPF_ERR_CUDA;
    hpf_status s = prop_input(p, p->xin, &x, (size_t)p->g.V * 4);
    if (s != HPF_OK) return s;
    prop_predict(p, x, out == Placed::kInPlace ? dphi : p->yout, p->stream, p->flag);
    if ((s = prop_launched(p)) != HPF_OK) return s;
    // in place: the wait status comes with the next synchronising call
    if (out == Placed::kInPlace) return HPF_OK;
    if ((s = prop_copy_out(p, dphi, p->yout, out_bytes)) != HPF_OK) return s;
    return prop_flag_status(p);  // the host copy has synchronised: the status is known
}

hpf_status hpf_prop_rollout(hpf_prop* p, const float* x, int32_t steps, float* phi_out) {
    if (!p || !phi_out || steps < 1) return HPF_ERR_INVALID;
    const int V = p->g.V;
    hpf_status s = prop_stage(p, p->xin, x, (size_t)V * 4);
    if (s != HPF_OK) return s;
    for (int k = 0; k < steps; ++k) {
        prop_predict(p, p->xin, p->yout, p->stream, p->flag);
        k_rollout_shift<<<(V + 255) / 256, 256, 0, p->stream>>>(p->xin, p->yout, V);
    }
    if ((s = prop_launched(p)) != HPF_OK) return s;
    if ((s = prop_copy_out(p, phi_out, p->xin + 2 * (size_t)V, sizeof(float) * 2 * V)) != HPF_OK)
        return s;
    cudaPointerAttributes a;
    const bool dev = cudaPointerGetAttributes(&a, phi_out) == cudaSuccess &&
                     (a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged);
    cudaGetLastError();
    return dev ? HPF_OK : prop_flag_status(p);
}

// Forward and backward of x against phi_next: device arrays of the current
// device are read in place (by the first kernel alone), host arrays go through
// the handle's staging buffers.
static hpf_status prop_gradients(hpf_prop* p, const float* x, const float* phi_next,
                                 const AdamArgs& adam) {
    hpf_status s = prop_input(p, p->xin, &x, (size_t)p->g.V * 4);
    if (s == HPF_OK) s = prop_input(p, p->tin, &phi_next, (size_t)p->g.V * 2);
    if (s != HPF_OK) return s;
    prop_forward(p, x, phi_next, p->stream, p->flag);
    prop_backward(p, adam);
    return HPF_OK;
}

hpf_status hpf_prop_backward(hpf_prop* p, const float* x, const float* phi_next, float* grads,
                             double* loss) {
    if (!p || !x || !phi_next) return HPF_ERR_INVALID;
    hpf_status s = prop_gradients(p, x, phi_next, AdamArgs{});
    if (s != HPF_OK) return s;
    if ((s = prop_launched(p)) != HPF_OK) return s;
    if ((s = prop_copy_out(p, grads, p->grads, sizeof(float) * p->np)) != HPF_OK) return s;
    return prop_read_loss(p, loss);
}

hpf_status hpf_prop_adam_step(hpf_prop* p, const float* grads, float lr) {
    if (!p || !grads || !(lr > 0.f)) return HPF_ERR_INVALID;
    hpf_status s = prop_stage(p, p->grads, grads, (size_t)p->np);
    if (s != HPF_OK) return s;
    k_adam<<<(p->np + 255) / 256, 256, 0, p->stream>>>(adam_args(p, lr), p->grads, p->np);
    pack_all_weights(p, p->stream);
    return prop_launched(p);
}

hpf_status hpf_prop_train_step(hpf_prop* p, const float* x, const float* phi_next, float lr,
                               double* loss) {
    if (!p || !x || !phi_next || !(lr > 0.f)) return HPF_ERR_INVALID;
    const int t = p->adam_t;
    hpf_status s = prop_gradients(p, x, phi_next, adam_args(p, lr));
    if (s != HPF_OK) {
        p->adam_t = t;  // nothing was launched
        return s;
    }
    pack_all_weights(p, p->stream);
    if ((s = prop_launched(p)) != HPF_OK) return s;
    return prop_read_loss(p, loss);
}

}  // extern "C"
