// k_judge.cu -- the density judge: how far the field force of a candidate
// density is from that of the reference, over all beads.
//
// One pass over the beads gathers both fields at once (sixteen corner loads in
// flight per bead) and sums |Fa - Fb|^2 and |Fb|^2 in FP64, one rounding per
// square: two force passes through memory, an error pass and a one-warp sum over
// 1216 partials took 18.6 + 18.6 + 37 + 74 us at 1M beads, this pass 43, the FP64
// pipe 74 % busy.  A call with its stencils and synchronisation takes 75.6 us; with
// a bead's squares in float-float instead (about 2^-45 relative, 37 us a pass),
// 69.6, which is not worth bits that the error pass had.  The last block to finish adds the block sums in order and writes
// them to the host.
#include "hpf_internal.cuh"

namespace hpf {

namespace {

constexpr int kJudgeBlock = 256;
// One wave of three blocks (80 registers: all sixteen corner loads of a bead in
// flight) on each of 152 SMs, and the same number on any other device, so that the
// sums are taken in the same order, to the same bits, everywhere.  A learned window of 1M
// beads with its judge: 1012 us at 304 or 456 blocks, 1019 at 608 (4 per SM),
// 1030 at 760 (5), 1034 at 1216 (48 registers, two waves).
constexpr int kJudgePerSM = 3;
constexpr int kJudgeGrid = kJudgePerSM * 152;

struct JudgeScratch {
    unsigned ticket;
    double part[kJudgeGrid][2];
};

__device__ __forceinline__ void block_sum2(double& e, double& r, double (*sh)[kJudgeBlock / 32]) {
    for (int o = 16; o > 0; o >>= 1) {
        e += __shfl_down_sync(0xffffffffu, e, o);
        r += __shfl_down_sync(0xffffffffu, r, o);
    }
    if ((threadIdx.x & 31) == 0) {
        sh[0][threadIdx.x >> 5] = e;
        sh[1][threadIdx.x >> 5] = r;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        e = sh[0][0];
        r = sh[1][0];
        for (int k = 1; k < kJudgeBlock / 32; ++k) {
            e += sh[0][k];
            r += sh[1][k];
        }
    }
}

__global__ void __launch_bounds__(kJudgeBlock, kJudgePerSM) k_judge(StateBuf st, const uint32_t* __restrict__ meta,
                                                       int n, MeshGeom g,
                                                       const float4* __restrict__ Ga,
                                                       const float4* __restrict__ Gb, int mode,
                                                       JudgeScratch* scratch, double* h_acc,
                                                       const int* flag, int* h_flag) {
    griddep_wait();
    __shared__ double sh[2][kJudgeBlock / 32];
    __shared__ bool s_last;
    double e = 0.0, r = 0.0;
    for (int i = blockIdx.x * kJudgeBlock + threadIdx.x; i < n; i += gridDim.x * kJudgeBlock) {
        const float x = st.x[i], y = st.y[i], z = st.z[i];
        const size_t off = (size_t)((meta[i] >> kTypeShift) & kTypeMask) * g.gnodes;
        float a[3] = {0.f, 0.f, 0.f}, b[3] = {0.f, 0.f, 0.f};
        if (mode == 0) {
            const AxisCoord cx = axis_gather(x, g.inv_h[0], (float)g.mx, g.inv_m[0]);
            const AxisCoord cy = axis_gather(y, g.inv_h[1], (float)g.my, g.inv_m[1]);
            const AxisCoord cz = axis_gather(z, g.inv_h[2], (float)g.mz, g.inv_m[2]);
            const FieldCorners ka = load_field(Ga + off, g, cx, cy, cz);
            const FieldCorners kb = load_field(Gb + off, g, cx, cy, cz);
            apply_field(ka, cx.f, cy.f, cz.f, a[0], a[1], a[2]);
            apply_field(kb, cx.f, cy.f, cz.f, b[0], b[1], b[2]);
        } else {
            gather_field_mode(Ga + off, g, mode, x, y, z, a[0], a[1], a[2]);
            gather_field_mode(Gb + off, g, mode, x, y, z, b[0], b[1], b[2]);
        }
        const double b0 = b[0], b1 = b[1], b2 = b[2];
        const double d0 = (double)a[0] - b0, d1 = (double)a[1] - b1, d2 = (double)a[2] - b2;
        e = fma(d0, d0, fma(d1, d1, fma(d2, d2, e)));
        r = fma(b0, b0, fma(b1, b1, fma(b2, b2, r)));
    }
    block_sum2(e, r, sh);
    if (threadIdx.x == 0) {
        scratch->part[blockIdx.x][0] = e;
        scratch->part[blockIdx.x][1] = r;
        __threadfence();
        s_last = atomicAdd(&scratch->ticket, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    e = r = 0.0;
    for (int k = threadIdx.x; k < (int)gridDim.x; k += kJudgeBlock) {
        e += __ldcg(&scratch->part[k][0]);
        r += __ldcg(&scratch->part[k][1]);
    }
    block_sum2(e, r, sh);
    if (threadIdx.x == 0) {
        h_acc[0] = e;
        h_acc[1] = r;
        *h_flag = *flag;
        scratch->ticket = 0u;
    }
}

}  // namespace

size_t judge_scratch_bytes() { return sizeof(JudgeScratch); }

void launch_judge(StateBuf st, const uint32_t* meta, int n, const MeshGeom& g, const float4* Ga,
                  const float4* Gb, int force_mode, void* scratch, double* h_acc, const int* flag,
                  int* h_flag, cudaStream_t s) {
    int blocks = (n + kJudgeBlock - 1) / kJudgeBlock;
    if (blocks > kJudgeGrid) blocks = kJudgeGrid;
    if (blocks < 1) blocks = 1;
    launch_pdl(k_judge, dim3(blocks), dim3(kJudgeBlock), 0, s, st, meta, n, g, Ga, Gb, force_mode,
               static_cast<JudgeScratch*>(scratch), h_acc, flag, h_flag);
}

}  // namespace hpf
