// k_state.cu -- loading the bead state into storage order and copying it out.
#include "hpf_internal.cuh"

namespace hpf {

// Tag-order input -> storage arrays + meta word.  err[0] counts species out
// of range, err[1] non-finite coordinates.
__global__ void k_stage_state(const float* __restrict__ pos, const float* __restrict__ vel,
                              const int32_t* __restrict__ type, int n, int S, StateBuf st,
                              uint32_t* __restrict__ meta, int* __restrict__ err) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float px = pos[3 * i], py = pos[3 * i + 1], pz = pos[3 * i + 2];
    const float ux = vel[3 * i], uy = vel[3 * i + 1], uz = vel[3 * i + 2];
    const int t = type[i];
    if (t < 0 || t >= S) atomicAdd(err + 0, 1);
    if (!(isfinite(px) && isfinite(py) && isfinite(pz) && isfinite(ux) && isfinite(uy) &&
          isfinite(uz)))
        atomicAdd(err + 1, 1);
    st.x[i] = px;
    st.y[i] = py;
    st.z[i] = pz;
    st.vx[i] = ux;
    st.vy[i] = uy;
    st.vz[i] = uz;
    meta[i] = (uint32_t)i | (((uint32_t)t & kTypeMask) << kTypeShift);
}

// Each bond must join consecutive tags; it sets bonded-to-next on the lower
// and bonded-to-previous on the upper bead.  err[2] counts malformed bonds,
// err[3] bonds given twice.
__global__ void k_mark_bonds(const int32_t* __restrict__ bonds, long long nb, int n,
                             uint32_t* __restrict__ meta, int* __restrict__ err) {
    const long long b = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= nb) return;
    const int a = bonds[2 * b], c = bonds[2 * b + 1];
    const int lo = a < c ? a : c, hi = a < c ? c : a;
    if (lo < 0 || hi >= n || hi - lo != 1) {
        atomicAdd(err + 2, 1);
        return;
    }
    const uint32_t old = atomicOr(meta + lo, kBondNext);
    if (old & kBondNext) atomicAdd(err + 3, 1);
    atomicOr(meta + hi, kBondPrev);
}

// The three components of a warp's beads to tag order: element e of the 96 is
// component e % 3 of bead e / 3, so that lanes side by side write words side by
// side wherever tags run on (whole chains do).  A component at a time, every
// store touched the sectors of all 32 beads for a third of their bytes.
// Measured for the read-back kernel: 125.9 -> 112.6 us at 8.1M beads, 14.1 ->
// 11.4 us at 1M, 6.1 -> 4.5 us at 10k.
__device__ __forceinline__ void store_tagged(float* __restrict__ out, uint32_t tag, float x, float y,
                                             float z) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const int e = 32 * k + lane, src = e / 3, c = e - 3 * src;
        const uint32_t t = __shfl_sync(0xffffffffu, tag, src);
        const float a = __shfl_sync(0xffffffffu, x, src), b = __shfl_sync(0xffffffffu, y, src),
                    d = __shfl_sync(0xffffffffu, z, src);
        if (t != 0xffffffffu) out[3 * t + c] = c == 0 ? a : (c == 1 ? b : d);
    }
}

// Storage order -> tag order, with a finiteness check of the state.  The last
// block to finish (ticket, left at zero) writes the error word to the mapped
// host word h_flag, which saves the read-back its copy: a frame of a small
// system is a few microseconds of work, and every copy on the stream costs
// about as much again.  Only a block that found something has to order the
// error word before its ticket; the beads' stores are covered by the end of the
// kernel.
__global__ void __launch_bounds__(256) k_unpermute(StateBuf st, const uint32_t* __restrict__ meta,
                                                   int n, float* __restrict__ pos_tag,
                                                   float* __restrict__ vel_tag, int* flag,
                                                   unsigned* ticket, volatile int* h_flag) {
    griddep_wait();
    const int i = blockIdx.x * 256 + threadIdx.x;
    uint32_t tag = 0xffffffffu;
    float x = 0.f, y = 0.f, z = 0.f, vx = 0.f, vy = 0.f, vz = 0.f;
    if (i < n) {
        tag = meta[i] & kTagMask;
        x = st.x[i];
        y = st.y[i];
        z = st.z[i];
        vx = st.vx[i];
        vy = st.vy[i];
        vz = st.vz[i];
    }
    if (pos_tag) store_tagged(pos_tag, tag, x, y, z);
    if (vel_tag) store_tagged(vel_tag, tag, vx, vy, vz);
    const bool any = __syncthreads_or(!(isfinite(x) && isfinite(y) && isfinite(z) && isfinite(vx) &&
                                        isfinite(vy) && isfinite(vz)));
    if (threadIdx.x != 0) return;
    if (any) {
        atomicOr(flag, kFlagNonFinite);
        __threadfence();
    }
    if (atomicAdd(ticket, 1u) != gridDim.x - 1) return;
    *ticket = 0u;
    __threadfence();
    *h_flag = atomicOr(flag, 0);
}

// New positions and velocities given in tag order, written in storage order
// (the inverse of k_unpermute); a non-finite value raises the device flag.
// With D, each bead's eight CIC weights of the new positions are also added
// to D[T] (the next field refresh and the observables need that density,
// which then costs no second pass over the beads).
__global__ void k_repermute(const float* __restrict__ pos_tag, const float* __restrict__ vel_tag,
                            const uint32_t* __restrict__ meta, int n, StateBuf st, MeshGeom g,
                            unsigned long long* __restrict__ D, int* __restrict__ flag) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const bool on = i < n;
    uint32_t m = 0;
    float x = 0.f, y = 0.f, z = 0.f;
    if (on) {
        m = meta[i];
        const uint32_t tag = m & kTagMask;
        x = pos_tag[3 * tag];
        y = pos_tag[3 * tag + 1];
        z = pos_tag[3 * tag + 2];
        const float vx = vel_tag[3 * tag], vy = vel_tag[3 * tag + 1], vz = vel_tag[3 * tag + 2];
        if (!(isfinite(x) && isfinite(y) && isfinite(z) && isfinite(vx) && isfinite(vy) &&
              isfinite(vz)))
            atomicOr(flag, kFlagNonFinite);
        st.x[i] = x;
        st.y[i] = y;
        st.z[i] = z;
        st.vx[i] = vx;
        st.vy[i] = vy;
        st.vz[i] = vz;
    }
    if (D) scatter_paired(D, g, x, y, z, m, on);
}

__global__ void k_order(const uint32_t* __restrict__ meta, int n, int32_t* __restrict__ order) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) order[i] = (int32_t)(meta[i] & kTagMask);
}

void launch_order(const uint32_t* meta, int n, int32_t* order, cudaStream_t s) {
    if (n <= 0) return;
    k_order<<<(n + 255) / 256, 256, 0, s>>>(meta, n, order);
}

__global__ void k_advance_counter(long long* step, long long by) { *step += by; }

void launch_advance_counter(long long* step, long long by, cudaStream_t s) {
    k_advance_counter<<<1, 1, 0, s>>>(step, by);
}

__global__ void k_set_counter(long long* step, long long v) { *step = v; }

void launch_set_counter(long long* step, long long v, cudaStream_t s) {
    k_set_counter<<<1, 1, 0, s>>>(step, v);
}

void launch_stage_state(const float* pos, const float* vel, const int32_t* type, int n, int S,
                        StateBuf st, uint32_t* meta, int* err, cudaStream_t s) {
    if (n <= 0) return;
    k_stage_state<<<(n + 255) / 256, 256, 0, s>>>(pos, vel, type, n, S, st, meta, err);
}

void launch_mark_bonds(const int32_t* bonds, long long nb, int n, uint32_t* meta, int* err,
                       cudaStream_t s) {
    if (nb <= 0) return;
    k_mark_bonds<<<(unsigned)((nb + 255) / 256), 256, 0, s>>>(bonds, nb, n, meta, err);
}

void launch_repermute(const float* pos_tag, const float* vel_tag, const uint32_t* meta, int n,
                      StateBuf st, const MeshGeom& g, unsigned long long* D, int* flag,
                      cudaStream_t s) {
    if (n <= 0) return;
    k_repermute<<<(n + 255) / 256, 256, 0, s>>>(pos_tag, vel_tag, meta, n, st, g, D, flag);
}

void launch_unpermute(StateBuf st, const uint32_t* meta, int n, float* pos_tag, float* vel_tag,
                      int* flag, unsigned* ticket, int* h_flag, cudaStream_t s) {
    if (n <= 0) return;
    launch_pdl(k_unpermute, dim3((n + 255) / 256), dim3(256), 0, s, st, meta, n, pos_tag, vel_tag,
               flag, ticket, (volatile int*)h_flag);
}

}  // namespace hpf
