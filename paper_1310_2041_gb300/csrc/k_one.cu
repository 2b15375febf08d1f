// k_one.cu -- one step per launch: the step kernel of schedules that refresh
// the field every step, one bead per thread.
//
// The field-period kernels (k_step.cu) keep beads on chip over many steps and
// pay for it once per launch: a segment's beads, their cell polynomials in
// shared memory, two CTAs of 256 threads per SM.  A single step amortises none
// of that, and the chain segment -> state -> corners of dependent loads at 16
// warps per SM was what such a launch took its time for.  Here the beads
// stream through shared memory ahead of their use (chunk_pipe.cuh), the eight
// corner loads of a bead are in flight while its noise and bonds are formed,
// and the polynomial stays in registers.  The arithmetic, operation by
// operation, is that of the field-period kernels: kWarp takes the order of
// the warp form's bond sums, else that of the halo form, so that a run gives
// the same bits whichever kernel its steps go through.  1M beads, step and
// deposit: 60 us with the warp kernel, 39 here, of which the deposit's
// reductions are 11.  No unit is full: the eight corner loads touch 22 sectors each
// (L1 data pipe 58 % of the launch), the L2 is 52 % busy with them and the deposit,
// and at 24 warps an SM a warp waits for its loads in 3.5 of the 11.8 cycles between
// its instructions.
#include "cell_poly.cuh"
#include "chunk_pipe.cuh"

namespace hpf {

namespace {

constexpr int kOneArrays = 7;  // x y z vx vy vz meta
// Beads (threads) of a CTA's chunk, and in a system of at most four small ones
// an SM.  Small systems are one chain of latencies, to which a chunk's gather
// and deposit on one SM add; 256 against 128, 20 steps of one launch and one
// field: 5k beads 134.9 / 123.8 us, 10k 135.8 / 124.9, 30k 158 / 150, 80k 204 / 201;
// past one chunk for every resident CTA the small ones lose: 120k 247 / 276, 1M
// 472 / 513.
constexpr int kChunk = 256;
constexpr int kSmallChunk = 128;
constexpr int kSmallPerSM = 4;
constexpr int kOnePerSM = 3;      // resident CTAs of 256 threads (80 registers; four, at 64, spill)

struct OneParams {
    const void* src[kOneArrays];
    StateBuf out;
    int n;
    long long step;
    MeshGeom g;
    const float4* G;
    StepConsts c;
    unsigned long long* D_next;
    int* flag;
};

template <int kC, int kTherm, bool kWarp>
__global__ void __launch_bounds__(kC, kOnePerSM * 256 / kC)
    k_step_one(const __grid_constant__ OneParams p) {
    using Pipe = ChunkPipe<kOneArrays, kC>;
    constexpr int kSpan = Pipe::kSpan;
    __shared__ __align__(128) float smem[kChunkStages * kOneArrays * kSpan];
    __shared__ __align__(8) unsigned long long bars[kChunkStages];
    const int tid = threadIdx.x;
    Pipe pipe;
    pipe.begin(smem, bars, p.n);
    griddep_wait();
    griddep_launch_dependents();
    const void* src = nullptr;
    if (tid < kOneArrays) src = p.src[tid];
    if (tid < 32) {
        __syncwarp();
        for (int i = 0; i < kChunkStages && i < pipe.count; ++i) pipe.issue(i, src);
    }
    __syncthreads();  // the barriers are initialised
    const MeshGeom& g = p.g;
    const StepConsts& c = p.c;
    for (int i = 0; i < pipe.count; ++i) {
        const bool ok = pipe.wait(i);
        const float(*s)[kSpan] = pipe.stage[i % kChunkStages];
        const int bead = pipe.bead0(i) + tid, e = tid + kChunkHalo;
        const bool live = ok && bead < p.n;
        float x = 0.f, y = 0.f, z = 0.f;
        uint32_t m = 0;
        if (live) {
            x = s[0][e];
            y = s[1][e];
            z = s[2][e];
            m = __float_as_uint(s[6][e]);
            float vx = s[3][e], vy = s[4][e], vz = s[5][e];
            const float s0 = __fmul_rn(x, g.inv_h[0]), s1 = __fmul_rn(y, g.inv_h[1]),
                        s2 = __fmul_rn(z, g.inv_h[2]);
            const float flx = floorf(s0), fly = floorf(s1), flz = floorf(s2);
            const Corners k = load_corners(p.G + (size_t)((m >> kTypeShift) & kTypeMask) * g.gnodes,
                                           g, flx, fly, flz);
            // while they arrive: the chain neighbours' bonds and the noise
            float nx = 0.f, ny = 0.f, nz = 0.f, qx = 0.f, qy = 0.f, qz = 0.f;
            if (kWarp) {
                // one bond of a bead lies inside its lane, the other crosses lanes
                const bool odd = (m & kSlotOdd) != 0;
                const float ax = x - s[0][e + 1], ay = y - s[1][e + 1], az = z - s[2][e + 1];
                const float bx = s[0][e - 1] - x, by = s[1][e - 1] - y, bz = s[2][e - 1] - z;
                if (odd) {
                    if (m & kBondNext) bond_force<kCrossBond>(ax, ay, az, c.two_k, c.r0, nx, ny, nz);
                    if (m & kBondPrev) bond_force<kLaneBond>(bx, by, bz, c.two_k, c.r0, qx, qy, qz);
                } else {
                    if (m & kBondNext) bond_force<kLaneBond>(ax, ay, az, c.two_k, c.r0, nx, ny, nz);
                    if (m & kBondPrev) bond_force<kCrossBond>(bx, by, bz, c.two_k, c.r0, qx, qy, qz);
                }
                nx = __fsub_rn(nx, qx);
                ny = __fsub_rn(ny, qy);
                nz = __fsub_rn(nz, qz);
            }
            const uint32_t tag = m & kTagMask;
            float gx = 0.f, gy = 0.f, gz = 0.f;
            bool coll = false;
            if (kTherm == 1) gauss3(c, tag, p.step, gx, gy, gz);
            if (kTherm == 2) {
                coll = andersen_collides(c, tag, p.step);
                if (coll) gauss3(c, tag, p.step, gx, gy, gz);
            }
            const float f0 = __fsub_rn(s0, flx), f1 = __fsub_rn(s1, fly), f2 = __fsub_rn(s2, flz);
            float4 lo, hi;
            cell_coefs(HPF_CORNERS(k, x), lo, hi);
            float fx = drag_field(c.fric, vx, cell_poly(lo, hi, f0, f1, f2));
            cell_coefs(HPF_CORNERS(k, y), lo, hi);
            float fy = drag_field(c.fric, vy, cell_poly(lo, hi, f0, f1, f2));
            cell_coefs(HPF_CORNERS(k, z), lo, hi);
            float fz = drag_field(c.fric, vz, cell_poly(lo, hi, f0, f1, f2));
            if (kTherm == 1) {
                fx = fmaf(c.sigma, gx, fx);
                fy = fmaf(c.sigma, gy, fy);
                fz = fmaf(c.sigma, gz, fz);
            }
            if (kWarp) {
                fx += nx;
                fy += ny;
                fz += nz;
            } else {
                if (m & kBondPrev)
                    bond_force<kChainBond>(x - s[0][e - 1], y - s[1][e - 1], z - s[2][e - 1], c.two_k,
                                           c.r0, fx, fy, fz);
                if (m & kBondNext)
                    bond_force<kChainBond>(x - s[0][e + 1], y - s[1][e + 1], z - s[2][e + 1], c.two_k,
                                           c.r0, fx, fy, fz);
            }
            if (kTherm == 2 && coll) {
                const float h = 0.5f * c.dt_m;
                vx = fmaf(h, fx, __fmul_rn(c.sig_v, gx));
                vy = fmaf(h, fy, __fmul_rn(c.sig_v, gy));
                vz = fmaf(h, fz, __fmul_rn(c.sig_v, gz));
            } else {
                vx = fmaf(c.dt_m, fx, vx);
                vy = fmaf(c.dt_m, fy, vy);
                vz = fmaf(c.dt_m, fz, vz);
            }
            x = fmaf(c.dt, vx, x);
            y = fmaf(c.dt, vy, y);
            z = fmaf(c.dt, vz, z);
            p.out.x[bead] = x;
            p.out.y[bead] = y;
            p.out.z[bead] = z;
            p.out.vx[bead] = vx;
            p.out.vy[bead] = vy;
            p.out.vz[bead] = vz;
            const bool finite = isfinite(x) && isfinite(y) && isfinite(z) && isfinite(vx) &&
                                isfinite(vy) && isfinite(vz);
            if (!finite) atomicOr(p.flag, kFlagNonFinite);
            else if (!(coord_in_range(x, g.inv_h[0]) && coord_in_range(y, g.inv_h[1]) &&
                       coord_in_range(z, g.inv_h[2])))
                atomicOr(p.flag, kFlagRange);
        }
        if (p.D_next) scatter_paired(p.D_next, g, x, y, z, m, live);
        if (__syncthreads_or(!ok)) {  // every thread is done with the stage
            if (tid == 0) atomicOr(p.flag, kFlagTimeout);
            pipe.drain(i);
            return;
        }
        if (tid < 32 && i + kChunkStages < pipe.count) pipe.issue(i + kChunkStages, src);
    }
}

}  // namespace

bool step_one_supports(const StepConsts& c) { return c.force_mode == 0 && bonded_level(c) == 0; }

void launch_step_one(StateBuf in, StateBuf out, const uint32_t* meta, int n, long long step,
                     const MeshGeom& g, const float4* G, const StepConsts& c, bool warp_order,
                     unsigned long long* D_next, int* flag, cudaStream_t s) {
    if (n <= 0) return;
    static std::once_flag once[64];
    static int sms[64];
    int dev = 0;
    cudaGetDevice(&dev);
    once_per_device(once, [dev] {
        cudaDeviceGetAttribute(&sms[dev & 63], cudaDevAttrMultiProcessorCount, dev);
    });
    const int n_sm = sms[dev & 63] > 0 ? sms[dev & 63] : 1;
    const bool small = n <= kSmallPerSM * kSmallChunk * n_sm;
    const int chunk = small ? kSmallChunk : kChunk;
    const int chunks = (n + chunk - 1) / chunk, cap = kOnePerSM * 256 / chunk * n_sm;
    const int blocks = chunks < cap ? chunks : cap;
    const OneParams p{{in.x, in.y, in.z, in.vx, in.vy, in.vz, meta}, out, n, step, g, G, c, D_next,
                      flag};
    const int th = step_thermostat(c);
#define HPF_ONE_C(C, T, W) launch_pdl(k_step_one<C, T, W>, dim3(blocks), dim3(C), 0, s, p)
#define HPF_ONE(T, W) small ? HPF_ONE_C(kSmallChunk, T, W) : HPF_ONE_C(kChunk, T, W)
    if (th == 1) warp_order ? HPF_ONE(1, true) : HPF_ONE(1, false);
    else if (th == 2) warp_order ? HPF_ONE(2, true) : HPF_ONE(2, false);
    else warp_order ? HPF_ONE(0, true) : HPF_ONE(0, false);
#undef HPF_ONE
#undef HPF_ONE_C
}

}  // namespace hpf
