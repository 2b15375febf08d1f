// k_step.cu -- field gather, bonds, Langevin velocity-Verlet (the fused field-period kernels).
#include "cell_poly.cuh"

namespace hpf {

constexpr int kHaloMax = 16;  // most steps fused into one launch

// Threads of a halo-form CTA (k_step): kStepBlock where the halo is at most
// kNarrowHalo beads a side, kWideBlock where the redundant rim would cost more
// than the finer CTAs give.  Four CTAs of 256 leave less of the chip idle in the last
// wave than two of 512 (160k beads, 4 steps: 318 CTAs for 304 places against 646
// for 608; 120 -> 110.5 us for 20 steps with their fields).  256 against 512
// threads, same steps: halo 2 to 10 -4 to -12 % (160k and 600k beads, bonds
// or angles), halo 15 and 16 0 to -12 %, halo 20 +2 % at 600k beads, halo 30
// +14 %.
constexpr int kStepBlock = 256;
constexpr int kWideBlock = 512;
constexpr int kNarrowHalo = kHaloMax;  // always met by bonds alone

int step_halo_max() { return kHaloMax; }

// ------------------------------------------------------------------ A4 + A5 forces
//
// Conservative force at the current positions, written in tag order.
__global__ void __launch_bounds__(256) k_forces(StateBuf st, const uint32_t* __restrict__ meta,
                                                int n, MeshGeom g, const float4* __restrict__ G,
                                                StepConsts c, int which,
                                                float* __restrict__ F_tag) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float x = st.x[i], y = st.y[i], z = st.z[i];
    const uint32_t m = meta[i];
    float fx = 0.f, fy = 0.f, fz = 0.f;
    if (which & HPF_FORCE_BOND) {
        if (m & kBondPrev)
            bond_force(x - st.x[i - 1], y - st.y[i - 1], z - st.z[i - 1], c.two_k, c.r0, fx, fy, fz);
        if (m & kBondNext)
            bond_force(x - st.x[i + 1], y - st.y[i + 1], z - st.z[i + 1], c.two_k, c.r0, fx, fy, fz);
        if (c.two_ka != 0.f) angle_forces_of(st, meta, i, m, c, fx, fy, fz);
        if (c.kd != 0.f) {
            int back, fwd;
            chain_reach(meta, i, m, back, fwd);
            dihedral_forces_of([&](int d) { return make_float3(st.x[i + d], st.y[i + d], st.z[i + d]); },
                               back, fwd, c, fx, fy, fz);
        }
    }
    if (which & HPF_FORCE_FIELD) {
        const int T = (m >> kTypeShift) & kTypeMask;
        gather_field_mode(G + (size_t)T * g.gnodes, g, c.force_mode, x, y, z, fx, fy, fz);
    }
    const uint32_t tag = m & kTagMask;
    F_tag[3 * tag] = fx;
    F_tag[3 * tag + 1] = fy;
    F_tag[3 * tag + 2] = fz;
}

void launch_forces(StateBuf st, const uint32_t* meta, int n, MeshGeom g, const float4* G,
                   StepConsts c, int which, float* F_tag, cudaStream_t s) {
    if (n <= 0) return;
    k_forces<<<(n + 255) / 256, 256, 0, s>>>(st, meta, n, g, G, c, which, F_tag);
}

// ------------------------------------------------------------------ A6 fused steps
//
// One CTA advances a window of kB consecutive beads (whole chains or
// not) by n_sub steps without leaving the chip: positions live in registers,
// bonded neighbours are exchanged through shared memory, and the frozen field
// is sampled through a per-bead cache.  A bead's update after k steps depends
// on beads up to k places away along its chain, so the outer `halo` beads on
// each side are recomputed redundantly (bit-identically, the noise is keyed by
// tag and step) and only the inner kB - 2 halo beads are written back.
//
// Field cache: inside one cell the interpolated gradient is the trilinear
// polynomial c0 + c1 fx + c2 fy + c3 fz + c4 fx fy + c5 fx fz + c6 fy fz
// + c7 fx fy fz of the cell offset f (per component).  A bead keeps the 24
// coefficients of its current cell in shared memory (six float4 planes, one
// slot per thread, conflict-free) and rebuilds them from the eight corners
// only when it enters another cell -- about once every 40 steps at kT = 1,
// h = 1, dt = 0.01 -- so most sub-steps read six shared float4s instead of
// gathering eight corners from L1/L2.
constexpr int kCachePlanes = 6;
constexpr size_t step_smem(int block) {
    return sizeof(float4) * kCachePlanes * block + sizeof(float) * 3 * 2 * block;
}

// The cell polynomial's coefficients from its corners into cache slot t
// (component-major: planes 2j, 2j + 1 hold c0..c7 of component j; kForce 1:
// planes 0 and 1 hold the polynomial of V).
template <int kForce>
__device__ __forceinline__ void store_cell_coefs(const Corners& k, float4* __restrict__ cache, int t,
                                                 int stride) {
    if (kForce == 1) {
        cell_coefs(HPF_CORNERS(k, w), cache[t], cache[stride + t]);
    } else {
        cell_coefs(HPF_CORNERS(k, x), cache[t], cache[stride + t]);
        cell_coefs(HPF_CORNERS(k, y), cache[2 * stride + t], cache[3 * stride + t]);
        cell_coefs(HPF_CORNERS(k, z), cache[4 * stride + t], cache[5 * stride + t]);
    }
}

// kForce 1: planes 0 and 1 hold the trilinear polynomial of V instead (the
// exact-energy-gradient force differentiates it).  kForce 2: the key is the
// nearest vertex and planes 0 and 1 hold its six staggered coefficients.
template <int kForce>
__device__ __forceinline__ void fill_cell_cache(const float4* __restrict__ Gt, const MeshGeom& g,
                                                float flx, float fly, float flz,
                                                float4* __restrict__ cache, int t,
                                                int stride) {
    if (kForce == 2) {
        float c[6];
        stag_vertex_coefs(Gt, g, flx, fly, flz, c);
        cache[t] = make_float4(c[0], c[1], c[2], c[3]);
        cache[stride + t] = make_float4(c[4], c[5], 0.f, 0.f);
        return;
    }
    store_cell_coefs<kForce>(load_corners(Gt, g, flx, fly, flz), cache, t, stride);
}

// The cache key of a mesh coordinate: its cell (floor), or its nearest
// vertex for the staggered force.
template <int kForce>
__device__ __forceinline__ float cache_key(float s) {
    return kForce == 2 ? stag_vertex(s) : floorf(s);
}

// Friction and field force of a bead with velocity (vx, vy, vz) from its cached
// cell, at the offset (fx, fy, fz).
template <int kForce>
__device__ __forceinline__ void eval_cell_cache(const float4* __restrict__ cache, int t, float fx,
                                                float fy, float fz, float fric, float vx, float vy,
                                                float vz, float& Fx, float& Fy, float& Fz,
                                                const MeshGeom& g, int stride) {
    if (kForce != 0) {
        Fx = __fmul_rn(-fric, vx);
        Fy = __fmul_rn(-fric, vy);
        Fz = __fmul_rn(-fric, vz);
    }
    if (kForce == 2) {
        const float4 lo = cache[t], hi = cache[stride + t];
        const float c[6] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y};
        stag_force(c, fx, fy, fz, g, Fx, Fy, Fz);
    } else if (kForce == 1) {
        // V = a0 + a1 fx + a2 fy + a3 fz + a4 fx fy + a5 fx fz + a6 fy fz + a7 fx fy fz;
        // F = -(1/h) dV/df per axis
        const float4 lo = cache[t], hi = cache[stride + t];
        const float dx = fmaf(fz, fmaf(fy, hi.w, hi.y), fmaf(fy, hi.x, lo.y));
        const float dy = fmaf(fz, fmaf(fx, hi.w, hi.z), fmaf(fx, hi.x, lo.z));
        const float dz = fmaf(fy, fmaf(fx, hi.w, hi.z), fmaf(fx, hi.y, lo.w));
        Fx = fmaf(-g.inv_h[0], dx, Fx);
        Fy = fmaf(-g.inv_h[1], dy, Fy);
        Fz = fmaf(-g.inv_h[2], dz, Fz);
    } else {
        Fx = drag_field(fric, vx, cell_poly(cache[0 * stride + t], cache[1 * stride + t], fx, fy, fz));
        Fy = drag_field(fric, vy, cell_poly(cache[2 * stride + t], cache[3 * stride + t], fx, fy, fz));
        Fz = drag_field(fric, vz, cell_poly(cache[4 * stride + t], cache[5 * stride + t], fx, fy, fz));
    }
}

// A warp reads shared positions of its own lanes and of the edge lanes of the
// two adjacent warps only, so each sub-step synchronises adjacent warp pairs
// (named barrier w + 1 joins warps w and w + 1) instead of the whole CTA.
// Every warp waits on its left pair first, then its right pair, so the waits
// form no cycle.  With two position buffers a warp can run at most one
// sub-step ahead of a neighbour, which has by then finished reading the buffer
// it is about to overwrite.
static_assert(kWideBlock / 32 <= 16, "named barriers 1..15 cover at most 16 warps");
template <int kB>
__device__ __forceinline__ void neighbour_sync(int w) {
    constexpr int kWarps = kB / 32;
    if (w > 0) asm volatile("bar.sync %0, 64;" ::"r"(w) : "memory");
    if (w + 1 < kWarps) asm volatile("bar.sync %0, 64;" ::"r"(w + 1) : "memory");
}

template <int kB, int kTherm, int kForce, int kBonded>
__global__ void __launch_bounds__(kB, 1024 / kB) k_step(StateBuf in, StateBuf out,
                                                        const uint32_t* __restrict__ meta, int n,
                                                        int halo, int n_sub, long long step0,
                                                        MeshGeom g, const float4* __restrict__ G,
                                                        StepConsts c,
                                                        unsigned long long* __restrict__ D_next,
                                                        int* __restrict__ flag) {
    griddep_wait();
    griddep_launch_dependents();
    extern __shared__ float4 smem4[];
    float4* cache = smem4;                                   // [kCachePlanes][kB]
    float* sx = reinterpret_cast<float*>(smem4 + kCachePlanes * kB);  // [2][block]
    float* sy = sx + 2 * kB;
    float* sz = sy + 2 * kB;
    const int t = threadIdx.x;
    const int payload = kB - 2 * halo;
    const long long i = (long long)blockIdx.x * payload - halo + t;
    const bool live = (i >= 0 && i < n);
    float x = 0.f, y = 0.f, z = 0.f, vx = 0.f, vy = 0.f, vz = 0.f;
    uint32_t m = 0;
    if (live) {
        x = in.x[i];
        y = in.y[i];
        z = in.z[i];
        vx = in.vx[i];
        vy = in.vy[i];
        vz = in.vz[i];
        m = meta[i];
    }
    // out-of-range threads only fill their shared-memory slot
    const bool has_prev = live && (m & kBondPrev) && t > 0;
    const bool has_next = live && (m & kBondNext) && t + 1 < kB;
    // bond flags of the whole window, for the angles centred at the neighbours
    // and the dihedrals through them
    __shared__ unsigned char s_bonds[kB];
    int back = 0, fwd = 0;  // consecutive bonds backwards / forwards inside the window (<= 3)
    if (kBonded >= 1) {
        s_bonds[t] = (unsigned char)((has_prev ? 1 : 0) | (has_next ? 2 : 0));
        __syncthreads();
    }
    if (kBonded == 2) {
        if (has_prev) {
            back = 1;
            if (s_bonds[t - 1] & 1) {
                back = 2;
                if (s_bonds[t - 2] & 1) back = 3;
            }
        }
        if (has_next) {
            fwd = 1;
            if (s_bonds[t + 1] & 2) {
                fwd = 2;
                if (s_bonds[t + 2] & 2) fwd = 3;
            }
        }
    }
    const uint32_t tag = m & kTagMask;
    const float4* __restrict__ Gt = G + (size_t)((m >> kTypeShift) & kTypeMask) * g.gnodes;
    float cfx = __int_as_float(0x7fc00000), cfy = cfx, cfz = cfx;  // cached cell: none
    for (int k = 0; k < n_sub; ++k) {
        const int b = k & 1;
        sx[b * kB + t] = x;
        sy[b * kB + t] = y;
        sz[b * kB + t] = z;
        neighbour_sync<kB>(t >> 5);
        const float s0 = __fmul_rn(x, g.inv_h[0]), s1 = __fmul_rn(y, g.inv_h[1]),
                    s2 = __fmul_rn(z, g.inv_h[2]);
        const float flx = cache_key<kForce>(s0), fly = cache_key<kForce>(s1),
                    flz = cache_key<kForce>(s2);
        if (flx != cfx || fly != cfy || flz != cfz) {
            fill_cell_cache<kForce>(Gt, g, flx, fly, flz, cache, t, kB);
            cfx = flx;
            cfy = fly;
            cfz = flz;
        }
        float fx, fy, fz;
        eval_cell_cache<kForce>(cache, t, __fsub_rn(s0, flx), __fsub_rn(s1, fly),
                                __fsub_rn(s2, flz), c.fric, vx, vy, vz, fx, fy, fz, g, kB);
        if (kTherm == 1) {
            float nx, ny, nz;
            gauss3(c, tag, step0 + k, nx, ny, nz);
            fx = fmaf(c.sigma, nx, fx);
            fy = fmaf(c.sigma, ny, fy);
            fz = fmaf(c.sigma, nz, fz);
        }
        const int tp = has_prev ? t - 1 : t, tn = has_next ? t + 1 : t;
        bond_force<kChainBond>(x - sx[b * kB + tp], y - sy[b * kB + tp], z - sz[b * kB + tp],
                               has_prev ? c.two_k : 0.0f, c.r0, fx, fy, fz);
        bond_force<kChainBond>(x - sx[b * kB + tn], y - sy[b * kB + tn], z - sz[b * kB + tn],
                               has_next ? c.two_k : 0.0f, c.r0, fx, fy, fz);
        if (kBonded >= 1) {
            // the three angles this bead belongs to: centred at t - 1, t and t + 1
            const int tp2 = (has_prev && t >= 2) ? t - 2 : t;
            const int tn2 = (has_next && t + 2 < kB) ? t + 2 : t;
            const bool left = has_prev && t >= 2 && (s_bonds[t - 1] & 1);
            const bool right = has_next && t + 2 < kB && (s_bonds[t + 1] & 2);
            const float xp = sx[b * kB + tp], yp = sy[b * kB + tp],
                        zp = sz[b * kB + tp];
            const float xn = sx[b * kB + tn], yn = sy[b * kB + tn],
                        zn = sz[b * kB + tn];
            float ax, ay, az, bx, by, bz;
            // centred at t: this bead takes minus both end shares
            angle_force(xp - x, yp - y, zp - z, xn - x, yn - y, zn - z,
                        (has_prev && has_next) ? c.two_ka : 0.0f, c, ax, ay, az, bx, by,
                        bz);
            fx -= ax + bx;
            fy -= ay + by;
            fz -= az + bz;
            // centred at t - 1 (ends t - 2 and t): this bead is end b
            angle_force(sx[b * kB + tp2] - xp, sy[b * kB + tp2] - yp,
                        sz[b * kB + tp2] - zp, x - xp, y - yp, z - zp,
                        left ? c.two_ka : 0.0f, c, ax, ay, az, bx, by, bz);
            fx += bx;
            fy += by;
            fz += bz;
            // centred at t + 1 (ends t and t + 2): this bead is end a
            angle_force(x - xn, y - yn, z - zn, sx[b * kB + tn2] - xn,
                        sy[b * kB + tn2] - yn, sz[b * kB + tn2] - zn,
                        right ? c.two_ka : 0.0f, c, ax, ay, az, bx, by, bz);
            fx += ax;
            fy += ay;
            fz += az;
        }
        if (kBonded == 2) {
            const int o = b * kB + t;
            dihedral_forces_of(
                [&](int d) { return make_float3(sx[o + d], sy[o + d], sz[o + d]); }, back, fwd, c,
                fx, fy, fz);
        }
        if (kTherm == 2 && andersen_collides(c, tag, step0 + k)) {
            // the on-step velocity redrawn, then the second half kick
            float nx, ny, nz;
            gauss3(c, tag, step0 + k, nx, ny, nz);
            const float h = 0.5f * c.dt_m;
            vx = fmaf(h, fx, __fmul_rn(c.sig_v, nx));
            vy = fmaf(h, fy, __fmul_rn(c.sig_v, ny));
            vz = fmaf(h, fz, __fmul_rn(c.sig_v, nz));
        } else {
            vx = fmaf(c.dt_m, fx, vx);
            vy = fmaf(c.dt_m, fy, vy);
            vz = fmaf(c.dt_m, fz, vz);
        }
        x = fmaf(c.dt, vx, x);
        y = fmaf(c.dt, vy, y);
        z = fmaf(c.dt, vz, z);
    }
    const bool mine = live && t >= halo && t < kB - halo;
    if (mine) {
        out.x[i] = x;
        out.y[i] = y;
        out.z[i] = z;
        out.vx[i] = vx;
        out.vy[i] = vy;
        out.vz[i] = vz;
        const bool finite = isfinite(x) && isfinite(y) && isfinite(z) && isfinite(vx) &&
                            isfinite(vy) && isfinite(vz);
        if (!finite) atomicOr(flag, kFlagNonFinite);
        else if (!(coord_in_range(x, g.inv_h[0]) && coord_in_range(y, g.inv_h[1]) &&
                   coord_in_range(z, g.inv_h[2])))
            atomicOr(flag, kFlagRange);
    }
    // a launch that ends on a refresh step deposits the final positions
    if (D_next) scatter_paired(D_next, g, x, y, z, m, mine);
}

template <int kB, int kTherm, int kForce, int kBonded>
static void launch_step_b(StateBuf in, StateBuf out, const uint32_t* meta, int n, int halo, int n_sub,
                          long long step0, MeshGeom g, const float4* G, StepConsts c,
                          unsigned long long* D_next, int* flag, cudaStream_t s) {
    static std::once_flag attr[64];
    once_per_device(attr, [] {
        cudaFuncSetAttribute(k_step<kB, kTherm, kForce, kBonded>,
                             cudaFuncAttributeMaxDynamicSharedMemorySize, (int)step_smem(kB));
    });
    const int payload = kB - 2 * halo;
    const int blocks = (n + payload - 1) / payload;
    launch_pdl(k_step<kB, kTherm, kForce, kBonded>, dim3(blocks), dim3(kB), step_smem(kB), s, in, out,
               meta, n, halo, n_sub, step0, g, G, c, D_next, flag);
}

template <int kTherm, int kForce, int kBonded>
static void launch_step_t(StateBuf in, StateBuf out, const uint32_t* meta, int n, int n_sub,
                          long long step0, MeshGeom g, const float4* G, StepConsts c,
                          unsigned long long* D_next, int* flag, cudaStream_t s) {
    // a bead's update after k sub-steps depends on beads up to k (bonds), 2k
    // (angles) or 3k (dihedrals) places away along its chain
    const int halo = (kBonded + 1) * n_sub;
    if (kBonded == 0 || halo <= kNarrowHalo)
        launch_step_b<kStepBlock, kTherm, kForce, kBonded>(in, out, meta, n, halo, n_sub, step0, g, G,
                                                           c, D_next, flag, s);
    else if constexpr (kBonded > 0)
        launch_step_b<kWideBlock, kTherm, kForce, kBonded>(in, out, meta, n, halo, n_sub, step0, g, G,
                                                           c, D_next, flag, s);
}

template <int kTherm, int kForce>
static void launch_step_a(StateBuf in, StateBuf out, const uint32_t* meta, int n, int n_sub,
                          long long step0, MeshGeom g, const float4* G, StepConsts c,
                          unsigned long long* D_next, int* flag, cudaStream_t s) {
    const int bonded = bonded_level(c);
    if (bonded == 2)
        launch_step_t<kTherm, kForce, 2>(in, out, meta, n, n_sub, step0, g, G, c, D_next, flag, s);
    else if (bonded == 1)
        launch_step_t<kTherm, kForce, 1>(in, out, meta, n, n_sub, step0, g, G, c, D_next, flag, s);
    else
        launch_step_t<kTherm, kForce, 0>(in, out, meta, n, n_sub, step0, g, G, c, D_next, flag, s);
}

void launch_step(StateBuf in, StateBuf out, const uint32_t* meta, int n, int n_sub,
                 long long step0, MeshGeom g, const float4* G, StepConsts c,
                 unsigned long long* D_next, int* flag, cudaStream_t s) {
    if (n <= 0 || n_sub <= 0) return;
    const int therm = step_thermostat(c);
#define HPF_HALO(T)                                                                        \
    if (c.force_mode == 2)                                                                   \
        launch_step_a<T, 2>(in, out, meta, n, n_sub, step0, g, G, c, D_next, flag, s);       \
    else if (c.force_mode == 1)                                                              \
        launch_step_a<T, 1>(in, out, meta, n, n_sub, step0, g, G, c, D_next, flag, s);       \
    else                                                                                     \
        launch_step_a<T, 0>(in, out, meta, n, n_sub, step0, g, G, c, D_next, flag, s);
    if (therm == 1) {
        HPF_HALO(1)
    } else if (therm == 2) {
        HPF_HALO(2)
    } else {
        HPF_HALO(0)
    }
#undef HPF_HALO
}

// ------------------------------------------------------------------ A6, warp form
//
// When every chain has at most 64 beads the sort also packs consecutive whole
// chains into segments of at most 64 beads, and one warp advances one segment
// for all n_sub steps on its own: lane l holds beads 2l and 2l + 1, so a
// bead's chain neighbours are either its partner in the same lane or the
// neighbouring lane's bead, exchanged with register shuffles.  No halo, no
// shared positions and no barrier: warps never wait for one another.  The
// field is sampled through the same per-bead cell cache as above (two slots
// per thread).  A persistent grid walks the segment list, whose length is
// read on the device so a re-sort needs no host synchronisation.
constexpr int kWarpBlock = 256;
constexpr size_t kWarpSmem = sizeof(float4) * kCachePlanes * 2 * kWarpBlock;
// The packed form (advance_pairs below) covers bonds with the interpolated-
// gradient force; it needs no shared cache.
__host__ __device__ constexpr bool pair_form(int force, int bonded) {
    return force == 0 && bonded == 0;
}
__host__ __device__ constexpr size_t warp_smem(int force, int bonded) {
    return pair_form(force, bonded) ? 0 : kWarpSmem;
}

struct Bead {
    float x, y, z, vx, vy, vz;
    uint32_t m;
    float cfx, cfy, cfz;  // cached cell (floor of the mesh coordinate), NaN: none
};

// The bead's cell: refill its cache of the cell polynomial when the bead
// has entered another cell; returns the offsets inside the cell.
template <int kForce, int kLerp = 0>
__device__ __forceinline__ void cell_check(Bead& b, const float4* __restrict__ G, const MeshGeom& g,
                                           float4* __restrict__ cache, int slot, float& f0,
                                           float& f1, float& f2,
                                           const float4* __restrict__ G2 = nullptr) {
    const float s0 = __fmul_rn(b.x, g.inv_h[0]), s1 = __fmul_rn(b.y, g.inv_h[1]),
                s2 = __fmul_rn(b.z, g.inv_h[2]);
    const float flx = cache_key<kForce>(s0), fly = cache_key<kForce>(s1),
                flz = cache_key<kForce>(s2);
    if (flx != b.cfx || fly != b.cfy || flz != b.cfz) {
        const size_t off = (size_t)((b.m >> kTypeShift) & kTypeMask) * g.gnodes;
        if (kLerp) {
            // the window's second field: its polynomial in planes 6..11
            store_cell_coefs<0>(load_corners(G2 + off, g, flx, fly, flz),
                                cache + kCachePlanes * 2 * kWarpBlock, slot, 2 * kWarpBlock);
        }
        fill_cell_cache<kForce>(G + off, g, flx,
                                fly, flz, cache, slot, 2 * kWarpBlock);
        b.cfx = flx;
        b.cfy = fly;
        b.cfz = flz;
    }
    f0 = __fsub_rn(s0, flx);
    f1 = __fsub_rn(s1, fly);
    f2 = __fsub_rn(s2, flz);
}

// Force on one bead: field (cached cell polynomial at offsets f), friction,
// noise (nx, ny, nz) and the bond force (bx, by, bz) already summed over its
// chain neighbours.
template <int kTherm, int kForce, int kLerp = 0>
__device__ __forceinline__ void bead_force(const Bead& b, float f0, float f1, float f2, float nx,
                                           float ny, float nz, float bx, float by, float bz,
                                           const StepConsts& c, const MeshGeom& g,
                                           const float4* __restrict__ cache, int slot, float a,
                                           float& fx, float& fy, float& fz) {
    if (kLerp) {
        // the field (1 - a) G0 + a G2: P0 + a (P2 - P0) of the two cached polynomials
        constexpr int st = 2 * kWarpBlock;
        const float4* c2 = cache + kCachePlanes * st;
        const float p0x = cell_poly(cache[0 * st + slot], cache[1 * st + slot], f0, f1, f2);
        const float p0y = cell_poly(cache[2 * st + slot], cache[3 * st + slot], f0, f1, f2);
        const float p0z = cell_poly(cache[4 * st + slot], cache[5 * st + slot], f0, f1, f2);
        const float p2x = cell_poly(c2[0 * st + slot], c2[1 * st + slot], f0, f1, f2);
        const float p2y = cell_poly(c2[2 * st + slot], c2[3 * st + slot], f0, f1, f2);
        const float p2z = cell_poly(c2[4 * st + slot], c2[5 * st + slot], f0, f1, f2);
        fx = drag_field(c.fric, b.vx, fmaf(a, p2x - p0x, p0x));
        fy = drag_field(c.fric, b.vy, fmaf(a, p2y - p0y, p0y));
        fz = drag_field(c.fric, b.vz, fmaf(a, p2z - p0z, p0z));
    } else {
        eval_cell_cache<kForce>(cache, slot, f0, f1, f2, c.fric, b.vx, b.vy, b.vz, fx, fy, fz, g,
                                2 * kWarpBlock);
    }
    if (kTherm == 1) {
        fx = fmaf(c.sigma, nx, fx);
        fy = fmaf(c.sigma, ny, fy);
        fz = fmaf(c.sigma, nz, fz);
    }
    fx += bx;
    fy += by;
    fz += bz;
}

// Kick of one bead by that force.  Andersen (kTherm 2): a colliding bead's
// on-step velocity is sqrt(kT/m) (nx, ny, nz) before the second half kick.
template <int kTherm, int kForce, int kLerp = 0>
__device__ __forceinline__ void kick_bead(Bead& b, float f0, float f1, float f2, float nx,
                                          float ny, float nz, float bx, float by, float bz,
                                          const StepConsts& c, const MeshGeom& g,
                                          const float4* __restrict__ cache, int slot,
                                          bool coll, float a = 0.f) {
    float fx, fy, fz;
    bead_force<kTherm, kForce, kLerp>(b, f0, f1, f2, nx, ny, nz, bx, by, bz, c, g, cache, slot, a,
                                      fx, fy, fz);
    if (kTherm == 2 && coll) {
        const float h = 0.5f * c.dt_m;
        b.vx = fmaf(h, fx, __fmul_rn(c.sig_v, nx));
        b.vy = fmaf(h, fy, __fmul_rn(c.sig_v, ny));
        b.vz = fmaf(h, fz, __fmul_rn(c.sig_v, nz));
    } else {
        b.vx = fmaf(c.dt_m, fx, b.vx);
        b.vy = fmaf(c.dt_m, fy, b.vy);
        b.vz = fmaf(c.dt_m, fz, b.vz);
    }
}

// ---- two beads a lane in packed FP32 (the interpolated-gradient force)
//
// A launch of the warp form is bound by instruction issue (63 % of the issue
// slots used at 16 warps per SM, about 550 instructions per warp and
// sub-step) and by the L1 data pipe (56 %, a third of it the reads of the
// shared polynomial cache).  Here every FP32 operation that a lane does for
// both of its beads is one packed instruction (add, multiply and
// multiply-add on float pairs), and the two cell polynomials live in 48
// registers, paired coefficient by coefficient, instead of shared memory: no
// loads per evaluation, and the L1 keeps the space.  91.4M -> 75.0M
// instructions and 124 -> 118 us per 10-step launch of 1M beads (L1 data pipe 56 ->
// 34 %), 108 with today's deposit, uniform segment bounds and fused friction.  What
// bounds it now is latency at 16 warps per SM (60 % of the issue slots used): the
// refills (a warp meets about one per sub-step; 1.3 of the 6.1 cycles between a warp's
// instructions) and dependent arithmetic.  Starting a refill's loads a
// sub-step's noise earlier was slower, whether as L1 prefetches (137 us: they
// do not fill the L1) or as asynchronous copies into shared memory (126 us).
// The rounding of every operation is the scalar form's, so the bits are too.
struct Pair {
    float2 x, y, z, vx, vy, vz;  // .x: bead 2 lane, .y: bead 2 lane + 1
    float2 cx, cy, cz;           // cached cells, NaN: none
    float2 kx[8], ky[8], kz[8];  // their polynomials, c0 .. c7 per component
    uint32_t m0, m1;
};

__device__ __forceinline__ float2 both(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 pair_sub(float2 a, float2 b) {  // a - b
    return __ffma2_rn(b, both(-1.0f), a);
}

// cell_poly of both beads.
__device__ __forceinline__ float2 pair_poly(const float2 (&c)[8], float2 fx, float2 fy, float2 fz) {
    float2 a = __ffma2_rn(fz, c[7], c[4]);
    a = __ffma2_rn(fy, a, c[1]);
    a = __ffma2_rn(fz, c[5], a);
    const float2 b = __ffma2_rn(fz, c[6], c[2]);
    float2 v = __ffma2_rn(fx, a, c[0]);
    v = __ffma2_rn(fy, b, v);
    return __ffma2_rn(fz, c[3], v);
}

template <int kBead>
__device__ __forceinline__ void pair_coefs(Pair& b, const Corners& k) {
    auto put = [](float2 (&c)[8], float4 lo, float4 hi) {
        const float v[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
#pragma unroll
        for (int j = 0; j < 8; ++j) (kBead == 0 ? c[j].x : c[j].y) = v[j];
    };
    float4 lo, hi;
    cell_coefs(HPF_CORNERS(k, x), lo, hi);
    put(b.kx, lo, hi);
    cell_coefs(HPF_CORNERS(k, y), lo, hi);
    put(b.ky, lo, hi);
    cell_coefs(HPF_CORNERS(k, z), lo, hi);
    put(b.kz, lo, hi);
}

__device__ __forceinline__ const float4* species_field(const float4* __restrict__ G,
                                                       const MeshGeom& g, uint32_t m) {
    return G + (size_t)((m >> kTypeShift) & kTypeMask) * g.gnodes;
}

// floor(s) of both for |s| < 2^22 (the coordinate range ends at 2^18): adding
// 1.5 2^23 rounded down leaves an integer ulp.
__device__ __forceinline__ float2 pair_floor(float2 s) {
    return __fadd2_rn(__fadd2_rd(s, both(12582912.0f)), both(-12582912.0f));
}

// Uniforms of two Philox words, as open_uniform: the float 1 + (r >> 9) 2^-23
// (its bits) minus 1 - 2^-24, exact.
__device__ __forceinline__ float2 pair_uniform(uint32_t r0, uint32_t r1) {
    return __fadd2_rn(make_float2(__uint_as_float(0x3f800000u | (r0 >> 9)),
                                  __uint_as_float(0x3f800000u | (r1 >> 9))),
                      both(-0.999999940395355224609375f));
}

// The Box-Muller radius sqrt(-2 ln u) of both (log_unit's two forms).
__device__ __forceinline__ float2 pair_radius(float2 u) {
    const float2 d = __ffma2_rn(u, both(-1.0f), both(1.0f));
    const float2 t = __ffma2_rn(__ffma2_rn(d, both(1.0f / 3.0f), both(0.5f)), d, both(1.0f));
    const float2 series = __fmul2_rn(d, t);
    const float2 l = __fmul2_rn(make_float2(d.x <= 0.015625f ? series.x : -__logf(u.x),
                                            d.y <= 0.015625f ? series.y : -__logf(u.y)),
                                both(2.0f));
    return __fmul2_rn(l, make_float2(rsqrtf(l.x), rsqrtf(l.y)));
}

// Minus gauss3 of both beads.
__device__ __forceinline__ void pair_gauss3_neg(const StepConsts& c, uint32_t tag0, uint32_t tag1,
                                            long long step, float2& gx, float2& gy, float2& gz) {
    uint32_t a0 = tag0 + c.tag_base, a1 = (uint32_t)step,
             a2 = (uint32_t)((unsigned long long)step >> 32), a3 = 0u;
    uint32_t b0 = tag1 + c.tag_base, b1 = a1, b2 = a2, b3 = 0u;
    philox4x32_10(a0, a1, a2, a3, c.rk0, c.rk1);
    philox4x32_10(b0, b1, b2, b3, c.rk0, c.rk1);
    const float2 a = pair_radius(pair_uniform(a0, b0));
    const float2 b = pair_radius(pair_uniform(a2, b2));
    const float2 t1 = __fmul2_rn(__fadd2_rn(pair_uniform(a1, b1), both(-0.5f)),
                                 both(6.28318530717958648f));
    const float2 t3 = __fmul2_rn(__fadd2_rn(pair_uniform(a3, b3), both(-0.5f)),
                                 both(6.28318530717958648f));
    float2 s1, k1;
    __sincosf(t1.x, &s1.x, &k1.x);
    __sincosf(t1.y, &s1.y, &k1.y);
    gx = __fmul2_rn(a, k1);
    gy = __fmul2_rn(a, s1);
    gz = __fmul2_rn(b, make_float2(__cosf(t3.x), __cosf(t3.y)));
}

// Minus the bond forces of a segment (warp_bonded_forces<0>), the lane's two bonds as
// a pair: the in-lane one (2l, 2l + 1) and the one to the next lane.  The pairs
// (dx, dy'), (dy, dx'), (dz, dz') give each its own order of |d|^2 (kLaneBond,
// kCrossBond).
__device__ __forceinline__ void pair_bonds(const Pair& b, bool p0, float2 two_k,
                                           const StepConsts& c, float2& wx, float2& wy,
                                           float2& wz) {
    const float dx = __shfl_down_sync(0xffffffffu, b.x.x, 1);
    const float dy = __shfl_down_sync(0xffffffffu, b.y.x, 1);
    const float dz = __shfl_down_sync(0xffffffffu, b.z.x, 1);
    const float2 A = make_float2(__fsub_rn(b.x.x, b.x.y), __fsub_rn(b.y.y, dy));
    const float2 B = make_float2(__fsub_rn(b.y.x, b.y.y), __fsub_rn(b.x.y, dx));
    const float2 C = make_float2(__fsub_rn(b.z.x, b.z.y), __fsub_rn(b.z.y, dz));
    const float2 rr = __ffma2_rn(C, C, __ffma2_rn(B, B, __fmul2_rn(A, A)));
    const float2 ir = make_float2(rsqrtf(fmaxf(rr.x, 1e-30f)), rsqrtf(fmaxf(rr.y, 1e-30f)));
    const float2 s = __fmul2_rn(two_k, __ffma2_rn(both(-c.r0), ir, both(1.0f)));
    const float2 fa = __fmul2_rn(s, A), fb = __fmul2_rn(s, B), fc = __fmul2_rn(s, C);
    const float ux = __shfl_up_sync(0xffffffffu, fb.y, 1);  // the previous lane's share
    const float uy = __shfl_up_sync(0xffffffffu, fa.y, 1);
    const float uz = __shfl_up_sync(0xffffffffu, fc.y, 1);
    wx = make_float2(p0 ? __fsub_rn(fa.x, ux) : fa.x, __fsub_rn(fb.y, fa.x));
    wy = make_float2(p0 ? __fsub_rn(fb.x, uy) : fb.x, __fsub_rn(fa.y, fb.x));
    wz = make_float2(p0 ? __fsub_rn(fc.x, uz) : fc.x, __fsub_rn(fc.y, fc.x));
}

// Minus the forces on a lane's two beads at their positions: field, friction,
// bonds and step `step`'s noise.  Opposite sums round alike, and with this sign
// friction and field are one fma, as in drag_field, without a negation.  The
// bonds come last: their shuffles then wait behind the refills (1M beads, 20 steps
// 255.0 -> 254.1 us).  (gx, gy, gz): minus the normals (Langevin), or with
// coll0, coll1 (Andersen: the bead collides) its normals.
struct PairForce {
    float2 nx, ny, nz, gx, gy, gz;
    bool coll0, coll1;
};

template <int kTherm>
__device__ __forceinline__ PairForce pair_force(Pair& b, bool p0, float2 two_k, long long step,
                                                const MeshGeom& g, const float4* __restrict__ G,
                                                const StepConsts& c) {
    PairForce r;
    const float2 s0 = __fmul2_rn(b.x, both(g.inv_h[0])), s1 = __fmul2_rn(b.y, both(g.inv_h[1])),
                 s2 = __fmul2_rn(b.z, both(g.inv_h[2]));
    const float2 l0 = pair_floor(s0), l1 = pair_floor(s1), l2 = pair_floor(s2);
    if (l0.x != b.cx.x || l1.x != b.cy.x || l2.x != b.cz.x)
        pair_coefs<0>(b, load_corners(species_field(G, g, b.m0), g, l0.x, l1.x, l2.x));
    if (l0.y != b.cx.y || l1.y != b.cy.y || l2.y != b.cz.y)
        pair_coefs<1>(b, load_corners(species_field(G, g, b.m1), g, l0.y, l1.y, l2.y));
    b.cx = l0;
    b.cy = l1;
    b.cz = l2;
    const float2 f0 = pair_sub(s0, l0), f1 = pair_sub(s1, l1), f2 = pair_sub(s2, l2);
    r.gx = r.gy = r.gz = both(0.f);
    r.coll0 = r.coll1 = false;
    const uint32_t t0 = b.m0 & kTagMask, t1 = b.m1 & kTagMask;
    if (kTherm == 1) pair_gauss3_neg(c, t0, t1, step, r.gx, r.gy, r.gz);
    if (kTherm == 2) {
        r.coll0 = andersen_collides(c, t0, step);
        r.coll1 = andersen_collides(c, t1, step);
        if (r.coll0) gauss3(c, t0, step, r.gx.x, r.gy.x, r.gz.x);
        if (r.coll1) gauss3(c, t1, step, r.gx.y, r.gy.y, r.gz.y);
    }
    const float2 fric = both(c.fric);
    r.nx = __ffma2_rn(fric, b.vx, pair_poly(b.kx, f0, f1, f2));
    r.ny = __ffma2_rn(fric, b.vy, pair_poly(b.ky, f0, f1, f2));
    r.nz = __ffma2_rn(fric, b.vz, pair_poly(b.kz, f0, f1, f2));
    if (kTherm == 1) {
        const float2 sigma = both(c.sigma);
        r.nx = __ffma2_rn(sigma, r.gx, r.nx);
        r.ny = __ffma2_rn(sigma, r.gy, r.ny);
        r.nz = __ffma2_rn(sigma, r.gz, r.nz);
    }
    float2 wx, wy, wz;
    pair_bonds(b, p0, two_k, c, wx, wy, wz);
    r.nx = __fadd2_rn(r.nx, wx);
    r.ny = __fadd2_rn(r.ny, wy);
    r.nz = __fadd2_rn(r.nz, wz);
    return r;
}

// Kick by those forces (a colliding bead: redrawn velocity, second half kick) and drift.
template <int kTherm>
__device__ __forceinline__ void pair_move(Pair& b, const PairForce& r, const StepConsts& c) {
    b.vx = __ffma2_rn(both(-c.dt_m), r.nx, b.vx);
    b.vy = __ffma2_rn(both(-c.dt_m), r.ny, b.vy);
    b.vz = __ffma2_rn(both(-c.dt_m), r.nz, b.vz);
    if (kTherm == 2) {
        const float h = -0.5f * c.dt_m;
        if (r.coll0) {
            b.vx.x = fmaf(h, r.nx.x, __fmul_rn(c.sig_v, r.gx.x));
            b.vy.x = fmaf(h, r.ny.x, __fmul_rn(c.sig_v, r.gy.x));
            b.vz.x = fmaf(h, r.nz.x, __fmul_rn(c.sig_v, r.gz.x));
        }
        if (r.coll1) {
            b.vx.y = fmaf(h, r.nx.y, __fmul_rn(c.sig_v, r.gx.y));
            b.vy.y = fmaf(h, r.ny.y, __fmul_rn(c.sig_v, r.gy.y));
            b.vz.y = fmaf(h, r.nz.y, __fmul_rn(c.sig_v, r.gz.y));
        }
    }
    b.x = __ffma2_rn(both(c.dt), b.vx, b.x);
    b.y = __ffma2_rn(both(c.dt), b.vy, b.y);
    b.z = __ffma2_rn(both(c.dt), b.vz, b.z);
}

__device__ __forceinline__ void finish_bead(const Bead& b, long long i, StateBuf out,
                                            const MeshGeom& g, int* flag) {
    out.x[i] = b.x;
    out.y[i] = b.y;
    out.z[i] = b.z;
    out.vx[i] = b.vx;
    out.vy[i] = b.vy;
    out.vz[i] = b.vz;
    const bool finite = isfinite(b.x) && isfinite(b.y) && isfinite(b.z) && isfinite(b.vx) &&
                        isfinite(b.vy) && isfinite(b.vz);
    if (!finite) atomicOr(flag, kFlagNonFinite);
    else if (!(coord_in_range(b.x, g.inv_h[0]) && coord_in_range(b.y, g.inv_h[1]) &&
               coord_in_range(b.z, g.inv_h[2])))
        atomicOr(flag, kFlagRange);
}

// The observables' bead terms of a segment's final state (what the next
// sub-step's force evaluation would form, never applied): F_n at the final
// positions with step `step`'s noise, the on-step velocity
// v_n = v + dt/(2m) F_n, |v_n|^2 and v_n added to the thread's float-float
// sums, and the energy of each bond once (the bond to the next bead: b0's to
// b1, b1's to the next lane's b0).  Bonds only, interpolated-gradient force,
// no Andersen redraw.
struct ObsArgs {
    float2* part;     // [gridDim.x][kBeadVals] float-float block partials
    float half_dt_m;  // dt / (2m)
    BondFF bond;
};

template <int kTherm>
__device__ __forceinline__ void observe_segment(Pair& b, bool a0, bool a1, bool p0, bool n0, bool n1,
                                                float2 two_k, long long step, const MeshGeom& g,
                                                const float4* __restrict__ G, const StepConsts& c,
                                                const ObsArgs& o, FF* acc) {
    const PairForce r = pair_force<kTherm>(b, p0, two_k, step, g, G, c);
    // the next lane's first bead (every lane takes part in the shuffles)
    const float qx = __shfl_down_sync(0xffffffffu, b.x.x, 1);
    const float qy = __shfl_down_sync(0xffffffffu, b.y.x, 1);
    const float qz = __shfl_down_sync(0xffffffffu, b.z.x, 1);
    float uh = acc[1].h, ul = acc[1].l;
    if (n0) bond_energy_ff(b.x.x, b.y.x, b.z.x, b.x.y, b.y.y, b.z.y, o.bond, uh, ul);
    if (n1) bond_energy_ff(b.x.y, b.y.y, b.z.y, qx, qy, qz, o.bond, uh, ul);
    acc[1] = FF{uh, ul};
    const float2 hf = both(-o.half_dt_m);
    const float2 ux = __ffma2_rn(hf, r.nx, b.vx), uy = __ffma2_rn(hf, r.ny, b.vy),
                 uz = __ffma2_rn(hf, r.nz, b.vz);
    if (a0) {
        acc[0] = ff_plus(acc[0], fmaf(ux.x, ux.x, fmaf(uy.x, uy.x, __fmul_rn(uz.x, uz.x))));
        acc[2] = ff_plus(acc[2], ux.x);
        acc[3] = ff_plus(acc[3], uy.x);
        acc[4] = ff_plus(acc[4], uz.x);
    }
    if (a1) {
        acc[0] = ff_plus(acc[0], fmaf(ux.y, ux.y, fmaf(uy.y, uy.y, __fmul_rn(uz.y, uz.y))));
        acc[2] = ff_plus(acc[2], ux.y);
        acc[3] = ff_plus(acc[3], uy.y);
        acc[4] = ff_plus(acc[4], uz.y);
    }
}

// One warp advances one segment by n_sub steps in packed form (the
// interpolated-gradient force).  kObs: also the observables' terms of the
// final state.
template <int kTherm, int kObs = 0>
__device__ __forceinline__ void advance_pairs(const StateBuf& in, const StateBuf& out,
                                              const uint32_t* __restrict__ meta, int base, int cnt,
                                              int n_sub, long long step0, const MeshGeom& g,
                                              const float4* __restrict__ G, const StepConsts& c,
                                              unsigned long long* __restrict__ D_next,
                                              int* __restrict__ flag, const ObsArgs* obs = nullptr,
                                              FF* obs_acc = nullptr) {
    const int lane = threadIdx.x & 31, j0 = 2 * lane;
    const bool a0 = j0 < cnt, a1 = j0 + 1 < cnt;
    const long long i = (long long)base + j0;
    Pair b;
    auto load = [&](const float* p) { return make_float2(a0 ? p[i] : 0.f, a1 ? p[i + 1] : 0.f); };
    b.x = load(in.x);
    b.y = load(in.y);
    b.z = load(in.z);
    b.vx = load(in.vx);
    b.vy = load(in.vy);
    b.vz = load(in.vz);
    b.m0 = a0 ? meta[i] : 0u;
    b.m1 = a1 ? meta[i + 1] : 0u;
    b.cx = b.cy = b.cz = both(__int_as_float(0x7fc00000));
#pragma unroll
    for (int j = 0; j < 8; ++j) b.kx[j] = b.ky[j] = b.kz[j] = both(0.f);
    // whole chains: every flagged neighbour is inside the segment
    const bool p0 = (b.m0 & kBondPrev) != 0, n0 = (b.m0 & kBondNext) != 0;
    const bool n1 = (b.m1 & kBondNext) != 0;  // b1's previous bond is b0's next
    const float2 two_k = make_float2(n0 ? c.two_k : 0.f, n1 ? c.two_k : 0.f);
    for (int k = 0; k < n_sub; ++k)
        pair_move<kTherm>(b, pair_force<kTherm>(b, p0, two_k, step0 + k, g, G, c), c);
    if constexpr (kObs != 0)
        observe_segment<kTherm>(b, a0, a1, p0, n0, n1, two_k, step0 + n_sub, g, G, c, *obs,
                                obs_acc);
    if (a0)
        finish_bead(Bead{b.x.x, b.y.x, b.z.x, b.vx.x, b.vy.x, b.vz.x, b.m0, 0.f, 0.f, 0.f}, i, out, g,
                    flag);
    if (a1)
        finish_bead(Bead{b.x.y, b.y.y, b.z.y, b.vx.y, b.vy.y, b.vz.y, b.m1, 0.f, 0.f, 0.f}, i + 1, out,
                    g, flag);
    if (D_next) {
        scatter_paired(D_next, g, b.x.x, b.y.x, b.z.x, b.m0, a0);
        scatter_paired(D_next, g, b.x.y, b.y.y, b.z.y, b.m1, a1);
    }
}

// One warp advances one segment (whole chains, base .. base + cnt) by n_sub
// steps with the polynomials in shared memory: the other force modes, and the
// interpolated fields of a learned window (two polynomials per bead).
template <int kTherm, int kForce, int kBonded, int kLerp = 0>
__device__ __forceinline__ void advance_segment(const StateBuf& in, const StateBuf& out,
                                                const uint32_t* __restrict__ meta, int base,
                                                int cnt, int n_sub, long long step0,
                                                const MeshGeom& g, const float4* __restrict__ G,
                                                const StepConsts& c,
                                                unsigned long long* __restrict__ D_next,
                                                int* __restrict__ flag, float4* wcache, int tid,
                                                const float4* __restrict__ G2 = nullptr,
                                                int lerp_j0 = 0, float lerp_inv_k = 0.f) {
    const int lane = tid & 31;
    const float nan = __int_as_float(0x7fc00000);
    const int j0 = 2 * lane, j1 = j0 + 1;
    const bool a0 = j0 < cnt, a1 = j1 < cnt;
    Bead b0{0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0u, nan, nan, nan};
    Bead b1 = b0;
    if (a0) {
        const long long i = (long long)base + j0;
        b0.x = in.x[i]; b0.y = in.y[i]; b0.z = in.z[i];
        b0.vx = in.vx[i]; b0.vy = in.vy[i]; b0.vz = in.vz[i];
        b0.m = meta[i];
    }
    if (a1) {
        const long long i = (long long)base + j1;
        b1.x = in.x[i]; b1.y = in.y[i]; b1.z = in.z[i];
        b1.vx = in.vx[i]; b1.vy = in.vy[i]; b1.vz = in.vz[i];
        b1.m = meta[i];
    }
    // whole chains: every flagged neighbour is inside the segment
    const bool p0 = (b0.m & kBondPrev) != 0, n0 = (b0.m & kBondNext) != 0;
    const bool n1 = (b1.m & kBondNext) != 0;  // b1's previous bond is b0's next
    for (int k = 0; k < n_sub; ++k) {
        float w0x, w0y, w0z, w1x, w1y, w1z;  // bonded forces on the lane's two beads
        warp_bonded_forces<kBonded>(b0.x, b0.y, b0.z, b1.x, b1.y, b1.z, p0, n0, n1, c, lane, w0x,
                                    w0y, w0z, w1x, w1y, w1z);
        // the two beads' phases side by side, so their independent work interleaves
        float f00, f01, f02, f10, f11, f12;
        cell_check<kForce, kLerp>(b0, G, g, wcache, tid, f00, f01, f02, G2);
        cell_check<kForce, kLerp>(b1, G, g, wcache, kWarpBlock + tid, f10, f11, f12, G2);
        float g0x = 0.f, g0y = 0.f, g0z = 0.f, g1x = 0.f, g1y = 0.f, g1z = 0.f;
        bool coll0 = false, coll1 = false;
        if (kTherm == 1) {
            gauss3(c, b0.m & kTagMask, step0 + k, g0x, g0y, g0z);
            gauss3(c, b1.m & kTagMask, step0 + k, g1x, g1y, g1z);
        }
        if (kTherm == 2) {
            coll0 = andersen_collides(c, b0.m & kTagMask, step0 + k);
            coll1 = andersen_collides(c, b1.m & kTagMask, step0 + k);
            if (coll0) gauss3(c, b0.m & kTagMask, step0 + k, g0x, g0y, g0z);
            if (coll1) gauss3(c, b1.m & kTagMask, step0 + k, g1x, g1y, g1z);
        }
        // window fraction of this sub-step (the learned field's interpolation)
        const float a = kLerp ? (float)(lerp_j0 + k) * lerp_inv_k : 0.f;
        kick_bead<kTherm, kForce, kLerp>(b0, f00, f01, f02, g0x, g0y, g0z, w0x, w0y, w0z, c, g,
                                         wcache, tid, coll0, a);
        kick_bead<kTherm, kForce, kLerp>(b1, f10, f11, f12, g1x, g1y, g1z, w1x, w1y, w1z, c, g,
                                         wcache, kWarpBlock + tid, coll1, a);
        b0.x = fmaf(c.dt, b0.vx, b0.x);
        b0.y = fmaf(c.dt, b0.vy, b0.y);
        b0.z = fmaf(c.dt, b0.vz, b0.z);
        b1.x = fmaf(c.dt, b1.vx, b1.x);
        b1.y = fmaf(c.dt, b1.vy, b1.y);
        b1.z = fmaf(c.dt, b1.vz, b1.z);
    }
    if (a0) finish_bead(b0, (long long)base + j0, out, g, flag);
    if (a1) finish_bead(b1, (long long)base + j1, out, g, flag);
    if (D_next) {
        scatter_paired(D_next, g, b0.x, b0.y, b0.z, b0.m, a0);
        scatter_paired(D_next, g, b1.x, b1.y, b1.z, b1.m, a1);
    }
}

// This warp's number in its block, from a shuffle: the compiler then knows it
// for the same in all lanes and keeps the segment's bounds and the replica's
// record in uniform registers.  At 128 registers a context's kernel then spills 16
// bytes (44 before), with the observables 4 (144), a batch's none: a 10-step launch of
// 1M beads took 109 -> 107.5 us, a 5-step launch of 8.1M 548 -> 536, 64 replicas' (4M
// beads, 10 steps) 462 -> 446.
__device__ __forceinline__ int uniform_warp() {
    return __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0);
}

// The segment a warp takes in the round that starts at segment r.  A block's
// warps take neighbouring segments (which share cells in L1), but those of a
// partial round are dealt out over all blocks, the later half's (the second
// CTA of an SM) on other schedulers, so that every SM gets its share.  A
// second or later round of less than two segments a block stays with neighbouring warps: it
// is over sooner that way (160k beads 75.2 / 77.5 us dealt out, 320k 105.6 /
// 110; two launches of 10 steps with their fields).  Together / dealt out:
// 5k beads 42.6 / 39.2, 40k 49.8 / 46.2, 120k 61.2 / 58.7, 240k 90.8 / 86.5,
// 1M 254.8 / 252.9; 200k with dihedrals, four launches, 214 / 189; two learned
// windows of 20 steps at 5k beads 216 / 197, 60k 277 / 244, 240k 415 / 407, 1M 1019 / 1017.
__device__ __forceinline__ int segment_of(int r, int total, int warp) {
    constexpr int kWarps = kWarpBlock / 32;
    const int rem = total - r, grid = (int)gridDim.x, block = (int)blockIdx.x;
    if (rem >= grid * kWarps || (r > 0 && rem < 2 * grid)) return r + block * kWarps + warp;
    const int slot = (warp + (2 * block >= grid ? kWarps - 2 : 0)) % kWarps;
    return r + slot * grid + block;
}

// All replicas of a batch in one persistent launch (a single context is a
// batch of one): the warps walk the concatenated segment lists; each
// segment's replica (warp-uniform) selects its record in the kernel parameter
// block.
template <int kTherm, int kCap, int kForce, int kBonded>
__global__ void __launch_bounds__(kWarpBlock, 2) k_step_warp_batch(
    const __grid_constant__ BatchStepParamsT<kCap> p) {
    griddep_wait();
    griddep_launch_dependents();
    extern __shared__ float4 wcache[];
    __shared__ int s_off[kCap + 1];
    const int tid = threadIdx.x;
    if (tid == 0) {
        int acc = 0;
        for (int r = 0; r < p.R; ++r) {
            s_off[r] = acc;
            acc += *p.rep[r].n_seg;
        }
        s_off[p.R] = acc;
    }
    __syncthreads();
    const int total = s_off[p.R];
    const int warps_total = gridDim.x * (kWarpBlock / 32);
    const long long step0 = p.step_dev ? *p.step_dev : p.step0;
    for (int r = 0, w; (w = segment_of(r, total, uniform_warp())) < total; r += warps_total) {
        int lo = 0;  // replica r with s_off[r] <= w < s_off[r + 1]
        if (kCap > 1) {
            int hi = p.R - 1;
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if (s_off[mid] <= w) lo = mid;
                else hi = mid - 1;
            }
            lo = __shfl_sync(0xffffffffu, lo, 0);
        }
        const BatchStepRep& rp = p.rep[kCap > 1 ? lo : 0];
        const int s = w - s_off[lo];
        unsigned long long* D = p.fuse ? rp.D[p.dnext] : nullptr;
        if constexpr (pair_form(kForce, kBonded))
            advance_pairs<kTherm>(rp.st[p.cur], rp.st[p.cur ^ 1], rp.meta, rp.seg_start[s],
                                           rp.seg_count[s], p.n_sub, step0, rp.g, rp.G, rp.c, D,
                                           p.flag);
        else
            advance_segment<kTherm, kForce, kBonded>(rp.st[p.cur], rp.st[p.cur ^ 1], rp.meta,
                                                     rp.seg_start[s], rp.seg_count[s], p.n_sub,
                                                     step0, rp.g, rp.G, rp.c, D, p.flag, wcache,
                                                     tid);
    }
}

// A single context's launch that also forms the observables' bead terms of
// its final state (bonds only, interpolated-gradient force, Langevin or no
// thermostat): each thread's float-float sums over its segments, then the
// block's, one partial per CTA for k_energy_final.
template <int kTherm>
__global__ void __launch_bounds__(kWarpBlock, 2) k_step_warp_obs(
    const __grid_constant__ SingleStepParams p, const ObsArgs o) {
    griddep_wait();
    griddep_launch_dependents();
    __shared__ FF sh[kBeadVals][kWarpBlock / 32];
    const int tid = threadIdx.x;
    const BatchStepRep& rp = p.rep[0];
    const int total = *rp.n_seg;
    const int warps_total = gridDim.x * (kWarpBlock / 32);
    const long long step0 = p.step0;
    FF acc[kBeadVals];
#pragma unroll
    for (int k = 0; k < kBeadVals; ++k) acc[k] = FF{0.f, 0.f};
    for (int r = 0, w; (w = segment_of(r, total, uniform_warp())) < total; r += warps_total)
        advance_pairs<kTherm, 1>(rp.st[p.cur], rp.st[p.cur ^ 1], rp.meta, rp.seg_start[w],
                                    rp.seg_count[w], p.n_sub, step0, rp.g, rp.G, rp.c,
                                    p.fuse ? rp.D[p.dnext] : nullptr, p.flag, &o, acc);
    const int wi = tid >> 5;
#pragma unroll
    for (int k = 0; k < kBeadVals; ++k) {
        acc[k] = warp_sum_ff(acc[k]);
        if ((tid & 31) == 0) sh[k][wi] = acc[k];
    }
    __syncthreads();
    if (tid < kBeadVals) {
        FF r = sh[tid][0];
#pragma unroll
        for (int j = 1; j < kWarpBlock / 32; ++j) r = ff_plus(r, sh[tid][j]);
        o.part[(size_t)blockIdx.x * kBeadVals + tid] = make_float2(r.h, r.l);
    }
}

// A learned window in one launch (a single context, interpolated-gradient
// force): the field at window step j is (1 - j/K) G0 + (j/K) G2, G0 the field
// of the true density at the window start and G2 that of the predicted
// density at its end -- the field of D(t) + (j/K) dphi, since the field is
// linear in the density.  Each bead caches both cells' polynomials (twelve
// planes); the launch's first sub-step is window step j0.
constexpr size_t kWarpSmemLerp = 2 * sizeof(float4) * kCachePlanes * 2 * kWarpBlock;

template <int kTherm, int kBonded>
__global__ void __launch_bounds__(kWarpBlock, 2) k_step_warp_lerp(
    const __grid_constant__ SingleStepParams p, const float4* __restrict__ G2, int j0,
    float inv_k) {
    griddep_wait();
    griddep_launch_dependents();
    extern __shared__ float4 wcache[];
    const int tid = threadIdx.x;
    const BatchStepRep& rp = p.rep[0];
    const int total = *rp.n_seg;
    const int warps_total = gridDim.x * (kWarpBlock / 32);
    for (int r = 0, w; (w = segment_of(r, total, tid >> 5)) < total; r += warps_total)
        advance_segment<kTherm, 0, kBonded, 1>(rp.st[p.cur], rp.st[p.cur ^ 1], rp.meta,
                                               rp.seg_start[w], rp.seg_count[w], p.n_sub,
                                               p.step0, rp.g, rp.G, rp.c,
                                               p.fuse ? rp.D[p.dnext] : nullptr, p.flag, wcache,
                                               tid, G2, j0, inv_k);
}

template <int kTherm, int kBonded>
static void launch_lerp_k(const SingleStepParams& p, const float4* G2, int j0, float inv_k,
                          int blocks, cudaStream_t s) {
    static std::once_flag once[64];
    once_per_device(once, [] {
        cudaFuncSetAttribute(k_step_warp_lerp<kTherm, kBonded>,
                             cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kWarpSmemLerp);
    });
    launch_pdl(k_step_warp_lerp<kTherm, kBonded>, blocks, kWarpBlock, kWarpSmemLerp, s, p, G2, j0,
               inv_k);
}

template <int kCap, int kTherm, int kForce>
static void warp_attrs_f() {
    cudaFuncSetAttribute(k_step_warp_batch<kTherm, kCap, kForce, 0>,
                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kWarpSmem);
    cudaFuncSetAttribute(k_step_warp_batch<kTherm, kCap, kForce, 1>,
                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kWarpSmem);
    cudaFuncSetAttribute(k_step_warp_batch<kTherm, kCap, kForce, 2>,
                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kWarpSmem);
}

template <int kCap, int kTherm>
static void warp_attrs_n() {
    warp_attrs_f<kCap, kTherm, 0>();
    warp_attrs_f<kCap, kTherm, 1>();
    warp_attrs_f<kCap, kTherm, 2>();
}

template <int kCap>
static void warp_attrs() {
    warp_attrs_n<kCap, 0>();
    warp_attrs_n<kCap, 1>();
    warp_attrs_n<kCap, 2>();
}

// The persistent grid of the current device (its SM count times the
// resident CTAs per SM), with the kernels' attributes set on first use.
static int warp_grid_cap() {
    static std::once_flag once[64];
    static int cap[64];
    int dev = 0;
    cudaGetDevice(&dev);
    once_per_device(once, [dev] {
        warp_attrs<HPF_MAX_REPLICAS>();
        warp_attrs<1>();
        int sms = 0, per_sm = 0;
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(
            &per_sm, k_step_warp_batch<1, HPF_MAX_REPLICAS, 1, 0>, kWarpBlock, kWarpSmem);
        cudaGetLastError();
        cap[dev & 63] = (sms > 0 ? sms : 1) * (per_sm > 0 ? per_sm : 1);
    });
    return cap[dev & 63];
}

// A context's launches use dependent launch; a batch's are captured into
// graphs and launched plainly.
template <int kCap>
static void launch_warp_k(void (*k)(const BatchStepParamsT<kCap>), const BatchStepParamsT<kCap>& p,
                          int blocks, size_t smem, cudaStream_t s) {
    if (kCap == 1) launch_pdl(k, blocks, kWarpBlock, smem, s, p);
    else k<<<blocks, kWarpBlock, smem, s>>>(p);
}

template <int kCap, int kTherm, int kForce>
static void launch_warp_f(const BatchStepParamsT<kCap>& p, int blocks, int bonded,
                          cudaStream_t s) {
#define HPF_WARP(B) \
    launch_warp_k(k_step_warp_batch<kTherm, kCap, kForce, B>, p, blocks, warp_smem(kForce, B), s)
    if (bonded == 2) HPF_WARP(2);
    else if (bonded == 1) HPF_WARP(1);
    else HPF_WARP(0);
#undef HPF_WARP
}

template <int kCap, int kTherm>
static void launch_warp_n(const BatchStepParamsT<kCap>& p, int blocks, int force, int bonded,
                          cudaStream_t s) {
    if (force == 2) launch_warp_f<kCap, kTherm, 2>(p, blocks, bonded, s);
    else if (force == 1) launch_warp_f<kCap, kTherm, 1>(p, blocks, bonded, s);
    else launch_warp_f<kCap, kTherm, 0>(p, blocks, bonded, s);
}

template <int kCap>
static void launch_warp(const BatchStepParamsT<kCap>& p, int blocks, int therm, int force,
                        cudaStream_t s) {
    const int bonded = bonded_level(p.rep[0].c);  // all replicas alike (checked at init)
    if (therm == 1) launch_warp_n<kCap, 1>(p, blocks, force, bonded, s);
    else if (therm == 2) launch_warp_n<kCap, 2>(p, blocks, force, bonded, s);
    else launch_warp_n<kCap, 0>(p, blocks, force, bonded, s);
}

void launch_step_warp_batch(const BatchStepParams& p, int max_seg_total, int therm,
                            cudaStream_t s) {
    if (max_seg_total <= 0 || p.n_sub <= 0) return;
    const int cap = warp_grid_cap();
    const int blocks = max_seg_total < cap ? max_seg_total : cap;
    launch_warp(p, blocks, therm, p.rep[0].c.force_mode, s);  // replicas share the force mode
}

void launch_step_warp_lerp(const SingleStepParams& p, const float4* G2, int j0, float inv_k,
                           int max_seg, int therm, cudaStream_t s) {
    if (max_seg <= 0 || p.n_sub <= 0) return;
    const int cap = warp_grid_cap();
    const int blocks = max_seg < cap ? max_seg : cap;
    const int bonded = bonded_level(p.rep[0].c);
    if (therm == 1) {
        if (bonded == 2) launch_lerp_k<1, 2>(p, G2, j0, inv_k, blocks, s);
        else if (bonded == 1) launch_lerp_k<1, 1>(p, G2, j0, inv_k, blocks, s);
        else launch_lerp_k<1, 0>(p, G2, j0, inv_k, blocks, s);
    } else if (therm == 2) {
        if (bonded == 2) launch_lerp_k<2, 2>(p, G2, j0, inv_k, blocks, s);
        else if (bonded == 1) launch_lerp_k<2, 1>(p, G2, j0, inv_k, blocks, s);
        else launch_lerp_k<2, 0>(p, G2, j0, inv_k, blocks, s);
    } else {
        if (bonded == 2) launch_lerp_k<0, 2>(p, G2, j0, inv_k, blocks, s);
        else if (bonded == 1) launch_lerp_k<0, 1>(p, G2, j0, inv_k, blocks, s);
        else launch_lerp_k<0, 0>(p, G2, j0, inv_k, blocks, s);
    }
}

int step_warp_grid_cap() { return warp_grid_cap(); }

int launch_step_warp_obs(const SingleStepParams& p, int max_seg, int therm, float2* part,
                         float half_dt_m, const BondFF& bond, cudaStream_t s) {
    if (max_seg <= 0 || p.n_sub <= 0) return 0;
    const int cap = warp_grid_cap();
    const int blocks = max_seg < cap ? max_seg : cap;
    const ObsArgs o{part, half_dt_m, bond};
    if (therm == 1) launch_pdl(k_step_warp_obs<1>, blocks, kWarpBlock, 0, s, p, o);
    else launch_pdl(k_step_warp_obs<0>, blocks, kWarpBlock, 0, s, p, o);
    return blocks;
}

void launch_step_warp_single(const SingleStepParams& p, int max_seg, int therm,
                             cudaStream_t s) {
    if (max_seg <= 0 || p.n_sub <= 0) return;
    const int cap = warp_grid_cap();
    const int blocks = max_seg < cap ? max_seg : cap;
    launch_warp(p, blocks, therm, p.rep[0].c.force_mode, s);
}


}  // namespace hpf
