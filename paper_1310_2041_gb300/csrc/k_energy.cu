// k_energy.cu -- the FP64 observables (kinetic, bonded and field energy,
// momentum, temperature) of the current step, reduced in a fixed order.
#include "hpf_internal.cuh"

namespace hpf {

// ------------------------------------------------------------------ A7 FP64 observables

constexpr int kRedBlock = 256;    // the bead and node kernels
constexpr int kFinalBlock = 1024;  // the one block that combines their partials (more than three species)
// Grid-stride shares (on average) of a bead or node thread: small, so that a
// million beads make about 2000 blocks, which the SMs take in several waves
// with little left over for the last one (at 8 beads a thread the 489 blocks
// of a million beads came to just over one wave of three blocks per SM); more
// beads give longer shares, so that the last block's sum over the blocks stays short.
constexpr int kPerThread = 2;
constexpr int kMaxBlocks = 2048;

// Exact unsigned 128-bit sums (the field energy's node sums).
struct U128 {
    unsigned long long lo, hi;
};
__device__ __forceinline__ void u128_add(U128& a, const U128& b) {
    const unsigned long long lo = a.lo + b.lo;
    a.hi += b.hi + (lo < a.lo ? 1ull : 0ull);
    a.lo = lo;
}
__device__ __forceinline__ U128 u128_mul(unsigned long long a, unsigned long long b) {
    return U128{a * b, __umul64hi(a, b)};
}
__device__ __forceinline__ double u128_to_double(const U128& v) {
    return (double)v.hi * 18446744073709551616.0 + (double)v.lo;
}
__device__ __forceinline__ U128 warp_sum_u128(U128 v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        u128_add(v, U128{__shfl_down_sync(0xffffffffu, v.lo, o),
                         __shfl_down_sync(0xffffffffu, v.hi, o)});
    return v;  // lane 0
}

// |d| in FP64 from an FP32 reciprocal-square-root seed and one Newton step
// y <- y (3 - r2 y^2) / 2 (relative error ~1.5 e0^2 ~ 3e-14 for the FP32
// seed's e0 ~ 1.4e-7); r2 = 0 gives 0.
__device__ __forceinline__ double norm_fp64(double r2) {
    if (!(r2 > 0.0)) return 0.0;
    double y = (double)rsqrtf((float)r2);
    y = y * fma(-0.5 * r2, y * y, 1.5);
    return r2 * y;
}

// Bond vector x[j] - x[i], exactly.
__device__ __forceinline__ FF3 bond_ff3(const StateBuf& st, int i, int j) {
    return FF3{ff_diff(st.x[j], st.x[i]), ff_diff(st.y[j], st.y[i]), ff_diff(st.z[j], st.z[i])};
}
__device__ __forceinline__ FF ff_of(const float (&v)[2]) { return FF{v[0], v[1]}; }

// Angle energy k (cos theta - cos0)^2 at the middle bead i of i - 1, i, i + 1.
__device__ __forceinline__ FF angle_energy_ff(const StateBuf& st, int i, const EnergyConsts& e) {
    const FF3 u = bond_ff3(st, i, i - 1), w = bond_ff3(st, i, i + 1);
    const FF c = ff_mul(ff_dot(u, w), ff_mul(ff_rsqrt(ff_dot(u, u)), ff_rsqrt(ff_dot(w, w))));
    const FF d = ff_plus(c, ff_neg(ff_of(e.ff_cos0)));
    return ff_mul(ff_of(e.ff_angle_k), ff_mul(d, d));
}

// Dihedral energy k [1 + cos(n phi - delta)] of the quadruplet i .. i + 3: cos
// phi = A.B / (|A||B|), sin phi = |b2| b1.B / (|A||B|) with A = b1 x b2, B =
// b2 x b3, and cos(n phi), sin(n phi) by the n-th power of cos phi + i sin phi.
// In FP64: the quadruplets that the float-float form leaves.
__device__ __noinline__ double dihedral_energy_fp64(const StateBuf& st, int i,
                                                    const EnergyConsts& e) {
    double b[3][3];  // bond vectors
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        b[k][0] = (double)st.x[i + k + 1] - st.x[i + k];
        b[k][1] = (double)st.y[i + k + 1] - st.y[i + k];
        b[k][2] = (double)st.z[i + k + 1] - st.z[i + k];
    }
    double A[3], B[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const int u = (a + 1) % 3, v = (a + 2) % 3;
        A[a] = b[0][u] * b[1][v] - b[0][v] * b[1][u];
        B[a] = b[1][u] * b[2][v] - b[1][v] * b[2][u];
    }
    const double AA = A[0] * A[0] + A[1] * A[1] + A[2] * A[2];
    const double BB = B[0] * B[0] + B[1] * B[1] + B[2] * B[2];
    const double L = norm_fp64(b[1][0] * b[1][0] + b[1][1] * b[1][1] + b[1][2] * b[1][2]);
    const double den = norm_fp64(AA) * norm_fp64(BB);
    const double cp = (A[0] * B[0] + A[1] * B[1] + A[2] * B[2]) / den;
    const double sp = L * (b[0][0] * B[0] + b[0][1] * B[1] + b[0][2] * B[2]) / den;
    double cn = cp, sn = sp;
    for (int k = 1; k < e.dih_n; ++k) {
        const double t = cn * cp - sn * sp;
        sn = sn * cp + cn * sp;
        cn = t;
    }
    return e.dih_k * (1.0 + cn * e.dih_cd + sn * e.dih_sd);
}

// a + s b with s near the value that leaves only a's part across b, rounded to 13
// bits so that s b is exact wherever b's components are FP32 numbers; ibb = 1 / b.b.
// cc: the length squared of the result.
__device__ __forceinline__ FF3 across(const FF3& a, const FF3& b, float ibb, float& cc) {
    const float d = fmaf(a.z.h, b.z.h, fmaf(a.y.h, b.y.h, __fmul_rn(a.x.h, b.x.h)));
    const float s = __uint_as_float((__float_as_uint(__fmul_rn(-d, ibb)) + 0x400u) & 0xfffff800u);
    auto add = [s](FF u, FF v) {
        const float p = __fmul_rn(s, v.h);
        return ff_plus(u, FF{p, fmaf(s, v.l, fmaf(s, v.h, -p))});
    };
    const FF3 c{add(a.x, b.x), add(a.y, b.y), add(a.z, b.z)};
    cc = fmaf(c.z.h, c.z.h, fmaf(c.y.h, c.y.h, __fmul_rn(c.x.h, c.x.h)));
    return c;
}

// The same in float-float; false where it would be less accurate than the FP64
// form.  In a nearly straight triplet the two halves of a cross product cancel,
// and with them goes what 48 bits have less than 53.  Adding a multiple of b2 to b1
// (and to b3) changes neither A, B nor b1.B, and without its part along b2
// nothing cancels.  FP64 takes over where even so |A| is below a fifth of the
// factors' product (within about 0.02 degrees of straight, exactly straight ones,
// whose angle is undefined, among them) or |A|^2 leaves the range in which FP32
// holds a product's low half (bonds below 3e-5 or beyond 3e7).  A lane there costs
// a launch 10 us, so the line must lie where thermal chains hardly come: with
// b1 +- b2 in place of the projection 1 in 4000 quadruplets crossed it.  Largest
// error per k against 80-bit arithmetic over 200,000 quadruplets each, n = 3, FP64
// form / this one: angles of 100 to 140 degrees 2.8e-13 / 1.0e-13, all angles alike
// 2.8e-13 / 1.0e-13, 177 to 179 degrees 2.5e-13 / 1.0e-13, 179 to 180 degrees
// 1.2e-11 / 8.6e-12 (b1 and b3 as they are: 1.0e-13, 1.3e-12, 2.4e-12, 1.7e-7).
__device__ __forceinline__ bool dihedral_energy_ff(const StateBuf& st, int i, const EnergyConsts& e,
                                                   FF& energy) {
    constexpr float kTau2 = 1.0f / 25.0f;
    constexpr float kLow = 8.673617379884035e-19f, kHigh = 1.2676506002282294e30f;  // 2^-60, 2^100
    const FF3 b2 = bond_ff3(st, i + 1, i + 2);
    const FF b22 = ff_dot(b2, b2);
    const float ibb = __fdividef(1.0f, b22.h);
    float c1, c3;
    const FF3 b1 = across(bond_ff3(st, i, i + 1), b2, ibb, c1);
    const FF3 b3 = across(bond_ff3(st, i + 2, i + 3), b2, ibb, c3);
    const FF3 A = ff_cross(b1, b2), B = ff_cross(b2, b3);
    const FF AA = ff_dot(A, A), BB = ff_dot(B, B);
    if (!(AA.h >= kTau2 * c1 * b22.h && BB.h >= kTau2 * c3 * b22.h && fminf(AA.h, BB.h) >= kLow &&
          fmaxf(AA.h, BB.h) <= kHigh))
        return false;
    const FF inv = ff_mul(ff_rsqrt(AA), ff_rsqrt(BB));
    const FF cp = ff_mul(ff_dot(A, B), inv);
    const FF sp = ff_mul(ff_mul(ff_mul(b22, ff_rsqrt(b22)), ff_dot(b1, B)), inv);
    FF cn = cp, sn = sp;
    for (int k = 1; k < e.dih_n; ++k) {
        const FF t = ff_plus(ff_mul(cn, cp), ff_neg(ff_mul(sn, sp)));
        sn = ff_plus(ff_mul(sn, cp), ff_mul(cn, sp));
        cn = t;
    }
    const FF v = ff_plus(ff_plus(FF{1.0f, 0.f}, ff_mul(cn, ff_of(e.ff_dih_cd))),
                         ff_mul(sn, ff_of(e.ff_dih_sd)));
    energy = ff_mul(ff_of(e.ff_dih_k), v);
    return true;
}

// Per bead: F_n with the terms the step kernel's kick uses (bonds, the field
// by a direct trilinear gather, friction, step n's noise), the on-step velocity
// v_n = v + dt/(2m) F_n, then kinetic energy, momentum and the bond energy of
// the bond to the next bead (each bond once).  The bond, cosine-angle and
// dihedral energies are formed in float-float (about 2^-46 per operation, like
// the FP64 forms they replace, whose lengths carried one Newton step from an
// FP32 seed: 3e-14), the harmonic angle's in FP64 for its arc tangent, all
// from the FP32 positions with exact differences (the FP64 pipe bound the
// angle and dihedral terms: 98 us for 200k beads with both); v_n and |v_n|^2 are FP32
// (the FP32 force already limits them to ~1e-7) and are summed in float-float
// over the thread's beads, its warp and its block, into one float-float
// partial per observable and block (kinetic energy without the factor m/2 and
// momentum without m, both applied in FP64 in energy_combine).
// Block blk of nb bead blocks (grid-stride over the beads within them).
// kBonded: bonded_level(c).
template <int kBonded>
__device__ __forceinline__ void energy_beads_block(const StateBuf& st,
                                                   const uint32_t* __restrict__ meta, int n,
                                                   const MeshGeom& g,
                                                   const float4* __restrict__ G,
                                                   const StepConsts& c, long long step,
                                                   const EnergyConsts& e,
                                                   float2* __restrict__ partials, int blk, int nb,
                                                   FF (*sh)[kRedBlock / 32]) {
    double ub = 0.0;           // harmonic angles and the dihedrals left to FP64
    float uh = 0.f, ul = 0.f;  // the other bonded energies, float-float
    FF kf{0.f, 0.f}, pfx{0.f, 0.f}, pfy{0.f, 0.f}, pfz{0.f, 0.f};
    for (int i = blk * kRedBlock + threadIdx.x; i < n; i += nb * kRedBlock) {
        const float x = st.x[i], y = st.y[i], z = st.z[i];
        const float vx = st.vx[i], vy = st.vy[i], vz = st.vz[i];
        const uint32_t m = meta[i];
        float fx = 0.f, fy = 0.f, fz = 0.f;
        if (m & kBondPrev)
            bond_force(x - st.x[i - 1], y - st.y[i - 1], z - st.z[i - 1], c.two_k, c.r0, fx, fy, fz);
        if (m & kBondNext) {
            const float xj = st.x[i + 1], yj = st.y[i + 1], zj = st.z[i + 1];
            bond_force(x - xj, y - yj, z - zj, c.two_k, c.r0, fx, fy, fz);
            bond_energy_ff(x, y, z, xj, yj, zj, bond_ff(e), uh, ul);
        }
        if (kBonded >= 1 && c.two_ka != 0.f) {
            angle_forces_of(st, meta, i, m, c, fx, fy, fz);
            if ((m & kBondPrev) && (m & kBondNext)) {  // the angle centred here, once
                if (e.angle_form == 1) {
                    // harmonic: theta = atan2(|u x w|, u.w)
                    const double ux = (double)st.x[i - 1] - x, uy = (double)st.y[i - 1] - y,
                                 uz = (double)st.z[i - 1] - z;
                    const double wx = (double)st.x[i + 1] - x, wy = (double)st.y[i + 1] - y,
                                 wz = (double)st.z[i + 1] - z;
                    const double qx = uy * wz - uz * wy, qy = uz * wx - ux * wz,
                                 qz = ux * wy - uy * wx;
                    const double d = atan2(norm_fp64(qx * qx + qy * qy + qz * qz),
                                           ux * wx + uy * wy + uz * wz) -
                                     e.theta0;
                    ub += e.angle_k * d * d;
                } else {
                    const FF u = ff_plus(FF{uh, ul}, angle_energy_ff(st, i, e));
                    uh = u.h;
                    ul = u.l;
                }
            }
        }
        if (kBonded == 2) {
            int back, fwd;
            chain_reach(meta, i, m, back, fwd);
            dihedral_forces_of(
                [&](int d) { return make_float3(st.x[i + d], st.y[i + d], st.z[i + d]); }, back,
                fwd, c, fx, fy, fz);
            if (fwd == 3) {  // the one starting here, once
                FF u;
                if (dihedral_energy_ff(st, i, e, u)) {
                    u = ff_plus(FF{uh, ul}, u);
                    uh = u.h;
                    ul = u.l;
                } else {
                    ub += dihedral_energy_fp64(st, i, e);
                }
            }
        }
        const float4* Gt = G + (size_t)((m >> kTypeShift) & kTypeMask) * g.gnodes;
        gather_field_mode(Gt, g, c.force_mode, x, y, z, fx, fy, fz);
        if (c.sigma > 0.f) {
            float nx, ny, nz;
            gauss3(c, m & kTagMask, step, nx, ny, nz);
            fx += c.sigma * nx;
            fy += c.sigma * ny;
            fz += c.sigma * nz;
        }
        fx -= c.fric * vx;
        fy -= c.fric * vy;
        fz -= c.fric * vz;
        const float hf = (float)e.half_dt_m;
        float ux = fmaf(hf, fx, vx), uy = fmaf(hf, fy, vy), uz = fmaf(hf, fz, vz);
        if (c.p_coll > 0.f && andersen_collides(c, m & kTagMask, step)) {
            // Andersen: this step's collision redraws the on-step velocity
            float nx, ny, nz;
            gauss3(c, m & kTagMask, step, nx, ny, nz);
            ux = c.sig_v * nx;
            uy = c.sig_v * ny;
            uz = c.sig_v * nz;
        }
        kf = ff_plus(kf, fmaf(ux, ux, fmaf(uy, uy, __fmul_rn(uz, uz))));
        pfx = ff_plus(pfx, ux);
        pfy = ff_plus(pfy, uy);
        pfz = ff_plus(pfz, uz);
    }
    FF v[kBeadVals] = {kf, ff_norm(uh, ul), pfx, pfy, pfz};
    if (kBonded >= 1) v[1] = ff_plus(v[1], ff_from_double(ub));
    const int w = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < kBeadVals; ++k) {
        v[k] = warp_sum_ff(v[k]);
        if ((threadIdx.x & 31) == 0) sh[k][w] = v[k];
    }
    __syncthreads();
    if (threadIdx.x < kBeadVals) {
        FF r = sh[threadIdx.x][0];
#pragma unroll
        for (int j = 1; j < kRedBlock / 32; ++j) r = ff_plus(r, sh[threadIdx.x][j]);
        partials[(size_t)blk * kBeadVals + threadIdx.x] = make_float2(r.h, r.l);
    }
}

// Per node: the exact integer sums behind the field energy, instantiated per
// species count (the kS (kS + 1) / 2 + 2 sums are register arrays).
// The field energy from exact integer sums.  With phi_K = phi_c D_K (D the
// int64 fixed-point density, non-negative) and T = sum_K D_K per node,
//   W / (rho0 h^3) = 1/2 kT phi_c^2 sum_KK' chi_KK' S_KK'
//                  + 1/2 inv_kappa (phi_c^2 sum T^2 - 2 phi_c sum T + nodes),
// S_KK' = sum over nodes of D_K D_K'.  Every product is below 2^126 and so is
// every sum (at most (sum D_K)(sum D_K') < 2^126), so the node sums are exact
// unsigned 128-bit integers, independent of order; FP64 enters only in the
// final combination.  Per block: the kS (kS + 1) / 2 pair sums (K <= K'),
// sum T^2 and sum T, each as (lo, hi).
template <int kS>
__device__ __forceinline__ void energy_nodes_block(const long long* __restrict__ D, int nodes,
                                                   unsigned long long* __restrict__ part, int blk,
                                                   int nn, U128 (*sh)[kRedBlock / 32]) {
    constexpr int kP = kS * (kS + 1) / 2;
    constexpr int kQ = kP + 2;
    U128 acc[kQ];
#pragma unroll
    for (int q = 0; q < kQ; ++q) acc[q] = U128{0ull, 0ull};
    for (int node = blk * kRedBlock + threadIdx.x; node < nodes; node += nn * kRedBlock) {
        unsigned long long d[kS];
        unsigned long long T = 0ull;
#pragma unroll
        for (int k = 0; k < kS; ++k) {
            d[k] = (unsigned long long)D[(size_t)k * nodes + node];
            T += d[k];
        }
        int q = 0;
#pragma unroll
        for (int k = 0; k < kS; ++k)
#pragma unroll
            for (int kp = k; kp < kS; ++kp) u128_add(acc[q++], u128_mul(d[k], d[kp]));
        u128_add(acc[kP], u128_mul(T, T));
        u128_add(acc[kP + 1], U128{T, 0ull});
    }
    const int w = threadIdx.x >> 5;
#pragma unroll
    for (int q = 0; q < kQ; ++q) {
        acc[q] = warp_sum_u128(acc[q]);
        if ((threadIdx.x & 31) == 0) sh[q][w] = acc[q];
    }
    __syncthreads();
    if (threadIdx.x < kQ) {
        U128 r = sh[threadIdx.x][0];
#pragma unroll
        for (int j = 1; j < kRedBlock / 32; ++j) u128_add(r, sh[threadIdx.x][j]);
        part[((size_t)blk * kQ + threadIdx.x) * 2] = r.lo;
        part[((size_t)blk * kQ + threadIdx.x) * 2 + 1] = r.hi;
    }
}

// The node sums alone (many species: their accumulators would not fit the
// register budget of the combined kernel below).
template <int kS>
__global__ void __launch_bounds__(kRedBlock) k_energy_nodes(const long long* __restrict__ D,
                                                            int nodes,
                                                            unsigned long long* __restrict__ part) {
    __shared__ U128 sh[kS * (kS + 1) / 2 + 2][kRedBlock / 32];
    energy_nodes_block<kS>(D, nodes, part, blockIdx.x, gridDim.x, sh);
    griddep_launch_dependents();
}

// One block of kB threads: the bead partials (float-float) and the node
// partials (exact 128-bit) summed over the blocks in a fixed order -- each
// thread a strided share of the blocks, its loads all in flight together, then
// its warp, then each value by one warp over the warps' sums -- and combined in
// FP64, the three independent parts by three warps, then written to the host.
template <int kS, int kB>
struct CombineSmem {
    static constexpr int kQ = kS * (kS + 1) / 2 + 2;
    FF f[kBeadVals][kB / 32];
    U128 u[kQ][kB / 32];
    double res[kBeadVals + kQ];
};

template <int kS, int kB>
__device__ __forceinline__ void energy_combine(const float2* bead_part, int nb,
                                               const unsigned long long* node_part, int nn,
                                               int nodes, const EnergyConsts& e,
                                               const EnergyOut& out, CombineSmem<kS, kB>& sh) {
    constexpr int kP = kS * (kS + 1) / 2;
    constexpr int kQ = kP + 2;
    constexpr int kW = kB / 32;
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    FF acc[kBeadVals];
#pragma unroll
    for (int k = 0; k < kBeadVals; ++k) acc[k] = FF{0.f, 0.f};
    for (int b = t; b < nb; b += kB) {
        float2 p[kBeadVals];
#pragma unroll
        for (int k = 0; k < kBeadVals; ++k) p[k] = __ldcg(&bead_part[(size_t)b * kBeadVals + k]);
#pragma unroll
        for (int k = 0; k < kBeadVals; ++k) acc[k] = ff_plus(acc[k], FF{p[k].x, p[k].y});
    }
    U128 qa[kQ];
#pragma unroll
    for (int q = 0; q < kQ; ++q) qa[q] = U128{0ull, 0ull};
    for (int b = t; b < nn; b += kB) {
        U128 p[kQ];
#pragma unroll
        for (int q = 0; q < kQ; ++q) {
            const ulonglong2 v =
                __ldcg(reinterpret_cast<const ulonglong2*>(node_part) + (size_t)b * kQ + q);
            p[q] = U128{v.x, v.y};
        }
#pragma unroll
        for (int q = 0; q < kQ; ++q) u128_add(qa[q], p[q]);
    }
#pragma unroll
    for (int k = 0; k < kBeadVals; ++k) {
        acc[k] = warp_sum_ff(acc[k]);
        if (lane == 0) sh.f[k][w] = acc[k];
    }
#pragma unroll
    for (int q = 0; q < kQ; ++q) {
        qa[q] = warp_sum_u128(qa[q]);
        if (lane == 0) sh.u[q][w] = qa[q];
    }
    __syncthreads();
    for (int v = w; v < kBeadVals + kQ; v += kW) {
        double r;
        if (v < kBeadVals)
            r = ff_to_double(warp_sum_ff(lane < kW ? sh.f[v][lane] : FF{0.f, 0.f}));
        else
            r = u128_to_double(warp_sum_u128(lane < kW ? sh.u[v - kBeadVals][lane] : U128{0ull, 0ull}));
        if (lane == 0) sh.res[v] = r;
    }
    __syncthreads();
    const double* res = sh.res;
    const double ke = 0.5 * e.mass * res[0], ub = res[1];
    if (t == 0) {
        double q_chi = 0.0;
        int q = 0;
        for (int k = 0; k < kS; ++k)
            for (int kp = k; kp < kS; ++kp, ++q)
                q_chi += (k == kp ? 1.0 : 2.0) * e.chi[k][kp] * res[kBeadVals + q];
        const double t2 = res[kBeadVals + kP], t1 = res[kBeadVals + kP + 1];
        const double pc = e.phi_c;
        const double w_f = e.w_scale * (0.5 * e.kT * pc * pc * q_chi +
                                        0.5 * e.inv_kappa * (pc * pc * t2 - 2.0 * pc * t1 +
                                                             (double)nodes));
        out.out6[0] = ke;
        out.out6[1] = ub;
        out.out6[2] = w_f;
        out.out6[3] = ke + ub + w_f;
    } else if (t == 32) {
        const double px = e.mass * res[2], py = e.mass * res[3], pz = e.mass * res[4];
        out.out6[4] = sqrt(px * px + py * py + pz * pz);
    } else if (t == 64) {
        out.out6[5] = e.n > 0 ? 2.0 * ke / (3.0 * (double)e.n) : 0.0;
        *out.h_flag = *out.flag;
        if (out.nh) {
            out.h_nh[0] = out.nh[0];
            out.h_nh[1] = out.nh[1];
        }
    }
}

// One launch for the bead and node sums and, with kN species (kN > 0), the
// observables: blocks 0 .. nb - 1 take the beads, the rest the nodes, so the
// two run side by side with the longer work first (200k beads with dihedrals: 29.2 ->
// 27.9 us against the nodes first), and the last of them to finish (ticket, left at zero)
// combines the partials of all.  A second launch of one block for that took
// 9 us more, half of it before its first load: 6.2 + 9.0 -> 12.1 us for 10k beads,
// 7.1 + 9.0 -> 13.0 for 70^3 nodes and given bead partials, 22.2 + 8.3 -> 29.2 for 200k
// beads with dihedrals, and the gap between the two.  nb bead blocks; nb_part partials of them (formed elsewhere when nb is
// 0).  kN 0: the beads alone.
template <int kN, int kBonded>
__global__ void __launch_bounds__(kRedBlock, kBonded == 0 ? 4 : 3) k_energy_main(
    StateBuf st, const uint32_t* __restrict__ meta, int n, MeshGeom g, const float4* __restrict__ G,
    StepConsts c, long long step, const __grid_constant__ EnergyConsts e, float2* bead_part, int nb,
    int nb_part, const long long* __restrict__ D, unsigned long long* node_part, int nn,
    unsigned* ticket, const __grid_constant__ EnergyOut out) {
    constexpr int kQ = kN * (kN + 1) / 2 + 2;
    constexpr int kS = kN > 0 ? kN : 1;  // without nodes the combination is not instantiated
    union Smem {
        U128 u[kQ][kRedBlock / 32];
        FF f[kBeadVals][kRedBlock / 32];
        CombineSmem<kS, kRedBlock> combine;
    };
    __shared__ __align__(16) unsigned char sm[sizeof(Smem)];
    __shared__ bool s_last;
    Smem& sh = *reinterpret_cast<Smem*>(sm);
    griddep_wait();
    griddep_launch_dependents();
    const int blk = (int)blockIdx.x;
    if (kN == 0 || blk < nb)
        energy_beads_block<kBonded>(st, meta, n, g, G, c, step, e, bead_part, blk, nb, sh.f);
    else
        energy_nodes_block<kS>(D, g.nodes, node_part, blk - nb, nn, sh.u);
    if constexpr (kN > 0) {
        if (threadIdx.x < 32) {  // the warp that wrote the block's partials
            __threadfence();
            __syncwarp();
            if (threadIdx.x == 0) s_last = atomicAdd(ticket, 1u) == gridDim.x - 1;
        }
        __syncthreads();
        if (!s_last) return;
        __threadfence();
        if (threadIdx.x == 0) *ticket = 0u;
        energy_combine<kS, kRedBlock>(bead_part, nb_part, node_part, nn, g.nodes, e, out, sh.combine);
    }
}

// The combination as a launch of its own (more than three species).
template <int kS>
__global__ void __launch_bounds__(kFinalBlock) k_energy_final(const float2* bead_part, int nb,
                                                              const unsigned long long* node_part,
                                                              int nn, int nodes,
                                                              const __grid_constant__ EnergyConsts e,
                                                              const __grid_constant__ EnergyOut out) {
    __shared__ CombineSmem<kS, kFinalBlock> sh;
    griddep_wait();  // launched programmatically after the partial sums
    energy_combine<kS, kFinalBlock>(bead_part, nb, node_part, nn, nodes, e, out, sh);
}

// Blocks of the energy reductions: each thread takes a grid-stride share,
// independent of the device so the summation order, and with it every FP64
// bit, is the same on any GPU.
static int energy_blocks(int count) {
    const int b = (count + kRedBlock * kPerThread - 1) / (kRedBlock * kPerThread);
    return b < kMaxBlocks ? b : kMaxBlocks;
}

int energy_launches(int n, int S) { return S <= 3 ? 1 : (n > 0 ? 3 : 2); }

// Doubles: the ticket (and padding), per node block S (S + 1) / 2 + 2 sums of
// two words, then the bead partials.
constexpr int kTicketWords = 2;

int energy_partials_needed(int n, int nodes, int S) {
    return kTicketWords + energy_blocks(nodes) * 2 * (S * (S + 1) / 2 + 2) +
           energy_blocks(n) * kBeadVals;
}

// The launches; nb_given >= 0: bead partials formed elsewhere.
static void launch_sums(StateBuf st, const uint32_t* meta, int n, MeshGeom g, const float4* G,
                        const StepConsts& c, long long step, const long long* D,
                        const EnergyConsts& e, const float2* given, int nb_given, double* partials,
                        const EnergyOut& out, cudaStream_t s) {
    const int nb = nb_given >= 0 ? 0 : energy_blocks(n);
    const int nn = energy_blocks(g.nodes);
    const int nb_part = nb_given >= 0 ? nb_given : nb;
    unsigned* ticket = reinterpret_cast<unsigned*>(partials);
    unsigned long long* node_part = reinterpret_cast<unsigned long long*>(partials + kTicketWords);
    // kBeadVals float-float pairs (one double's room each) per block
    float2* bead_part = nb_given >= 0
                            ? const_cast<float2*>(given)
                            : reinterpret_cast<float2*>(node_part + (size_t)nn * 2 *
                                                                        (e.S * (e.S + 1) / 2 + 2));
    // up to three species: one launch; more species: the beads, the node sums
    // and the combination in launches of their own
    const int bonded = bonded_level(c);
#define HPF_MAIN_B(k, B, blocks)                                                                 \
    launch_pdl(k_energy_main<k, B>, dim3(blocks), dim3(kRedBlock), 0, s, st, meta, n, g, G, c, step, \
               e, bead_part, nb, nb_part, D, node_part, nn, ticket, out)
#define HPF_MAIN(k, blocks)                         \
    if (bonded == 2) HPF_MAIN_B(k, 2, blocks);      \
    else if (bonded == 1) HPF_MAIN_B(k, 1, blocks); \
    else HPF_MAIN_B(k, 0, blocks);
    if (e.S <= 3) {
        if (e.S == 1) {
            HPF_MAIN(1, nn + nb)
        } else if (e.S == 2) {
            HPF_MAIN(2, nn + nb)
        } else {
            HPF_MAIN(3, nn + nb)
        }
        return;
    }
    if (nb > 0) {
        HPF_MAIN(0, nb)
    }
#undef HPF_MAIN
#undef HPF_MAIN_B
    switch (e.S) {
#define HPF_NODES(k)                                                                         \
    case k:                                                                                  \
        k_energy_nodes<k><<<nn, kRedBlock, 0, s>>>(D, g.nodes, node_part);                   \
        launch_pdl(k_energy_final<k>, dim3(1), dim3(kFinalBlock), 0, s,                      \
                   (const float2*)bead_part, nb_part, (const unsigned long long*)node_part, nn, \
                   g.nodes, e, out);                                                         \
        break;
        HPF_NODES(4) HPF_NODES(5) HPF_NODES(6) HPF_NODES(7) HPF_NODES(8)
#undef HPF_NODES
    }
}

void launch_energy(StateBuf st, const uint32_t* meta, int n, MeshGeom g, const float4* G,
                   StepConsts c, long long step, const long long* D, const EnergyConsts& e,
                   double* partials, const EnergyOut& out, cudaStream_t s) {
    launch_sums(st, meta, n, g, G, c, step, D, e, nullptr, -1, partials, out, s);
}

// The node sums and the combination, with bead partials formed elsewhere
// (nb_bead CTAs' worth, by the step launch that ended at this state).
int energy_nodes_launches(int S) { return S <= 3 ? 1 : 2; }

void launch_energy_nodes_only(int n, MeshGeom g, const long long* D, const EnergyConsts& e,
                              const float2* bead_part, int nb_bead, double* partials,
                              const EnergyOut& out, cudaStream_t s) {
    launch_sums(StateBuf{}, nullptr, n, g, nullptr, StepConsts{}, 0, D, e, bead_part, nb_bead,
                partials, out, s);
}

}  // namespace hpf
