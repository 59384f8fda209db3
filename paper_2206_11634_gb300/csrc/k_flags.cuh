// Node classification and local refilling (templated on storage and lattice).
//
// k_flags (one CTA per brick): sorts the brick's list, classifies its nodes
// (§2.3.1: solid when M_j >= c0, Eq. (26), owner = largest M_j, ties to the
// lower index), and refills the nodes the particles uncovered since the last
// step (§2.3.3, Eq. (30)).  M is evaluated in FP32 against a certified
// error band and re-evaluated in FP64 inside it, so the flags equal those of
// an exact FP64 evaluation.
#pragma once

#include "lbm_internal.cuh"

namespace lbmmb {

__device__ __forceinline__ void quat_rot(const double q[4], const double v[3], double r[3]) {
    const double w = q[0], x = q[1], y = q[2], z = q[3];
    const double R00 = 1 - 2 * (y * y + z * z), R01 = 2 * (x * y - w * z), R02 = 2 * (x * z + w * y);
    const double R10 = 2 * (x * y + w * z), R11 = 1 - 2 * (x * x + z * z), R12 = 2 * (y * z - w * x);
    const double R20 = 2 * (x * z - w * y), R21 = 2 * (y * z + w * x), R22 = 1 - 2 * (x * x + y * y);
    r[0] = R00 * v[0] + R01 * v[1] + R02 * v[2];
    r[1] = R10 * v[0] + R11 * v[1] + R12 * v[2];
    r[2] = R20 * v[0] + R21 * v[1] + R22 * v[2];
}

template <typename C>
__device__ __forceinline__ C feq_i(int ex, int ey, int ez, C w, C rho, C ux, C uy, C uz) {
    const C eu = ex * ux + ey * uy + ez * uz;
    const C uu = ux * ux + uy * uy + uz * uz;
    return w * rho * (C(1) + C(3) * eu + C(4.5) * eu * eu - C(1.5) * uu);
}
// The same equilibrium in offset form: f^eq_i - w_i rho0 for density
// rho = rho0 + drho.
template <typename C>
__device__ __forceinline__ C geq_i(int ex, int ey, int ez, C w, C drho, C rho, C ux, C uy, C uz) {
    const C eu = ex * ux + ey * uy + ez * uz;
    const C uu = ux * ux + uy * uy + uz * uz;
    return w * (drho + rho * (C(3) * eu + C(4.5) * eu * eu - C(1.5) * uu));
}

// Per-brick solid marks written by the flag pass (brick_solid): bit 7 when
// the brick holds a solid node, bits 0-5 when one lies on its low-x, high-x,
// low-y, high-y, low-z or high-z face.
constexpr uint32_t kSolidAny = 0x80u;

// M in FP64 out of line: few nodes need it, and inline it and the refill held
// registers that other CTAs can use.
__device__ __noinline__ inline double metaball64_far(const Params &P, const DevParticle &p, int x, int y, int z) {
    return metaball64(P, p, (double)x, (double)y, (double)z);
}

// Local refilling, §2.3.3.  Reading: f_i' at x_new counts as known
// (Eq. (30)) when it streams in from x_new + e_i and that node was a fluid
// node of the previous step; then f_i = f_i'(x_new+e_i) + 6 w_i rho0
// e_i.u_w, else f_i = f^eq_i(rho0, u_new); u_w = u_new is the surface
// velocity at x_new of the particle that uncovered it.  The values become
// the node's post-collision populations.
template <typename S, int Q>
__device__ __noinline__ void refill_node(const Params &P, int x, int y, int z, long long n, int old) {
    using L = Lat<Q>;
    using Cd = Codec<S>;
    using C = typename Cd::C;
    const DevParticle &pj = P.parts[old - 1];
    double r[3] = {minimg_d(P, 0, (double)x - pj.x[0]), minimg_d(P, 1, (double)y - pj.x[1]),
                   minimg_d(P, 2, (double)z - pj.x[2])};
    const C ux = (C)(pj.v[0] + pj.w[1] * r[2] - pj.w[2] * r[1]);
    const C uy = (C)(pj.v[1] + pj.w[2] * r[0] - pj.w[0] * r[2]);
    const C uz = (C)(pj.v[2] + pj.w[0] * r[1] - pj.w[1] * r[0]);
    const C rho0 = (C)P.rho0;
    S *A = (S *)P.fA;
    const long long N = P.N;
#pragma unroll
    for (int i = 0; i < Q; i++) {
        const int ex = L::e(i, 0), ey = L::e(i, 1), ez = L::e(i, 2);
        int sx = x + ex, sy = y + ey, sz = z + ez;
        bool in = true;
        if (sx < 0 || sx >= P.nx) { if (P.per[0]) sx = (sx + P.nx) % P.nx; else in = false; }
        if (sy < 0 || sy >= P.ny) { if (P.per[1]) sy = (sy + P.ny) % P.ny; else in = false; }
        if (sz < 0 || sz >= P.nz) { if (P.per[2]) sz = (sz + P.nz) % P.nz; else in = false; }
        const C w = (C)L::w(i);
        // offset form (g = f - w rho0; opposite directions share w)
        C g;
        const long long nb = (long long)sx + (long long)P.nx * ((long long)sy + (long long)P.ny * sz);
        if (i != 0 && in && P.flag_old[nb] == 0) {
            const int io = L::opp(i);
            g = Cd::ld_plain(A + (long long)io * N + nb, w, rho0) +
                C(6) * w * rho0 * (ex * ux + ey * uy + ez * uz);
        } else {
            g = geq_i<C>(ex, ey, ez, w, C(0), rho0, ux, uy, uz);
        }
        Cd::st(A + (long long)i * N + n, g, w, rho0);
    }
    atomicAdd(&P.counters[CNT_NREFILL], 1);
}

template <typename S, int Q>
__device__ __forceinline__ void flags_brick(const Params &P, SmemParticles &sp, int b) {
    const int tid = threadIdx.x;
    const int cnt = brick_count(P, b);
    // the list's slots are read in the same round as its count (slots past
    // the count hold stale ids and are not used)
    const int raw_id = tid < MAXPB ? P.blist[b * MAXPB + tid] : 0;
    __syncthreads();  // the previous brick's use of sp and of the list is over
    // ascending particle order makes the list, and hence every sum over it,
    // independent of the scatter's atomic order: lane s of warp 0 places its
    // id at its rank (ids are distinct)
    if (tid < 32) {
        const int id = tid < cnt ? raw_id : 0x7fffffff;
        int rank = 0;
        for (int o = 0; o < cnt; o++) rank += __shfl_sync(0xffffffffu, id, o) < id;
        if (tid < cnt) {
            P.blist[b * MAXPB + rank] = id;
            sp.id[rank] = id;
        }
        if (tid == 0) sp.n = cnt;
    }
    constexpr bool kF64 = sizeof(typename Codec<S>::C) == 8;
    __shared__ unsigned s_faces, s_far;
    if (tid == 0) s_faces = s_far = 0u;
    __syncthreads();
    int bxi, byi, bzi;
    brick_coords(P, b, bxi, byi, bzi);
    const int bx0 = bxi * BX, by0 = byi * BY, bz0 = bzi * BZ;
    const int lx = tid % BX, ly = (tid / BX) % BY, lz = tid / (BX * BY);
    const int x = bx0 + lx, y = by0 + ly, z = bz0 + lz;
    const bool active = x < P.nx && y < P.ny && z < P.nz;
    const long long n = (long long)x + (long long)P.nx * ((long long)y + (long long)P.ny * z);
    // the previous flag (the refill below needs it), issued with the
    // particles' loads so that the two latencies overlap
    const uint16_t old = active ? P.flag_old[n] : (uint16_t)0;
    if (kF64) {
        // listed particles (a bit each) whose FP32 positions the error band of
        // metaball32 does not cover: farther than it says, many box lengths
        // away along a periodic axis
        for (int t = tid; t < cnt * MAXCP; t += BRICK) {
            const DevParticle &p = P.parts[sp.id[t / MAXCP]];
            const int k = t % MAXCP;
            if (k < p.ncp && (fabsf(p.cpw_hl[k][0][0] - (float)bx0) > kBandReach ||
                              fabsf(p.cpw_hl[k][1][0] - (float)by0) > kBandReach ||
                              fabsf(p.cpw_hl[k][2][0] - (float)bz0) > kBandReach))
                atomicOr(&s_far, 1u << (t / MAXCP));
        }
    }
    if (cnt > 0) load_particle_records(P, sp, cnt, bx0, by0, bz0);

    // owner: the covering particle with the largest M, ties to the lower
    // index (the list is ascending); with one cover its FP32 decision is
    // enough, several covers compare their M in FP64.  Kept as running
    // values, so no per-thread array is indexed at run time.
    int own = -1;
    if (active && cnt > 0) {
        int own_s = -1;
        // FP64 lattices: thresholds at which FP32 has no band left
        const bool exact = kF64 && !(P.c0_f > 1e-30f && P.c0_f < 1e30f);
        double own_M = -1.0;  // FP64 M of the current owner, < 0 until computed
        for (int s = 0; s < cnt; s++) {
            if (!in_bound(P, sp, s, lx, ly, lz)) continue;  // outside s: M < c0 there
            bool unsure;
            const float M = metaball32(P, sp, s, (float)lx, (float)ly, (float)lz, unsure);
            bool inside;
            double Md = -1.0;
            if (unsure || exact || (kF64 && ((s_far >> s) & 1u))) {
                Md = metaball64_far(P, P.parts[sp.id[s]], x, y, z);
                inside = Md >= P.c0;
            } else {
                inside = M >= P.c0_f;
            }
            if (!inside) continue;
            if (own_s < 0) {
                own_s = s;
                own_M = Md;
                continue;
            }
            if (own_M < 0.0) own_M = metaball64_far(P, P.parts[sp.id[own_s]], x, y, z);
            if (Md < 0.0) Md = metaball64_far(P, P.parts[sp.id[s]], x, y, z);
            if (Md > own_M) {
                own_s = s;
                own_M = Md;
            }
        }
        if (own_s >= 0) own = sp.id[own_s];
    }
    const uint16_t fl = own >= 0 ? (uint16_t)(own + 1) : (uint16_t)0;
    if (active) P.flag_new[n] = fl;
    // where the brick holds solid nodes now: bit 7 anywhere, bits 0-5 on its
    // faces (low x, high x, low y, high y, low z, high z; a high face is the
    // last node inside the box on a ragged edge).  The near sweep takes the
    // plain path for a brick none of whose nodes has a solid neighbour.
    {
        uint32_t m = 0;
        if (active && fl != 0) {
            m = kSolidAny;
            if (lx == 0) m |= 1u;
            if (lx == BX - 1 || x == P.nx - 1) m |= 2u;
            if (ly == 0) m |= 4u;
            if (ly == BY - 1 || y == P.ny - 1) m |= 8u;
            if (lz == 0) m |= 16u;
            if (lz == BZ - 1 || z == P.nz - 1) m |= 32u;
        }
        m = __reduce_or_sync(0xffffffffu, m);
        if ((tid & 31) == 0 && m) atomicOr(&s_faces, m);
        __syncthreads();
        if (tid == 0 && P.brick_solid) P.brick_solid[b] = (uint8_t)s_faces;
    }

    if (active && fl == 0 && old != 0) refill_node<S, Q>(P, x, y, z, n, old);
}

// Persistent grid over the bricks listed this step and in the two steps
// before; a brick listed in several of these lists is visited once (its most
// recent listing).
// The entries are handed out from a per-step counter, as in the near sweep
// (thread 0 claims the next ones while the current brick runs; s_next
// alternates between two slots): this step's one at a time, the older ones,
// nearly all of which are listed again, eight at a time, a lane each, until few
// are left (one at a time a CTA spent two barriers and three dependent loads on
// each of them).
struct Claim {
    int first, size;
};
template <typename S, int Q>
__device__ __forceinline__ void flags_work(const Params &P, SmemParticles &sp, Claim *s_next, int blk, int ctas) {
    const int t = P.step;
    const int r0 = t % 3, r1 = (t + 2) % 3, r2 = (t + 1) % 3;
    const int c0 = P.counters[CNT_LISTED];
    const int c1 = t >= 1 ? P.wl_count[r1] : 0;
    const int c2 = t >= 2 ? P.wl_count[r2] : 0;
    if (blk == 0 && threadIdx.x == 0) P.wl_count[r0] = c0;  // read by the next two steps
    const int total = c0 + c1 + c2;
    const int lane = threadIdx.x & 31;
    Claim nxt = {0, 1};
    if (threadIdx.x == 0) nxt.first = atomicAdd(&P.counters[CNT_FLAGS_NEXT], 1);
    for (int k = 0;; k ^= 1) {
        if (threadIdx.x == 0) s_next[k] = nxt;
        __syncthreads();
        const Claim c = s_next[k];
        if (c.first >= total) break;
        if (threadIdx.x == 0) {
            nxt.size = c.first >= c0 && total - c.first >= 16 * ctas ? 8 : 1;
            nxt.first = atomicAdd(&P.counters[CNT_FLAGS_NEXT], nxt.size);
        }
        const int w = c.first + lane;
        int b = -1;  // the lane's brick (every warp holds the same)
        if (lane < c.size && w < total) {
            if (w < c0) {
                b = P.wl_list[r0 * P.nbricks + w];
            } else if (w < c0 + c1) {
                b = P.wl_list[r1 * P.nbricks + (w - c0)];
                if (P.stamp[b] == t) b = -1;      // also listed this step
            } else {
                b = P.wl_list[r2 * P.nbricks + (w - c0 - c1)];
                if (P.stamp[b] >= t - 1) b = -1;  // listed again since
            }
        }
        for (unsigned m = __ballot_sync(0xffffffffu, b >= 0); m; m &= m - 1)
            flags_brick<S, Q>(P, sp, __shfl_sync(0xffffffffu, b, __ffs(m) - 1));
    }
}
// (Four CTAs per SM at 64 registers: 8 at 32 registers left more room to the
// plain sweep beside them, 755 -> 717 us a step for 200 metaballs in 256^3, but
// spilled where one brick's latency counts, 139 -> 145 us for one metaball.)
template <typename S, int Q>
__global__ void __launch_bounds__(BRICK, 4) k_flags(Params P) {
    __shared__ SmemParticles sp;
    __shared__ Claim s_next[2];
    flags_work<S, Q>(P, sp, s_next, blockIdx.x, gridDim.x);
}

// Every node to f^eq(rho0, u0).
template <typename S, int Q>
__global__ void k_init(Params P, S *f) {
    using L = Lat<Q>;
    using C = typename Codec<S>::C;
    const C rho0 = (C)P.rho0, ux = (C)P.u0[0], uy = (C)P.u0[1], uz = (C)P.u0[2];
    for (long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x; n < P.N; n += (long long)gridDim.x * blockDim.x) {
#pragma unroll
        for (int i = 0; i < Q; i++) {
            const C w = (C)L::w(i);
            Codec<S>::st(f + (long long)i * P.N + n, geq_i<C>(L::e(i, 0), L::e(i, 1), L::e(i, 2), w, C(0), rho0, ux, uy, uz),
                         w, rho0);
        }
    }
}

// FP32 to FP64, and FP64 to FP32 rounded to nearest even, without the FP64
// pipe (a conversion there holds its sub-partition for 64 cycles a warp, as
// any FP64 instruction): the same bits as the casts, which take the values
// outside FP32's normal range.
__device__ __forceinline__ double to_double(double v) { return v; }
__device__ __forceinline__ double to_double(float v) {
    const uint32_t b = __float_as_uint(v), e = (b >> 23) & 255u;
    if (e == 0u || e == 255u) return (double)v;
    const unsigned long long m = ((unsigned long long)(b & 0x7fffffffu) + (896ull << 23)) << 29;
    return __longlong_as_double((long long)(m | ((unsigned long long)(b & 0x80000000u) << 32)));
}
template <typename C> __device__ __forceinline__ C from_double(double v);
template <> __device__ __forceinline__ double from_double<double>(double v) { return v; }
template <> __device__ __forceinline__ float from_double<float>(double v) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    const uint32_t hi = (uint32_t)(b >> 32), e = (hi >> 20) & 2047u;
    if (e < 897u || e > 1149u) return (float)v;  // not certain to round to a normal FP32 value
    const unsigned long long r = b + 0x0fffffffull + ((b >> 29) & 1ull);
    return __uint_as_float((hi & 0x80000000u) | (((uint32_t)(r >> 29) - (896u << 23)) & 0x7fffffffu));
}

// Stored populations -> FP64 [Q][N] (and back).  Bound by HBM once the
// conversions leave the FP64 pipe: 256^3 FP32, 3.83 GB: get 0.81 -> 0.64 ms, set
// 0.72 -> 0.59 ms (6.0 and 6.5 TB/s).
template <typename S, int Q>
__global__ void k_get_pop(Params P, const S *f, double *out) {
    using L = Lat<Q>;
    using C = typename Codec<S>::C;
    for (long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x; n < P.N; n += (long long)gridDim.x * blockDim.x) {
        C v[Q];  // every load before the stores, which might alias them
#pragma unroll
        for (int i = 0; i < Q; i++) v[i] = Codec<S>::ldf(f + (long long)i * P.N + n, (C)L::w(i), (C)P.rho0);
#pragma unroll
        for (int i = 0; i < Q; i++) out[(long long)i * P.N + n] = to_double(v[i]);
    }
}
template <typename S, int Q>
__global__ void k_set_pop(Params P, S *f, const double *in) {
    using L = Lat<Q>;
    using C = typename Codec<S>::C;
    for (long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x; n < P.N; n += (long long)gridDim.x * blockDim.x) {
        double v[Q];
#pragma unroll
        for (int i = 0; i < Q; i++) v[i] = in[(long long)i * P.N + n];
#pragma unroll
        for (int i = 0; i < Q; i++)
            Codec<S>::stf(f + (long long)i * P.N + n, from_double<C>(v[i]), (C)L::w(i), (C)P.rho0);
    }
}

// ---------------------------------------------------------------------------
// Macroscopic fields of the stored populations: rho = sum f, u = (sum f e -
// F/2)/rho (the velocity of the collision that produced them), in FP64.
//
// An FP64 warp instruction, conversions to and from FP64 included, holds its
// sub-partition for 64 cycles on this GPU (0.5 cycles per node and SM), while
// a node's memory traffic (FP32 D3Q19: 76 B in, 34 B out) takes 5.2 of those
// cycles.  The sums as FP64 additions of converted values (about 130 FP64
// instructions a node) took 3.77 ms at 256^3.  So below FP64 storage the sums
// run in FP32, in parts that add up exactly (all but 2^-54), and nine FP64 instructions are left: the density's sum
// with rho0 and the division.  Measured at 256^3, FP32, the call: 3.77 ->
// 0.56 ms (one 64-bit integer per value instead of the three FP32 parts
// below: 0.87).
//
// The sums: with 2^(E - 126) above the node's largest magnitude, adding and
// taking off 1.5 2^23 u rounds a value to a multiple of u, so a value splits
// exactly into a multiple of u1 = 2^(E - 145) (at most 2^19 of them), one of
// u2 = 2^-20 u1 (at most 2^19) and a rest of at most u2 / 2 (Rump, Ogita and
// Oishi's extraction, SIAM J. Sci. Comput. 31, 2008).  Q <= 19 such multiples
// add up exactly in FP32 in any order.  The rests, up to 2^(E - 166) each, add up
// with 18 roundings of up to 2^(E - 186), and their sum is rounded to u3 =
// 2^(E - 182): together under 2^(E - 181), 2^-54 of the largest value, which is
// 2^(E - 127) at least (a single FP64 sum's roundings are 18 of 2^-53 of it).
// ---------------------------------------------------------------------------
constexpr int kFieldEmin = 56, kFieldEmax = 240;  // the exponent fields E that the units stay normal for
__device__ __forceinline__ float exp2_field(int e) { return __uint_as_float((uint32_t)e << 23); }  // 2^(e - 127)

// a 2^e2 rounded to nearest even (|a| < 2^63, the result in FP64's normal
// range), without the FP64 pipe.
__device__ __forceinline__ double fixed_double(long long a, int e2) {
    if (a == 0) return 0.0;
    const unsigned long long mag = a < 0 ? 0ull - (unsigned long long)a : (unsigned long long)a;
    const int lz = __clzll((long long)mag);
    const unsigned long long n = mag << lz;  // bit 63 set
    unsigned long long m = n >> 11;          // 53 bits, the leading one included
    const uint32_t rem = (uint32_t)n & 0x7ffu;
    m += (rem > 0x400u || (rem == 0x400u && ((uint32_t)m & 1u))) ? 1ull : 0ull;
    const unsigned long long bits = ((unsigned long long)(1023 + 63 - lz + e2 - 1) << 52) + m;
    return __longlong_as_double((long long)(bits | (a < 0 ? 0x8000000000000000ull : 0ull)));
}
// FP64 to FP32 by truncation, for magnitudes within FP32's normal range.
__device__ __forceinline__ float trunc_float(double v) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    const uint32_t hi = (uint32_t)(b >> 32);
    return __uint_as_float((hi & 0x80000000u) | (((uint32_t)(b >> 29) - (896u << 23)) & 0x7fffffffu));
}

// Exponent field of an FP64 value (0 for zero): comparisons by it do not go
// through the FP64 pipe, as FP64 ones do.
__device__ __forceinline__ uint32_t exponent64(double v) {
    return ((uint32_t)((unsigned long long)__double_as_longlong(v) >> 32) >> 20) & 2047u;
}

// a u1 + b u2 + c as FP64, rounded once; c to the nearest u3 = 2^-17 u2
__device__ __forceinline__ double field_sum(float a, float b, float c, int E) {
    const int ia = __float2int_rn(a * exp2_field(272 - E));
    const int ib = __float2int_rn(b * exp2_field(292 - E));
    const int ic = __float2int_rn(c * exp2_field(309 - E));
    return fixed_double((long long)ia * (1ll << 37) + ((long long)ib * (1ll << 17) + ic), E - 182);
}

// Density and momentum (sum g e - F/2) of a node's FP32 offsets, E their
// largest exponent field.
template <int Q>
__device__ __forceinline__ void field_moments(const Params &P, float (&g)[Q], int E, double &r, double m[3]) {
    using L = Lat<Q>;
    float s[3], x[3], y[3], z[3];
#pragma unroll
    for (int p = 0; p < 3; p++) {
        // parts 0 and 1: the multiples of u1 and u2; part 2: what is left
        const float big = 1.5f * exp2_field(E - (p == 0 ? 145 : 165) + 127 + 23);
        s[p] = x[p] = y[p] = z[p] = 0.f;
#pragma unroll
        for (int i = 0; i < Q; i++) {
            float t = g[i];
            if (p < 2) {
                t = __fsub_rn(__fadd_rn(big, g[i]), big);
                g[i] = __fsub_rn(g[i], t);
            }
            s[p] = __fadd_rn(s[p], t);
            if (L::e(i, 0)) x[p] = __fadd_rn(x[p], L::e(i, 0) > 0 ? t : -t);
            if (L::e(i, 1)) y[p] = __fadd_rn(y[p], L::e(i, 1) > 0 ? t : -t);
            if (L::e(i, 2)) z[p] = __fadd_rn(z[p], L::e(i, 2) > 0 ? t : -t);
        }
    }
    r = P.rho0 + field_sum(s[0], s[1], s[2], E);
    m[0] = field_sum(x[0], x[1], x[2], E);
    m[1] = field_sum(y[0], y[1], y[2], E);
    m[2] = field_sum(z[0], z[1], z[2], E);
    for (int a = 0; a < 3; a++)
        if (exponent64(P.F[a])) m[a] -= 0.5 * P.F[a];
}

// u = m / r: an FP32 quotient, its FP64 residual, and the residual's share by
// 1/r to 2^-43 (one Newton step from the FP32 reciprocal): within 0.51 ulp of
// the quotient.  Two FP64 instructions a component and two for 1/r; operands
// outside the range that the FP32 steps hold are divided.
__device__ __forceinline__ void field_velocity(double r, const double m[3], double u[3]) {
    // 2^-50 <= r < 2^50
    const bool mid = exponent64(r) - 973u < 100u && (__double_as_longlong(r) >> 63) == 0;
    const float r0 = __frcp_rn(mid ? trunc_float(r) : 1.0f);
    const double r0d = to_double(r0);
    const double r1 = fma(r0d, fma(-r, r0d, 1.0), r0d);
#pragma unroll
    for (int a = 0; a < 3; a++) {
        const uint32_t e = exponent64(m[a]);
        if (e == 0u && mid) {
            u[a] = 0.0;  // m is zero (sums and forces of normal values)
        } else if (e - 957u < 130u && mid) {  // 2^-66 <= |m| < 2^64
            const double q = to_double(trunc_float(m[a]) * r0);
            u[a] = fma(fma(-q, r, m[a]), r1, q);
        } else {
            u[a] = m[a] / r;
        }
    }
}

template <typename S, int Q>
__global__ void __launch_bounds__(256, 4) k_fields(Params P, const S *f, const uint16_t *flags, double *rho, double *u,
                                                uint16_t *fl_out) {
    using L = Lat<Q>;
    using C = typename Codec<S>::C;
    for (long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x; n < P.N; n += (long long)gridDim.x * blockDim.x) {
        const uint16_t fl = flags[n];
        double r = 0, m[3] = {0, 0, 0}, uu[3] = {0, 0, 0};
        if (rho || u) {
            // the loads do not wait for the flag
            C g[Q];
#pragma unroll
            for (int i = 0; i < Q; i++) g[i] = Codec<S>::ld_plain(f + (long long)i * P.N + n, (C)L::w(i), (C)P.rho0);
            if (fl == 0) {
                bool done = false;
                if constexpr (sizeof(C) == 4) {
                    uint32_t top = 0;
#pragma unroll
                    for (int i = 0; i < Q; i++) top = max(top, __float_as_uint(g[i]) & 0x7fffffffu);
                    const int E = top ? (int)(top >> 23) : kFieldEmin;
                    if (E >= kFieldEmin && E <= kFieldEmax) {
                        field_moments<Q>(P, g, E, r, m);
                        field_velocity(r, m, uu);
                        done = true;
                    }
                }
                if (!done) {  // FP64 storage, or offsets outside the range above (not finite, too)
#pragma unroll
                    for (int i = 0; i < Q; i++) {
                        const double gi = (double)g[i];
                        r += gi;
                        m[0] += gi * L::e(i, 0);
                        m[1] += gi * L::e(i, 1);
                        m[2] += gi * L::e(i, 2);
                    }
                    r += P.rho0;
                    uu[0] = (m[0] - 0.5 * P.F[0]) / r;
                    uu[1] = (m[1] - 0.5 * P.F[1]) / r;
                    uu[2] = (m[2] - 0.5 * P.F[2]) / r;
                }
            }
        }
        if (fl_out) fl_out[n] = fl;
        if (rho) rho[n] = r;
        if (u) {
            u[n] = uu[0];
            u[P.N + n] = uu[1];
            u[2 * P.N + n] = uu[2];
        }
    }
}

// Health scan: non-finite populations or |u| > 0.5 at a fluid node.
template <typename S, int Q>
__global__ void k_check(Params P, const S *f, const uint16_t *flags) {
    using L = Lat<Q>;
    using C = typename Codec<S>::C;
    bool bad = false;
    for (long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x; n < P.N; n += (long long)gridDim.x * blockDim.x) {
        if (flags[n] != 0) continue;
        float r = P.rho0_f, mx = 0, my = 0, mz = 0;
#pragma unroll
        for (int i = 0; i < Q; i++) {
            const float gi = (float)Codec<S>::ld_plain(f + (long long)i * P.N + n, (C)L::w(i), (C)P.rho0);
            r += gi;
            mx += gi * L::e(i, 0);
            my += gi * L::e(i, 1);
            mz += gi * L::e(i, 2);
        }
        const float u2 = (mx * mx + my * my + mz * mz) / (r * r);
        if (!(r > 0.f) || !isfinite(r) || !(u2 <= 0.25f)) bad = true;
    }
    if (__syncthreads_or(bad) && threadIdx.x == 0) atomicOr(&P.status[ST_ERR], ERRB_DIVERGED);
}

}  // namespace lbmmb
