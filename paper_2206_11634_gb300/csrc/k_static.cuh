// The fixed-geometry sweep.
//
// When every particle is fixed (fixed = 1) the node flags, the particle links
// and their geometry (q of Eq. (27), the lever arm from the centroid to the
// wall point x_w and the wall velocity there) cannot change.  Once the flag
// pass has run for three steps, k_static_build records them: per node whether
// the plain path may take it (sskip), and for every fluid node with particle
// links its link directions and each link's geometry.  The missing force
// points (§2.3.5 item 2, Eqs. (31)-(32)) depend on the geometry only, so their
// fixed-point force/torque totals are summed once (smf).  Every later step is
// two kernels that run concurrently on disjoint nodes: k_static_plain over the
// nodes the plain path takes (the pull, BGK and stores of k_sweep_plain, over
// aligned 256-node spans, no brick lists) and k_static_links over the link
// nodes (VIBB of Eqs. (19)-(25) and the momentum exchange of Eqs. (28)-(29)
// with the recorded geometry).  The arithmetic is the near sweep's
// (link_geometry, link_update, solid_links, collide_store), so a step gives
// the same bits either way.  Lattices below FP64 only (the force totals are
// the fixed-point ones).
#pragma once

#include "k_sweep.cuh"

namespace lbmmb {

// ---------------------------------------------------------------------------
// build: one CTA per brick listed this step (no other brick holds a solid
// node or a node next to one), after sskip, scount and smf were cleared
// ---------------------------------------------------------------------------
struct StaticBuildScratch {
    uint32_t nf[BRICK][19];  // the node's flag and its neighbours' (index i: y = x - e_i)
    unsigned long long fix[BRICK / 32][MAXPB][6];  // each warp's missing-force terms
};

template <typename S, int Q>
__device__ __forceinline__ void static_build_brick(const Params &P, SmemParticles &sp, StaticBuildScratch &bs,
                                                   int b) {
    using L = Lat<Q>;
    using C = typename Codec<S>::C;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    int bxi, byi, bzi;
    brick_coords(P, b, bxi, byi, bzi);
    const int bx0 = bxi * BX, by0 = byi * BY, bz0 = bzi * BZ;
    const int lx = tid % BX, ly = (tid / BX) % BY, lz = tid / (BX * BY);
    const int x = bx0 + lx, y = by0 + ly, z = bz0 + lz;
    const bool active = x < P.nx && y < P.ny && z < P.nz;
    const int n = x + P.nx * (y + P.ny * z);
    const int cnt = brick_count(P, b);
    __syncthreads();  // the previous brick is done with the shared state
    load_smem_particles(P, sp, b, bx0, by0, bz0);
    for (int e = lane; e < cnt * 6; e += 32) bs.fix[warp][e / 6][e % 6] = 0ull;
    __syncwarp();

    constexpr uint32_t kWall = 0xFFFFFFFFu;
    {
        int xs[3], ys[3], zs[3];
        neighbour_coords(P, x, y, z, xs, ys, zs);
        bs.nf[tid][0] = active ? (uint32_t)P.flag_new[n] : 1u;
#pragma unroll
        for (int i = 1; i < Q; i++) {
            const int sx = xs[1 - L::e(i, 0)], sy = ys[1 - L::e(i, 1)], sz = zs[1 - L::e(i, 2)];
            const bool wall = (sx | sy | sz) < 0;
            bs.nf[tid][i] = (!active || wall) ? kWall : (uint32_t)P.flag_new[sx + P.nx * (sy + P.ny * sz)];
        }
    }
    const uint32_t own = bs.nf[tid][0];
    const bool fluid = active && own == 0;
    uint32_t links = 0;
    if (fluid) {
        for (int i = 1; i < Q; i++)
            if (bs.nf[tid][i] != 0 && bs.nf[tid][i] != kWall) links |= 1u << i;
    }
    if (active) P.sskip[n] = (uint8_t)((!fluid || links) ? 1 : 0);

    if (links) {
        const int k = __popc(links);
        const int node = atomicAdd(&P.scount[0], 1);
        const int base = atomicAdd(&P.scount[1], k);
        if (node >= P.snode_cap || base + k > P.slink_cap) {
            atomicOr(&P.status[ST_ERR], ERRB_STATIC_CAPACITY);
        } else {
            StaticNode sn;
            sn.n = n;
            sn.mask = links;
            sn.base = base;
            P.snodes[node] = sn;
            C Mf_cache = 0;
            int Mf_slot = -1;
            int r = 0;
            uint32_t m = links;
            while (m) {
                const int i = __ffs(m) - 1;
                m &= m - 1;
                const int j = (int)bs.nf[tid][i] - 1;
                const int s = slot_of(sp, j);
                StaticLink rec;
                if (s < 0) {  // cannot happen for a consistent brick list
                    atomicOr(&P.status[ST_ERR], ERRB_BRICK_OVERFLOW);
                    rec.q = 0.f;
                    for (int a = 0; a < 3; a++) rec.r[a] = rec.uw[a] = 0.f;
                } else {
                    const LinkGeom<C> g = link_geometry<S, Q>(P, sp, i, s, lx, ly, lz, bx0, by0, bz0, &Mf_cache,
                                                              &Mf_slot);
                    rec.q = (float)g.q;
                    for (int a = 0; a < 3; a++) {
                        rec.r[a] = (float)g.r[a];
                        rec.uw[a] = (float)g.uw[a];
                    }
                }
                // x_ff = x - d = x + e_i is the neighbour on the far side
                const bool ff_ok = bs.nf[tid][L::opp(i)] == 0;
                rec.jf = (j & 0xFFFF) | (ff_ok ? (int)0x80000000u : 0);
                P.slinks[base + r] = rec;
                r++;
            }
        }
    }

    // missing force points of the solid nodes: their totals once
    if (active && !fluid && P.missing_force) {
        const int owner = (int)own - 1;
        const ForceSink<C> sink{nullptr, bs.fix[warp]};
        for (int s = 0; s < sp.n; s++) {
            const int j = sp.id[s];
            uint32_t cand = 0;
            for (int i = 1; i < Q; i++) {
                const uint32_t f = bs.nf[tid][i];
                const bool seen = (f == 0 && j == owner) || f == (uint32_t)(j + 1);
                if (!seen) cand |= 1u << i;
            }
            if (cand) solid_links<S, Q>(P, sp, s, j == owner, cand, lx, ly, lz, bx0, by0, bz0, sink);
        }
    }
    __syncwarp();
    for (int e = lane; e < cnt * 6; e += 32) {
        const unsigned long long v = bs.fix[warp][e / 6][e % 6];
        if (v) atomicAdd(&P.smf[sp.id[e / 6] * 6 + e % 6], v);
    }
}

template <typename S, int Q>
__global__ void __launch_bounds__(BRICK) k_static_build(Params P) {
    if (sizeof(typename Codec<S>::C) == 8) return;  // FP64 lattices keep the near sweep
    __shared__ SmemParticles sp;
    __shared__ StaticBuildScratch bs;
    const int listed = P.counters[CNT_LISTED];
    for (int w = blockIdx.x; w < listed; w += gridDim.x)
        static_build_brick<S, Q>(P, sp, bs, P.wl_list[(P.step % 3) * P.nbricks + w]);
}

// ---------------------------------------------------------------------------
// plain nodes: one CTA per 256 consecutive nodes
// ---------------------------------------------------------------------------
// The node's skip mark is loaded together with its pulls (which stay in the
// box either way), so the two latencies overlap; a skipped node stores
// nothing.
template <typename S, int Q, bool kForce>
__device__ __forceinline__ void static_plain_node(const Params &P, int n) {
    if (n >= P.N) return;
    const bool skip = P.sskip[n] != 0;
    const int z = (int)fast_quot((uint32_t)n, P.by_nxy), r = n - z * P.nx * P.ny;
    const int y = (int)fast_quot((uint32_t)r, P.by_nx), x = r - y * P.nx;
    typename Codec<S>::C fin[Q];
    plain_pull<S, Q, true>(P, x, y, z, n, fin);
    if (!skip) collide_store<S, Q, kForce, true>(P, fin, (S *)P.fB, P.N, n);
}
// Step t's two kernels, then step t + 1's, all on one stream as programmatic
// dependent launches: a kernel's CTAs come up while the one before still runs.
// The first of a step waits for the whole of step t - 1, then lets the second
// start, which runs beside it on other nodes (ordered by the step's gate,
// lbm_internal.cuh) and whose completion stands for the whole step.  On two
// streams with events between them, and a memset a step, a step of the 48^3
// drag box took 22.6 us, most of it gaps; this way 7.5, and 11.1 with the
// kernels one after the other.  While all CTAs of the plain kernel run at once
// (four per SM) the link kernel, the longer chain of loads, comes first; beyond
// that the plain kernel, whose CTAs then have no gate to pass.  Plain kernel
// first and second, us a step: 48^3 FP32 8.5 and 7.5, FP16 10.8 and 10.2; 64^3 12.1
// and 12.6, 14.1 and 14.5; 96^3 25.6 and 27.0.
//
// The last CTA clears the step counters and force totals of the next step's
// region (the binning, which clears it otherwise, does not run here); they
// are those of step t - 1, whose kernels are done.
template <typename S, int Q, bool kForce>
__global__ void __launch_bounds__(BRICK, 4) k_static_plain(Params P) {
    if (P.links_first) {
        pdl_launch_dependents();
        gate_pass(P.gate);
    } else {
        pdl_wait();
        gate_open(P.gate);
    }
    if (blockIdx.x == gridDim.x - 1) {
        int *tail = static_cast<int *>(P.bin_next) + P.nbricks;
        const int words = (int)(P.bin_next_bytes / 4) - P.nbricks;
        for (int k = threadIdx.x; k < words; k += BRICK) tail[k] = 0;
    }
    static_plain_node<S, Q, kForce>(P, blockIdx.x * BRICK + (int)threadIdx.x);
    if (P.links_first) pdl_wait();
}

// ---------------------------------------------------------------------------
// link nodes: one warp per kPer listed link nodes
// ---------------------------------------------------------------------------
// A warp's links in a queue (lane order, then direction order): the lane's
// node and direction, then the link's result.
struct StaticScratch {
    unsigned short entry[BRICK / 32][kLinkQueue];  // (lane << 5) | direction
    int rec[BRICK / 32][kLinkQueue];               // link record, then (as float bits) its result
    int node[BRICK / 32][32];                      // node index of each lane
};

// One link of node n (direction i, record r): the node's own populations,
// x_ff's and the record fetched in one round, the unknown and the momentum
// exchange with the recorded geometry; the force/torque terms in fixed point.
// Coherent loads: the kernel can be up before the step before has written them.
template <typename S, int Q>
__device__ __forceinline__ float static_link(const Params &P, int n, int i, int r, int &j, LinkTerms &lt) {
    using L = Lat<Q>;
    using Cd = Codec<S>;
    using C = typename Cd::C;
    const S *A = (const S *)P.fA;
    const long long N = P.N;
    const C rho0 = Prm<C>::rho0(P);
    const StaticLink rec = P.slinks[r];
    const int nxy = P.nx * P.ny;
    const int z = n / nxy, rr = n - z * nxy;
    const int y = rr / P.nx, x = rr - y * P.nx;
    const int io = L::opp(i);
    // x_ff = x - d = x + e_i; beyond a wall the wrapped node is read and its
    // values are not used (the record says so), so no load waits for the record
    int fx = x + lat_e<Q>(i, 0), fy = y + lat_e<Q>(i, 1), fz = z + lat_e<Q>(i, 2);
    if (fx < 0) fx += P.nx; else if (fx >= P.nx) fx -= P.nx;
    if (fy < 0) fy += P.ny; else if (fy >= P.ny) fy -= P.ny;
    if (fz < 0) fz += P.nz; else if (fz >= P.nz) fz -= P.nz;
    const int nff = fx + P.nx * (fy + P.ny * fz);
    FFData<C> ff;
    ff.drho = 0;
    ff.m[0] = ff.m[1] = ff.m[2] = 0;
    ff.g_io = 0;
    C fown_io = 0, drho_f = 0, m_f[3] = {0, 0, 0};
#pragma unroll
    for (int k = 0; k < Q; k++) {
        const C fk = Cd::ld_plain(A + (long long)k * N + n, (C)L::w(k), rho0);
        drho_f += fk;
        m_f[0] += fk * L::e(k, 0);
        m_f[1] += fk * L::e(k, 1);
        m_f[2] += fk * L::e(k, 2);
        if (k == io) fown_io = fk;
        if (P.vibb) {
            const C gk = Cd::ld_plain(A + (long long)k * N + nff, (C)L::w(k), rho0);
            ff.drho += gk;
            ff.m[0] += gk * L::e(k, 0);
            ff.m[1] += gk * L::e(k, 1);
            ff.m[2] += gk * L::e(k, 2);
            if (k == io) ff.g_io = gk;
        }
    }
    ff.ok = rec.jf < 0;  // bit 31
    C u_f[3];
    const C inv_rho_f = rcp_w<C>(rho0 + drho_f);  // as the near sweep's link_coop
    for (int a = 0; a < 3; a++) u_f[a] = (m_f[a] - C(0.5) * Prm<C>::F(P, a)) * inv_rho_f;
    LinkGeom<C> g;
    g.q = (C)rec.q;
    for (int a = 0; a < 3; a++) {
        g.r[a] = (C)rec.r[a];
        g.uw[a] = (C)rec.uw[a];
    }
    C dP[3];
    const C fin = link_update<S, Q>(P, i, g, ff, fown_io, drho_f, u_f, dP);
    C t[6];
    force_terms<C>(dP, g.r, t);
    j = rec.jf & 0xFFFF;
    lt.s = j;
#pragma unroll
    for (int c = 0; c < 6; c++) lt.t[c] = (long long)to_fixed<C>(t[c]);
    return (float)fin;
}

// The warp's link terms of one round added to the particles' totals: per
// particle met, the exact 64-bit sums over the warp by 32-bit reductions (as
// warp_add_terms) and one atomic each.  (Shared-memory atomics per link, 64
// bits wide, are compare-and-swap loops: they took most of the link kernel.)
__device__ __forceinline__ void static_add_terms(const Params &P, const LinkTerms &lt, int lane) {
    unsigned todo = __ballot_sync(0xffffffffu, lt.s >= 0);
    while (todo) {
        const int j = __shfl_sync(0xffffffffu, lt.s, __ffs(todo) - 1);
        const bool mine = lt.s == j;
        todo &= ~__ballot_sync(0xffffffffu, mine);
        unsigned long long out = 0;
#pragma unroll
        for (int c = 0; c < 6; c++) {
            const long long v = mine ? lt.t[c] : 0ll;
            const unsigned lo = (unsigned)v & 0x1FFFFFu, mid = (unsigned)(v >> 21) & 0x1FFFFFu;
            const int hi = (int)(v >> 42);
            const unsigned long long sum =
                (unsigned long long)__reduce_add_sync(0xffffffffu, lo) +
                ((unsigned long long)__reduce_add_sync(0xffffffffu, mid) << 21) +
                ((unsigned long long)(long long)__reduce_add_sync(0xffffffffu, hi) << 42);
            if (lane == c) out = sum;
        }
        if (lane < 6 && out) atomicAdd(&P.Ffix[j * 6 + lane], out);
    }
}

// The lane's link node of warp wg (no links past the list's end).
template <int kPer>
__device__ __forceinline__ StaticNode static_node(const Params &P, int wg) {
    const int lane = threadIdx.x & 31, idx = wg * kPer + lane;
    StaticNode sn;
    sn.n = 0;
    sn.mask = 0u;
    sn.base = 0;
    if (lane < kPer && idx < P.snodes_n) sn = P.snodes[idx];
    return sn;
}
template <typename S, int Q, bool kForce>
__device__ __forceinline__ void static_links_warp(const Params &P, StaticScratch &ss, const StaticNode &sn) {
    using L = Lat<Q>;
    using Cd = Codec<S>;
    using C = typename Cd::C;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const S *A = (const S *)P.fA;
    S *B = (S *)P.fB;
    const long long N = P.N;
    const C rho0 = Prm<C>::rho0(P);
    const bool has = sn.mask != 0u;  // every listed node has links
    __syncwarp();  // the previous round of the warp is done with its queue
    ss.node[warp][lane] = sn.n;
    const uint32_t links = sn.mask;
    const int mine = __popc(links);
    int incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += v;
    }
    const int first = incl - mine;
    const int total = __shfl_sync(0xffffffffu, incl, 31);
    {
        uint32_t m = links;
        for (int k = 0; m; k++) {
            const int i = __ffs(m) - 1;
            m &= m - 1;
            ss.entry[warp][first + k] = (unsigned short)((lane << 5) | i);
            ss.rec[warp][first + k] = sn.base + k;
        }
    }
    __syncwarp();
    for (int r = 0; r < total; r += 32) {
        const int e = r + lane;
        LinkTerms lt;
        lt.s = -1;
        if (e < total) {
            const int ent = ss.entry[warp][e];
            int j;
            ss.rec[warp][e] =
                __float_as_int(static_link<S, Q>(P, ss.node[warp][ent >> 5], ent & 31, ss.rec[warp][e], j, lt));
        }
        static_add_terms(P, lt, lane);
    }
    __syncwarp();
    if (has) {
        const int n = sn.n;
        const int nxy = P.nx * P.ny;
        const int z = n / nxy, rr = n - z * nxy;
        const int y = rr / P.nx, x = rr - y * P.nx;
        int xs[3], ys[3], zs[3];
        neighbour_coords(P, x, y, z, xs, ys, zs);
        C fin[Q];
        int k = first;
#pragma unroll
        for (int i = 0; i < Q; i++) {
            if (links & (1u << i)) {  // link results are offsets g
                fin[i] = Cd::g_to_v((C)__int_as_float(ss.rec[warp][k]), (C)L::w(i));
                k++;
            } else {
                const int sx = xs[1 - L::e(i, 0)], sy = ys[1 - L::e(i, 1)], sz = zs[1 - L::e(i, 2)];
                const bool wall = (sx | sy | sz) < 0;
                const S *ptr = wall ? A + (long long)L::opp(i) * N + n
                                    : A + (long long)i * N + (sx + P.nx * (sy + P.ny * sz));
                fin[i] = Cd::ldv_s(ptr, (C)L::w(i), rho0);
            }
        }
        collide_store<S, Q, kForce>(P, fin, B, N, n);  // collide-space values
    }
}

// The step's constant parts: the missing-force-point totals and the link
// count (threads t of nt).
__device__ __forceinline__ void static_constants(const Params &P, int t, int nt) {
    for (int k = t; k < P.np * 6; k += nt)
        if (P.smf[k]) atomicAdd(&P.Ffix[k], P.smf[k]);
    if (t == 0) atomicAdd(&P.counters[CNT_NLINKS], P.scount[1]);
}

template <typename S, int Q, bool kForce, int kPer>
__global__ void __launch_bounds__(BRICK, kNearCtasPerSm) k_static_links(Params P) {
    if (sizeof(typename Codec<S>::C) == 8) return;
    __shared__ StaticScratch ss;
    const int warps = (P.snodes_n + kPer - 1) / kPer;
    int wg = blockIdx.x * (BRICK / 32) + (int)(threadIdx.x >> 5);
    StaticNode sn = static_node<kPer>(P, wg);  // (recorded before any of these steps: read before the wait)
    if (P.links_first) {
        pdl_wait();
        gate_open(P.gate);
    } else {
        pdl_launch_dependents();
        gate_pass(P.gate);
    }
    if (blockIdx.x == gridDim.x - 1) static_constants(P, threadIdx.x, BRICK);
    while (wg < warps) {
        static_links_warp<S, Q, kForce>(P, ss, sn);
        wg += gridDim.x * (BRICK / 32);
        sn = static_node<kPer>(P, wg);
    }
    if (!P.links_first) pdl_wait();
}

// ---------------------------------------------------------------------------
// batched lattices: the same two kernels over all cases
// ---------------------------------------------------------------------------

// The two kernels of a step wait for one another as the single lattice's do
// (k_static_plain).  The step's parity comes with the launch: step numbers are
// not needed here, and counting a step's CTAs down to advance a device
// counter, one atomic on one address per CTA, took 7 % of a step (64 boxes,
// FP32, ms a step: 1.558, without it 1.453; FP16 1.208, 1.103).

// plain_chunk spans per CTA as k_sweep_plain_batch; the CTA holding a case's
// first span also clears that case's per-step region for the next step (the
// binning, which clears it otherwise, does not run in fixed-geometry steps).
// Compiled for five CTAs per SM (48 registers, 8 bytes spilled): no particle
// kernel needs the SM slots here, and it measured 1 % faster than four on the
// 64-case batch (six spilled 88 bytes and was 2-6 % slower).
template <typename S, int Q, bool kForce>
__global__ void __launch_bounds__(BRICK, 5) k_static_plain_batch(BatchArgs B) {
    pdl_wait();
    gate_open(B.gate);
    const int total = B.span_off[B.ncases];
    const Params *row = B.tab + (size_t)B.parity * B.ncases;
    const int g0 = blockIdx.x * B.plain_chunk;
    const int g1 = min(total, g0 + B.plain_chunk);
    // the case's parameters in shared memory (re-read when the CTA's spans
    // cross into the next case): loads from there cannot alias the stores
    // to the populations, so they stay in registers
    __shared__ Params sP;
    int cur = -1;
    for (int g = g0; g < g1; g++) {
        const int c = B.span_case[g];
        if (c != cur) {
            __syncthreads();
            const int *src = reinterpret_cast<const int *>(row + c);
            int *dst = reinterpret_cast<int *>(&sP);
            for (int k = threadIdx.x; k < (int)(sizeof(Params) / 4); k += blockDim.x) dst[k] = src[k];
            __syncthreads();
            cur = c;
        }
        const Params &P = sP;
        if (g == B.span_off[c]) {
            int4 *zp = static_cast<int4 *>(P.bin_next);
            const long long n16 = P.bin_next_bytes / 16;
            for (long long k = threadIdx.x; k < n16; k += blockDim.x) zp[k] = make_int4(0, 0, 0, 0);
        }
        static_plain_node<S, Q, kForce>(P, (g - B.span_off[c]) * BRICK + (int)threadIdx.x);
    }
}

// One warp per kStaticNodesPerWarp link nodes of a case (each case at least one
// warp, which also adds the case's constant parts).
template <typename S, int Q, bool kForce>
__global__ void __launch_bounds__(BRICK, kNearCtasPerSm) k_static_links_batch(BatchArgs B) {
    __shared__ StaticScratch ss;
    pdl_launch_dependents();
    const int warps = B.swarp_off[B.ncases];
    const int gw = blockIdx.x * (BRICK / 32) + (int)(threadIdx.x >> 5);
    const int c = case_of(B.swarp_off, B.ncases, min(gw, warps - 1));  // whose warp range holds gw
    const Params &P = B.tab[(size_t)B.parity * B.ncases + c];
    const int wl = gw - B.swarp_off[c];
    const StaticNode sn = static_node<kStaticNodesPerWarp>(P, wl);  // (recorded before any of these steps)
    gate_pass(B.gate);
    if (gw < warps) {
        if (wl == 0) static_constants(P, threadIdx.x & 31, 32);
        if (wl * kStaticNodesPerWarp < P.snodes_n) static_links_warp<S, Q, kForce>(P, ss, sn);
    }
    pdl_wait();
}

}  // namespace lbmmb
