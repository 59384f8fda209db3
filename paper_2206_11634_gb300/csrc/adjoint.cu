// Discrete adjoint of the lattice sweep around one fixed metaball (the C ABI
// of include/lbm_adjoint.h): d(mean drag)/d(control points, weights) with
// the node flags frozen.
//
// Forward step (offset form g = f - w rho0, as the main sweep): for every
// fluid node, pull g_i from x - e_i, or, on a particle link (x - e_i solid),
// take the VIBB unknown of Eqs. (19)-(25) from the node's own post-collision
// populations and those of x_ff = x + e_i (halfway bounce-back when x_ff is
// solid); collide (BGK + Guo, Eqs. (15)-(18)); the drag of the step is the
// x component of Eq. (28) summed over the links (u_w = 0; its constant part
// cancels over the closed link set, as in the main sweep).
//
// Adjoint of one step, for lambda' = dJ/dg+(t+1):
//   A1  per fluid node: lambda_in = (dBGK/dg_in)^T lambda' (the equilibrium
//       and forcing depend on the pulled values g_in only through their
//       density and momentum, so this is (1 - omega) lambda' + a + b.e_j with
//       a and b from those four numbers), plus the drag's direct dependence
//       on the pulled link values;
//   A2  the pull, transposed: node n stores lambda_in_j(n) into
//       dJ/dg+(t)_j(n - e_j) when n - e_j is a fluid node, and writes dJ/dg+(t)
//       itself in the directions whose neighbour is solid (its links); every
//       entry of a fluid node has exactly one writer;
//   A3  per VIBB link: its value depends on the node's and x_ff's populations
//       through their density, momentum and one population each, and on q.
//       The two single populations' entries of dJ/dg+(t) are written by the
//       link's own node (its link direction, and its push to x_ff), so their
//       shares are added there; the density and momentum shares, (A, B) with
//       A + B.e_k in every direction k, are summed per node beside dJ/dg+(t)
//       and added when the next adjoint step reads it.
//
// What A1 and A3 need of the forward run is kept step by step: a node's four
// moments of the pulled values (16 bytes, instead of a whole state of 76 and
// a second gather with its link values) and nine partial derivatives per link
// (by reverse differentiation of the VIBB value, where the value is formed).
// A workspace too small for every step's (lbm_adj_workspace_sizes) keeps a
// state every ceil(sqrt(T)) steps instead, and each segment is run forward again
// from it.
//
// A step, forward or adjoint, is two kernels on disjoint nodes in programmatic
// dependent launches, ordered as the fixed-geometry sweep's (k_static.cuh): one
// over 256-node spans for the nodes without links, then one for the fluid nodes
// with links, whose links are spread over a warp's lanes.  96^3, T = 500, on a
// GB300: forward 28 us a step (44 with the links of a node one after another in
// its thread), adjoint 29 (113, with a recomputed forward step, a second gather
// and a separate atomic scatter per link); 32^3: 5.7 and 6.5 (18 and 42).
//
// Finally dJ/dq goes through Eq. (27) and Eq. (4) to the control points and
// weights (FP64).
#include <algorithm>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <new>
#include <vector>

#include "lbm_adjoint.h"
#include "k_plain.cuh"

using namespace lbmmb;

namespace {

constexpr int Q = 19;
using L19 = Lat<19>;
constexpr size_t kAlign = 256;
size_t align_up(size_t v) { return (v + kAlign - 1) / kAlign * kAlign; }

// ---------------------------------------------------------------------------
// the pieces of the step
// ---------------------------------------------------------------------------
struct AdjConst {
    int nx, ny, nz;
    long long N;
    FastDiv by_nxy, by_nx;
    float rho0, omega, gfac;
    float F[3], Fg[3];  // body force, and gfac times it
};

// f^eq_i - w_i rho0 for density rho = rho0 + drho, velocity u (Eq. (16))
__device__ __forceinline__ float geq_f(float ex, float ey, float ez, float w, float drho, float rho, float ux, float uy,
                                       float uz) {
    const float eu = ux * ex + uy * ey + uz * ez;
    const float uu = ux * ux + uy * uy + uz * uz;
    return (drho + rho * (eu * 3.0f + eu * eu * 4.5f - uu * 1.5f)) * w;
}
// its derivatives along d: dr with rho following drho, u[3]
__device__ __forceinline__ void geq_grad(const float d[3], float w, float rho, const float u[3], float &g_dr,
                                         float g_u[3]) {
    const float eu = u[0] * d[0] + u[1] * d[1] + u[2] * d[2];
    const float uu = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
    g_dr = w * (1.0f + (eu * 3.0f + eu * eu * 4.5f - uu * 1.5f));
    const float c = w * rho, ce = c * (3.0f + 9.0f * eu);
#pragma unroll
    for (int a = 0; a < 3; a++) g_u[a] = ce * d[a] - 3.0f * c * u[a];
}

// What a link's value is formed from: the density offset, momentum and io
// population (post-collision) of the fluid node x_f and of x_ff.
struct LinkState {
    float drf, mf[3], gf, drff, mff[3], gff;
};
// Derivatives of a link's value by those (gf: 2q, gff: 1 - 2q) and by q.
struct LinkGrad {
    float4 f, ff;  // by (drf, mf) and (drff, mff)
    float q;
};

// The VIBB unknown of a link whose direction into the solid is d (index io),
// u_w = 0 (a fixed particle): u = (m - F/2)/rho of the two nodes.  kGrad: its
// derivatives too, by reverse differentiation (about three times the value's
// arithmetic; forward-mode dual numbers took eleven tangents through it).
template <bool kGrad>
__device__ __forceinline__ float vibb_f(const AdjConst &A, int io, float q, const LinkState &s, LinkGrad &g) {
    const float d[3] = {(float)lat_e<19>(io, 0), (float)lat_e<19>(io, 1), (float)lat_e<19>(io, 2)};
    const float w = (float)lat_w<19>(io);
    const float rf = s.drf + A.rho0, rff = s.drff + A.rho0;
    const float irf = 1.0f / rf, irff = 1.0f / rff;
    float uf[3], uff[3], us[3], ud[3];
#pragma unroll
    for (int a = 0; a < 3; a++) {
        uf[a] = (s.mf[a] - 0.5f * A.F[a]) * irf;
        uff[a] = (s.mff[a] - 0.5f * A.F[a]) * irff;
    }
    const float geqf = geq_f(d[0], d[1], d[2], w, s.drf, rf, uf[0], uf[1], uf[2]);
    const float geqff = geq_f(d[0], d[1], d[2], w, s.drff, rff, uff[0], uff[1], uff[2]);
    const float q2 = q * 2.0f, one_m2q = 1.0f - q2;
    const float fneq = q2 * (s.gf - geqf) + one_m2q * (s.gff - geqff);  // Eq. (21)
    const bool near = q <= 0.5f;                                        // Eqs. (22)-(23)
    const float c_f = near ? q2 : (1.0f - q) / q;  // u* = c_f u_f + c_ff u_ff, u_w = 0
    const float c_ff = near ? one_m2q : 0.0f;
    const float drd = near ? q2 * s.drf + one_m2q * s.drff : s.drf;
    const float b = (1.0f - q) / (1.0f + q);  // Eq. (24), u_w = 0
#pragma unroll
    for (int a = 0; a < 3; a++) {
        us[a] = c_f * uf[a] + c_ff * uff[a];
        ud[a] = (us[a] + 2.0f * (b * uff[a])) * (1.0f / 3.0f);  // Eq. (25)
    }
    const float rd = drd + A.rho0;
    const float val = geq_f(d[0], d[1], d[2], w, drd, rd, ud[0], ud[1], ud[2]) + fneq;  // Eqs. (20), (19)
    if (kGrad) {
        float gd_dr, gd_u[3], gf_dr, gf_u[3], gff_dr, gff_u[3];
        geq_grad(d, w, rd, ud, gd_dr, gd_u);
        geq_grad(d, w, rf, uf, gf_dr, gf_u);
        geq_grad(d, w, rff, uff, gff_dr, gff_u);
        const float iq = 1.0f / q, i1q = 1.0f / (1.0f + q);
        float uf_b[3], uff_b[3], q_b = 2.0f * (s.gf - geqf) - 2.0f * (s.gff - geqff), su_f = 0.f, su_ff = 0.f;
        float du = 0.f, bu = 0.f;
#pragma unroll
        for (int a = 0; a < 3; a++) {
            const float us_b = gd_u[a] * (1.0f / 3.0f);
            uf_b[a] = c_f * us_b - q2 * gf_u[a];
            uff_b[a] = (c_ff + 2.0f * b) * us_b - one_m2q * gff_u[a];
            su_f += uf[a] * uf_b[a];
            su_ff += uff[a] * uff_b[a];
            // u* by q: 2 (u_f - u_ff), or -u_f / q^2
            du += us_b * (near ? 2.0f * (uf[a] - uff[a]) : -iq * iq * uf[a]);
            bu += us_b * uff[a];
        }
        q_b += du - 4.0f * i1q * i1q * bu;  // db/dq = -2 / (1 + q)^2
        if (near) q_b += 2.0f * (s.drf - s.drff) * gd_dr;
        g.q = q_b;
        g.f.x = (near ? q2 : 1.0f) * gd_dr - q2 * gf_dr - su_f * irf;
        g.f.y = uf_b[0] * irf;
        g.f.z = uf_b[1] * irf;
        g.f.w = uf_b[2] * irf;
        g.ff.x = c_ff * gd_dr - one_m2q * gff_dr - su_ff * irff;
        g.ff.y = uff_b[0] * irff;
        g.ff.z = uff_b[1] * irff;
        g.ff.w = uff_b[2] * irff;
    }
    return val;
}

// Population i of an array of 19 (its offset is the same for all threads).
// Within it the span kernels address by 32-bit byte offsets, which the load
// and store units add to the base themselves; boxes of 2^30 nodes and more
// (kWide) by 64-bit ones.
template <typename T, bool kWide>
struct Pop {
    T *base;
    __device__ __forceinline__ T &operator[](unsigned n) const {
        return kWide ? base[n] : *reinterpret_cast<T *>((uintptr_t)base + (size_t)(n * 4u));
    }
};
template <bool kWide = true, typename T>
__device__ __forceinline__ Pop<T, kWide> pop(T *p, const AdjConst &A, int i) {
    return Pop<T, kWide>{p + (long long)i * A.N};
}

// ---------------------------------------------------------------------------
// device data
// ---------------------------------------------------------------------------
// Node kinds: a fluid node with links and a solid node are left out of the
// span kernels; kShared marks the others that are some link's x_ff (the
// adjoint adds the link's shares there).
enum NodeKind : uint8_t { kPlain = 0, kLeftOut = 1, kShared = 2 };

struct AdjDev {
    AdjConst c;
    const uint8_t *kind;      // [N] NodeKind
    // fluid nodes with links: node, link directions (the unknowns), first link
    const int *n_node, *n_base;
    const uint32_t *n_mask;
    int nnodes;
    const int *l_nf, *l_dir, *l_nff;  // [L] node, direction (unknown), x_ff node or -1; a node's links in
                                      // direction order
    float *l_q;               // [L]
    double *l_dqdMf, *l_dqdMs;  // [L] dq/dM at x_f and x_s (0 where q was clamped)
    double *l_dJdq;           // [L]
    int nlinks;
    const double *cp;         // [ncp][3] world
    const double *K;          // [ncp]
    int ncp;
    unsigned long long *J_fix;  // sum of the window's drag (2^-40 units)
    double *grad;             // [ncp][4]: dJ/dx, dJ/dy, dJ/dz, dJ/dK
    float inv_W;
    StepGate gate;
};
// What a forward step keeps for the adjoint (mom NULL: nothing).
struct Kept {
    float4 *mom;              // [N] density offset and momentum of the pulled values
    float4 *l_f, *l_ff;       // [L] LinkGrad
    float *l_gq;              // [L]
};

__device__ __forceinline__ int wrapi(int v, int n) { return v < 0 ? v + n : (v >= n ? v - n : v); }

// The rows next to node (x, y, z): nx (y' + ny z') and x' for offsets -1, 0, 1.
struct Around {
    int xs[3], row[3][3];
};
__device__ __forceinline__ Around around(const AdjConst &A, int n) {
    const int z = (int)fast_quot((uint32_t)n, A.by_nxy), r = n - z * A.nx * A.ny;
    const int y = (int)fast_quot((uint32_t)r, A.by_nx), x = r - y * A.nx;
    Around o;
    int ys[3], zs[3];
#pragma unroll
    for (int k = 0; k < 3; k++) {
        o.xs[k] = wrapi(x + k - 1, A.nx);
        ys[k] = wrapi(y + k - 1, A.ny);
        zs[k] = wrapi(z + k - 1, A.nz);
    }
#pragma unroll
    for (int b = 0; b < 3; b++)
#pragma unroll
        for (int c = 0; c < 3; c++) o.row[b][c] = A.nx * (ys[b] + A.ny * zs[c]);
    return o;
}
// node n - e_i
__device__ __forceinline__ int upstream(const Around &o, int i) {
    return o.xs[1 - L19::e(i, 0)] + o.row[1 - L19::e(i, 1)][1 - L19::e(i, 2)];
}

// The 256-node span of a block; every other launch runs through the lattice
// from its end, so that it starts with what the launch before touched last
// (two states and the adjoint of a 96^3 box are about the size of L2).
__device__ __forceinline__ int span_node(bool reverse) {
    const unsigned b = reverse ? gridDim.x - 1 - blockIdx.x : blockIdx.x;
    return (int)(b * 256u + threadIdx.x);
}

__global__ void __launch_bounds__(256) k_adj_init(AdjDev D, float *S, float ux, float uy, float uz) {
    for (long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x; n < D.c.N; n += (long long)gridDim.x * blockDim.x)
#pragma unroll
        for (int i = 0; i < Q; i++)
            S[(long long)i * D.c.N + n] = geq_f((float)L19::e(i, 0), (float)L19::e(i, 1), (float)L19::e(i, 2),
                                                (float)L19::w(i), 0.f, D.c.rho0, ux, uy, uz);
}

// q of every link for the control points of this forward run (Eq. (27) with
// M of Eq. (4), FP64, periodic minimum image), and dq/dM for the gradient.
__global__ void k_adj_q(AdjDev D) {
    const AdjConst &A = D.c;
    for (int L = blockIdx.x * blockDim.x + threadIdx.x; L < D.nlinks; L += gridDim.x * blockDim.x) {
        const long long n = D.l_nf[L];
        const int io = L19::opp(D.l_dir[L]);
        const int x = (int)(n % A.nx), y = (int)((n / A.nx) % A.ny), z = (int)(n / ((long long)A.nx * A.ny));
        const double pf[3] = {(double)x, (double)y, (double)z};
        const double ps[3] = {pf[0] + lat_e<19>(io, 0), pf[1] + lat_e<19>(io, 1), pf[2] + lat_e<19>(io, 2)};
        const int dims[3] = {A.nx, A.ny, A.nz};
        double Mf = 0.0, Ms = 0.0;
        for (int c = 0; c < D.ncp; c++) {
            double rf2 = 0.0, rs2 = 0.0;
            for (int a = 0; a < 3; a++) {
                double df = pf[a] - D.cp[3 * c + a], ds = ps[a] - D.cp[3 * c + a];
                df -= dims[a] * rint(df / dims[a]);
                ds -= dims[a] * rint(ds / dims[a]);
                rf2 += df * df;
                rs2 += ds * ds;
            }
            Mf += D.K[c] / rf2;
            Ms += D.K[c] / rs2;
        }
        const double den = Ms - Mf;
        double q = (1.0 - Mf) / den;  // c0 = 1 (Eq. (26) with the surface of Eq. (4))
        double dqf = (1.0 - Ms) / (den * den), dqs = -(1.0 - Mf) / (den * den);
        if (!(q > 0.0)) { q = 0.0; dqf = dqs = 0.0; }
        if (q > 1.0) { q = 1.0; dqf = dqs = 0.0; }
        D.l_q[L] = (float)q;
        D.l_dqdMf[L] = dqf;
        D.l_dqdMs[L] = dqs;
    }
}

// The collided population along e, less (1 - omega) times the pulled one:
// omega g^eq + Guo's term (Eqs. (15)-(16), Eq. (18)'s half-force shift).  The
// roundings are spelled out: over hundreds of steps another order of them
// drifts the drag by 1e-5 (sharing the even parts of opposite directions, as
// collide_values does, would too).
template <bool kForce>
__device__ __forceinline__ float collide_h(const AdjConst &A, float w, float eu, float uu, float eF, float uF,
                                           float drho, float rho) {
    const float p = __fmaf_rn(-uu, 1.5f, __fmaf_rn(eu, 3.0f, __fmul_rn(__fmul_rn(eu, eu), 4.5f)));
    const float g = __fmul_rn(__fmaf_rn(rho, p, drho), w);
    if (!kForce) return __fmul_rn(g, A.omega);
    const float t = __fmaf_rn(__fsub_rn(eF, uF), 3.0f, __fmul_rn(eu, __fmul_rn(9.0f, eF)));
    return __fmaf_rn(t, __fmul_rn(A.gfac, w), __fmul_rn(g, A.omega));
}

// Collision of the pulled values: the new populations of node n, and its
// moments for the adjoint.
template <bool kForce, bool kWide>
__device__ __forceinline__ void adj_collide(const AdjConst &A, const float (&g)[Q], int n, float *R, float4 *mom) {
    float drho = 0.f, mx = 0.f, my = 0.f, mz = 0.f;
#pragma unroll
    for (int i = 0; i < Q; i++) {
        drho += g[i];
        mx = add_e(mx, L19::e(i, 0), g[i]);
        my = add_e(my, L19::e(i, 1), g[i]);
        mz = add_e(mz, L19::e(i, 2), g[i]);
    }
    if (mom) __stcs(&mom[n], make_float4(drho, mx, my, mz));
    const float rho = drho + A.rho0, ir = 1.0f / rho;
    const float ux = (kForce ? __fmaf_rn(0.5f, A.F[0], mx) : mx) * ir, uy = (kForce ? __fmaf_rn(0.5f, A.F[1], my) : my) * ir,
                uz = (kForce ? __fmaf_rn(0.5f, A.F[2], mz) : mz) * ir;
    const float uu = __fmaf_rn(uz, uz, __fmaf_rn(ux, ux, __fmul_rn(uy, uy)));
    const float uF = kForce ? __fmaf_rn(uz, A.F[2], __fmaf_rn(ux, A.F[0], __fmul_rn(uy, A.F[1]))) : 0.f;
    const float om1 = 1.0f - A.omega;
    pop<kWide>(R, A, 0)[(unsigned)n] =
        __fmaf_rn(om1, g[0], collide_h<kForce>(A, (float)L19::w(0), 0.f, uu, 0.f, uF, drho, rho));
#pragma unroll
    for (int i = 1; i < Q; i += 2) {
        const int ex = L19::e(i, 0), ey = L19::e(i, 1), ez = L19::e(i, 2);
        const float eu = dot_e(ex, ey, ez, ux, uy, uz);
        const float eF = kForce ? dot_e(ex, ey, ez, A.F[0], A.F[1], A.F[2]) : 0.f;
        const float w = (float)L19::w(i);
        pop<kWide>(R, A, i)[(unsigned)n] = __fmaf_rn(om1, g[i], collide_h<kForce>(A, w, eu, uu, eF, uF, drho, rho));
        pop<kWide>(R, A, i + 1)[(unsigned)n] = __fmaf_rn(om1, g[i + 1], collide_h<kForce>(A, w, -eu, uu, -eF, uF, drho, rho));
    }
}

// Forward step S -> R, the nodes without links.  (S is not __restrict__: the
// kernel is up before the step before has written it, which the read-only path
// does not allow.)  Four CTAs per SM: with five and six (48 and 40 registers)
// the pulled values are spilled; 96^3 at 4 / 5 / 6: 28.1, 28.9, 31.6 us a step.
template <bool kForce, bool kWide>
__global__ void __launch_bounds__(256, 4) k_adj_step(AdjDev D, const float *S, float *R, Kept kept, int reverse) {
    pdl_wait();
    gate_open(D.gate);
    const AdjConst &A = D.c;
    const int n = span_node(reverse != 0);
    if (n < A.N) {
        const bool take = D.kind[n] != kLeftOut;
        const Around o = around(A, n);
        float gin[Q];
#pragma unroll
        for (int i = 0; i < Q; i++) gin[i] = pop<kWide>(S, A, i)[(unsigned)upstream(o, i)];
        if (take) adj_collide<kForce, kWide>(A, gin, n, R, kept.mom);
    }
}

// Forward step S -> R, the nodes with links: a warp takes kLinkNodes of them,
// its lanes evaluate their links (both nodes' populations in one round of
// loads), then each node takes its links' values, pulls the rest and collides.
// The drag of a step in the window is Eq. (28)'s x component over the links,
// in fixed point (exact in any order).
constexpr int kLinkNodes = 4;
template <bool kForce>
__global__ void __launch_bounds__(256, 2) k_adj_step_links(AdjDev D, const float *S, float *R, Kept kept, int window) {
    __shared__ unsigned short s_ent[8][kLinkNodes * 18];
    __shared__ float s_val[8][kLinkNodes * 18];
    pdl_launch_dependents();
    const AdjConst &A = D.c;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int w0 = (blockIdx.x * 8 + warp) * kLinkNodes;
    // (the node list is lbm_adj_init's: read before the gate)
    const bool has = lane < kLinkNodes && w0 + lane < D.nnodes;
    const int n = has ? D.n_node[w0 + lane] : 0, base = has ? D.n_base[w0 + lane] : 0;
    const uint32_t lm = has ? D.n_mask[w0 + lane] : 0u;
    gate_pass(D.gate);
    if (w0 >= D.nnodes) {
        pdl_wait();
        return;
    }
    const int first_link = __shfl_sync(0xffffffffu, base, 0);
    const int first = base - first_link;  // the nodes' links follow one another
    int total = __popc(lm);
#pragma unroll
    for (int o = 1; o < kLinkNodes; o <<= 1) total += __shfl_xor_sync(0xffffffffu, total, o);
    total = __shfl_sync(0xffffffffu, total, 0);
    uint32_t m = lm;
    for (int k = first; m; k++) {
        const int i = __ffs(m) - 1;
        m &= m - 1;
        s_ent[warp][k] = (unsigned short)((lane << 5) | i);
    }
    __syncwarp();
    long long drag = 0;
    for (int r = 0; r < total; r += 32) {
        const int e = r + lane;
        const int ent = e < total ? s_ent[warp][e] : 0;
        const int nf = __shfl_sync(0xffffffffu, n, ent >> 5);
        if (e < total) {
            const int L = first_link + e, i = ent & 31, io = L19::opp(i);
            const int nff = D.l_nff[L];
            const int at = nff < 0 ? nf : nff;
            const float q = D.l_q[L];
            LinkState s = {};
#pragma unroll
            for (int k = 0; k < Q; k++) {
                const float a = pop(S, A, k)[(unsigned)nf], b = pop(S, A, k)[(unsigned)at];
                s.drf += a;
                s.drff += b;
                s.mf[0] = add_e(s.mf[0], L19::e(k, 0), a);
                s.mf[1] = add_e(s.mf[1], L19::e(k, 1), a);
                s.mf[2] = add_e(s.mf[2], L19::e(k, 2), a);
                s.mff[0] = add_e(s.mff[0], L19::e(k, 0), b);
                s.mff[1] = add_e(s.mff[1], L19::e(k, 1), b);
                s.mff[2] = add_e(s.mff[2], L19::e(k, 2), b);
                if (k == io) {
                    s.gf = a;
                    s.gff = b;
                }
            }
            float v = s.gf;  // halfway bounce-back, u_w = 0
            if (nff >= 0) {
                LinkGrad g;
                if (kept.mom) {
                    v = vibb_f<true>(A, io, q, s, g);
                    kept.l_f[L] = g.f;
                    kept.l_ff[L] = g.ff;
                    kept.l_gq[L] = g.q;
                } else {
                    v = vibb_f<false>(A, io, q, s, g);
                }
            }
            s_val[warp][e] = v;
            if (window) {
                const float dx = (float)lat_e<19>(io, 0);
                drag += __float2ll_rn(dx * (s.gf + v) * (float)(1ull << kForceFixBits));
            }
        }
    }
    __syncwarp();
    if (has) {
        const Around o = around(A, n);
        float gin[Q];
        int k = first;
#pragma unroll
        for (int i = 0; i < Q; i++) {
            if ((lm >> i) & 1u) gin[i] = s_val[warp][k++];
            else gin[i] = pop(S, A, i)[(unsigned)upstream(o, i)];
        }
        adj_collide<kForce, true>(A, gin, n, R, kept.mom);
    }
    if (window) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) drag += __shfl_xor_sync(0xffffffffu, drag, o);
        if (lane == 0 && drag) atomicAdd(D.J_fix, (unsigned long long)drag);
    }
    pdl_wait();
}

// ---------------------------------------------------------------------------
// adjoint step
// ---------------------------------------------------------------------------
// a = sum_i lambda_i dh_i/d(drho), b = sum_i lambda_i dh_i/dm for the part h_i
// of the collided population i that depends on the pulled values through
// their density offset and momentum (omega g^eq_i + Guo's term, u = (m + F/2)
// / rho), differentiated by hand: with P_i = 3 e.u + 4.5 (e.u)^2 - 1.5 u.u,
//   dh_i/d(drho) at fixed u = omega w_i (1 + P_i),
//   dh_i/du = omega w_i rho (3 e_i + 9 (e_i.u) e_i - 3 u)
//             + gfac w_i (9 (e_i.F) e_i - 3 F),
// and du/dm = I / rho, du/d(drho) = -u / rho.  The sums over the directions,
// with S = w_i (lambda_i + lambda_i') and D = w_i (lambda_i - lambda_i') of a
// pair of opposite ones:
//   sl = sum S, p = sum (3 e.u D + 4.5 (e.u)^2 S),
//   V = sum e (omega rho (3 D + 9 e.u S) + 9 gfac e.F S).
struct BackSums {
    float sl, p, V[3];
};
// the terms of one pair (S, D) along e
template <bool kForce>
__device__ __forceinline__ void back_pair(const AdjConst &A, float S, float D, float eu, float eFg, float om_rho,
                                          float &sl, float &p, float &t) {
    const float seu = S * eu;
    sl += S;
    p += eu * (3.0f * D + 4.5f * seu);
    t = om_rho * (3.0f * D + 9.0f * seu);
    if (kForce) t += 9.0f * eFg * S;
}
__device__ __forceinline__ float4 back_ab(const AdjConst &A, const BackSums &s, float om_rho, float ir,
                                          const float u[3]) {
    const float uu = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
    float b[3], gu = 0.f;
#pragma unroll
    for (int c = 0; c < 3; c++) {
        const float g = s.V[c] - 3.0f * s.sl * (om_rho * u[c] + A.Fg[c]);
        b[c] = g * ir;
        gu += g * u[c];
    }
    return make_float4(A.omega * (s.sl * (1.0f - 1.5f * uu) + s.p) - gu * ir, b[0], b[1], b[2]);
}

// Adjoint step lamN -> lamT, the nodes without links: every neighbour is
// fluid, so lambda_in goes to all of them.  share/share_next: the density and
// momentum shares that this step's reader adds (and clears for the step after
// the next) and that the link kernel sums for the next step.
// Four CTAs per SM: 96^3 at 3 / 4: 33.6, 31.2 us a step.
template <bool kForce, bool kWide>
__global__ void __launch_bounds__(256, 4) k_adj_back(AdjDev D, const float4 *mom, const float *lamN, float *lamT,
                                                      float4 *share, int reverse) {
    pdl_wait();
    gate_open(D.gate);
    const AdjConst &A = D.c;
    const int n = span_node(reverse != 0);
    if (n < A.N) {
        const uint8_t kind = D.kind[n];
        const float4 mo = __ldcs(&mom[n]);
        float lam[Q];
#pragma unroll
        for (int i = 0; i < Q; i++) lam[i] = pop<kWide>(lamN, A, i)[(unsigned)n];
        if (kind != kLeftOut) {
            if (kind == kShared) {
                const float4 x = share[n];
                share[n] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                for (int i = 0; i < Q; i++)
                    lam[i] = add_e(add_e(add_e(lam[i] + x.x, L19::e(i, 0), x.y), L19::e(i, 1), x.z), L19::e(i, 2), x.w);
            }
            const float rho = mo.x + A.rho0, ir = 1.0f / rho, om_rho = A.omega * rho;
            const float u[3] = {(mo.y + 0.5f * A.F[0]) * ir, (mo.z + 0.5f * A.F[1]) * ir, (mo.w + 0.5f * A.F[2]) * ir};
            BackSums s = {};
            s.sl = (float)L19::w(0) * lam[0];
#pragma unroll
            for (int i = 1; i < Q; i += 2) {
                const int ex = L19::e(i, 0), ey = L19::e(i, 1), ez = L19::e(i, 2);
                const float w = (float)L19::w(i);
                float t;
                back_pair<kForce>(A, w * (lam[i] + lam[i + 1]), w * (lam[i] - lam[i + 1]),
                                  dot_e(ex, ey, ez, u[0], u[1], u[2]), dot_e(ex, ey, ez, A.Fg[0], A.Fg[1], A.Fg[2]),
                                  om_rho, s.sl, s.p, t);
                s.V[0] = add_e(s.V[0], ex, t);
                s.V[1] = add_e(s.V[1], ey, t);
                s.V[2] = add_e(s.V[2], ez, t);
            }
            const float4 ab = back_ab(A, s, om_rho, ir, u);
            const float om1 = 1.0f - A.omega;
            const Around o = around(A, n);
            pop<kWide>(lamT, A, 0)[(unsigned)n] = om1 * lam[0] + ab.x;
#pragma unroll
            for (int j = 1; j < Q; j += 2) {
                const float eb = dot_e(L19::e(j, 0), L19::e(j, 1), L19::e(j, 2), ab.y, ab.z, ab.w);
                pop<kWide>(lamT, A, j)[(unsigned)upstream(o, j)] = om1 * lam[j] + (ab.x + eb);
                pop<kWide>(lamT, A, j + 1)[(unsigned)upstream(o, j + 1)] = om1 * lam[j + 1] + (ab.x - eb);
            }
        }
    }
}

// Adjoint step, the nodes with links: one warp per node, lane i its direction
// i, so a node's links and their kept derivatives are read in one round.
__global__ void __launch_bounds__(256) k_adj_back_links(AdjDev D, Kept kept, const float *lamN, float *lamT,
                                                         float4 *share, float4 *share_next, int window) {
    pdl_launch_dependents();
    const AdjConst &A = D.c;
    const int lane = threadIdx.x & 31;
    const int w = blockIdx.x * 8 + (threadIdx.x >> 5);
    // (the node list and the links are lbm_adj_init's, q the forward call's:
    // read before the gate)
    const bool has = w < D.nnodes;
    const int n = has ? D.n_node[w] : 0, base = has ? D.n_base[w] : 0;
    const uint32_t lm = has ? D.n_mask[w] : 0u;
    const bool dir = lane < Q;
    const bool link = dir && ((lm >> lane) & 1u);
    const int L = base + __popc(lm & ((1u << lane) - 1u));
    const int nff = link ? D.l_nff[L] : -1;
    const float q = link ? D.l_q[L] : 0.f;
    gate_pass(D.gate);
    if (!has) {
        pdl_wait();
        return;
    }
    const int ei[3] = {dir ? lat_e<19>(lane, 0) : 0, dir ? lat_e<19>(lane, 1) : 0, dir ? lat_e<19>(lane, 2) : 0};
    const float ex = (float)ei[0], ey = (float)ei[1], ez = (float)ei[2];
    const float wi = dir ? (float)lat_w<19>(lane) : 0.f;
    const float4 mo = kept.mom[n];
    const float4 x = share[n];
    float lam = dir ? lamN[(long long)lane * A.N + n] : 0.f;
    float gq = 0.f;
    float4 gf = make_float4(0.f, 0.f, 0.f, 0.f), gff = gf;
    if (link) {
        gq = kept.l_gq[L];
        gf = kept.l_f[L];
        gff = kept.l_ff[L];
    }
    __syncwarp();
    if (lane == 0) share[n] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (dir) lam += x.x + ex * x.y + ey * x.z + ez * x.w;
    const float rho = mo.x + A.rho0, ir = 1.0f / rho, om_rho = A.omega * rho;
    const float u[3] = {(mo.y + 0.5f * A.F[0]) * ir, (mo.z + 0.5f * A.F[1]) * ir, (mo.w + 0.5f * A.F[2]) * ir};
    // a lane's direction by itself: S = D = w_i lambda_i
    BackSums s = {};
    float t;
    back_pair<true>(A, wi * lam, wi * lam, u[0] * ex + u[1] * ey + u[2] * ez, A.Fg[0] * ex + A.Fg[1] * ey + A.Fg[2] * ez,
                    om_rho, s.sl, s.p, t);
    s.V[0] = ex * t;
    s.V[1] = ey * t;
    s.V[2] = ez * t;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        s.sl += __shfl_xor_sync(0xffffffffu, s.sl, o);
        s.p += __shfl_xor_sync(0xffffffffu, s.p, o);
#pragma unroll
        for (int c = 0; c < 3; c++) s.V[c] += __shfl_xor_sync(0xffffffffu, s.V[c], o);
    }
    const float4 ab = back_ab(A, s, om_rho, ir, u);
    float v = (1.0f - A.omega) * lam + ab.x + ab.y * ex + ab.z * ey + ab.w * ez;
    // the drag's x component of a link along its opposite direction: -e_x
    if (link && window) v -= D.inv_W * ex;
    const bool vibb = link && nff >= 0;
    // the share of x_ff's single population goes with this node's push along
    // the link's opposite direction
    const float vff = vibb ? v * (1.0f - 2.0f * q) : 0.f;
    const int io = lane == 0 ? 0 : ((lane & 1) ? lane + 1 : lane - 1);
    const float from = __shfl_sync(0xffffffffu, vff, io & 31);
    if (link) {
        // dJ/dg+(t) of this node's own opposite population: the halfway
        // link's value, or the VIBB share 2q, and the drag's dependence on it
        float acc = nff < 0 ? v : v * (2.0f * q);
        if (window) acc -= D.inv_W * ex;
        lamT[(long long)io * A.N + n] = acc;
    } else if (dir) {
        const int z = (int)fast_quot((uint32_t)n, A.by_nxy), r = n - z * A.nx * A.ny;
        const int y = (int)fast_quot((uint32_t)r, A.by_nx), xx = r - y * A.nx;
        const int t = wrapi(xx - ei[0], A.nx) + A.nx * (wrapi(y - ei[1], A.ny) + A.ny * wrapi(z - ei[2], A.nz));
        lamT[(long long)lane * A.N + t] = v + (lane > 0 ? from : 0.f);
    }
    float4 own = make_float4(0.f, 0.f, 0.f, 0.f);
    if (vibb) {
        D.l_dJdq[L] += (double)v * (double)gq;
        own = make_float4(v * gf.x, v * gf.y, v * gf.z, v * gf.w);
        atomicAdd(&share_next[nff], make_float4(v * gff.x, v * gff.y, v * gff.z, v * gff.w));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        own.x += __shfl_xor_sync(0xffffffffu, own.x, o);
        own.y += __shfl_xor_sync(0xffffffffu, own.y, o);
        own.z += __shfl_xor_sync(0xffffffffu, own.z, o);
        own.w += __shfl_xor_sync(0xffffffffu, own.w, o);
    }
    if (lane == 0) atomicAdd(&share_next[n], own);
    pdl_wait();
}

// dJ/dq -> dJ/d(control point position, weight) through Eq. (27) and Eq. (4).
__global__ void __launch_bounds__(256) k_adj_grad(AdjDev D) {
    __shared__ double sg[LBM_MAX_CP][4];
    const AdjConst &A = D.c;
    for (int k = threadIdx.x; k < D.ncp * 4; k += blockDim.x) sg[k / 4][k % 4] = 0.0;
    __syncthreads();
    const int dims[3] = {A.nx, A.ny, A.nz};
    for (int L = blockIdx.x * blockDim.x + threadIdx.x; L < D.nlinks; L += gridDim.x * blockDim.x) {
        const double G = D.l_dJdq[L];
        if (G == 0.0) continue;
        const double gf = G * D.l_dqdMf[L], gs = G * D.l_dqdMs[L];
        if (gf == 0.0 && gs == 0.0) continue;
        const long long n = D.l_nf[L];
        const int io = L19::opp(D.l_dir[L]);
        const double pf[3] = {(double)(n % A.nx), (double)((n / A.nx) % A.ny), (double)(n / ((long long)A.nx * A.ny))};
        const double ps[3] = {pf[0] + lat_e<19>(io, 0), pf[1] + lat_e<19>(io, 1), pf[2] + lat_e<19>(io, 2)};
        for (int c = 0; c < D.ncp; c++) {
            double rf[3], rs[3], rf2 = 0.0, rs2 = 0.0;
            for (int a = 0; a < 3; a++) {
                rf[a] = pf[a] - D.cp[3 * c + a];
                rs[a] = ps[a] - D.cp[3 * c + a];
                rf[a] -= dims[a] * rint(rf[a] / dims[a]);
                rs[a] -= dims[a] * rint(rs[a] / dims[a]);
                rf2 += rf[a] * rf[a];
                rs2 += rs[a] * rs[a];
            }
            // M = sum K / |x - x_c|^2:  dM/dK_c = 1/r^2,  dM/dx_c = 2 K_c (x - x_c) / r^4
            atomicAdd(&sg[c][3], gf / rf2 + gs / rs2);
            const double cf = gf * 2.0 * D.K[c] / (rf2 * rf2), cs = gs * 2.0 * D.K[c] / (rs2 * rs2);
            for (int a = 0; a < 3; a++) atomicAdd(&sg[c][a], cf * rf[a] + cs * rs[a]);
        }
    }
    __syncthreads();
    for (int k = threadIdx.x; k < D.ncp * 4; k += blockDim.x) atomicAdd(&D.grad[k], sg[k / 4][k % 4]);
}

}  // namespace

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
struct lbm_adj {
    lbm_config cfg;
    int T, W, K, C;          // steps, window, checkpoint interval, checkpoints
    bool keep_all;           // every step's kept data is held, else one segment's
    int ncp, nlinks, nnodes;
    long long N;
    size_t S;                // bytes of one state (19 N floats)
    size_t kept;             // bytes that one step keeps for the adjoint
    char *ws;
    cudaStream_t stream;
    size_t o_state[2], o_ckpt, o_kept, o_lam[2], o_share[2], o_kind, o_nnode, o_nbase, o_nmask, o_lnf, o_ldir, o_lnff,
        o_lq, o_dqf, o_dqs, o_dJdq, o_cp, o_K, o_J, o_grad, o_gate, total;
    unsigned gate_id;        // steps issued (the gate's numbers)
    bool have_forward;
    char err[256];
};

namespace {

thread_local char g_adj_error[256] = "no error";

int afail(lbm_adj *a, int code, const char *fmt, ...) {
    char *buf = a ? a->err : g_adj_error;
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, 256, fmt, ap);
    va_end(ap);
    return code;
}
int acheck(lbm_adj *a, cudaError_t e, const char *what) {
    if (e == cudaSuccess) return LBM_OK;
    return afail(a, LBM_ERR_CUDA, "%s: %s", what, cudaGetErrorString(e));
}

const char *adj_check(const lbm_config *c, const lbm_particle *p, int T, int W) {
    if (!c || !p) return "config or particle is NULL";
    if (c->nx < 4 || c->ny < 4 || c->nz < 4) return "nx, ny, nz must be >= 4";
    if ((long long)c->nx * c->ny * c->nz >= (1LL << 31)) return "lattice must hold fewer than 2^31 nodes";
    if (!c->periodic[0] || !c->periodic[1] || !c->periodic[2]) return "the adjoint needs a fully periodic box";
    if (c->lattice != 19) return "the adjoint runs D3Q19";
    if (!(c->tau > 0.5)) return "tau must be > 1/2";
    if (!(c->rho0 > 0.0)) return "rho0 must be > 0";
    if (c->c0 != 1.0 && c->c0 != 0.0) return "the adjoint takes the surface M = 1 (c0 = 1)";
    if (p->n_cp < 1 || p->n_cp > LBM_MAX_CP) return "n_cp out of range";
    if (T < 1 || W < 1 || W > T) return "need T >= 1 and 1 <= W <= T";
    return nullptr;
}

// World control points of the particle (x + R(q) cp).
void world_cps(const lbm_particle *p, std::vector<double> &cp) {
    double q[4] = {p->q[0], p->q[1], p->q[2], p->q[3]};
    const double qn = std::sqrt(q[0] * q[0] + q[1] * q[1] + q[2] * q[2] + q[3] * q[3]);
    for (double &v : q) v /= qn;
    const double w = q[0], x = q[1], y = q[2], z = q[3];
    const double R[9] = {1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                         2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                         2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)};
    cp.assign(3 * (size_t)p->n_cp, 0.0);
    for (int k = 0; k < p->n_cp; k++)
        for (int a = 0; a < 3; a++)
            cp[3 * k + a] = p->x[a] + R[3 * a] * p->cp[k][0] + R[3 * a + 1] * p->cp[k][1] + R[3 * a + 2] * p->cp[k][2];
}

// The node kinds from the frozen flags (M >= 1, periodic minimum image), the
// fluid nodes with links (node, directions, first link) and the links, in node
// then direction order.
struct Links {
    std::vector<uint8_t> kind;
    std::vector<int> node, base, nf, dir, nff;
    std::vector<uint32_t> mask;
};
void classify_links(const lbm_config *c, const lbm_particle *p, Links &k) {
    std::vector<uint8_t> solid;
    const int nx = c->nx, ny = c->ny, nz = c->nz;
    const long long N = (long long)nx * ny * nz;
    std::vector<double> cp;
    world_cps(p, cp);
    solid.assign((size_t)N, 0);
    const int dims[3] = {nx, ny, nz};
    for (int z = 0; z < nz; z++)
        for (int y = 0; y < ny; y++)
            for (int x = 0; x < nx; x++) {
                const double pt[3] = {(double)x, (double)y, (double)z};
                double M = 0.0;
                for (int k = 0; k < p->n_cp; k++) {
                    double r2 = 0.0;
                    for (int a = 0; a < 3; a++) {
                        double d = pt[a] - cp[3 * k + a];
                        d -= dims[a] * std::rint(d / dims[a]);
                        r2 += d * d;
                    }
                    M += p->K[k] / r2;
                }
                solid[x + (size_t)nx * (y + (size_t)ny * z)] = M >= 1.0;
            }
    k = Links();
    k.kind.assign((size_t)N, kPlain);
    auto wrap = [](int v, int n) { return v < 0 ? v + n : (v >= n ? v - n : v); };
    for (int z = 0; z < nz; z++)
        for (int y = 0; y < ny; y++)
            for (int x = 0; x < nx; x++) {
                const long long n = x + (long long)nx * (y + (long long)ny * z);
                if (solid[(size_t)n]) {
                    k.kind[(size_t)n] = kLeftOut;
                    continue;
                }
                uint32_t mask = 0;
                const int base = (int)k.nf.size();
                for (int i = 1; i < Q; i++) {
                    const int ex = L19::e(i, 0), ey = L19::e(i, 1), ez = L19::e(i, 2);
                    const long long s = wrap(x - ex, nx) + (long long)nx * (wrap(y - ey, ny) + (long long)ny * wrap(z - ez, nz));
                    if (!solid[(size_t)s]) continue;
                    const long long f2 = wrap(x + ex, nx) + (long long)nx * (wrap(y + ey, ny) + (long long)ny * wrap(z + ez, nz));
                    mask |= 1u << i;
                    k.nf.push_back((int)n);
                    k.dir.push_back(i);
                    k.nff.push_back(solid[(size_t)f2] ? -1 : (int)f2);
                }
                if (mask) {
                    k.kind[(size_t)n] = kLeftOut;
                    k.node.push_back((int)n);
                    k.base.push_back(base);
                    k.mask.push_back(mask);
                }
            }
    for (int f2 : k.nff)
        if (f2 >= 0 && k.kind[(size_t)f2] == kPlain) k.kind[(size_t)f2] = kShared;
}

// keep_all: room for every step's kept data (96^3: 14.5 MB a step), so that the
// adjoint runs no forward step again; else a state every ceil(sqrt(T)) steps
// and one segment's data.
void adj_layout(lbm_adj *a, bool keep_all) {
    size_t o = 0;
    a->keep_all = keep_all;
    auto take = [&](size_t bytes) {
        size_t at = o;
        o = align_up(o + bytes);
        return at;
    };
    const size_t L = (size_t)std::max(1, a->nlinks), N = (size_t)a->N, M = (size_t)std::max(1, a->nnodes);
    a->o_state[0] = take(a->S);
    a->o_state[1] = take(a->S);
    a->o_ckpt = take(a->keep_all ? 0 : a->S * (size_t)a->C);
    a->o_kept = take(a->kept * (size_t)(a->keep_all ? a->T : a->K));
    a->o_lam[0] = take(a->S);
    a->o_lam[1] = take(a->S);
    a->o_share[0] = take(N * 16);
    a->o_share[1] = take(N * 16);
    a->o_kind = take(N);
    a->o_nnode = take(M * 4);
    a->o_nbase = take(M * 4);
    a->o_nmask = take(M * 4);
    a->o_lnf = take(L * 4);
    a->o_ldir = take(L * 4);
    a->o_lnff = take(L * 4);
    a->o_lq = take(L * 4);
    a->o_dqf = take(L * 8);
    a->o_dqs = take(L * 8);
    a->o_dJdq = take(L * 8);
    a->o_cp = take((size_t)a->ncp * 24);
    a->o_K = take((size_t)a->ncp * 8);
    a->o_J = take(8);
    a->o_grad = take((size_t)a->ncp * 32);
    a->o_gate = take(4);
    a->total = o;
}

void adj_sizes(lbm_adj *a, const lbm_config *c, int T, int W, int ncp, const Links &k) {
    a->cfg = *c;
    a->T = T;
    a->W = W;
    a->K = std::max(1, (int)std::ceil(std::sqrt((double)T)));
    a->C = (T + a->K - 1) / a->K;
    a->ncp = ncp;
    a->nlinks = (int)k.nf.size();
    a->nnodes = (int)k.node.size();
    a->N = (long long)c->nx * c->ny * c->nz;
    a->S = align_up((size_t)Q * (size_t)a->N * 4);
    const size_t L = (size_t)std::max(1, a->nlinks);
    a->kept = align_up((size_t)a->N * 16) + 2 * align_up(L * 16) + align_up(L * 4);
}

AdjDev adj_dev(lbm_adj *a) {
    AdjDev D;
    const lbm_config &c = a->cfg;
    D.c.nx = c.nx; D.c.ny = c.ny; D.c.nz = c.nz; D.c.N = a->N;
    D.c.rho0 = (float)c.rho0;
    D.c.omega = (float)(1.0 / c.tau);
    D.c.gfac = (float)(1.0 - 0.5 / c.tau);
    for (int k = 0; k < 3; k++) {
        D.c.F[k] = (float)c.force[k];
        D.c.Fg[k] = D.c.gfac * D.c.F[k];
    }
    D.c.by_nxy = fast_div((uint32_t)(c.nx * c.ny));
    D.c.by_nx = fast_div((uint32_t)c.nx);
    char *w = a->ws;
    D.kind = reinterpret_cast<const uint8_t *>(w + a->o_kind);
    D.n_node = reinterpret_cast<const int *>(w + a->o_nnode);
    D.n_base = reinterpret_cast<const int *>(w + a->o_nbase);
    D.n_mask = reinterpret_cast<const uint32_t *>(w + a->o_nmask);
    D.nnodes = a->nnodes;
    D.l_nf = reinterpret_cast<const int *>(w + a->o_lnf);
    D.l_dir = reinterpret_cast<const int *>(w + a->o_ldir);
    D.l_nff = reinterpret_cast<const int *>(w + a->o_lnff);
    D.l_q = reinterpret_cast<float *>(w + a->o_lq);
    D.l_dqdMf = reinterpret_cast<double *>(w + a->o_dqf);
    D.l_dqdMs = reinterpret_cast<double *>(w + a->o_dqs);
    D.l_dJdq = reinterpret_cast<double *>(w + a->o_dJdq);
    D.nlinks = a->nlinks;
    D.cp = reinterpret_cast<const double *>(w + a->o_cp);
    D.K = reinterpret_cast<const double *>(w + a->o_K);
    D.ncp = a->ncp;
    D.J_fix = reinterpret_cast<unsigned long long *>(w + a->o_J);
    D.grad = reinterpret_cast<double *>(w + a->o_grad);
    D.inv_W = 1.0f / (float)a->W;
    D.gate.word = reinterpret_cast<unsigned *>(w + a->o_gate);
    D.gate.id = 0;  // set per step
    return D;
}

Kept kept_slot(lbm_adj *a, int slot) {
    char *p = a->ws + a->o_kept + a->kept * (size_t)slot;
    const size_t L = (size_t)std::max(1, a->nlinks);
    Kept k;
    k.mom = reinterpret_cast<float4 *>(p);
    p += align_up((size_t)a->N * 16);
    k.l_f = reinterpret_cast<float4 *>(p);
    p += align_up(L * 16);
    k.l_ff = reinterpret_cast<float4 *>(p);
    p += align_up(L * 16);
    k.l_gq = reinterpret_cast<float *>(p);
    return k;
}

float *state(lbm_adj *a, size_t off) { return reinterpret_cast<float *>(a->ws + off); }

unsigned span_grid(const lbm_adj *a) { return (unsigned)((a->N + 255) / 256); }

// The link kernels run with no link node too: their completion stands for the
// step's.
unsigned link_grid(const lbm_adj *a, int per_block) {
    return (unsigned)std::max(1, (a->nnodes + per_block - 1) / per_block);
}

// One forward step S -> R on the stream, one adjoint step lamN -> lamT.
template <bool kForce, bool kWide>
void forward_step_t(lbm_adj *a, const AdjDev &D, const float *S, float *R, const Kept &kept, int window, int t) {
    launch_pdl(k_adj_step<kForce, kWide>, dim3(span_grid(a)), 256, a->stream, D, S, R, kept, t & 1);
    launch_pdl(k_adj_step_links<kForce>, dim3(link_grid(a, 8 * kLinkNodes)), 256, a->stream, D, S, R, kept, window);
}
template <bool kForce, bool kWide>
void adjoint_step_t(lbm_adj *a, const AdjDev &D, const Kept &kept, const float *lamN, float *lamT, float4 *share,
                    float4 *share_next, int window, int t) {
    launch_pdl(k_adj_back<kForce, kWide>, dim3(span_grid(a)), 256, a->stream, D, kept.mom, lamN, lamT, share, t & 1);
    launch_pdl(k_adj_back_links, dim3(link_grid(a, 8)), 256, a->stream, D, kept, lamN, lamT, share, share_next, window);
}
template <typename... X>
void forward_step(lbm_adj *a, AdjDev D, const X &...x) {
    D.gate.id = ++a->gate_id;
    const bool force = a->cfg.force[0] != 0.0 || a->cfg.force[1] != 0.0 || a->cfg.force[2] != 0.0;
    const bool wide = a->N >= (1ll << 30);
    if (wide) force ? forward_step_t<true, true>(a, D, x...) : forward_step_t<false, true>(a, D, x...);
    else force ? forward_step_t<true, false>(a, D, x...) : forward_step_t<false, false>(a, D, x...);
}
template <typename... X>
void adjoint_step(lbm_adj *a, AdjDev D, const X &...x) {
    D.gate.id = ++a->gate_id;
    const bool force = a->cfg.force[0] != 0.0 || a->cfg.force[1] != 0.0 || a->cfg.force[2] != 0.0;
    const bool wide = a->N >= (1ll << 30);
    if (wide) force ? adjoint_step_t<true, true>(a, D, x...) : adjoint_step_t<false, true>(a, D, x...);
    else force ? adjoint_step_t<true, false>(a, D, x...) : adjoint_step_t<false, false>(a, D, x...);
}

}  // namespace

extern "C" {

int lbm_adj_workspace_sizes(const lbm_config *cfg, const lbm_particle *p, int T, int W, size_t *least, size_t *keep) {
    if (const char *m = adj_check(cfg, p, T, W)) return afail(nullptr, LBM_ERR_BAD_ARG, "%s", m);
    if (!least || !keep) return afail(nullptr, LBM_ERR_BAD_ARG, "least or keep is NULL");
    Links k;
    classify_links(cfg, p, k);
    lbm_adj a;
    adj_sizes(&a, cfg, T, W, p->n_cp, k);
    adj_layout(&a, true);
    *keep = a.total;
    adj_layout(&a, false);
    *least = std::min(a.total, *keep);  // (a short run's steps may take less than its checkpoints)
    return LBM_OK;
}

int lbm_adj_workspace_size(const lbm_config *cfg, const lbm_particle *p, int T, int W, size_t *bytes) {
    size_t keep;
    if (!bytes) return afail(nullptr, LBM_ERR_BAD_ARG, "bytes is NULL");
    return lbm_adj_workspace_sizes(cfg, p, T, W, bytes, &keep);
}

int lbm_adj_init(const lbm_config *cfg, const lbm_particle *p, int T, int W, void *dev_ws, size_t ws_bytes,
                 void *cuda_stream, lbm_adj **out) {
    if (!out) return afail(nullptr, LBM_ERR_BAD_ARG, "out is NULL");
    *out = nullptr;
    if (const char *m = adj_check(cfg, p, T, W)) return afail(nullptr, LBM_ERR_BAD_ARG, "%s", m);
    if (!dev_ws || reinterpret_cast<uintptr_t>(dev_ws) % kAlign)
        return afail(nullptr, LBM_ERR_BAD_ARG, "workspace NULL or not 256-byte aligned");
    Links k;
    classify_links(cfg, p, k);
    lbm_adj *a = new (std::nothrow) lbm_adj();
    if (!a) return afail(nullptr, LBM_ERR_BAD_ARG, "out of host memory");
    adj_sizes(a, cfg, T, W, p->n_cp, k);
    // every step's kept data if there is room
    adj_layout(a, true);
    const size_t keep = a->total;
    if (ws_bytes < keep) adj_layout(a, false);
    if (ws_bytes < a->total) {
        const size_t need = std::min(a->total, keep);
        delete a;
        return afail(nullptr, LBM_ERR_WS_TOO_SMALL, "workspace of %zu bytes, %zu needed", ws_bytes, need);
    }
    a->ws = static_cast<char *>(dev_ws);
    a->stream = static_cast<cudaStream_t>(cuda_stream);
    a->have_forward = false;
    a->gate_id = 0;
    std::snprintf(a->err, sizeof(a->err), "no error");
    int rc = acheck(a, cudaMemsetAsync(a->ws + a->o_gate, 0, 4, a->stream), "cudaMemsetAsync");
    auto up = [&](size_t off, const void *src, size_t bytes) {
        if (rc == LBM_OK && bytes)
            rc = acheck(a, cudaMemcpyAsync(a->ws + off, src, bytes, cudaMemcpyHostToDevice, a->stream), "cudaMemcpyAsync");
    };
    const size_t Lb = k.nf.size() * 4, Mb = k.node.size() * 4;
    up(a->o_kind, k.kind.data(), k.kind.size());
    up(a->o_nnode, k.node.data(), Mb);
    up(a->o_nbase, k.base.data(), Mb);
    up(a->o_nmask, k.mask.data(), Mb);
    up(a->o_lnf, k.nf.data(), Lb);
    up(a->o_ldir, k.dir.data(), Lb);
    up(a->o_lnff, k.nff.data(), Lb);
    if (rc == LBM_OK) rc = acheck(a, cudaStreamSynchronize(a->stream), "cudaStreamSynchronize");
    if (rc != LBM_OK) {
        std::snprintf(g_adj_error, sizeof(g_adj_error), "%s", a->err);
        delete a;
        return rc;
    }
    *out = a;
    return LBM_OK;
}

int lbm_adj_forward(lbm_adj *a, const double *cp_world, const double *K, double *J) {
    if (!a) return afail(nullptr, LBM_ERR_BAD_ARG, "handle is NULL");
    if (!cp_world || !K) return afail(a, LBM_ERR_BAD_ARG, "cp_world and K are required");
    for (int c = 0; c < a->ncp; c++)
        if (!(K[c] >= 0.0)) return afail(a, LBM_ERR_BAD_ARG, "negative weight");
    int rc = acheck(a, cudaMemcpyAsync(a->ws + a->o_cp, cp_world, (size_t)a->ncp * 24, cudaMemcpyHostToDevice, a->stream),
                    "cudaMemcpyAsync");
    if (rc == LBM_OK)
        rc = acheck(a, cudaMemcpyAsync(a->ws + a->o_K, K, (size_t)a->ncp * 8, cudaMemcpyHostToDevice, a->stream),
                    "cudaMemcpyAsync");
    if (rc == LBM_OK) rc = acheck(a, cudaMemsetAsync(a->ws + a->o_J, 0, 8, a->stream), "cudaMemsetAsync");
    if (rc != LBM_OK) return rc;
    const AdjDev D = adj_dev(a);
    const int lgrid = std::max(1, std::min(1024, (a->nlinks + 255) / 256));
    if (a->nlinks > 0) k_adj_q<<<lgrid, 256, 0, a->stream>>>(D);
    // state 0, and every K-th state of a run that keeps checkpoints, is
    // written where the adjoint's segments start from
    float *buf[2] = {state(a, a->o_state[0]), state(a, a->o_state[1])};
    auto ckpt = [&](int c) { return state(a, a->o_ckpt + a->S * (size_t)c); };
    float *src = a->keep_all ? buf[0] : ckpt(0);
    k_adj_init<<<1216, 256, 0, a->stream>>>(D, src, (float)a->cfg.u0[0], (float)a->cfg.u0[1], (float)a->cfg.u0[2]);
    const Kept none = {};
    for (int t = 0; t < a->T; t++) {
        const bool mark = !a->keep_all && (t + 1) % a->K == 0 && t + 1 < a->T;
        float *dst = mark ? ckpt((t + 1) / a->K) : (src == buf[0] ? buf[1] : buf[0]);
        forward_step(a, D, src, dst, a->keep_all ? kept_slot(a, t) : none, t >= a->T - a->W ? 1 : 0, t);
        src = dst;
    }
    long long jfix = 0;
    rc = acheck(a, cudaGetLastError(), "forward launch");
    if (rc == LBM_OK)
        rc = acheck(a, cudaMemcpyAsync(&jfix, a->ws + a->o_J, 8, cudaMemcpyDeviceToHost, a->stream), "cudaMemcpyAsync");
    if (rc == LBM_OK) rc = acheck(a, cudaStreamSynchronize(a->stream), "cudaStreamSynchronize");
    if (rc != LBM_OK) return rc;
    if (J) *J = std::ldexp((double)jfix, -kForceFixBits) / a->W;
    a->have_forward = true;
    return LBM_OK;
}

int lbm_adj_backward(lbm_adj *a, double *dJ_dcp, double *dJ_dK) {
    if (!a) return afail(nullptr, LBM_ERR_BAD_ARG, "handle is NULL");
    if (!a->have_forward) return afail(a, LBM_ERR_BAD_ARG, "no forward run to differentiate");
    const AdjDev D = adj_dev(a);
    int rc = acheck(a, cudaMemsetAsync(a->ws + a->o_dJdq, 0, (size_t)std::max(1, a->nlinks) * 8, a->stream), "cudaMemsetAsync");
    if (rc == LBM_OK) rc = acheck(a, cudaMemsetAsync(a->ws + a->o_lam[0], 0, a->S, a->stream), "cudaMemsetAsync");
    for (int k = 0; k < 2; k++)
        if (rc == LBM_OK)
            rc = acheck(a, cudaMemsetAsync(a->ws + a->o_share[k], 0, (size_t)a->N * 16, a->stream), "cudaMemsetAsync");
    if (rc == LBM_OK) rc = acheck(a, cudaMemsetAsync(a->ws + a->o_grad, 0, (size_t)a->ncp * 32, a->stream), "cudaMemsetAsync");
    if (rc != LBM_OK) return rc;
    float *lamN = state(a, a->o_lam[0]), *lamT = state(a, a->o_lam[1]);
    float4 *share = reinterpret_cast<float4 *>(a->ws + a->o_share[0]);
    float4 *share_next = reinterpret_cast<float4 *>(a->ws + a->o_share[1]);
    float *buf[2] = {state(a, a->o_state[0]), state(a, a->o_state[1])};
    for (int c = a->keep_all ? 0 : a->C - 1; c >= 0; c--) {
        const int t0 = a->keep_all ? 0 : c * a->K, t1 = a->keep_all ? a->T : std::min(a->T, t0 + a->K);
        if (!a->keep_all) {
            // the segment's kept data, from its checkpoint
            const float *src = state(a, a->o_ckpt + a->S * (size_t)c);
            for (int t = t0; t < t1; t++) {
                float *dst = src == buf[0] ? buf[1] : buf[0];
                forward_step(a, D, src, dst, kept_slot(a, t - t0), 0, t);
                src = dst;
            }
        }
        for (int t = t1 - 1; t >= t0; t--) {
            const int window = t >= a->T - a->W ? 1 : 0;
            const Kept kept = kept_slot(a, t - t0);
            adjoint_step(a, D, kept, lamN, lamT, share, share_next, window, t);
            std::swap(lamN, lamT);
            std::swap(share, share_next);
        }
    }
    if (a->nlinks > 0) k_adj_grad<<<std::max(1, std::min(256, (a->nlinks + 255) / 256)), 256, 0, a->stream>>>(D);
    std::vector<double> g((size_t)a->ncp * 4);
    rc = acheck(a, cudaGetLastError(), "adjoint launch");
    if (rc == LBM_OK)
        rc = acheck(a, cudaMemcpyAsync(g.data(), a->ws + a->o_grad, g.size() * 8, cudaMemcpyDeviceToHost, a->stream),
                    "cudaMemcpyAsync");
    if (rc == LBM_OK) rc = acheck(a, cudaStreamSynchronize(a->stream), "cudaStreamSynchronize");
    if (rc != LBM_OK) return rc;
    for (int c = 0; c < a->ncp; c++) {
        if (dJ_dcp)
            for (int k = 0; k < 3; k++) dJ_dcp[3 * c + k] = g[4 * (size_t)c + k];
        if (dJ_dK) dJ_dK[c] = g[4 * (size_t)c + 3];
    }
    return LBM_OK;
}

int lbm_adj_info(const lbm_adj *a, int *nlinks, int *checkpoint_every) {
    if (!a) return afail(nullptr, LBM_ERR_BAD_ARG, "handle is NULL");
    if (nlinks) *nlinks = a->nlinks;
    if (checkpoint_every) *checkpoint_every = a->K;
    return LBM_OK;
}

int lbm_adj_destroy(lbm_adj *a) {
    if (!a) return LBM_OK;
    cudaStreamSynchronize(a->stream);
    delete a;
    return LBM_OK;
}

const char *lbm_adj_last_error(const lbm_adj *a) { return a ? a->err : g_adj_error; }

}  // extern "C"
