// Isothermal nonideal fluid (Sec. "Nonideal Fluids and two-phase flow"; derivative
// stencil of Appendix A), with the van der Waals, the Peng-Robinson type (Eq. cspreos)
// or the Carnahan-Starling equation of state.
//
// Per step, from the post-collision state src:
//   k_ni_density  rho of the streamed populations, sum_i f_i(x - c_i), and
//                 mu_nid(rho), F_nid(rho) of each node
//   k_ni_fields   per node: grad2 rho (3) and the scalar S whose gradient holds the force's isotropic
//                 terms,
//                   S = -F + (1 - eta) (theta_hat / 2) lap F + kappa [-(1/2)|grad2 rho|^2 - rho lap rho]
//   k_ni_force    g^nid of Eq. (gradientFinal) at the node, from its stencil
//                 neighbours' fields:
//                   rho g = -[rho grad2 mu + mu grad2 rho - eta grad2 F
//                             - (1 - eta) grad4 F + kappa grad2_b I_ab],
//                   grad4 = grad2 - (theta_hat / 2) grad2 lap,
//                   I_ab = [-(1/2)|grad rho|^2 - rho lap rho] delta_ab + grad_a rho grad_b rho,
//                 which is -[rho grad2 mu + mu grad2 rho + grad2 S + kappa grad2_b (grad_a rho grad_b rho)]
//   k_ni_step     the pull step with the forced BGK collision of
//                 Eq. (multiphaseEvolution), alpha = 2: u = j / rho + g / 2,
//                 f^eq = f^eq(rho, u, theta_0), F_i = g.(c_i - u)/theta_0 f^eq_i,
//                 f' = f + 2 beta (f^eq - f) + (1 - beta) F_i.
// With 16-bit storage and nx even the two gathering passes run on x pairs (k_ni_density2x,
// k_ni_step2x: the x-pair gather of k_step2x, packed FP32x2 arithmetic); with FP32 fields and nx
// even the two stencil passes do too (k_ni_fields2x, k_ni_force2x: the pair's 24 distinct
// neighbours loaded once for both nodes).
// The stencil is the 15-velocity bcc set of Appendix A: rest, (+-1, 0, 0) and
// permutations (on the node's own sub-lattice), (+-1/2, +-1/2, +-1/2) (on the
// other); weights 14/36, 1/36, 2/36; theta_hat = 1/6.  The fields are in
// the storage codec's compute type: FP64 for FP64 storage, FP32 otherwise.
#include <math.h>

#include "lb_ctx.h"
#include "lb_eos.cuh"
#include "lb_kernels.cuh"

namespace gblb {

constexpr double kHatTheta = 1.0 / 6.0;
constexpr int kStencil = 14;  // moving stencil velocities (the rest one only enters lap)

// Doubled velocity and weight of moving stencil velocity k: 6 sc-1 then 8 bcc-1/2.
template <class F>
__device__ __forceinline__ void stencil(int k, int& cx, int& cy, int& cz, F& w) {
    if (k < 6) {
        cx = cy = cz = 0;
        const int v = (k & 1) ? -2 : 2;
        if (k < 2)
            cx = v;
        else if (k < 4)
            cy = v;
        else
            cz = v;
        w = F(1.0 / 36.0);
    } else {
        const int j = k - 6;
        cx = (j & 1) ? -1 : 1;
        cy = (j & 2) ? -1 : 1;
        cz = (j & 4) ? -1 : 1;
        w = F(2.0 / 36.0);
    }
}

constexpr int kNiThreads = 128;

// Field arrays in the compute type F over the n = 2 nx ny nz nodes (field index q, n even).  The
// arrays of two fields hold the nodes in pairs (2p, 2p + 1), p = q >> 1, as four values
// {u(2p), u(2p + 1), v(2p), v(2p + 1)}: an x pair (x even, nx even) reads both nodes' u and v
// in one 16-byte load, and a warp's loads of 32 pairs are contiguous.
//   RF = {rho, F_nid}, MU[q] = mu_nid                              (density pass)
//   C = {grad2_x rho, grad2_y rho}, D = {grad2_z rho, S}           (field pass)
//   G[a n + q] = g^nid_a                                           (force pass)
template <class F>
struct NiFields {
    F* RF;
    F* C;
    F* D;
    F* MU;
    F* G;
};

// Index of u (v = 0) or v (v = 1) of node q in an array of two fields.
__device__ __forceinline__ uint32_t ni_pair_at(uint32_t q, int v) { return 4 * (q >> 1) + 2 * v + (q & 1); }

// Four values of one pair in the field type (the 16-byte load of a pair with F = float).
template <class F>
struct alignas(4 * sizeof(F)) NiQuad {
    F x, y, z, w;
};
// u (v = 0) or v (v = 1) of the pair's node c.
template <class F>
__device__ __forceinline__ F quad_at(const NiQuad<F>& r, int v, int c) {
    return v ? (c ? r.w : r.z) : (c ? r.y : r.x);
}

// a in [0, n] (wrap_up) or in [-1, n) (wrap_dn) back into [0, n): the stencil's offsets are +-1.
__device__ __forceinline__ uint32_t wrap_up(int a, int n) { return (uint32_t)(a == n ? 0 : a); }
__device__ __forceinline__ uint32_t wrap_dn(int a, int n) { return (uint32_t)(a < 0 ? n - 1 : a); }

// Field index of node (s, z, y, x): ((s nz + z) ny + y) nx + x, below 2^32 (checked when the mode is enabled).
__device__ __forceinline__ uint32_t ni_index(const Dims& d, int s, int z, int y, int x) {
    return (((uint32_t)s * (uint32_t)d.nz + (uint32_t)z) * (uint32_t)d.ny + (uint32_t)y) * (uint32_t)d.nx + (uint32_t)x;
}

// Field indices of the 14 moving stencil neighbours of node (s, z, y, x), in the order of
// stencil(): the sc-1 links +x, -x, +y, -y, +z, -z on the node's own sub-lattice, then the
// bcc-1/2 links on the other, whose +1/2 neighbour along an axis has index coordinate + s and
// whose -1/2 neighbour has + s - 1.  32-bit: 2 nx ny nz < 2^32 (checked when the mode is enabled).
__device__ __forceinline__ void ni_neighbors(const Dims& d, int s, int z, int y, int x, uint32_t (&m)[kStencil]) {
    const uint32_t nx = (uint32_t)d.nx, nxy = nx * (uint32_t)d.ny, pl = (uint32_t)d.plane;
    const uint32_t own = (uint32_t)s * pl, oth = (uint32_t)(1 - s) * pl;
    const uint32_t xs = (uint32_t)x, ys = (uint32_t)y * nx, zs = (uint32_t)z * nxy;
    m[0] = own + zs + ys + wrap_up(x + 1, d.nx);
    m[1] = own + zs + ys + wrap_dn(x - 1, d.nx);
    m[2] = own + zs + wrap_up(y + 1, d.ny) * nx + xs;
    m[3] = own + zs + wrap_dn(y - 1, d.ny) * nx + xs;
    m[4] = own + wrap_up(z + 1, d.nz) * nxy + ys + xs;
    m[5] = own + wrap_dn(z - 1, d.nz) * nxy + ys + xs;
    const uint32_t X[2] = {wrap_up(x + s, d.nx), wrap_dn(x + s - 1, d.nx)};
    const uint32_t Y[2] = {wrap_up(y + s, d.ny) * nx, wrap_dn(y + s - 1, d.ny) * nx};
    const uint32_t Z[2] = {wrap_up(z + s, d.nz) * nxy, wrap_dn(z + s - 1, d.nz) * nxy};
#pragma unroll
    for (int j = 0; j < 8; ++j) m[6 + j] = oth + Z[(j >> 2) & 1] + Y[(j >> 1) & 1] + X[j & 1];
}

template <class Codec>
__global__ void __launch_bounds__(kNiThreads) k_ni_density(const typename Codec::raw_t* src, Dims d, EntryGrid g,
                                                           Consts<typename Codec::R> K, NiEosT<typename Codec::R> e,
                                                           NiFields<typename Codec::R> fl) {
    using R = typename Codec::R;
    int s, z, y, x;
    const bool active = entry_node<kNode>(d, g, s, z, y, x);
    pdl_begin();
    if (!active) return;
    R v[kQ];
    pull_node<Codec, LoadCA, true>(src, d, s, z, y, x, v);
    R dr = 0;  // rho - 1 = sum_i (f_i - w_i)
    static_for<kQ>([&](auto I) { dr += Codec::dev(v[I], K.w[vel(I).shell] * R(1.0 / Codec::kScale)); });
    const R r = R(1) + dr;
    R mu, Fe;
    ni_eos<R>(r, e, mu, Fe);
    const uint32_t qq = ni_index(d, s, z, y, x);
    fl.RF[ni_pair_at(qq, 0)] = r;
    fl.RF[ni_pair_at(qq, 1)] = Fe;
    fl.MU[qq] = mu;
}

// Every moving stencil term of a first derivative carries w_k c_ka / 2 = +-1/36 (sc-1: 1/36 x +-1,
// bcc-1/2: 2/36 x +-1/2), so the passes sum the neighbours' values with signs and apply the weight
// once; grad2 X = (1 / (36 theta_hat)) sum_k sgn(c_ka) (X(x + c_k) - X(x)) over the k with c_ka != 0.
// The signs sum to zero; close values subtract exactly, so the differences round less than the values.
constexpr double kGradScale = 1.0 / (36.0 * kHatTheta);

// acc += v for sign > 0, acc -= v otherwise (the sign is a compile-time constant after unrolling).
template <class F>
__device__ __forceinline__ void add_signed(F& acc, F v, int sign) {
    acc = sign > 0 ? acc + v : acc - v;
}

// The field pass at one node from its rho0, F0 and its neighbours' rn, Fn (in the order of
// stencil()): grad2 rho and S.  lap X = (2 / theta_hat) sum_k w_k (X(x + c_k) - X(x)) = (1/3) [sum_sc dX +
// 2 sum_bcc dX].
template <class F>
__device__ __forceinline__ void ni_fields_node(const NiEosT<F>& e, F r0, F F0, const F (&rn)[kStencil],
                                               const F (&Fn)[kStencil], F (&g)[3], F& S) {
    F gsum[3] = {F(0), F(0), F(0)}, lr[2] = {F(0), F(0)}, lF[2] = {F(0), F(0)};
#pragma unroll
    for (int k = 0; k < kStencil; ++k) {
        int cx, cy, cz;
        F w;
        stencil(k, cx, cy, cz, w);
        const F dr = rn[k] - r0;
        if (cx) add_signed(gsum[0], dr, cx);
        if (cy) add_signed(gsum[1], dr, cy);
        if (cz) add_signed(gsum[2], dr, cz);
        const int sh = k < 6 ? 0 : 1;  // sc-1 or bcc-1/2
        lr[sh] += dr;
        lF[sh] += Fn[k] - F0;
    }
    const F gs = F(kGradScale);
    for (int b = 0; b < 3; ++b) g[b] = gsum[b] * gs;
    const F lap = F(1.0 / 3.0) * (lr[0] + F(2) * lr[1]);
    const F iso = F(-0.5) * (g[0] * g[0] + g[1] * g[1] + g[2] * g[2]) - r0 * lap;
    const F lapF = F(1.0 / 3.0) * (lF[0] + F(2) * lF[1]);
    S = fma((F(1) - e.eta) * F(0.5 * kHatTheta), lapF, e.kappa * iso) - F0;
}

template <class F>
__global__ void __launch_bounds__(kNiThreads) k_ni_fields(Dims d, EntryGrid gr, NiEosT<F> e, NiFields<F> fl) {
    int s, z, y, x;
    const bool active = entry_node<kNode, true>(d, gr, s, z, y, x);
    pdl_begin();
    if (!active) return;
    const uint32_t q = ni_index(d, s, z, y, x);
    uint32_t nb[kStencil];
    ni_neighbors(d, s, z, y, x, nb);
    F rn[kStencil], Fn[kStencil];
#pragma unroll
    for (int k = 0; k < kStencil; ++k) {
        rn[k] = fl.RF[ni_pair_at(nb[k], 0)];
        Fn[k] = fl.RF[ni_pair_at(nb[k], 1)];
    }
    F g[3], S;
    ni_fields_node<F>(e, fl.RF[ni_pair_at(q, 0)], fl.RF[ni_pair_at(q, 1)], rn, Fn, g, S);
    fl.C[ni_pair_at(q, 0)] = g[0];
    fl.C[ni_pair_at(q, 1)] = g[1];
    fl.D[ni_pair_at(q, 0)] = g[2];
    fl.D[ni_pair_at(q, 1)] = S;
}

// A stencil neighbour's fields as the force pass uses them.
template <class F>
struct NiNb {
    F mu, S, g[3];
};

// One stencil neighbour's terms of the force sums, k its stencil velocity (doubled c: sc-1 +-2
// along one axis; bcc-1/2 +-1 along each), o the node itself.  With sgn(c_a) = c_a / |c_a|:
//   dmu_a, t_a += sgn(c_a) (mu - mu_0), sgn(c_a) (S - S_0)                        (c_a != 0)
//   tau_a += sum_b sgn(c_b) grad_a rho grad_b rho;
// each sum times 1 / (36 theta_hat) is the grad2 of Appendix A.
template <class F>
struct NiForceSums {
    F dmu[3], dS[3], tau[3];
};
template <class F>
__device__ __forceinline__ void ni_sums_zero(NiForceSums<F>& a) {
    for (int b = 0; b < 3; ++b) a.dmu[b] = a.dS[b] = a.tau[b] = F(0);
}
template <class F>
__device__ __forceinline__ void ni_force_term(NiForceSums<F>& a, int k, const NiNb<F>& v, F mu0, F S0) {
    int cc[3];
    F w;
    stencil(k, cc[0], cc[1], cc[2], w);
    const F dmu = v.mu - mu0, dS = v.S - S0;
    F cg = F(0);  // sum_b sgn(c_b) grad_b rho
    bool first = true;
    for (int b = 0; b < 3; ++b) {
        if (cc[b] == 0) continue;
        add_signed(a.dmu[b], dmu, cc[b]);
        add_signed(a.dS[b], dS, cc[b]);
        if (first)
            cg = cc[b] > 0 ? v.g[b] : -v.g[b];
        else
            add_signed(cg, v.g[b], cc[b]);
        first = false;
    }
    for (int b = 0; b < 3; ++b) a.tau[b] = fma(v.g[b], cg, a.tau[b]);
}

// g^nid from the sums and the node's own rho, mu and grad2 rho:
//   rho g = -[rho grad2 mu + mu grad2 rho + grad2 S + kappa grad2_b (grad_a rho grad_b rho)].
template <class F>
__device__ __forceinline__ void ni_force_finish(const NiEosT<F>& e, const NiForceSums<F>& a, F r0, F mu0,
                                                const F (&g2r)[3], F (&g)[3]) {
    const F gs = F(kGradScale), inv_r0 = F(1) / r0;
    for (int b = 0; b < 3; ++b) {
        const F rg = -(r0 * (a.dmu[b] * gs) + mu0 * g2r[b] + fma(e.kappa, a.tau[b], a.dS[b]) * gs);
        g[b] = rg * inv_r0;
    }
}

// g^nid of every node into G (a pass of its own: folded into the step, the stencil sums raise the
// step's register count and the fused step ran slower than the two passes).
template <class F>
__global__ void __launch_bounds__(kNiThreads) k_ni_force(Dims d, EntryGrid gr, NiEosT<F> e, NiFields<F> fl) {
    int s, z, y, x;
    const bool active = entry_node<kNode, true>(d, gr, s, z, y, x);
    pdl_begin();
    if (!active) return;
    const uint32_t q = ni_index(d, s, z, y, x);
    uint32_t nb[kStencil];
    ni_neighbors(d, s, z, y, x, nb);
    const F mu0 = fl.MU[q], S0 = fl.D[ni_pair_at(q, 1)];
    NiForceSums<F> a;
    ni_sums_zero(a);
#pragma unroll
    for (int k = 0; k < kStencil; ++k) {
        const uint32_t m = nb[k];
        const NiNb<F> v{fl.MU[m], fl.D[ni_pair_at(m, 1)],
                        {fl.C[ni_pair_at(m, 0)], fl.C[ni_pair_at(m, 1)], fl.D[ni_pair_at(m, 0)]}};
        ni_force_term<F>(a, k, v, mu0, S0);
    }
    const F g2r[3] = {fl.C[ni_pair_at(q, 0)], fl.C[ni_pair_at(q, 1)], fl.D[ni_pair_at(q, 0)]};
    F g[3];
    ni_force_finish<F>(e, a, fl.RF[ni_pair_at(q, 0)], mu0, g2r, g);
    const size_t n = 2 * (size_t)d.plane;
    for (int b = 0; b < 3; ++b) fl.G[b * n + q] = g[b];
}

// Two x-adjacent nodes (x even, nx even) per thread in the stencil passes; q is the even node's field
// index, q >> 1 the pair's.
// The stencil neighbours of the pair (x, x + 1) on sub-lattice S lie in 15 pairs (pair indices):
//   0-2    the own row's pairs at x - 2, x, x + 2 (wrapped)
//   3-6    the rows +y, -y, +z, -z at x
//   7-10   the other sub-lattice's rows c = 0..3 of the bcc-1/2 links at x (y side c & 1, z side
//          c >> 1; side 0 is the +1/2 one)
//   11-14  the same rows at x - 2 (S = 0) or x + 2 (S = 1)
constexpr int kPairPos = 15;
template <int S>
__device__ __forceinline__ void ni_pair_positions(const Dims& d, int z, int y, int x, uint32_t q,
                                                  uint32_t (&p)[kPairPos]) {
    const uint32_t nx = (uint32_t)d.nx, nxy = nx * (uint32_t)d.ny, pl = (uint32_t)d.plane;
    const uint32_t own = (uint32_t)S * pl, oth = (uint32_t)(1 - S) * pl, hx = nx / 2;
    const uint32_t xs = (uint32_t)x, ys = (uint32_t)y * nx, zs = (uint32_t)z * nxy;
    const bool first = x == 0, last = x + 2 == d.nx;
    auto left = [&](uint32_t r) { return first ? r + hx - 1 : r - 1; };   // the pair at x - 2 of r's row
    auto right = [&](uint32_t r) { return last ? r + 1 - hx : r + 1; };  // the pair at x + 2
    const uint32_t pq = q >> 1;
    p[0] = left(pq);
    p[1] = pq;
    p[2] = right(pq);
    p[3] = (own + zs + wrap_up(y + 1, d.ny) * nx + xs) >> 1;
    p[4] = (own + zs + wrap_dn(y - 1, d.ny) * nx + xs) >> 1;
    p[5] = (own + wrap_up(z + 1, d.nz) * nxy + ys + xs) >> 1;
    p[6] = (own + wrap_dn(z - 1, d.nz) * nxy + ys + xs) >> 1;
    const uint32_t Y[2] = {wrap_up(y + S, d.ny) * nx, wrap_dn(y + S - 1, d.ny) * nx};
    const uint32_t Z[2] = {wrap_up(z + S, d.nz) * nxy, wrap_dn(z + S - 1, d.nz) * nxy};
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        p[7 + c] = (oth + Z[c >> 1] + Y[c & 1] + xs) >> 1;
        p[11 + c] = S ? right(p[7 + c]) : left(p[7 + c]);
    }
}

// 2 x (pair position) + node within it of stencil neighbour k of node x + h.
template <int S>
__host__ __device__ constexpr int ni_pair_src(int h, int k) {
    if (k == 0) return h ? 2 * 2 + 0 : 2 * 1 + 1;  // +x: x + 1, x + 2
    if (k == 1) return h ? 2 * 1 + 0 : 2 * 0 + 1;  // -x: x - 1, x
    if (k < 6) return 2 * (k + 1) + h;             // +-y, +-z: the same x
    const int c = (k - 6) >> 1;
    const int o = ((k - 6) & 1) ? S - 1 + h : S + h;  // x offset of the bcc-1/2 neighbour
    return o < 0 ? 2 * (11 + c) + 1 : o == 0 ? 2 * (7 + c) : o == 1 ? 2 * (7 + c) + 1 : 2 * (11 + c);
}

template <class F>
struct alignas(2 * sizeof(F)) NiDuo {
    F x, y;
};

template <class F, int S>
__device__ __forceinline__ void ni_fields_pair(const Dims& d, const NiEosT<F>& e, const NiFields<F>& fl, int z, int y, int x, uint32_t q) {
    uint32_t p[kPairPos];
    ni_pair_positions<S>(d, z, y, x, q, p);
    const NiQuad<F>* RF = reinterpret_cast<const NiQuad<F>*>(fl.RF);
    NiQuad<F> rf[kPairPos];
#pragma unroll
    for (int i = 0; i < kPairPos; ++i) rf[i] = RF[p[i]];
    F g[2][3], S_[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        F rn[kStencil], Fn[kStencil];
#pragma unroll
        for (int k = 0; k < kStencil; ++k) {
            const int src = ni_pair_src<S>(h, k);
            rn[k] = quad_at(rf[src >> 1], 0, src & 1);
            Fn[k] = quad_at(rf[src >> 1], 1, src & 1);
        }
        ni_fields_node<F>(e, quad_at(rf[1], 0, h), quad_at(rf[1], 1, h), rn, Fn, g[h], S_[h]);
    }
    const uint32_t pq = q >> 1;
    reinterpret_cast<NiQuad<F>*>(fl.C)[pq] = NiQuad<F>{g[0][0], g[1][0], g[0][1], g[1][1]};
    reinterpret_cast<NiQuad<F>*>(fl.D)[pq] = NiQuad<F>{g[0][2], g[1][2], S_[0], S_[1]};
}

// k_ni_fields for an x pair.
template <class F>
__global__ void __launch_bounds__(kNiThreads) k_ni_fields2x(Dims d, EntryGrid gr, NiEosT<F> e, NiFields<F> fl) {
    int s, z, y, x;
    const bool active = entry_node<kPair, true>(d, gr, s, z, y, x);
    pdl_begin();
    if (!active) return;
    const uint32_t q = ni_index(d, s, z, y, x);
    if (s)
        ni_fields_pair<F, 1>(d, e, fl, z, y, x, q);
    else
        ni_fields_pair<F, 0>(d, e, fl, z, y, x, q);
}

template <class F, int S>
__device__ __forceinline__ void ni_force_pair(const Dims& d, const NiEosT<F>& e, const NiFields<F>& fl, int z, int y,
                                              int x, uint32_t q) {
    uint32_t p[kPairPos];
    ni_pair_positions<S>(d, z, y, x, q, p);
    const NiQuad<F>* C = reinterpret_cast<const NiQuad<F>*>(fl.C);
    const NiQuad<F>* D = reinterpret_cast<const NiQuad<F>*>(fl.D);
    const NiDuo<F>* MU = reinterpret_cast<const NiDuo<F>*>(fl.MU);
    NiQuad<F> qc[kPairPos], qd[kPairPos];
    NiDuo<F> qm[kPairPos];
#pragma unroll
    for (int i = 0; i < kPairPos; ++i) {
        qc[i] = C[p[i]];
        qd[i] = D[p[i]];
        qm[i] = MU[p[i]];
    }
    NiForceSums<F> a[2];
    ni_sums_zero(a[0]);
    ni_sums_zero(a[1]);
#pragma unroll
    for (int k = 0; k < kStencil; ++k) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int src = ni_pair_src<S>(h, k), i = src >> 1, c = src & 1;
            const NiNb<F> v{c ? qm[i].y : qm[i].x, quad_at(qd[i], 1, c),
                            {quad_at(qc[i], 0, c), quad_at(qc[i], 1, c), quad_at(qd[i], 0, c)}};
            ni_force_term<F>(a[h], k, v, h ? qm[1].y : qm[1].x, quad_at(qd[1], 1, h));
        }
    }
    const NiQuad<F> rf = reinterpret_cast<const NiQuad<F>*>(fl.RF)[q >> 1];
    F g[2][3];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const F g2r[3] = {quad_at(qc[1], 0, h), quad_at(qc[1], 1, h), quad_at(qd[1], 0, h)};
        ni_force_finish<F>(e, a[h], quad_at(rf, 0, h), h ? qm[1].y : qm[1].x, g2r, g[h]);
    }
    const size_t n = 2 * (size_t)d.plane;
    for (int b = 0; b < 3; ++b) *reinterpret_cast<NiDuo<F>*>(fl.G + b * n + q) = NiDuo<F>{g[0][b], g[1][b]};
}

// k_ni_force for an x pair.  Bound by the L1 traffic of its 15 pairs and the latency of the loads: five
// values of a neighbour instead of seven (mu, F, lap F, iso and the gradient apart) take the 160 x 200 x 200
// step with FP16 storage from 0.99 to 0.92 ms, FP32 from 1.30 to 1.23.  64 registers (8 blocks per SM),
// without spills: 1.180 ms for the 256 x 256 x 128 step, against 1.186 with 80 (6 blocks).
template <class F>
__global__ void __launch_bounds__(kNiThreads, 8) k_ni_force2x(Dims d, EntryGrid gr, NiEosT<F> e, NiFields<F> fl) {
    int s, z, y, x;
    const bool active = entry_node<kPair, true>(d, gr, s, z, y, x);
    pdl_begin();
    if (!active) return;
    const uint32_t q = ni_index(d, s, z, y, x);
    if (s)
        ni_force_pair<F, 1>(d, e, fl, z, y, x, q);
    else
        ni_force_pair<F, 0>(d, e, fl, z, y, x, q);
}

// The forced relaxation of a node as collide's sink: with G_i = (1 - beta) g.(c_i - u) / theta0 the new
// value is (1 - 2 beta) v + f^eq_i (2 beta + G_i) for FP64, and for the deviation codecs, whose f^eq_i / w_i
// is 1 + h^eq_i, (1 - 2 beta) v + h^eq_i (2 beta + G_i) + kScale G_i.  H = (1 - beta) g / theta0, hu = H.u; the
// direction's H.c is formed for the +c of a pair and used for both.
template <class Codec, class VGet, class Out>
struct NiForcedSink {
    using R = typename Codec::R;
    R hx, hy, hz, hu, tb, omb;
    VGet vget;
    Out out;
    R hc;
    template <class I>
    __device__ __forceinline__ void operator()(I i, R veq) {
        constexpr Vel c = vel(I::value);
        R G;
        if constexpr (c.shell == 0) {
            G = -hu;
        } else if constexpr (I::value % 2 == 1) {
            hc = R(0);
            bool first = true;
            auto term = [&](auto C2, R h) {
                constexpr int k = decltype(C2)::value;
                if constexpr (k != 0) {
                    hc = first ? R(0.5 * k) * h : fma(R(0.5 * k), h, hc);
                    first = false;
                }
            };
            term(std::integral_constant<int, c.x>{}, hx);
            term(std::integral_constant<int, c.y>{}, hy);
            term(std::integral_constant<int, c.z>{}, hz);
            G = hc - hu;
        } else {
            G = -hc - hu;
        }
        const R v = vget(i);
        if constexpr (Codec::stores_f)
            out(i, fma(veq, tb + G, omb * v));
        else
            out(i, fma(veq, tb + G, fma(omb, v, R(Codec::kScale) * G)));
    }
};

// State of the forced step: u = j / rho + g / 2 (the temperature is theta_0 throughout).
template <class R>
__device__ __forceinline__ NodeState<R> ni_state(const NodeSums<R>& m, R gx, R gy, R gz) {
    NodeState<R> st;
    st.drho = m.drho;
    st.rho = R(1) + m.drho;
    const R inv_rho = recip_newton(st.rho);
    st.ux = fma(R(0.5), gx, m.jx * inv_rho);
    st.uy = fma(R(0.5), gy, m.jy * inv_rho);
    st.uz = fma(R(0.5), gz, m.jz * inv_rho);
    st.eta = R(0);
    return st;
}

template <class Codec, class VGet, class KS, class Out>
__device__ __forceinline__ void ni_collide(const NodeState<typename Codec::R>& st, const StepConsts<KS>& K,
                                           typename Codec::R tb, typename Codec::R gx, typename Codec::R gy,
                                           typename Codec::R gz, VGet vget, Out out) {
    using R = typename Codec::R;
    const R k = (R(1) - R(0.5) * tb) * R(K.inv_theta0);  // (1 - beta) / theta0
    const R hx = gx * k, hy = gy * k, hz = gz * k;
    NiForcedSink<Codec, VGet, Out> sink{hx, hy, hz, fma(hx, st.ux, fma(hy, st.uy, hz * st.uz)), tb, R(1) - tb,
                                        vget, out, R(0)};
    collide<Codec, true, false, true>(st, K, R(Codec::kScale), R(0), vget, sink);
}

// The pull step with the forced BGK collision; g^nid from G.
template <class Codec>
__global__ void __launch_bounds__(kNiThreads) k_ni_step(const typename Codec::raw_t* src, typename Codec::raw_t* dst,
                                                        Dims d, EntryGrid g, StepConsts<typename Codec::R> K,
                                                        typename Codec::R tb, const typename Codec::R* G, int* err) {
    using R = typename Codec::R;
    int s, z, y, x;
    const bool active = entry_node<kNode>(d, g, s, z, y, x);
    pdl_begin();
    if (!active) return;
    const uint32_t q = ni_index(d, s, z, y, x);
    const size_t n = 2 * (size_t)d.plane;
    const R gx = LoadCA::load(G + q), gy = LoadCA::load(G + n + q), gz = LoadCA::load(G + 2 * n + q);
    R v[kQ];
    pull_node<Codec, LoadCA, true>(src, d, s, z, y, x, v);
    auto vget = [&](auto I) { return v[I]; };
    const NodeState<R> st = ni_state(node_sums<Codec>(K, vget), gx, gy, gz);
    if (!state_ok(st)) atomicOr(err, 1);
    typename Codec::raw_t* o = dst + (size_t)s * (kQ - 1) * d.plane + q;
    ni_collide<Codec>(st, K, tb, gx, gy, gz, vget, [&](auto I, R val) { o[(size_t)I * d.plane] = Codec::to_raw(val); });
}

// k_ni_density for an x pair (16-bit storage, nx even).
template <class Codec, bool WIDE>
__global__ void __launch_bounds__(kStepThreads) k_ni_density2x(const typename Codec::raw_t* src, Dims d, EntryGrid g,
                                                               Consts<float> K, NiEosT<float> e, NiFields<float> fl) {
    int s, z, y, x;
    const bool active = entry_node<kPair>(d, g, s, z, y, x);
    pdl_begin();
    if (!active) return;
    const uint32_t q = ni_index(d, s, z, y, x);
    typename Codec::pair_t pv[kQ];
    pull_pair<Codec, WIDE>(src, d, s, z, y, x, pv);
    constexpr float inv_scale = (float)(1.0 / Codec::kScale);
    F2 dr(0.f);  // rho - 1 = sum_i (f_i - w_i), in the population order of k_ni_density
    static_for<kQ>([&](auto I) { dr += F2(Codec::unpack2(pv[I])) * F2(K.w[vel(I).shell] * inv_scale); });
    const F2 r = F2(1.f) + dr;
    float mu0, F0, mu1, F1;
    ni_eos<float>(r.v.x, e, mu0, F0);
    ni_eos<float>(r.v.y, e, mu1, F1);
    *reinterpret_cast<float4*>(fl.RF + 2 * (size_t)q) = make_float4(r.v.x, r.v.y, F0, F1);
    *reinterpret_cast<float2*>(fl.MU + q) = make_float2(mu0, mu1);
}

// k_ni_step for an x pair (16-bit storage, nx even).  Bound by the latency of its arithmetic: 4 blocks per SM
// (128 registers, 76 bytes of spills) take the 160 x 200 x 200 step from 1.04 to 0.99 ms against 3.
template <class Codec, bool WIDE>
__global__ void __launch_bounds__(kStepThreads, 4) k_ni_step2x(const typename Codec::raw_t* src,
                                                               typename Codec::raw_t* dst, Dims d, EntryGrid g,
                                                               StepConsts<float2> K, float tb, const float* G, int* err) {
    using P = typename Codec::pair_t;
    using C2 = Codec2<Codec>;
    int s, z, y, x;
    const bool active = entry_node<kPair>(d, g, s, z, y, x);
    pdl_begin();
    if (!active) return;
    const uint32_t q = ni_index(d, s, z, y, x);
    const size_t n = 2 * (size_t)d.plane;
    P pv[kQ];
    pull_pair<Codec, WIDE>(src, d, s, z, y, x, pv);
    auto vget = [&](auto I) { return F2(Codec::unpack2(pv[I])); };
    auto ld = [&](size_t off) { return F2(LoadCA::load(reinterpret_cast<const float2*>(G + off + q))); };
    const F2 gx = ld(0), gy = ld(n), gz = ld(2 * n);
    const NodeState<F2> st = ni_state(node_sums<C2>(K, vget), gx, gy, gz);
    if (!state_ok(st)) atomicOr(err, 1);
    keep_packed<Codec>(pv);
    typename Codec::raw_t* o = dst + (size_t)s * (kQ - 1) * d.plane + q;
    ni_collide<C2>(st, K, F2(tb), gx, gy, gz, vget, [&](auto I, F2 val) {
        *reinterpret_cast<P*>(o + (size_t)I * d.plane) = Codec::to_raw2(val.v);
    });
}

template <class F>
static cudaError_t ni_codec(int prec, F&& f) {
    switch (prec) {
        case kF64: return f(CodecF64{});
        case kF32: return f(CodecF32{});
        case kF16: return f(CodecF16{});
        case kBF16: return f(CodecBF16{});
        default: return cudaErrorInvalidValue;
    }
}

// The field arrays RF, C, D (2 values per node each), MU (1) and G (3), in the field type.
size_t nonideal_doubles(const Dims& d, int prec) {
    const size_t values = (size_t)10 * 2 * d.plane;
    return prec == kF64 ? values : (values + 1) / 2;
}

cudaError_t launch_nonideal_step(int prec, const void* src, void* dst, const Dims& d, const LaunchConsts& c,
                                 double twobeta, int kind, const double eos[4], double* work, int* err,
                                 cudaStream_t st) {
    const int64_t n = 2 * d.plane;
    if (d.plane >= ((int64_t)1 << 30)) return cudaErrorInvalidValue;  // 32-bit entries
    if (kind < kVdW || kind > kCarnahanStarling) return cudaErrorInvalidValue;
    const NiEos e64{eos[0], eos[1], c.theta0, eos[2], eos[3], kind};
    return ni_codec(prec, [&](auto codec) {
        using C = decltype(codec);
        using R = typename C::R;
        const Consts<R>* K = &consts_of<C>(c);
        const NiEosT<R> e = ni_eos_in<R>(e64);
        // field arrays in the compute type: RF, C, D (2 values per node each; 16-byte aligned, n
        // is even), then MU (1) and G (3)
        NiFields<R> fl;
        fl.RF = reinterpret_cast<R*>(work);
        fl.C = fl.RF + 2 * n;
        fl.D = fl.C + 2 * n;
        fl.MU = fl.D + 2 * n;
        fl.G = fl.MU + n;
        const auto* in = static_cast<const typename C::raw_t*>(src);
        auto* out = static_cast<typename C::raw_t*>(dst);
        // x pairs with nx even: the gathering passes with 16-bit storage, the stencil passes with FP32 fields
        const bool even = d.nx % 2 == 0, wide = wide_offsets(d);
        const EntryGrid gn = entry_grid<kNode>(d), gp = entry_grid<kPair>(d);
        constexpr bool kPairs = sizeof(typename C::raw_t) == 2;
        cudaError_t err_ = cudaSuccess;
        auto ok = [&](cudaError_t e_) { return (err_ = e_) == cudaSuccess; };
        bool gathered = false;
        if constexpr (kPairs) {
            if (even) {
                if (!ok(launch_linear(wide ? k_ni_density2x<C, true> : k_ni_density2x<C, false>, gp.entries, st, in, d, gp,
                                      *K, e, fl)))
                    return err_;
                gathered = true;
            }
        }
        if (!gathered && !ok(launch_linear(k_ni_density<C>, gn.entries, st, in, d, gn, *K, e, fl))) return err_;
        bool fields = false;
        if constexpr (sizeof(R) == 4) {
            if (even) {
                if (!ok(launch_linear(k_ni_fields2x<R>, gp.entries, st, d, gp, e, fl)) ||
                    !ok(launch_linear(k_ni_force2x<R>, gp.entries, st, d, gp, e, fl)))
                    return err_;
                fields = true;
            }
        }
        if (!fields && (!ok(launch_linear(k_ni_fields<R>, gn.entries, st, d, gn, e, fl)) ||
                        !ok(launch_linear(k_ni_force<R>, gn.entries, st, d, gn, e, fl))))
            return err_;
        if constexpr (kPairs) {
            if (even)
                return launch_linear(wide ? k_ni_step2x<C, true> : k_ni_step2x<C, false>, gp.entries, st, in, out, d, gp,
                                     pair_consts<C>(c), (float)twobeta, (const float*)fl.G, err);
        }
        return launch_linear(k_ni_step<C>, gn.entries, st, in, out, d, gn, (step_consts<C, 1>(c)), (R)twobeta,
                             (const R*)fl.G, err);
    });
}

}  // namespace gblb
