// Shared device code of the RD3Q41 solver: the velocity table, the storage
// codecs and the fused per-node collision (moments, energy-conserving
// equilibrium, BGK relaxation).
//
// Model: arXiv:1909.08406.  Velocity shells and weights: Sec. IV, Table I.
// Moments: Sec. II.  Rest-state equilibrium to O(eta^3) and the velocity
// series Eq. (feqGenU3): Sec. V.  BGK update: Sec. II.
//
// The per-node arithmetic is organised around the +-c pairs of the velocity
// set: for a pair the equilibrium splits into an even part (shared) and an odd
// part (sign-flipped), so each pair costs one dot product, a handful of FMAs
// and two relaxations.  All shell-dependent quantities are folded into six
// per-node shell constants.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>
#include <string.h>

#include <type_traits>
#include <utility>

namespace gblb {

constexpr int kQ = 41;
constexpr int kShells = 6;  // rest, sc-1, sc-2, fcc-1, bcc-1, bcc-1/2

// Doubled velocity components 2 c_i, ordered rest then +-c pairs (2k+1, 2k+2).
struct Vel {
    int x, y, z, shell;
};

__host__ __device__ constexpr Vel vel(int i) {
    constexpr Vel t[kQ] = {
        {0, 0, 0, 0},
        // sc-1
        {2, 0, 0, 1}, {-2, 0, 0, 1}, {0, 2, 0, 1}, {0, -2, 0, 1}, {0, 0, 2, 1}, {0, 0, -2, 1},
        // sc-2
        {4, 0, 0, 2}, {-4, 0, 0, 2}, {0, 4, 0, 2}, {0, -4, 0, 2}, {0, 0, 4, 2}, {0, 0, -4, 2},
        // fcc-1
        {2, 2, 0, 3}, {-2, -2, 0, 3}, {2, -2, 0, 3}, {-2, 2, 0, 3},
        {2, 0, 2, 3}, {-2, 0, -2, 3}, {2, 0, -2, 3}, {-2, 0, 2, 3},
        {0, 2, 2, 3}, {0, -2, -2, 3}, {0, 2, -2, 3}, {0, -2, 2, 3},
        // bcc-1
        {2, 2, 2, 4}, {-2, -2, -2, 4}, {2, 2, -2, 4}, {-2, -2, 2, 4},
        {2, -2, 2, 4}, {-2, 2, -2, 4}, {-2, 2, 2, 4}, {2, -2, -2, 4},
        // bcc-1/2
        {1, 1, 1, 5}, {-1, -1, -1, 5}, {1, 1, -1, 5}, {-1, -1, 1, 5},
        {1, -1, 1, 5}, {-1, 1, -1, 5}, {-1, 1, 1, 5}, {1, -1, -1, 5},
    };
    return t[i];
}

// The velocity table as data, for lookups with a run-time index.
struct VelTable {
    Vel v[kQ];
};
__host__ __device__ constexpr VelTable make_vel_table() {
    VelTable t{};
    for (int i = 0; i < kQ; ++i) t.v[i] = vel(i);
    return t;
}
static __constant__ VelTable c_vel = make_vel_table();

// Per-shell lattice constants in the compute type.
template <class R>
struct Consts {
    R w[kShells];    // weight of one velocity of the shell
    R c2[kShells];   // c^2 of the shell
    R p1[kShells];   // rest equilibrium f~/(w rho) = 1 + eta p1 + eta^2 p2 + eta^3 p3
    R p2[kShells];
    R p3[kShells];
    // Shell sums of the momentum projection as cubics in eta: with R_s = f~_s / (w_s rho) and
    // n2, n4, n22 the sums over shell s of c_x^2, c_x^4, c_x^2 c_y^2,
    //   pj[0](eta) = sum_s w_s n2_s R_s,       pj[1](eta) = sum_s w_s n2_s c_s^2 R_s,
    //   pj[2](eta) = sum_s w_s n4_s R_s,       pj[3](eta) = sum_s w_s n22_s R_s,
    // pj[j](eta) = pj[j][0] + eta (pj[j][1] + eta (pj[j][2] + eta pj[j][3])).
    R pj[4][4];
    R m2[4];         // M_2  (1+eta)^2 = m2[0] + m2[1] eta + m2[2] eta^2 + m2[3] eta^3
    R m2p[4];        // M_2' (1+eta)^2 likewise
    R theta0;
    R inv_3theta0;
};

// What the series step needs, in the type it is used in: S = float or double, or float2 with each
// constant twice, so that the packed two-node kernels read a constant pair in one load.
// Deviation codecs (FP32 arithmetic), with the stored scale folded in:
//   w = w_s / kScale, de = w_s (c_s^2 - 3 theta_0) / kScale, j2 = 2 w[2], j5 = w[5] / 2,
//   rp = (unused, p1, p2, p3)
// FP64, which stores f:
//   w = 2 w_s (w[0] = w_0), de = c_s^2 - 3 theta_0, rp = w_s (1, p1, p2, p3): w_s R_s as a cubic
template <class S>
struct StepConsts {
    S w[kShells], de[kShells], c2[kShells], j2, j5;
    S rp[kShells][4];
    S m2[4], m2p[4];                // as in Consts
    S pj0[4], pj1[4], pj3[4];       // Consts::pj
    S pq[4];                        // pj[2] - 3 pj[3]
    S inv_theta0, inv_3theta0;
};

template <int... Is, class F>
__device__ __forceinline__ void static_for_impl(std::integer_sequence<int, Is...>, F&& f) {
    (f(std::integral_constant<int, Is>{}), ...);
}
template <int N, class F>
__device__ __forceinline__ void static_for(F&& f) {
    static_for_impl(std::make_integer_sequence<int, N>{}, f);
}

// ---------------------------------------------------------------------------
// Storage codecs.  value(): stored element -> working value v (f, or
// kScale * h); dev(v, w / kScale): deviation f - w; relax(): new working value
// from v and x = 2 beta kScale h^eq; to_raw(): rounding to the storage type.
// ---------------------------------------------------------------------------
struct CodecF64 {  // stores f_i
    using raw_t = double;
    using R = double;
    using KS = double;  // type of the lattice constants
    static constexpr bool stores_f = true;
    static constexpr double kScale = 1.0;
    static __device__ __forceinline__ R value(raw_t r) { return r; }
    static __device__ __forceinline__ R dev(R v, R w) { return v - w; }
    static __device__ __forceinline__ R relax(R v, R omb, R x, R w, R tb) { return fma(omb, v, w * (tb + x)); }
    static __device__ __forceinline__ raw_t to_raw(R v) { return v; }
};

struct CodecF32 {  // stores h_i = f_i / w_i - 1
    using raw_t = float;
    using R = float;
    using KS = float;
    static constexpr bool stores_f = false;
    static constexpr double kScale = 1.0;
    using pair_t = float2;
    static __device__ __forceinline__ pair_t pack2(raw_t a, raw_t b) { return make_float2(a, b); }
    static __device__ __forceinline__ float2 unpack2(pair_t p) { return p; }
    static __device__ __forceinline__ R value(raw_t r) { return r; }
    static __device__ __forceinline__ R dev(R v, R w) { return w * v; }
    static __device__ __forceinline__ R relax(R v, R omb, R x, R, R) { return fmaf(omb, v, x); }
    static __device__ __forceinline__ raw_t to_raw(R v) { return v; }
};

// FP16 stores 2^8 h_i: the power-of-two scale is exact and moves FP16's
// subnormal range (|x| < 6.1e-5) down to |h| < 2.4e-7, while |h| up to 255
// stays finite.  The scale is folded into the per-shell constants, so the
// working value v is the stored (scaled) number.
struct CodecF16 {
    using raw_t = __half;
    using R = float;
    using KS = float;
    static constexpr bool stores_f = false;
    static constexpr double kScale = 256.0;
    static __device__ __forceinline__ R value(raw_t r) { return __half2float(r); }
    static __device__ __forceinline__ R dev(R v, R w) { return w * v; }
    static __device__ __forceinline__ R relax(R v, R omb, R x, R, R) { return fmaf(omb, v, x); }
    static __device__ __forceinline__ raw_t to_raw(R v) { return __float2half_rn(v); }
    // two stored elements kept packed in one register
    using pair_t = __half2;
    static __device__ __forceinline__ pair_t pack2(raw_t a, raw_t b) { return __halves2half2(a, b); }
    static __device__ __forceinline__ float2 unpack2(pair_t p) { return __half22float2(p); }
    // (hi of a, lo of b): the pair that starts at an odd element between two aligned pairs
    static __device__ __forceinline__ pair_t straddle(pair_t a, pair_t b) {
        return __halves2half2(__high2half(a), __low2half(b));
    }
    static __device__ __forceinline__ pair_t to_raw2(float2 v) { return __float22half2_rn(v); }
};

struct CodecBF16 {
    using raw_t = __nv_bfloat16;
    using R = float;
    using KS = float;
    static constexpr bool stores_f = false;
    static constexpr double kScale = 1.0;
    static __device__ __forceinline__ R value(raw_t r) { return __bfloat162float(r); }
    static __device__ __forceinline__ R dev(R v, R w) { return w * v; }
    static __device__ __forceinline__ R relax(R v, R omb, R x, R, R) { return fmaf(omb, v, x); }
    static __device__ __forceinline__ raw_t to_raw(R v) { return __float2bfloat16_rn(v); }
    using pair_t = __nv_bfloat162;
    static __device__ __forceinline__ pair_t pack2(raw_t a, raw_t b) { return __halves2bfloat162(a, b); }
    static __device__ __forceinline__ float2 unpack2(pair_t p) { return __bfloat1622float2(p); }
    static __device__ __forceinline__ pair_t straddle(pair_t a, pair_t b) {
        return __halves2bfloat162(__high2bfloat16(a), __low2bfloat16(b));
    }
    static __device__ __forceinline__ pair_t to_raw2(float2 v) { return __float22bfloat162_rn(v); }
};

// ---------------------------------------------------------------------------
// Two nodes per thread: F2 carries one float per node and maps every
// arithmetic operation onto Blackwell's packed FP32x2 instructions
// (__fadd2_rn, __fmul2_rn, __ffma2_rn; each lane rounds exactly as the scalar
// FP32 operation does), halving the FP32 instruction count of the collision.
// ---------------------------------------------------------------------------
struct F2 {
    float2 v;
    __device__ __forceinline__ F2() {}
    __device__ __forceinline__ F2(float s) : v(make_float2(s, s)) {}
    __device__ __forceinline__ F2(double s) : v(make_float2((float)s, (float)s)) {}
    __device__ __forceinline__ F2(int s) : v(make_float2((float)s, (float)s)) {}
    __device__ __forceinline__ F2(float a, float b) : v(make_float2(a, b)) {}
    __device__ __forceinline__ F2(float2 x) : v(x) {}
};
__device__ __forceinline__ F2 operator+(F2 a, F2 b) { return F2(__fadd2_rn(a.v, b.v)); }
__device__ __forceinline__ F2 operator-(F2 a) { return F2(make_float2(-a.v.x, -a.v.y)); }
__device__ __forceinline__ F2 operator-(F2 a, F2 b) { return F2(__fadd2_rn(a.v, (-b).v)); }
__device__ __forceinline__ F2 operator*(F2 a, F2 b) { return F2(__fmul2_rn(a.v, b.v)); }
__device__ __forceinline__ F2 operator/(F2 a, F2 b) { return F2(a.v.x / b.v.x, a.v.y / b.v.y); }
__device__ __forceinline__ F2& operator+=(F2& a, F2 b) {
    a = a + b;
    return a;
}
using ::fma;  // keep the scalar overloads visible next to the F2 one
__device__ __forceinline__ F2 fma(F2 a, F2 b, F2 c) { return F2(__ffma2_rn(a.v, b.v, c.v)); }

// Reciprocals of the node scalars (1/rho, theta0/theta, ...).  FP64 keeps the IEEE division.
// recip: the FP32 hardware approximation (within 2 ulp).
__device__ __forceinline__ double recip(double x) { return 1.0 / x; }
__device__ __forceinline__ float recip(float x) { return __fdividef(1.0f, x); }
__device__ __forceinline__ F2 recip(F2 x) { return F2(__fdividef(1.0f, x.v.x), __fdividef(1.0f, x.v.y)); }
// recip_newton: the approximation and one step of Newton's iteration, r + r (1 - x r).  The approximation is
// biased near 1, where these numbers lie: mean relative error -1.1e-8 over [0.99, 1.01], -1.5e-8 over [1, 1.001].
// After the step the mean, rms and largest errors over 2^20 numbers are the rounded quotient's.
__device__ __forceinline__ double recip_newton(double x) { return 1.0 / x; }
__device__ __forceinline__ float recip_newton(float x) {
    const float r = recip(x);
    return fmaf(r, fmaf(-x, r, 1.0f), r);
}
__device__ __forceinline__ F2 recip_newton(F2 x) {
    const F2 r = recip(x);
    return fma(r, fma(-x, r, F2(1.0f)), r);
}
// The reciprocals of rho and theta / theta0 in a time step with the codec's storage.  FP32 keeps the populations
// to 2^-24, and the bias adds up over the steps: error of h against 64 bits after 100 steps, 21 x 95 x 12, 5.2e-7
// with the Newton step, 2.3e-6 without; 33 x 18 x 20, 1.2e-6 and 3.8e-6; a 256^3 step takes 1.604 ms (1.593), a
// 512^3 one 12.58 (12.58).  The rounding of 16-bit storage (2^-11, 2^-8) hides the bias: the errors are the
// same with and without, and the Newton step would cost 5% of the BF16 step at 256^3 (1.119 against 1.063 ms)
// and 2% of the stochastic one at 512^3.
template <class Codec>
__device__ __forceinline__ typename Codec::R recip_step(typename Codec::R x) {
    return sizeof(typename Codec::raw_t) == 2 ? recip(x) : recip_newton(x);
}

// A product rounded by itself (not contracted into a following addition).
__device__ __forceinline__ double mul(double a, double b) { return a * b; }
__device__ __forceinline__ float mul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ F2 mul(F2 a, F2 b) { return a * b; }

// Two-node codec over a one-node storage codec: same storage, F2 arithmetic.
template <class Base>
struct Codec2 {
    using raw_t = typename Base::raw_t;
    using R = F2;
    using KS = float2;
    static constexpr bool stores_f = Base::stores_f;
    static constexpr double kScale = Base::kScale;
};

// Moments of one node from the deviations d_i = f_i - w_i (Sec. II):
// drho = rho - 1, j = rho u, dk = <f, c^2> - 3 theta_0.
template <class R>
struct NodeMoments {
    R drho, jx, jy, jz, dk;
};

// dget(I) returns d_I for a compile-time population index I.
template <class R, class G>
__device__ __forceinline__ NodeMoments<R> moments_from(G&& dget) {
    NodeMoments<R> m;
    m.drho = dget(std::integral_constant<int, 0>{});
    m.jx = R(0);
    m.jy = R(0);
    m.jz = R(0);
    m.dk = R(0);
    static_for<20>([&](auto K) {
        constexpr int ip = 2 * K + 1, im = 2 * K + 2;
        constexpr Vel c = vel(ip);
        const R dp = dget(std::integral_constant<int, ip>{});
        const R dm = dget(std::integral_constant<int, im>{});
        const R s = dp + dm;
        const R df = dp - dm;
        m.drho += s;
        // c2 components are doubled: c = c2 / 2
        if constexpr (c.x != 0) m.jx = fma(R(0.5 * c.x), df, m.jx);
        if constexpr (c.y != 0) m.jy = fma(R(0.5 * c.y), df, m.jy);
        if constexpr (c.z != 0) m.jz = fma(R(0.5 * c.z), df, m.jz);
        constexpr double csq = 0.25 * (c.x * c.x + c.y * c.y + c.z * c.z);
        m.dk = fma(R(csq), s, m.dk);
    });
    return m;
}

template <class R>
__device__ __forceinline__ NodeMoments<R> moments_from_dev(const R (&d)[kQ]) {
    return moments_from<R>([&](auto I) { return d[I]; });
}

// Primitive variables of a node: rho, u, eta = theta / theta_0 - 1.
template <class R>
struct NodeState {
    R drho, rho, ux, uy, uz, eta;
};

template <class R, class KS>
__device__ __forceinline__ NodeState<R> state_from_moments(const NodeMoments<R>& m, const Consts<KS>& K) {
    NodeState<R> st;
    st.drho = m.drho;
    st.rho = R(1) + m.drho;
    const R inv_rho = recip(st.rho);
    st.ux = m.jx * inv_rho;
    st.uy = m.jy * inv_rho;
    st.uz = m.jz * inv_rho;
    const R usq = st.ux * st.ux + st.uy * st.uy + st.uz * st.uz;
    // theta = (<f,c^2>/rho - u^2)/3  =>  eta = (dk - 3 theta0 drho - rho u^2) / (3 theta0 rho)
    st.eta = (m.dk - R(3) * K.theta0 * m.drho - st.rho * usq) * inv_rho * K.inv_3theta0;
    return st;
}

template <class R>
__device__ __forceinline__ bool state_ok(const NodeState<R>& st) {
    // rho > 0, theta > 0 and both finite (NaN fails every comparison)
    return st.rho > R(0) && st.rho < R(1e30) && st.eta > R(-1) && st.eta < R(1e30) && st.ux == st.ux &&
           st.uy == st.uy && st.uz == st.uz && fabs(st.ux) < R(1e30) && fabs(st.uy) < R(1e30) &&
           fabs(st.uz) < R(1e30);
}

// Two nodes: rho > 0, theta > 0 and |rho| + |eta| + |u_x| + |u_y| + |u_z| below 1e30 for both (a NaN
// or an infinity in any of them fails the last comparison).
__device__ __forceinline__ bool state_ok(const NodeState<F2>& st) {
    const float ma = st.rho.v.x + st.eta.v.x + fabsf(st.ux.v.x) + fabsf(st.uy.v.x) + fabsf(st.uz.v.x);
    const float mb = st.rho.v.y + st.eta.v.y + fabsf(st.ux.v.y) + fabsf(st.uy.v.y) + fabsf(st.uz.v.y);
    return st.rho.v.x > 0.f && st.rho.v.y > 0.f && st.eta.v.x > -1.f && st.eta.v.y > -1.f && ma < 1e30f &&
           mb < 1e30f;
}

// Moments of one node as the fused step uses them: drho = rho - 1, j = rho u and
// de = <f, c^2 - 3 theta_0>, summed by shells.
template <class R>
struct NodeSums {
    R drho, jx, jy, jz, de;
};

// Sums of the working values v = vget(I).  Per +-c pair one sum and one difference; the pair sums are
// added up by shell and weighted once per shell, and the differences are combined along the axes of
// the fcc and bcc shells first (the four diagonals give all three components in seven additions):
// about 100 operations a node, 115 in FP64, against 163 when every deviation is weighted and enters
// drho, j and dk by itself.  FP64 stores f: its pair sums are deviations, (f+ - 2w) + f-, both steps
// exact or within the rounding of f.  Every multiply-add is written as one, so that the scalar and the
// packed two-node forms round alike.
template <class Codec, class VGet>
__device__ __forceinline__ NodeSums<typename Codec::R> node_sums(const StepConsts<typename Codec::KS>& K, VGet&& vget) {
    using R = typename Codec::R;
    constexpr bool kF = Codec::stores_f;
    // sum and difference of the pair ip, ip + 1
    auto pair = [&](auto IP, R& S, R& D) {
        constexpr int ip = decltype(IP)::value;
        const R vp = vget(std::integral_constant<int, ip>{}), vm = vget(std::integral_constant<int, ip + 1>{});
        if constexpr (kF)
            S = (vp - R(K.w[vel(ip).shell])) + vm;
        else
            S = vp + vm;
        D = vp - vm;
    };
    NodeSums<R> m;
    {
        const R v0 = vget(std::integral_constant<int, 0>{});
        if constexpr (kF) {
            m.drho = v0 - R(K.w[0]);
            m.de = m.drho * R(K.de[0]);
        } else {
            m.drho = R(K.w[0]) * v0;
            m.de = R(K.de[0]) * v0;
        }
    }
    // a finished shell's sum H enters drho and de
    auto shell = [&](int s, R H) {
        if constexpr (kF) {
            m.drho = m.drho + H;
            m.de = fma(H, R(K.de[s]), m.de);
        } else {
            m.drho = fma(R(K.w[s]), H, m.drho);
            m.de = fma(R(K.de[s]), H, m.de);
        }
    };
    {  // sc-1 (pairs 1, 3, 5) and sc-2 (7, 9, 11), axis by axis
        R H1, H2;
        auto axis = [&](auto A, R& j) {
            constexpr int k = decltype(A)::value;
            R S1, D1, S2, D2;
            pair(std::integral_constant<int, 1 + 2 * k>{}, S1, D1);
            pair(std::integral_constant<int, 7 + 2 * k>{}, S2, D2);
            if constexpr (kF)
                j = fma(R(2), D2, D1);
            else
                j = fma(R(K.w[1]), D1, R(K.j2) * D2);
            H1 = k == 0 ? S1 : H1 + S1;
            H2 = k == 0 ? S2 : H2 + S2;
        };
        axis(std::integral_constant<int, 0>{}, m.jx);
        axis(std::integral_constant<int, 1>{}, m.jy);
        axis(std::integral_constant<int, 2>{}, m.jz);
        shell(1, H1);
        shell(2, H2);
    }
    {  // fcc-1: (1, 1, 0), (1, -1, 0) and likewise in the xz and yz planes
        R H;
        auto plane = [&](auto IP, R& ja, R& jb) {
            constexpr int ip = decltype(IP)::value;
            R S1, D1, S2, D2;
            pair(std::integral_constant<int, ip>{}, S1, D1);
            pair(std::integral_constant<int, ip + 2>{}, S2, D2);
            const R p = D1 + D2, n = D1 - D2, S = S1 + S2;
            ja = kF ? ja + p : fma(R(K.w[3]), p, ja);
            jb = kF ? jb + n : fma(R(K.w[3]), n, jb);
            H = ip == 13 ? S : H + S;
        };
        plane(std::integral_constant<int, 13>{}, m.jx, m.jy);
        plane(std::integral_constant<int, 17>{}, m.jx, m.jz);
        plane(std::integral_constant<int, 21>{}, m.jy, m.jz);
        shell(3, H);
    }
    {  // bcc-1 (pairs 25 ..) and bcc-1/2 (33 ..) along the diagonals (1,1,1) (1,1,-1) (1,-1,1) (-1,1,1)
        R H4, H5;
        auto diag = [&](auto KD) {
            constexpr int k = decltype(KD)::value;
            R S4, D4, S5, D5;
            pair(std::integral_constant<int, 25 + 2 * k>{}, S4, D4);
            pair(std::integral_constant<int, 33 + 2 * k>{}, S5, D5);
            H4 = k == 0 ? S4 : H4 + S4;
            H5 = k == 0 ? S5 : H5 + S5;
            return kF ? fma(R(0.5), D5, D4) : fma(R(K.j5), D5, R(K.w[4]) * D4);
        };
        const R E0 = diag(std::integral_constant<int, 0>{}), E1 = diag(std::integral_constant<int, 1>{});
        const R p = E0 + E1, r = E0 - E1;
        m.jx = m.jx + p;
        m.jy = m.jy + p;
        m.jz = m.jz + r;
        const R E2 = diag(std::integral_constant<int, 2>{}), E3 = diag(std::integral_constant<int, 3>{});
        const R q = E2 - E3, t = E2 + E3;
        m.jx = m.jx + q;
        m.jy = m.jy - q;
        m.jz = m.jz + t;
        shell(4, H4);
        shell(5, H5);
    }
    return m;
}

// Primitive variables from the shell sums: eta = (de / rho - u^2) / (3 theta_0).
template <class Codec, class R, class KS>
__device__ __forceinline__ NodeState<R> state_from_sums(const NodeSums<R>& m, const StepConsts<KS>& K) {
    NodeState<R> st;
    st.drho = m.drho;
    st.rho = R(1) + m.drho;
    const R inv_rho = recip_step<Codec>(st.rho);
    st.ux = m.jx * inv_rho;
    st.uy = m.jy * inv_rho;
    st.uz = m.jz * inv_rho;
    const R usq = fma(st.ux, st.ux, fma(st.uy, st.uy, st.uz * st.uz));
    st.eta = fma(m.de, inv_rho, -usq) * R(K.inv_3theta0);
    return st;
}

template <class Codec, class VGet>
__device__ __forceinline__ NodeState<typename Codec::R> node_state(const StepConsts<typename Codec::KS>& K, VGet&& vget) {
    return state_from_sums<Codec>(node_sums<Codec>(K, vget), K);
}

// Equilibrium (Eq. feqGenU3, with the optional momentum projection) and BGK relaxation of one node, in
// the fewest operations: v[i] the working values, tb = 2 beta kScale, omb = 1 - 2 beta; sink(I, value)
// receives the new working value of population I.
//
// With up = u / theta, a = up.c and per shell R_s = f~_s / (w_s rho), C_s, D_s (see
// equilibrium_relax_g), a pair's relaxation is
//   v'_+- = omb v_+- + T +- P (a (D_s + a^2 / 6) + c.v),  T = B_s + P a^2 / 2,
//   P = tb rho R_s,  B_s = tb (rho R_s - 1) + P C_s      (deviation codecs)
//   P = tb w_s rho R_s,  B_s = P (1 + C_s)               (FP64, which stores f)
// i.e. four multiply-adds for the pair's common terms and two for each population.  Pairs of one
// direction in two shells (sc-1 and sc-2, bcc-1 and bcc-1/2) share a and a^2: with a = k a_1 the factors
// k and k^2 go into the shell constants.  The projection v = dj / (rho theta) is odd in u along each
// axis: v_a = -up_a (K0 + K1 up_a^2).  About 300 operations a node, against 520 for the direct form.
// RELAX false: sink receives tb h^eq_i (f^eq_i for FP64), no relaxation.  ISO: theta = theta_0 (st.eta is
// not read), where every cubic in eta is its constant term.
template <class Codec, bool PROJECT, bool RELAX = true, bool ISO = false, class VGet, class Sink>
__device__ __forceinline__ void collide(const NodeState<typename Codec::R>& st,
                                        const StepConsts<typename Codec::KS>& K, typename Codec::R tb,
                                        typename Codec::R omb, VGet&& vget, Sink&& sink) {
    using R = typename Codec::R;
    constexpr bool kF = Codec::stores_f;
    const R eta = ISO ? R(0) : st.eta;
    const R it1 = ISO ? R(1) : recip_step<Codec>(R(1) + eta);                // theta_0 / theta
    const R it = ISO ? R(K.inv_theta0) : it1 * R(K.inv_theta0);              // 1 / theta
    const R usq = fma(st.ux, st.ux, fma(st.uy, st.uy, st.uz * st.uz));
    const R g = usq * it;
    const R r2 = it1 * it1;
    auto cubic = [&](const typename Codec::KS(&c)[4]) {
        if constexpr (ISO) return R(c[0]);
        return fma(eta, fma(eta, fma(eta, R(c[3]), R(c[2])), R(c[1])), R(c[0]));
    };
    const R M2 = ISO ? cubic(K.m2) : mul(cubic(K.m2), r2);
    const R A1 = (R(2.5) * M2) * recip(fma(R(2.5), M2, R(1)));
    // A2 = 5 A1 (1 - M2) - (3 + M2' - 5 M2)
    const R A2 = fma(fma(R(-5), M2, R(5)), A1, fma(R(5), M2, fma(-cubic(K.m2p), r2, R(-3))));
    const R nga = (g * A1) * (it * R(-1.0 / 6.0));  // -g A1 / (6 theta)
    const R hg = R(-0.5) * g;
    const R cg = fma(-hg, A1, hg);                  // -g (1 - A1) / 2
    const R gA2 = g * A2;
    const R upx = mul(st.ux, it), upy = mul(st.uy, it), upz = mul(st.uz, it);
    const R x2 = upx * upx, y2 = upy * upy, z2 = upz * upz;
    R vx = R(0), vy = R(0), vz = R(0);
    if constexpr (PROJECT) {
        const R Sp = fma(gA2 * R(1.0 / 6.0), cubic(K.pj0), nga * cubic(K.pj1));
        const R nit = -it;
        const R K0 = nit * fma((it * g) * R(0.5), cubic(K.pj3), Sp);
        const R K1 = (nit * R(1.0 / 6.0)) * cubic(K.pq);
        vx = mul(upx, fma(K1, x2, K0));
        vy = mul(upy, fma(K1, y2, K0));
        vz = mul(upz, fma(K1, z2, K0));
    }
    const R tbr = tb * st.rho, tbd = tb * st.drho, one_cg = R(1) + cg,
            one_dg = fma(gA2, R(1.0 / 6.0), R(1));
    // P and B of shell s
    auto shell = [&](int s, R& P, R& B) {
        if constexpr (kF) {
            P = tbr * cubic(K.rp[s]);
            B = P * fma(nga, R(K.c2[s]), one_cg);
        } else if constexpr (ISO) {
            P = tbr;
            B = fma(P, fma(nga, R(K.c2[s]), cg), tbd);
        } else {
            const R rm1 = eta * fma(eta, fma(eta, R(K.rp[s][3]), R(K.rp[s][2])), R(K.rp[s][1]));
            const R tr = fma(tbr, rm1, tbd);  // tb (rho R_s - 1)
            P = fma(tbr, rm1, tbr);
            B = fma(P, fma(nga, R(K.c2[s]), cg), tr);
        }
    };
    auto Dof = [&](int s) { return fma(nga, R(K.c2[s]), one_dg); };
    {
        R P, B;
        shell(0, P, B);
        if constexpr (RELAX)
            sink(std::integral_constant<int, 0>{}, fma(omb, vget(std::integral_constant<int, 0>{}), B));
        else
            sink(std::integral_constant<int, 0>{}, B);
    }
    // pair ip, ip + 1 along a_1 (its square sq, projection cv = c_1.v): half = k^2 P / 2, odd = k P
    auto pair = [&](auto IP, R a, R sq, R cv, R B, R half, R odd, R sixth, R Ds) {
        const R T = fma(half, sq, B);
        const R m = fma(a, fma(sq, sixth, Ds), cv);
        constexpr std::integral_constant<int, decltype(IP)::value> p{};
        constexpr std::integral_constant<int, decltype(IP)::value + 1> n{};
        if constexpr (RELAX) {
            sink(p, fma(odd, m, fma(omb, vget(p), T)));
            sink(n, fma(odd, -m, fma(omb, vget(n), T)));
        } else {
            sink(p, fma(odd, m, T));
            sink(n, fma(odd, -m, T));
        }
    };
    {
        R P1, B1, P2, B2;
        shell(1, P1, B1);
        shell(2, P2, B2);
        const R h1 = R(0.5) * P1, o2 = R(2) * P2, D1 = Dof(1), D2 = Dof(2);
        const R s1 = R(1.0 / 6.0), s2 = R(4.0 / 6.0);
        pair(std::integral_constant<int, 1>{}, upx, x2, vx, B1, h1, P1, s1, D1);
        pair(std::integral_constant<int, 3>{}, upy, y2, vy, B1, h1, P1, s1, D1);
        pair(std::integral_constant<int, 5>{}, upz, z2, vz, B1, h1, P1, s1, D1);
        pair(std::integral_constant<int, 7>{}, upx, x2, vx, B2, o2, o2, s2, D2);
        pair(std::integral_constant<int, 9>{}, upy, y2, vy, B2, o2, o2, s2, D2);
        pair(std::integral_constant<int, 11>{}, upz, z2, vz, B2, o2, o2, s2, D2);
    }
    const R axy = upx + upy, dxy = upx - upy, cxy = vx + vy, exy = vx - vy;
    {
        R P, B;
        shell(3, P, B);
        const R h = R(0.5) * P, Ds = Dof(3), s6 = R(1.0 / 6.0);
        auto fcc = [&](auto IP, R a, R cv) { pair(IP, a, a * a, cv, B, h, P, s6, Ds); };
        fcc(std::integral_constant<int, 13>{}, axy, cxy);
        fcc(std::integral_constant<int, 15>{}, dxy, exy);
        fcc(std::integral_constant<int, 17>{}, upx + upz, vx + vz);
        fcc(std::integral_constant<int, 19>{}, upx - upz, vx - vz);
        fcc(std::integral_constant<int, 21>{}, upy + upz, vy + vz);
        fcc(std::integral_constant<int, 23>{}, upy - upz, vy - vz);
    }
    {
        R P4, B4, P5, B5;
        shell(4, P4, B4);
        shell(5, P5, B5);
        const R h4 = R(0.5) * P4, h5 = R(0.125) * P5, o5 = R(0.5) * P5;
        const R D4 = Dof(4), D5 = Dof(5), s4 = R(1.0 / 6.0), s5 = R(1.0 / 24.0);
        // the two shells' pairs along the diagonals (1,1,1) (1,1,-1) (1,-1,1) (-1,1,1)
        auto diagonals = [&](auto&& f) {
            f(std::integral_constant<int, 0>{}, axy + upz, cxy + vz);
            f(std::integral_constant<int, 2>{}, axy - upz, cxy - vz);
            f(std::integral_constant<int, 4>{}, dxy + upz, exy + vz);
            f(std::integral_constant<int, 6>{}, upz - dxy, vz - exy);
        };
        auto bcc = [&](auto KD, R a, R sq, R cv) {
            pair(std::integral_constant<int, 25 + decltype(KD)::value>{}, a, sq, cv, B4, h4, P4, s4, D4);
        };
        auto half = [&](auto KD, R a, R sq, R cv) {
            pair(std::integral_constant<int, 33 + decltype(KD)::value>{}, a, sq, cv, B5, h5, o5, s5, D5);
        };
        if constexpr (kF) {  // bound by its operations: a, a^2 and c.v serve both shells
            diagonals([&](auto KD, R a, R cv) {
                const R sq = a * a;
                bcc(KD, a, sq, cv);
                half(KD, a, sq, cv);
            });
        } else {  // bound by registers: one shell's constants at a time
            diagonals([&](auto KD, R a, R cv) { bcc(KD, a, a * a, cv); });
            diagonals([&](auto KD, R a, R cv) { half(KD, a, a * a, cv); });
        }
    }
}

// Equilibrium (Eq. feqGenU3, with the optional momentum projection) and BGK
// relaxation of one node.  v[i] are the working values of the node's incoming
// populations (f or h, see the codec), tb = 2 beta, omb = 1 - 2 beta.
// sink(I, value) receives the new working value of population I.
template <class Codec, bool PROJECT, class VGet, class Sink>
__device__ __forceinline__ void equilibrium_relax_g(const NodeState<typename Codec::R>& st,
                                                    const Consts<typename Codec::KS>& K, typename Codec::R tb,
                                                    typename Codec::R omb, VGet&& vget, Sink&& sink) {
    using R = typename Codec::R;
    const R rho = st.rho, eta = st.eta;
    const R inv_1pe = recip(R(1) + eta);             // theta_0 / theta
    const R inv_theta = inv_1pe / K.theta0;          // 1 / theta
    const R usq = st.ux * st.ux + st.uy * st.uy + st.uz * st.uz;
    const R g = usq * inv_theta;                     // u^2 / theta
    // M_2, M_2' from their exact polynomials; A_1, A_2 (Sec. V)
    const R r2 = inv_1pe * inv_1pe;
    const R M2 = (K.m2[0] + eta * (K.m2[1] + eta * (K.m2[2] + eta * K.m2[3]))) * r2;
    const R M2p = (K.m2p[0] + eta * (K.m2p[1] + eta * (K.m2p[2] + eta * K.m2p[3]))) * r2;
    const R A1 = R(2.5) * M2 * recip(R(1) + R(2.5) * M2);
    const R A2 = R(5) * A1 * (R(1) - M2) - (R(3) + M2p - R(5) * M2);
    // rest-state factors per shell: f~_s = w_s rho R_s, R_s - 1 = eta (p1 + eta (p2 + eta p3));
    // per-shell even constant C_s and odd factor D_s of the series
    //   X_i = C_s + a^2/2 + a D_s + a^3/6,  a = u.c/theta
    //   C_s = -g (1 - A1)/2 - g c_s^2 A1 / (6 theta),  D_s = 1 + g A2 / 6 - g c_s^2 A1 / (6 theta)
    // They are formed where a shell is used (the populations are ordered by shell), which keeps
    // only one shell's factors live at a time.
    const R gA1_6t = g * A1 * inv_theta * R(1.0 / 6.0);
    const R cg = R(-0.5) * g * (R(1) - A1);
    const R dg = g * A2 * R(1.0 / 6.0);
    auto rest_m1 = [&](int s) { return eta * (K.p1[s] + eta * (K.p2[s] + eta * K.p3[s])); };
    auto dm1 = [&](int s) { return dg - gA1_6t * K.c2[s]; };
    const R upx = st.ux * inv_theta, upy = st.uy * inv_theta, upz = st.uz * inv_theta;
    // momentum projection v = dj / (rho theta), dj = rho u - sum_i f^eq_i c_i in closed form:
    //   dj_a = -(u_a/theta) S - [S4 u_a^3 + 3 S22 u_a (u^2 - u_a^2)] / (6 theta^3), with the shell sums
    //   S = sum_s f~_s n2_s (D_s - 1) = rho [dg pj[0] - (g A1 / 6 theta) pj[1]], S4 = rho pj[2],
    //   S22 = rho pj[3] (f~_s = w_s rho R_s, D_s - 1 = dg - (g A1 / 6 theta) c_s^2)
    R vx = R(0), vy = R(0), vz = R(0);
    if constexpr (PROJECT) {
        R S, S4, S22;
        {
            auto pj = [&](int j) { return K.pj[j][0] + eta * (K.pj[j][1] + eta * (K.pj[j][2] + eta * K.pj[j][3])); };
            S = rho * (dg * pj(0) - gA1_6t * pj(1));
            S4 = rho * pj(2);
            S22 = rho * pj(3);
        }
        const R it3 = inv_theta * inv_theta * inv_theta * R(1.0 / 6.0);
        const R ux2 = st.ux * st.ux, uy2 = st.uy * st.uy, uz2 = st.uz * st.uz;
        const R djx = -upx * S - it3 * st.ux * (S4 * ux2 + R(3) * S22 * (usq - ux2));
        const R djy = -upy * S - it3 * st.uy * (S4 * uy2 + R(3) * S22 * (usq - uy2));
        const R djz = -upz * S - it3 * st.uz * (S4 * uz2 + R(3) * S22 * (usq - uz2));
        const R k = inv_theta * recip(rho);
        vx = djx * k;
        vy = djy * k;
        vz = djz * k;
    }
    // rest population: a = 0
    {
        const R rm1 = rest_m1(0);
        const R P0 = tb * (rho + rho * rm1);
        const R x0 = fma(P0, cg - gA1_6t * K.c2[0], tb * (st.drho + rho * rm1));
        sink(std::integral_constant<int, 0>{},
             Codec::relax(vget(std::integral_constant<int, 0>{}), omb, x0, K.w[0], tb));
    }
    R P, B, Ds;  // factors of the current shell
    static_for<20>([&](auto KK) {
        constexpr int ip = 2 * KK + 1, im = 2 * KK + 2;
        constexpr Vel c = vel(ip);
        constexpr int s = c.shell;
        if constexpr (KK == 0 || vel(ip - 2).shell != s) {
            const R rm1 = rest_m1(s);
            P = tb * (rho + rho * rm1);
            B = fma(P, cg - gA1_6t * K.c2[s], tb * (st.drho + rho * rm1));
            Ds = R(1) + dm1(s);
        }
        // p_s = D_s u / theta + v
        R a = R(0), q = R(0);
        if constexpr (c.x != 0) {
            a = fma(R(0.5 * c.x), upx, a);
            q = fma(R(0.5 * c.x), fma(Ds, upx, vx), q);
        }
        if constexpr (c.y != 0) {
            a = fma(R(0.5 * c.y), upy, a);
            q = fma(R(0.5 * c.y), fma(Ds, upy, vy), q);
        }
        if constexpr (c.z != 0) {
            a = fma(R(0.5 * c.z), upz, a);
            q = fma(R(0.5 * c.z), fma(Ds, upz, vz), q);
        }
        const R a2 = a * a;
        const R t = fma(R(0.5) * P, a2, B);
        const R o = fma(P * R(1.0 / 6.0), a2 * a, P * q);
        sink(std::integral_constant<int, ip>{},
             Codec::relax(vget(std::integral_constant<int, ip>{}), omb, t + o, K.w[s], tb));
        sink(std::integral_constant<int, im>{},
             Codec::relax(vget(std::integral_constant<int, im>{}), omb, t - o, K.w[s], tb));
    });
}

__device__ __forceinline__ double expm1_of(double x) { return expm1(x); }
__device__ __forceinline__ float expm1_of(float x) { return expm1f(x); }

__device__ __forceinline__ double log1p_of(double x) { return log1p(x); }
__device__ __forceinline__ float log1p_of(float x) { return log1pf(x); }

// phi(y) = (1 + y) ln(1 + y) - y, the entropy change along the path per unit population.  For
// |y| < 1/8 its series sum_{n >= 2} (-y)^n / (n (n - 1)) (to y^8 in FP32, y^18 in FP64: below
// the unit roundoff of y^2 / 2), else the formula (cancellation at most 16 ulp there).
template <class R>
__device__ __forceinline__ R path_phi(R y) {
    constexpr int N = sizeof(R) == 8 ? 18 : 8;
    if (fabs(y) < R(0.125)) {
        R s = R(0);
#pragma unroll
        for (int n = N; n >= 2; --n) s = fma(s, -y, R(1.0 / (n * (n - 1.0))));
        return s * y * y;
    }
    return (R(1) + y) * log1p_of(y) - y;
}

// Entropic path length alpha of one node (Sec. "Droplet Collision": the update with alpha beta,
// alpha such that the H theorem holds, from x_i = f^eq_i / f_i - 1): the nontrivial root of
// Delta H(alpha) = H(f + alpha (f^eq - f)) - H(f), H = sum_i f_i ln(f_i / w_i).  For an f^eq
// with the moments of f whose logarithm is a sum of collision invariants (the exact entropic
// equilibrium: ln(f^eq_i / w_i) = ln rho + X_i), sum_i f_i x_i (1 + ln(f^eq_i / w_i)) vanishes
// and, with ln(f_i / w_i) = ln(f^eq_i / w_i) - ln(1 + x_i),
//   Delta H(alpha) = sum_i f_i [phi(alpha x_i) - alpha x_i ln(1 + x_i)],
//   d/dalpha     = sum_i f_i x_i [ln(1 + alpha x_i) - ln(1 + x_i)],
// both free of cancellation as x -> 0 (alpha -> 2).  Newton from 2, kept inside (0, alpha_max),
// alpha_max = min over x_i < 0 of -1/x_i; left of Delta H's minimum it doubles alpha instead.
// fw[i] = f_i / w_i, lx[i] = ln(1 + x_i).  Returns 2 (plain BGK) when f = f^eq or when Newton
// does not converge (no root below alpha_max).
template <class R>
__device__ __forceinline__ R entropic_path(const Consts<R>& K, const R (&x)[kQ], const R (&lx)[kQ],
                                           const R (&fw)[kQ]) {
    constexpr bool kDouble = sizeof(R) == 8;
    constexpr int MAXIT = kDouble ? 40 : 30;
    const R tol = kDouble ? R(1e-14) : R(1e-6);
    R amax = R(0), xmax = R(0);  // amax as 1 / alpha_max = max over i of -x_i
#pragma unroll
    for (int i = 0; i < kQ; ++i) {
        amax = fmax(amax, -x[i]);
        xmax = fmax(xmax, fabs(x[i]));
    }
    if (!(xmax > R(0))) return R(2);
    const bool bounded = amax > R(0);
    const R alim = bounded ? R(1) / amax : R(0);
    R a = (!bounded || alim > R(2)) ? R(2) : R(0.5) * alim;
    bool conv = false;
#pragma unroll 1
    for (int it = 0; it < MAXIT; ++it) {
        R g = R(0), dg = R(0);
        static_for<kQ>([&](auto I) {
            const R f = K.w[vel(I).shell] * fw[I], y = a * x[I];
            g = fma(f, path_phi(y) - y * lx[I], g);
            dg = fma(f * x[I], log1p_of(y) - lx[I], dg);
        });
        R an;
        if (!(dg > R(0)))
            an = (!bounded || R(2) * a < alim) ? R(2) * a : R(0.5) * (a + alim);
        else
            an = a - g / dg;
        if (bounded && !(an < alim)) an = R(0.5) * (a + alim);
        if (!(an > R(0))) an = R(0.5) * a;
        conv = dg > R(0) && fabs(an - a) <= tol * an;
        a = an;
        if (conv) break;
    }
    return conv ? a : R(2);
}

// (1 + a)(1 + b) - 1
template <class R>
__device__ __forceinline__ R join(R a, R b) {
    return fma(a, b, a + b);
}

// expm1 of +-l / 2, and sinh(l / 2), cosh(l / 2) - 1, from one exponential: with h = expm1(|l| / 2) and
// r = 1 / (1 + h), expm1(-|l| / 2) = -h r, sinh = h (1 + r) / 2, cosh - 1 = h^2 r / 2 (no cancellation).
template <class R>
struct HalfAngle {
    R p, m, s, c;
    __device__ __forceinline__ explicit HalfAngle(R l) {
        const R h = expm1_of(R(0.5) * fabs(l)), r = R(1) / (R(1) + h), hr = h * r;
        const bool neg = l < R(0);
        p = neg ? -hr : h;
        m = neg ? h : -hr;
        const R sh = R(0.5) * (h + hr);
        s = neg ? -sh : sh;
        c = R(0.5) * (h * hr);
    }
};

// Exact entropic equilibrium (Eqs. (discreteentropiceq) and
// (fivelagrangemultipliersystem)) and BGK relaxation of one node.
//   f^eq_i = w_i rho exp(X_i),  X_i = l0 + l.c_i + l4 (c_i^2 - 3 theta_0),
// with the five multipliers fixed by <f^eq, (1, c, c^2)> = (rho, rho u,
// rho u^2 + 3 rho theta).  Divided by rho and written for the deviations this
// is  sum_i w_i expm1(X_i) phi_i = t,  phi = (1, c, c^2 - 3 theta_0),
// t = (0, u, u^2 + 3 theta_0 eta), which keeps full relative precision of the
// small deviations in FP32.  Newton's method starts from the solution of the
// linearised system (J = diag(1, theta_0, theta_0, theta_0, 6 theta_0^2) at
// rest); once the residual is below `tol` one more step is taken (quadratic
// convergence then leaves round-off), and `ok` is cleared if that does not
// happen within MAXIT steps.
//
// The exponential of X_i is a product of one factor per axis and one of the shell, so the sums over
// a shell's directions are products of hyperbolic functions: with S = sinh l_a, C = cosh l_a - 1 (and
// s, c of l_a / 2), the sum over the fcc directions of the xy plane is 4 (1 + C_x)(1 + C_y), its first
// moment 4 S_x (1 + C_y), its cross moment 4 S_x S_y, and likewise for the others.  A Newton step takes
// six exponentials and about 250 operations for residual and Jacobian, against 41 exponentials and
// about 900 summed direction by direction (64^3 FP32: 44 us a step against 117).  Sums of
// exponentials are kept as deviations throughout (join).
// PATH: the relaxation factor 2 beta becomes alpha beta with the entropic path length alpha of
// entropic_path (tb and 1 - omb scaled by alpha / 2).
template <class Codec, bool PATH = false, class VGet, class Sink>
__device__ __forceinline__ void entropic_relax(const NodeState<typename Codec::R>& st,
                                               const Consts<typename Codec::KS>& K, typename Codec::R tb,
                                               typename Codec::R omb, VGet&& vget, Sink&& sink, bool& ok) {
    using R = typename Codec::R;
    constexpr bool kDouble = sizeof(R) == 8;
    constexpr int MAXIT = kDouble ? 20 : 12;
    const R tol = kDouble ? R(1e-10) : R(3e-5);
    const R th0 = K.theta0;
    const R usq = st.ux * st.ux + st.uy * st.uy + st.uz * st.uz;
    const R t4 = usq + R(3) * th0 * st.eta;
    R l[5] = {R(0), st.ux / th0, st.uy / th0, st.uz / th0, t4 / (R(6) * th0 * th0)};
    const R tgt[5] = {R(0), st.ux, st.uy, st.uz, t4};
    // shell deviations E_s = expm1(l0 + l4 (c_s^2 - 3 theta_0)), c^2 = 0, 1, 4, 2, 3, 3/4
    auto shells = [&](R (&E)[kShells]) {
        const R g = expm1_of(l[4]);
        E[0] = expm1_of(fma(R(-3) * th0, l[4], l[0]));
        E[1] = join(E[0], g);
        E[3] = join(E[1], g);
        E[4] = join(E[3], g);
        E[2] = join(E[4], g);
        E[5] = join(E[0], expm1_of(R(0.75) * l[4]));
    };
    const R w1 = R(2) * K.w[1], w2 = R(2) * K.w[2], w3 = R(4) * K.w[3], w4 = R(8) * K.w[4], w5 = R(8) * K.w[5];
    bool conv = false;
#pragma unroll 1
    for (int it = 0; it < MAXIT; ++it) {
        R E[kShells];
        shells(E);
        R s[3], c[3], S[3], C[3];  // of l_a / 2 and of l_a
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const HalfAngle<R> h(l[1 + a]);
            s[a] = h.s;
            c[a] = h.c;
            S[a] = R(2) * fma(h.s, h.c, h.s);
            C[a] = R(2) * (h.s * h.s);
        }
        // residual F and Jacobian J (upper triangle) of sum w exp(X) phi phi^T
        R F[5], A[5][5];
        const R p0 = K.c2[0] - R(3) * th0, p1 = K.c2[1] - R(3) * th0, p2 = K.c2[2] - R(3) * th0,
                p3 = K.c2[3] - R(3) * th0, p4 = K.c2[4] - R(3) * th0, p5 = K.c2[5] - R(3) * th0;
        // Q: the shells' sums of w expm1(X) over their directions
        const R cyz = join(C[1], C[2]), cxz = join(C[0], C[2]), cxy = join(C[0], C[1]);
        const R hyz = join(c[1], c[2]), hxz = join(c[0], c[2]), hxy = join(c[0], c[1]);
        const R cxyz = join(C[0], cyz), hxyz = join(c[0], hyz);
        R C2[3];  // cosh(2 l_a) - 1
#pragma unroll
        for (int a = 0; a < 3; ++a) C2[a] = R(2) * (S[a] * S[a]);
        const R Q0 = K.w[0] * E[0];
        const R Q1 = w1 * (join(E[1], C[0]) + join(E[1], C[1]) + join(E[1], C[2]));
        const R Q2 = w2 * (join(E[2], C2[0]) + join(E[2], C2[1]) + join(E[2], C2[2]));
        const R Q3 = w3 * (join(E[3], cyz) + join(E[3], cxz) + join(E[3], cxy));
        const R Q4 = w4 * join(E[4], cxyz), Q5 = w5 * join(E[5], hxyz);
        F[0] = (Q0 + Q1) + (Q2 + Q3) + (Q4 + Q5);
        F[4] = fma(p0, Q0, fma(p1, Q1, fma(p2, Q2, fma(p3, Q3, fma(p4, Q4, p5 * Q5)))));
        // sums of w exp(X) over each shell's directions weigh the second moments
        const R T0 = Q0 + K.w[0], T1 = fma(R(3), w1, Q1), T2 = fma(R(3), w2, Q2), T3 = fma(R(3), w3, Q3), T4 = Q4 + w4,
                T5 = Q5 + w5;
        A[0][0] = (T0 + T1) + (T2 + T3) + (T4 + T5);
        A[0][4] = fma(p0, T0, fma(p1, T1, fma(p2, T2, fma(p3, T3, fma(p4, T4, p5 * T5)))));
        A[4][4] = fma(p0 * p0, T0, fma(p1 * p1, T1, fma(p2 * p2, T2, fma(p3 * p3, T3, fma(p4 * p4, T4, p5 * p5 * T5)))));
        const R W1 = fma(w1, E[1], w1), W2 = fma(w2, E[2], w2), W3 = fma(w3, E[3], w3), W4 = fma(w4, E[4], w4),
                W5 = fma(w5, E[5], w5);
        const R H5 = R(0.25) * W5;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const R yz = a == 0 ? cyz : a == 1 ? cxz : cxy, hh = a == 0 ? hyz : a == 1 ? hxz : hxy;
            const R o1 = C[(a + 1) % 3], o2 = C[(a + 2) % 3];
            // the other two axes' factors (1 + C) and (1 + C)(1 + C')
            const R two = R(2) + (o1 + o2), both = R(1) + yz, hboth = R(1) + hh;
            const R m1 = W1 * S[a], m2 = R(4) * W2 * fma(S[a], C[a], S[a]),  // 2 sinh(2 l) = 4 S (1 + C)
                m3 = W3 * (S[a] * two), m4 = W4 * (S[a] * both), m5 = R(0.5) * W5 * (s[a] * hboth);
            const R odd = (m1 + m2) + (m3 + m4) + m5;
            F[1 + a] = odd;
            A[0][1 + a] = odd;
            A[1 + a][4] = fma(p1, m1, fma(p2, m2, fma(p3, m3, fma(p4, m4, p5 * m5))));
            A[1 + a][1 + a] = fma(W1, C[a], W1) + R(4) * fma(W2, C2[a], W2) + W3 * fma(C[a], two, two) +
                              fma(W4, cxyz, W4) + fma(H5, hxyz, H5);
        }
        auto cross = [&](int a, int b, int d) {
            return (S[a] * S[b]) * (W3 + fma(W4, C[d], W4)) + (s[a] * s[b]) * fma(H5, c[d], H5);
        };
        A[1][2] = cross(0, 1, 2);
        A[1][3] = cross(0, 2, 1);
        A[2][3] = cross(1, 2, 0);
        R res = R(0), x[5];
#pragma unroll
        for (int k = 0; k < 5; ++k) {
            x[k] = tgt[k] - F[k];
            res = fmax(res, fabs(x[k]));
        }
        conv = res <= tol;
        if (!(res <= R(1e30))) break;  // NaN or infinity (fmax drops a NaN: see below)
        // solve J d = -F (symmetric positive definite: elimination on the upper triangle)
        R inv[5];
#pragma unroll
        for (int k = 0; k < 5; ++k) {
            inv[k] = R(1) / A[k][k];
#pragma unroll
            for (int r = k + 1; r < 5; ++r) {
                const R f = A[k][r] * inv[k];
#pragma unroll
                for (int q = r; q < 5; ++q) A[r][q] = fma(-f, A[k][q], A[r][q]);
                x[r] = fma(-f, x[k], x[r]);
            }
        }
#pragma unroll
        for (int k = 4; k >= 0; --k) {
            R sum = x[k];
#pragma unroll
            for (int q = k + 1; q < 5; ++q) sum = fma(-A[k][q], x[q], sum);
            x[k] = sum * inv[k];
        }
#pragma unroll
        for (int k = 0; k < 5; ++k) l[k] += x[k];
        if (conv) break;
    }
    // a NaN multiplier (fmax above ignores NaN residuals) fails here
    if (!conv || !(l[0] + l[1] + l[2] + l[3] + l[4] == l[0] + l[1] + l[2] + l[3] + l[4])) ok = false;

    R E[kShells];
    shells(E);
    // axis factors as deviations: half links h, unit links e = (1 + h)^2 - 1, double ones
    R h[3][2], e[3][2];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const HalfAngle<R> ha(l[1 + a]);
        h[a][0] = ha.p;
        h[a][1] = ha.m;
#pragma unroll
        for (int d = 0; d < 2; ++d) e[a][d] = fma(h[a][d], h[a][d], R(2) * h[a][d]);
    }
    // em(I): expm1(X_I)
    auto em_of = [&](auto I) {
        constexpr Vel c = vel(decltype(I)::value);
        if constexpr (c.shell == 0) return E[0];
        constexpr int sx = c.x < 0, sy = c.y < 0, sz = c.z < 0;
        if constexpr (c.shell == 1 || c.shell == 2) {
            constexpr int a = c.x != 0 ? 0 : c.y != 0 ? 1 : 2, d = c.x + c.y + c.z < 0;
            if constexpr (c.shell == 1)
                return join(E[1], e[a][d]);
            else
                return join(E[2], fma(e[a][d], e[a][d], R(2) * e[a][d]));
        } else if constexpr (c.shell == 3) {
            if constexpr (c.z == 0)
                return join(E[3], join(e[0][sx], e[1][sy]));
            else if constexpr (c.y == 0)
                return join(E[3], join(e[0][sx], e[2][sz]));
            else
                return join(E[3], join(e[1][sy], e[2][sz]));
        } else if constexpr (c.shell == 4) {
            return join(E[4], join(join(e[0][sx], e[1][sy]), e[2][sz]));
        } else {
            return join(E[5], join(join(h[0][sx], h[1][sy]), h[2][sz]));
        }
    };
    if constexpr (PATH) {
        // h_i and x_i = f^eq_i / f_i - 1 = (h^eq_i - h_i) / (1 + h_i), h^eq = rho expm1(X) + drho
        auto h_of = [&](auto I) {
            if constexpr (Codec::stores_f)
                return vget(I) / K.w[vel(I).shell] - R(1);
            else
                return vget(I) * R(1.0 / Codec::kScale);
        };
        R x[kQ], lx[kQ], fw[kQ];
        static_for<kQ>([&](auto I) {
            const R heq = st.rho * em_of(I) + st.drho, hi = h_of(I);
            fw[I] = R(1) + hi;
            x[I] = (heq - hi) / fw[I];
            lx[I] = log1p_of(x[I]);
        });
        const R half_alpha = R(0.5) * entropic_path<R>(K, x, lx, fw);
        const R tba = tb * half_alpha, omba = R(1) - (R(1) - omb) * half_alpha;
        // relaxation towards h^eq = h + x (1 + h)
        static_for<kQ>([&](auto I) {
            const R heq = fma(x[I], fw[I], h_of(I));
            sink(I, Codec::relax(vget(I), omba, tba * heq, K.w[vel(I).shell], tba));
        });
    } else {
        // relaxation towards h^eq = rho expm1(X) + drho (FP64: f^eq = w rho (1 + expm1(X)))
        const R tbr = tb * st.rho, tbd = tb * st.drho;
        static_for<kQ>([&](auto I) {
            if constexpr (Codec::stores_f) {
                const R wr = K.w[vel(I).shell] * tbr;
                sink(I, fma(wr, em_of(I), fma(omb, vget(I), wr)));
            } else {
                sink(I, fma(tbr, em_of(I), fma(omb, vget(I), tbd)));
            }
        });
    }
}

// Constants of the step with equilibrium kind EQ: the entropic kinds add the lattice constants.
template <class R>
struct EntropicConsts {
    StepConsts<R> sums;
    Consts<R> lattice;
};
template <class R, int EQ>
using StepK = std::conditional_t<(EQ >= 2), EntropicConsts<R>, StepConsts<R>>;

template <class Codec, int EQ>
__device__ __forceinline__ NodeState<typename Codec::R> step_state(const StepK<typename Codec::R, EQ>& K,
                                                                   const typename Codec::R (&v)[kQ]) {
    auto vget = [&](auto I) { return v[I]; };
    if constexpr (EQ >= 2)
        return node_state<Codec>(K.sums, vget);
    else
        return node_state<Codec>(K, vget);
}

template <class Codec, int EQ, class Sink>
__device__ __forceinline__ void step_relax(const NodeState<typename Codec::R>& st,
                                           const StepK<typename Codec::R, EQ>& K, typename Codec::R tb,
                                           typename Codec::R omb, const typename Codec::R (&v)[kQ], Sink&& sink,
                                           bool& ok) {
    if constexpr (EQ >= 2)
        entropic_relax<Codec, EQ == 3>(st, K.lattice, tb, omb, [&](auto I) { return v[I]; }, sink, ok);
    else
        collide<Codec, EQ == 1>(st, K, tb, omb, [&](auto I) { return v[I]; }, sink);
}

// Equilibrium of a node's fields (initial states, wall columns), term by term: sink receives
// tb h^eq_i (f^eq_i for FP64).
template <class Codec, int EQ, class Sink>
__device__ __forceinline__ void equilibrium_of(const NodeState<typename Codec::R>& st,
                                               const Consts<typename Codec::KS>& K, typename Codec::R tb, Sink&& sink,
                                               bool& ok) {
    using R = typename Codec::R;
    auto zero = [](auto) { return R(0); };
    if constexpr (EQ >= 2)
        entropic_relax<Codec, EQ == 3>(st, K, tb, R(0), zero, sink, ok);
    else
        equilibrium_relax_g<Codec, EQ == 1>(st, K, tb, R(0), zero, sink);
}

// ---------------------------------------------------------------------------
// Stochastic rounding of the BF16 store (lb_set_stochastic_rounding).  A BF16
// number is the upper half of an FP32 bit pattern; adding 16 uniform random
// bits r to the lower half and truncating rounds the magnitude up with
// probability (lower half) / 2^16, so the stored value is unbiased:
//   SR(v; r) = upper half of (bits(v) + r).
// The bits come from a counter-based generator:
//   step key    k_t = H(H(lo(seed) ^ H(hi(seed))) + t),  t = steps since enabling
//   node pair   s_0 = H(k_t ^ (q >> 1)),  q = s nx ny nz + (z ny + y) nx + x
//   population  s_(i+1) = 1664525 s_i + 1013904223 (mod 2^32), i = 0..40 in the
//               library's population order,  w_i = s_(i+1) ^ (s_(i+1) >> 16)
//   r = low 16 bits of w_i for even q, high 16 bits for odd q
// where H is the 32-bit PCG hash of Jarzynski and Olano (Hash Functions for GPU
// Rendering, JCGT 9(3), 2020) and the recurrence is the Numerical Recipes
// linear congruential generator.  The two nodes of an x pair share one word.
// ---------------------------------------------------------------------------
__host__ __device__ constexpr uint32_t pcg_hash(uint32_t x) {
    const uint32_t state = x * 747796405u + 2891336453u;
    const uint32_t word = ((state >> ((state >> 28u) + 4u)) ^ state) * 277803737u;
    return (word >> 22u) ^ word;
}
constexpr uint32_t kSrLcgA = 1664525u, kSrLcgC = 1013904223u;
// s_n = sr_lcg_a(n) s_0 + sr_lcg_c(n) after n steps of the recurrence
__host__ __device__ constexpr uint32_t sr_lcg_a(int n) {
    uint32_t a = 1u;
    for (int k = 0; k < n; ++k) a *= kSrLcgA;
    return a;
}
__host__ __device__ constexpr uint32_t sr_lcg_c(int n) {
    uint32_t c = 0u;
    for (int k = 0; k < n; ++k) c = c * kSrLcgA + kSrLcgC;
    return c;
}
inline uint32_t sr_step_key(uint64_t seed, uint32_t t) {
    return pcg_hash(pcg_hash((uint32_t)seed ^ pcg_hash((uint32_t)(seed >> 32))) + t);
}
// w_I of a node pair with first state s0
template <int I>
__device__ __forceinline__ uint32_t sr_word(uint32_t s0) {
    constexpr uint32_t A = sr_lcg_a(I + 1), C = sr_lcg_c(I + 1);
    const uint32_t s = A * s0 + C;
    return s ^ (s >> 16);
}
__device__ __forceinline__ __nv_bfloat16 sr_bf16(float v, uint32_t r16) {
    return __ushort_as_bfloat16((unsigned short)((__float_as_uint(v) + r16) >> 16));
}
// the pair (v.x, v.y) of nodes q (even) and q + 1 with one word w
__device__ __forceinline__ __nv_bfloat162 sr_bf16x2(float2 v, uint32_t w) {
    const uint32_t lo = __float_as_uint(v.x) + (w & 0xFFFFu);
    const uint32_t hi = __float_as_uint(v.y) + (w >> 16);
    const uint32_t packed = __byte_perm(lo, hi, 0x7632);
    __nv_bfloat162 r;
    memcpy(&r, &packed, 4);
    return r;
}

// Geometry of one population buffer.
struct Dims {
    int nx, ny, nz;
    int64_t plane;  // nx * ny * nz
    int64_t rows;   // 2 * ny * nz
};

// Division of n < 2^31 by a run-time constant d >= 1 as one multiply and shift
// (Granlund and Montgomery, division by invariant integers using
// multiplication, 1994): with 2^k >= d and m = ceil(2^(31+k) / d),
// floor(n / d) = (n m) >> (31 + k).  Proof: write n = q d + r and
// m d = 2^(31+k) + e with 0 <= e < d <= 2^k; then
// n m / 2^(31+k) = q + (r + n e / 2^(31+k)) / d, and n e / 2^(31+k) < 1,
// so the bracket stays below d.  m < 2^32 because d > 2^(k-1) for the
// smallest such k.
struct FastDiv {
    uint32_t m, sh;
};

inline FastDiv make_fastdiv(uint32_t d) {
    uint32_t k = 0;
    while ((1ull << k) < d) ++k;
    FastDiv f;
    f.m = (uint32_t)(((1ull << (31 + k)) + d - 1) / d);
    f.sh = 31 + k;
    return f;
}

__device__ __forceinline__ uint32_t fdiv(uint32_t n, FastDiv f) { return (uint32_t)(((uint64_t)n * f.m) >> f.sh); }

// coordinate of (a) wrapped into [0, n) for a in [-2, n + 1]
__device__ __forceinline__ int wrap(int a, int n) {
    a = a < 0 ? a + n : a;
    a = a < 0 ? a + n : a;
    a = a >= n ? a - n : a;
    a = a >= n ? a - n : a;
    return a;
}

}  // namespace gblb
