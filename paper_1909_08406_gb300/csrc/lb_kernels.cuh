// Kernel templates of the RD3Q41 solver.  Each translation unit that includes
// this header instantiates the kernels for the codecs it needs (FP32-family
// kernels are compiled with double-precision-use warnings enabled).
#pragma once

#include "lb_common.cuh"
#include "lb_launch.h"

namespace gblb {

constexpr int kStepThreads = 128;

// Load paths: the read-only (non-coherent) path for kernels whose inputs are complete before their
// launch, ordinary loads for kernels that start before the kernel that writes their inputs has ended
// (pdl_begin: a non-coherent load may be moved across the wait), and L2-coherent loads for
// persistent kernels that read, after a grid barrier, what other CTAs wrote.  The last two must not be
// moved across the wait or the barrier.  The intrinsics for the 32- and 64-bit types and for the unsigned
// integers are volatile, those for __half, __nv_bfloat16 and their pairs are not (cuda_fp16.hpp,
// cuda_bf16.hpp): the 16-bit types are loaded as integers of their size.
template <class T>
struct LoadWord {
    using type = T;
};
template <>
struct LoadWord<__half> {
    using type = unsigned short;
};
template <>
struct LoadWord<__nv_bfloat16> {
    using type = unsigned short;
};
template <>
struct LoadWord<__half2> {
    using type = unsigned int;
};
template <>
struct LoadWord<__nv_bfloat162> {
    using type = unsigned int;
};
template <class T, class F>
__device__ __forceinline__ T load_as_word(const T* p, F&& load) {
    using W = typename LoadWord<T>::type;
    static_assert(sizeof(W) == sizeof(T), "one word per value");
    static_assert(std::is_same<W, float>::value || std::is_same<W, float2>::value || std::is_same<W, double>::value ||
                      std::is_same<W, unsigned short>::value || std::is_same<W, unsigned int>::value,
                  "a type whose load intrinsic is volatile");
    const W w = load(reinterpret_cast<const W*>(p));
    T v;
    memcpy(&v, &w, sizeof v);
    return v;
}
struct LoadCA {
    template <class T>
    static __device__ __forceinline__ T load(const T* p) {
        return load_as_word(p, [](auto* q) { return __ldca(q); });
    }
};
struct LoadNC {
    template <class T>
    static __device__ __forceinline__ T load(const T* p) {
        return __ldg(p);
    }
};
struct LoadCG {
    template <class T>
    static __device__ __forceinline__ T load(const T* p) {
        return load_as_word(p, [](auto* q) { return __ldcg(q); });
    }
};

template <class T>
struct SameTypeOf {
    using type = T;
};
template <class T>
using SameType = typename SameTypeOf<T>::type;  // a parameter that takes no part in deduction

// Entries of the direct step kernels.  Thread p takes entry p of the grid's x-fastest order, so only
// the last block has idle threads whatever nx is (a block per row chunk left 22% of them idle at
// nx = 150 or 200 and ran 24.9 and 27.4 GMLUPS there with 16-bit storage, against 30.7 and 32.2).
// An entry is a node (kNode), the nodes (y, x) and (y + 1, x) of two rows, y even (kRows; ny even),
// or the nodes x and x + 1, x even (kPair; nx even).
enum EntryKind { kNode, kRows, kPair };

struct EntryGrid {
    uint32_t entries;  // of both sub-lattices, < 2^31
    FastDiv fx, fy;    // by the entries per row, by the rows (row pairs) per plane
};

template <int KIND>
inline EntryGrid entry_grid(const Dims& d) {
    const uint32_t wx = (uint32_t)(KIND == kPair ? d.nx / 2 : d.nx), wy = (uint32_t)(KIND == kRows ? d.ny / 2 : d.ny);
    return EntryGrid{2u * wx * wy * (uint32_t)d.nz, make_fastdiv(wx), make_fastdiv(wy)};
}

// ZSY: rows in (z, s, y) order, so that the two sub-lattices of a plane are visited together.
template <int KIND, bool ZSY = false>
__device__ __forceinline__ bool entry_node(const Dims& d, const EntryGrid& g, int& s, int& z, int& y, int& x) {
    const uint32_t p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= g.entries) return false;
    const uint32_t wx = KIND == kPair ? (uint32_t)d.nx >> 1 : (uint32_t)d.nx;
    const uint32_t wy = KIND == kRows ? (uint32_t)d.ny >> 1 : (uint32_t)d.ny;
    const uint32_t row = fdiv(p, g.fx), zs = fdiv(row, g.fy);
    x = (int)(p - row * wx) * (KIND == kPair ? 2 : 1);
    y = (int)(row - zs * wy) * (KIND == kRows ? 2 : 1);
    if constexpr (ZSY) {
        z = (int)(zs >> 1);
        s = (int)(zs & 1u);
    } else {
        s = zs >= (uint32_t)d.nz;
        z = (int)zs - (s ? d.nz : 0);
    }
    return true;
}

// Base pointers and offsets of the two sub-lattices' populations.  Offsets into a population buffer are
// 32-bit and hold the sub-lattice's start (one add forms a load's offset, one multiply-add its address);
// with WIDE, for grids of 42 nx ny nz >= 2^32 elements, the start is in the base pointers.
template <class T, bool WIDE>
struct SubBases {
    const T *own, *oth;
    uint32_t o_own, o_oth;
    __device__ __forceinline__ SubBases(const T* src, const Dims& d, int s) {
        if constexpr (WIDE) {
            own = src + (size_t)s * kQ * d.plane;
            oth = src + (size_t)(1 - s) * kQ * d.plane;
            o_own = o_oth = 0;
        } else {
            own = oth = src;
            o_own = s ? (uint32_t)kQ * (uint32_t)d.plane : 0u;
            o_oth = s ? 0u : (uint32_t)kQ * (uint32_t)d.plane;
        }
    }
};
template <class T, bool WIDE>
__device__ __forceinline__ T* dst_base(T* dst, const Dims& d, int s) {
    return WIDE ? dst + (size_t)s * kQ * d.plane : dst;
}
inline bool wide_offsets(const Dims& d) { return (uint64_t)(kQ + 1) * (uint64_t)d.plane >= ((uint64_t)1 << 32); }

// Waits for the previous kernel's results.  Launched with the programmatic attribute (launch_entries), a
// step's launch overlaps the previous step's tail: 33 x 18 x 20 nodes, FP32, 100 steps in a row, 2.7 us a
// step against 5.1 without.  Steps do not trigger their successors early (launch_dependents at the start
// of the kernel: 4.4 us, the waiting blocks of later steps take the SMs' slots).
__device__ __forceinline__ void pdl_begin() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

// The gather of one node: v[i] = f*_i(x - c_i, t) in the codec's working value.
template <class Codec, class Ld, bool WIDE>
__device__ __forceinline__ void pull_node(const typename Codec::raw_t* src, const Dims& d, int s, int z, int y, int x,
                                          typename Codec::R (&v)[kQ]) {
    using T = typename Codec::raw_t;
    const uint32_t nx = (uint32_t)d.nx, nxy = nx * (uint32_t)d.ny, plane = (uint32_t)d.plane;
    const SubBases<T, WIDE> b(src, d, s);

    // coordinate / offset of the upwind cell for a shift delta = k - 2 (source = x - delta)
    uint32_t xs[5], yo[5], zo[5];
#pragma unroll
    for (int k = 0; k < 5; ++k) {
        xs[k] = (uint32_t)wrap(x - (k - 2), d.nx);
        yo[k] = (uint32_t)wrap(y - (k - 2), d.ny) * nx;
        zo[k] = (uint32_t)wrap(z - (k - 2), d.nz) * nxy + b.o_own;
    }
    // half links: component +1/2 has delta = 1 - s, component -1/2 has delta = -s
    const uint32_t hxp = s ? xs[2] : xs[3], hxm = s ? xs[1] : xs[2];
    const uint32_t hyp = s ? yo[2] : yo[3], hym = s ? yo[1] : yo[2];
    const uint32_t sub = b.o_oth - b.o_own;
    const uint32_t hzp = (s ? zo[2] : zo[3]) + sub, hzm = (s ? zo[1] : zo[2]) + sub;

    static_for<kQ>([&](auto I) {
        constexpr Vel c = vel(I);
        if constexpr (c.shell == 5) {
            const uint32_t off = (c.z > 0 ? hzp : hzm) + (c.y > 0 ? hyp : hym) + (c.x > 0 ? hxp : hxm);
            v[I] = Codec::value(Ld::load(b.oth + (size_t)I * plane + off));
        } else {
            const uint32_t off = zo[c.z / 2 + 2] + yo[c.y / 2 + 2] + xs[c.x / 2 + 2];
            v[I] = Codec::value(Ld::load(b.own + (size_t)I * plane + off));
        }
    });
}

// Fused pull update (Sec. II) of one node (s, z, y, x): gather f*_i(x - c_i, t)
// for all 41 velocities, compute the moments, the equilibrium and the BGK
// relaxation, and write the 41 post-collision values.  Integer links stay on
// the sub-lattice (shifts 0, +-1, +-2 cells); the bcc-1/2 links come from the
// other sub-lattice: for A (s = 0) a component +1/2 reads cell r - 1 and -1/2
// reads cell r; for B (s = 1) +1/2 reads cell r and -1/2 reads cell r + 1.
// SR: BF16 storage with the stochastic store of lb_common.cuh, step key sr_key.
template <class Codec, int EQ, class Ld = LoadNC, bool SR = false, bool WIDE = true>
__device__ __forceinline__ void step_node(const typename Codec::raw_t* __restrict__ src,
                                          typename Codec::raw_t* __restrict__ dst, const Dims& d,
                                          const StepK<typename Codec::R, EQ>& K, typename Codec::R tb,
                                          int* __restrict__ err, int s, int z, int y, int x, uint32_t sr_key = 0) {
    using R = typename Codec::R;
    using T = typename Codec::raw_t;
    const uint32_t nx = (uint32_t)d.nx, nxy = nx * (uint32_t)d.ny, plane = (uint32_t)d.plane;
    R v[kQ];
    pull_node<Codec, Ld, WIDE>(src, d, s, z, y, x, v);

    const NodeState<R> st = step_state<Codec, EQ>(K, v);
    bool ok = state_ok(st);

    const uint32_t qn = (uint32_t)z * nxy + (uint32_t)y * nx + (uint32_t)x;
    T* out = dst_base<T, WIDE>(dst, d, s) + (SubBases<T, WIDE>(src, d, s).o_own + qn);
    if constexpr (SR) {
        const uint32_t q = (s ? plane : 0u) + qn;
        const uint32_t s0 = pcg_hash(sr_key ^ (q >> 1));
        step_relax<Codec, EQ>(st, K, tb * R(Codec::kScale), R(1) - tb, v,
                              [&](auto I, R val) {
                                  const uint32_t w = sr_word<decltype(I)::value>(s0);
                                  out[(size_t)I * plane] = sr_bf16(val, (q & 1u) ? (w >> 16) : (w & 0xFFFFu));
                              },
                              ok);
    } else {
        step_relax<Codec, EQ>(st, K, tb * R(Codec::kScale), R(1) - tb, v,
                              [&](auto I, R val) { out[(size_t)I * plane] = Codec::to_raw(val); }, ok);
    }
    if (!ok) atomicOr(err, 1);
}

// One node per thread.  EQ: equilibrium kind (see step_relax).
// FP32 arithmetic fits 80 registers (6 blocks per SM), FP64 128 (4).
template <class Codec, int EQ>
constexpr int step_min_blocks() {
    return EQ >= 2 ? 1 : sizeof(typename Codec::R) == 8 ? 4 : 6;
}
template <class Codec, int EQ, bool WIDE, bool SR = false>
__global__ void __launch_bounds__(kStepThreads, step_min_blocks<Codec, EQ>()) k_step(const typename Codec::raw_t* __restrict__ src,
                                                       typename Codec::raw_t* __restrict__ dst, Dims d, EntryGrid g,
                                                       StepK<typename Codec::R, EQ> K, typename Codec::R tb,
                                                       int* __restrict__ err, uint32_t sr_key) {
    int s, z, y, x;
    const bool active = entry_node<kNode>(d, g, s, z, y, x);
    pdl_begin();
    if (active) step_node<Codec, EQ, LoadCA, SR, WIDE>(src, dst, d, K, tb, err, s, z, y, x, sr_key);
}

// Nodes (s, z, y, x) and (s, z, y + 1, x) (y even), packed FP32x2 arithmetic.
template <class Codec, bool PROJECT, class Ld, bool WIDE = true>
__device__ __forceinline__ void step_node2(const typename Codec::raw_t* __restrict__ src,
                                           typename Codec::raw_t* __restrict__ dst, const Dims& d,
                                           const StepConsts<float2>& K, float tb, int* __restrict__ err, int s, int z,
                                           int y, int x) {
    using T = typename Codec::raw_t;
    using C2 = Codec2<Codec>;
    const uint32_t nx = (uint32_t)d.nx, nxy = (uint32_t)d.nx * (uint32_t)d.ny;
    const uint32_t plane = (uint32_t)d.plane;
    const SubBases<T, WIDE> b(src, d, s);

    // source coordinates: x - delta for delta = k - 2; rows y + k - 2 for k = 0..5 (covers
    // y - delta for the first node and y + 1 - delta for the second); planes z - delta
    uint32_t xs[5], yo[6], zo[5];
#pragma unroll
    for (int k = 0; k < 5; ++k) {
        xs[k] = (uint32_t)wrap(x - (k - 2), d.nx);
        zo[k] = (uint32_t)wrap(z - (k - 2), d.nz) * nxy + b.o_own;
    }
#pragma unroll
    for (int k = 0; k < 6; ++k) yo[k] = (uint32_t)wrap(y + k - 2, d.ny) * nx;
    // half links: delta = 1 - s for a +1/2 component, -s for -1/2; the row index is 2 - delta
    const uint32_t hxp = s ? xs[2] : xs[3], hxm = s ? xs[1] : xs[2];
    const uint32_t sub = b.o_oth - b.o_own;
    const uint32_t hzp = (s ? zo[2] : zo[3]) + sub, hzm = (s ? zo[1] : zo[2]) + sub;
    // rows of the +1/2 and -1/2 components for the first and the second node
    const uint32_t hyp[2] = {s ? yo[2] : yo[1], s ? yo[3] : yo[2]}, hym[2] = {s ? yo[3] : yo[2], s ? yo[4] : yo[3]};

    // the two nodes' stored values stay packed (one register per population for 16-bit
    // storage) and are widened to FP32 where they are used
    typename Codec::pair_t pv[kQ];
    static_for<kQ>([&](auto I) {
        constexpr Vel c = vel(I);
        uint32_t oa, ob;
        const T* base;
        if constexpr (c.shell == 5) {
            const uint32_t xz = (c.z > 0 ? hzp : hzm) + (c.x > 0 ? hxp : hxm);
            oa = xz + (c.y > 0 ? hyp[0] : hym[0]);
            ob = xz + (c.y > 0 ? hyp[1] : hym[1]);
            base = b.oth;
        } else {
            const uint32_t xz = zo[c.z / 2 + 2] + xs[c.x / 2 + 2];
            oa = xz + yo[2 - c.y / 2];
            ob = xz + yo[3 - c.y / 2];
            base = b.own;
        }
        const T* p = base + (size_t)I * plane;
        pv[I] = Codec::pack2(Ld::load(p + oa), Ld::load(p + ob));
    });
    auto vget = [&](auto I) { return F2(Codec::unpack2(pv[I])); };

    const NodeState<F2> st = node_state<C2>(K, vget);
    if (!state_ok(st)) atomicOr(err, 1);

    T* outa = dst_base<T, WIDE>(dst, d, s) + (b.o_own + (uint32_t)z * nxy + (uint32_t)y * nx + (uint32_t)x);
    collide<C2, PROJECT>(st, K, F2(tb * (float)Codec::kScale), F2(1.f - tb), vget, [&](auto I, F2 val) {
        T* p = outa + (size_t)I * plane;
        p[0] = Codec::to_raw(val.v.x);
        p[nx] = Codec::to_raw(val.v.y);
    });
}

// Two rows per thread (FP32 arithmetic, any storage except FP64; ny even).
template <class Codec, bool PROJECT, int MINB, bool WIDE>
__global__ void __launch_bounds__(kStepThreads, MINB) k_step2(const typename Codec::raw_t* __restrict__ src,
                                                              typename Codec::raw_t* __restrict__ dst, Dims d,
                                                              EntryGrid g, StepConsts<float2> K, float tb,
                                                              int* __restrict__ err) {
    int s, z, y, x;
    const bool active = entry_node<kRows>(d, g, s, z, y, x);
    pdl_begin();
    if (active) step_node2<Codec, PROJECT, LoadCA, WIDE>(src, dst, d, K, tb, err, s, z, y, x);
}

// The gather of the x pair (s, z, y, x), (s, z, y, x + 1), x even, nx even, 16-bit storage.  Each plane is
// read as aligned pairs of 16-bit values: one 32-bit load when the plane's x shift is even, two loads
// and a byte permute when it is odd.
template <class Codec, bool WIDE>
__device__ __forceinline__ void pull_pair(const typename Codec::raw_t* src, const Dims& d, int s, int z, int y, int x,
                                          typename Codec::pair_t (&pv)[kQ]) {
    using T = typename Codec::raw_t;
    using P = typename Codec::pair_t;
    const uint32_t nx = (uint32_t)d.nx, nxy = nx * (uint32_t)d.ny, plane = (uint32_t)d.plane;
    const SubBases<T, WIDE> b(src, d, s);
    uint32_t yo[5], zo[5];
#pragma unroll
    for (int k = 0; k < 5; ++k) {
        yo[k] = (uint32_t)wrap(y - (k - 2), d.ny) * nx;
        zo[k] = (uint32_t)wrap(z - (k - 2), d.nz) * nxy + b.o_own;
    }
    const uint32_t sub = b.o_oth - b.o_own;
    const uint32_t hyp = s ? yo[2] : yo[3], hym = s ? yo[1] : yo[2];
    const uint32_t hzp = (s ? zo[2] : zo[3]) + sub, hzm = (s ? zo[1] : zo[2]) + sub;
    // aligned pair starts: x - 2, x, x + 2 (periodic; nx even keeps them even)
    const uint32_t xm = (uint32_t)wrap(x - 2, d.nx), x0 = (uint32_t)x, xq = (uint32_t)wrap(x + 2, d.nx);
    // half links along x: A's +1/2 component straddles the pairs x - 2 and x, B's -1/2 one the pairs x
    // and x + 2; the other two are the pair x itself (both pairs of the permute at x, a whole taken)
    const uint32_t hlo = s ? x0 : xm, hhi = s ? xq : x0;
    const uint32_t sel_p = s ? 0x7654u : 0x5432u, sel_m = s ? 0x5432u : 0x3210u;

    static_for<kQ>([&](auto I) {
        constexpr Vel c = vel(I);
        const T* base = (c.shell == 5 ? b.oth : b.own) + (size_t)I * plane;
        auto ld = [&](uint32_t off) { return LoadCA::load(reinterpret_cast<const P*>(base + off)); };
        if constexpr (c.shell == 5) {
            const uint32_t row = (c.z > 0 ? hzp : hzm) + (c.y > 0 ? hyp : hym);
            const P lo = ld(row + (c.x > 0 ? hlo : x0)), hi = ld(row + (c.x > 0 ? x0 : hhi));
            uint32_t wl, wh;
            memcpy(&wl, &lo, 4);
            memcpy(&wh, &hi, 4);
            const uint32_t w = __byte_perm(wl, wh, c.x > 0 ? sel_p : sel_m);
            memcpy(&pv[I], &w, 4);
        } else {
            const uint32_t row = zo[c.z / 2 + 2] + yo[c.y / 2 + 2];
            if constexpr (c.x == 4)
                pv[I] = ld(row + xm);
            else if constexpr (c.x == 2)
                pv[I] = Codec::straddle(ld(row + xm), ld(row + x0));
            else if constexpr (c.x == 0)
                pv[I] = ld(row + x0);
            else if constexpr (c.x == -2)
                pv[I] = Codec::straddle(ld(row + x0), ld(row + xq));
            else
                pv[I] = ld(row + xq);
        }
    });
}

// The values stay packed from here to their use: without the barrier the compiler keeps the 82 widened
// numbers of the moment sums alive and spills more.
template <class Codec>
__device__ __forceinline__ void keep_packed(typename Codec::pair_t (&pv)[kQ]) {
    static_for<kQ>([&](auto I) {
        uint32_t w;
        memcpy(&w, &pv[I], sizeof w);
        asm volatile("" : "+r"(w));
        memcpy(&pv[I], &w, sizeof w);
    });
}

// Two x-adjacent nodes (s, z, y, x) and (s, z, y, x + 1), x even, per thread (16-bit storage, nx
// even), packed FP32x2 arithmetic; the two results of a plane are written with one 32-bit store.
//
// Bound by the latency of its dependent arithmetic at the warps that fit: 128 registers (4 blocks, 16
// warps per SM, 24 bytes of spills); 32.9 GMLUPS on 256^3 with FP16 storage, 80% of the copy bandwidth
// (a block per row chunk with the next row prefetched into L2: 32.2; 168 registers, 12 warps: 29.4).
// SR: BF16 storage with the stochastic store of lb_common.cuh, step key sr_key (one word per
// population and x pair).
template <class Codec, bool PROJECT, bool WIDE, bool SR = false>
__global__ void __launch_bounds__(kStepThreads, 4) k_step2x(const typename Codec::raw_t* __restrict__ src,
                                                            typename Codec::raw_t* __restrict__ dst, Dims d,
                                                            EntryGrid g, StepConsts<float2> K, float tb,
                                                            int* __restrict__ err, uint32_t sr_key) {
    using T = typename Codec::raw_t;
    using P = typename Codec::pair_t;
    using C2 = Codec2<Codec>;
    int s, z, y, x;
    const bool active = entry_node<kPair>(d, g, s, z, y, x);
    pdl_begin();
    if (!active) return;
    P pv[kQ];
    pull_pair<Codec, WIDE>(src, d, s, z, y, x, pv);
    auto vget = [&](auto I) { return F2(Codec::unpack2(pv[I])); };
    const NodeState<F2> st = node_state<C2>(K, vget);
    if (!state_ok(st)) atomicOr(err, 1);
    keep_packed<Codec>(pv);
    const uint32_t plane = (uint32_t)d.plane;
    const uint32_t qn = ((uint32_t)z * (uint32_t)d.ny + (uint32_t)y) * (uint32_t)d.nx + (uint32_t)x;
    T* out = dst_base<T, WIDE>(dst, d, s) + (SubBases<T, WIDE>(src, d, s).o_own + qn);
    uint32_t s0 = 0;
    if constexpr (SR) s0 = pcg_hash(sr_key ^ (((s ? plane : 0u) + qn) >> 1));
    collide<C2, PROJECT>(st, K, F2(tb * (float)Codec::kScale), F2(1.f - tb), vget, [&](auto I, F2 val) {
        P* o = reinterpret_cast<P*>(out + (size_t)I * plane);
        if constexpr (SR)
            *o = sr_bf16x2(val.v, sr_word<decltype(I)::value>(s0));
        else
            *o = Codec::to_raw2(val.v);
    });
}

// Entries that leave an SM fewer than this many warps: where the choice of the kernel is the library's, it
// takes one node per thread there (the same bits), as latency counts, not work per thread.  Microseconds a
// step, one node against two: FP16 pairs 2.39 to 2.69 at 12 x 6 x 6, 2.55 to 2.79 at 24 x 20 x 20, 3.52 to
// 3.48 at 28^3, 4.68 to 3.59 at 40 x 30 x 30; FP32 rows 2.26 to 2.90, 2.48 to 2.92, 3.69 to 3.87, 4.43 to 4.18.
constexpr int64_t kSms = 152;
template <int KIND>
inline bool few_entries(const Dims& d) {
    const int64_t warps = KIND == kPair ? 4 : 8;
    return d.plane < kSms * warps * 32;  // entries of two nodes: as many as cells
}

// Launches `kern`, one thread per entry, with the programmatic attribute (pdl_begin).  Blocks of
// 128 threads, smaller ones where those would leave fewer than eight per SM, down to a warp, so that the
// last wave is short.
template <class... A>
inline cudaError_t launch_linear(void (*kern)(A...), uint32_t entries, cudaStream_t st, const SameType<A>&... args) {
    constexpr uint32_t kEnough = (uint32_t)kSms * 8u;
    const uint32_t th = entries >= kEnough * 128u ? 128u : entries >= kEnough * 64u ? 64u : 32u;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((entries + th - 1) / th);
    cfg.blockDim = dim3(th);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, args...);
}

template <int KIND, class T, class... A>
inline cudaError_t launch_entries(void (*kern)(const T*, T*, Dims, EntryGrid, A...), const void* src, void* dst,
                                  const Dims& d, cudaStream_t st, const SameType<A>&... args) {
    if (d.plane >= ((int64_t)1 << 30)) return cudaErrorInvalidValue;  // 32-bit entries (such a state exceeds the memory)
    const EntryGrid g = entry_grid<KIND>(d);
    return launch_linear(kern, g.entries, st, static_cast<const T*>(src), static_cast<T*>(dst), d, g, args...);
}

// Populations = equilibrium of the given float64 fields, for nodes
// q in [q0, q0 + count), q = s * plane + (z * ny + y) * nx + x.  Field
// pointers are indexed by q - q0 (u component c at c * ustride + q - q0).
template <class Codec, int EQ>
__global__ void __launch_bounds__(256) k_init(typename Codec::raw_t* __restrict__ dst, Dims d, Consts<typename Codec::R> K,
                                              double theta0, double inv_theta0, int64_t q0, int64_t count,
                                              const double* __restrict__ rho, const double* __restrict__ u,
                                              int64_t ustride, const double* __restrict__ theta,
                                              int* __restrict__ err) {
    using R = typename Codec::R;
    const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= count) return;
    const int64_t q = q0 + k;
    const int s = q >= d.plane;
    const int64_t node = q - s * d.plane;
    NodeState<R> st;
    st.drho = (R)(rho[k] - 1.0);
    st.rho = (R)rho[k];
    st.ux = (R)u[k];
    st.uy = (R)u[ustride + k];
    st.uz = (R)u[2 * ustride + k];
    st.eta = (R)((theta[k] - theta0) * inv_theta0);
    bool ok = state_ok(st);
    typename Codec::raw_t* out = dst + (int64_t)s * kQ * d.plane + node;
    equilibrium_of<Codec, EQ>(st, K, R(Codec::kScale),
                              [&](auto I, R val) { out[(int64_t)I * d.plane] = Codec::to_raw(val); }, ok);
    if (!ok) atomicOr(err, 1);
}

// An FP32 number as the FP64 number of the same value, by integer operations where it is normal:
// GB300's FP64 pipe, which also carries the conversions, takes two lanes per clock and SM, and the
// kernels below are bound by it before HBM if they convert in it (export of 129 M FP16 values
// 0.54 ms with, 0.30 ms without).  The call keeps the conversion out of the normal numbers' path.
static __device__ __noinline__ double widen_rare(float v) { return (double)v; }
__device__ __forceinline__ double widen(float v) {
    const uint32_t u = __float_as_uint(v), e = (u >> 23) & 0xffu;
    if (e - 1u < 254u)
        return __hiloint2double((int)((u & 0x80000000u) | (((u & 0x7fffffffu) >> 3) + 0x38000000u)), (int)(u << 29));
    return widen_rare(v);
}

template <class Codec>
__device__ __forceinline__ NodeMoments<typename Codec::R> node_moments_at(const typename Codec::raw_t* __restrict__ src,
                                                                          const Dims& d, int64_t q,
                                                                          const Consts<typename Codec::R>& K) {
    using R = typename Codec::R;
    const int s = q >= d.plane;
    const int64_t node = q - s * d.plane;
    const typename Codec::raw_t* base = src + (int64_t)s * kQ * d.plane + node;
    R dv[kQ];
    constexpr R inv_scale = R(1.0 / Codec::kScale);
    static_for<kQ>([&](auto I) {
        dv[I] = Codec::dev(Codec::value(base[(int64_t)I * d.plane]), K.w[vel(I).shell] * inv_scale);
    });
    return moments_from_dev(dv);
}

// Moments of nodes q in [q0, q0 + count) into float64 fields indexed by q - q0.
template <class Codec>
__global__ void __launch_bounds__(256) k_moments(const typename Codec::raw_t* __restrict__ src, Dims d,
                                                 Consts<typename Codec::R> K, double theta0, int64_t q0, int64_t count,
                                                 double* __restrict__ rho, double* __restrict__ u, int64_t ustride,
                                                 double* __restrict__ theta) {
    using R = typename Codec::R;
    const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= count) return;
    const NodeMoments<R> m = node_moments_at<Codec>(src, d, q0 + k, K);
    const NodeState<R> st = state_from_moments(m, K);
    auto to_f64 = [](R v) {
        if constexpr (sizeof(R) == 4)
            return widen(v);
        else
            return v;
    };
    if (rho) rho[k] = 1.0 + to_f64(m.drho);
    if (u) {
        u[k] = to_f64(st.ux);
        u[ustride + k] = to_f64(st.uy);
        u[2 * ustride + k] = to_f64(st.uz);
    }
    if (theta) theta[k] = fma(to_f64(st.eta), theta0, theta0);
}

constexpr int kRedThreads = 256;

// The five sums (drho, jx, jy, jz, dk) of the V consecutive nodes that start at node q, as FP64
// additions to acc.  V = 2 (FP32 arithmetic): one aligned two-element load per population, packed
// FP32x2 arithmetic; each node's five values are the ones V = 1 forms.
template <class Codec, int V>
__device__ __forceinline__ void add_node_sums(const typename Codec::raw_t* __restrict__ src, const Dims& d, int64_t q,
                                              const Consts<typename Codec::R>& K, double (&acc)[5]) {
    if constexpr (V == 1) {
        const NodeMoments<typename Codec::R> m = node_moments_at<Codec>(src, d, q, K);
        acc[0] += (double)m.drho;
        acc[1] += (double)m.jx;
        acc[2] += (double)m.jy;
        acc[3] += (double)m.jz;
        acc[4] += (double)m.dk;
    } else {
        using P = typename Codec::pair_t;
        const int s = q >= d.plane;
        const typename Codec::raw_t* base = src + (int64_t)s * (kQ - 1) * d.plane + q;
        P v[kQ];
        static_for<kQ>([&](auto I) { v[I] = __ldg(reinterpret_cast<const P*>(base + (int64_t)I * d.plane)); });
        constexpr float inv_scale = (float)(1.0 / Codec::kScale);
        const NodeMoments<F2> m = moments_from<F2>(
            [&](auto I) { return F2(K.w[vel(I).shell] * inv_scale) * F2(Codec::unpack2(v[I])); });
        const F2 part[5] = {m.drho, m.jx, m.jy, m.jz, m.dk};
#pragma unroll
        for (int k = 0; k < 5; ++k) {
            acc[k] += widen(part[k].v.x);
            acc[k] += widen(part[k].v.y);
        }
    }
}

template <class Codec>
constexpr int sum_width() {
    return sizeof(typename Codec::R) == 4 ? 2 : 1;
}
// Resident blocks per SM that the summing kernel's registers are sized for (80 and up to 128 a
// thread, so that a node's 41 loads are in flight together); its grid is one wave of them.
template <class Codec>
constexpr int sum_blocks_per_sm() {
    return sizeof(typename Codec::raw_t) == 2 ? 3 : 2;
}
// The paired loads need an even number of nodes in every plane and an aligned base.
template <class Codec>
inline bool sum_vector_ok(const void* src, const Dims& d) {
    constexpr int V = sum_width<Codec>();
    return V > 1 && ((int64_t)d.nx * d.ny) % V == 0 &&
           reinterpret_cast<uintptr_t>(src) % (V * sizeof(typename Codec::raw_t)) == 0;
}

// Per-block FP64 partial sums of (drho, jx, jy, jz, dk) over all nodes, in a
// fixed order (grid-stride loop, then a shared-memory tree): deterministic
// for a given grid size.
// Over the planes [z0, z0 + nzr) of both sub-lattices (all of them: z0 = 0, nzr = nz).
template <class Codec, int V>
__global__ void __launch_bounds__(kRedThreads, sum_blocks_per_sm<Codec>())
    k_conserved(const typename Codec::raw_t* __restrict__ src, Dims d, Consts<typename Codec::R> K,
                double* __restrict__ partials, int64_t z0, int64_t nzr) {
    double acc[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
    const int64_t nxy = (int64_t)d.nx * d.ny, span = nzr * nxy, n = 2 * span;
    for (int64_t j = ((int64_t)blockIdx.x * kRedThreads + threadIdx.x) * V; j < n;
         j += (int64_t)gridDim.x * kRedThreads * V) {
        const int64_t q = j < span ? z0 * nxy + j : d.plane + z0 * nxy + (j - span);
        add_node_sums<Codec, V>(src, d, q, K, acc);
    }
    __shared__ double sh[5][kRedThreads];
#pragma unroll
    for (int k = 0; k < 5; ++k) sh[k][threadIdx.x] = acc[k];
    __syncthreads();
    for (int w = kRedThreads / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w)
#pragma unroll
            for (int k = 0; k < 5; ++k) sh[k][threadIdx.x] += sh[k][threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0)
#pragma unroll
        for (int k = 0; k < 5; ++k) partials[(int64_t)blockIdx.x * 5 + k] = sh[k][0];
}

// Sum of the per-block partials in a fixed order: thread t adds blocks t, t + 256, ..., then a
// shared-memory tree; sh[k][0] holds the five sums.
__device__ __forceinline__ void reduce_partials(const double* __restrict__ partials, int nblocks,
                                                double (&sh)[5][kRedThreads]) {
    double acc[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
    for (int b = threadIdx.x; b < nblocks; b += kRedThreads)
#pragma unroll
        for (int k = 0; k < 5; ++k) acc[k] += partials[(int64_t)b * 5 + k];
#pragma unroll
    for (int k = 0; k < 5; ++k) sh[k][threadIdx.x] = acc[k];
    __syncthreads();
    for (int w = kRedThreads / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w)
#pragma unroll
            for (int k = 0; k < 5; ++k) sh[k][threadIdx.x] += sh[k][threadIdx.x + w];
        __syncthreads();
    }
}

// c d of an FP64 number d and c = chi + clo as an FP32 number, |error| below (1/2 + 2^-20) ulp:
// d splits exactly into its upper 24 and lower 29 bits (integer operations), the product is formed
// in two FP32 terms.  Exponents outside [-70, 60] (and zero, infinities, NaN) take FP64 arithmetic.
static __device__ __noinline__ float scale_rare(double d, float chi, float clo) {
    return (float)(d * ((double)chi + (double)clo));
}
__device__ __forceinline__ float scale_to_float(double d, float chi, float clo) {
    const uint32_t h = (uint32_t)__double2hiint(d), l = (uint32_t)__double2loint(d);
    const uint32_t e = (h >> 20) & 0x7ffu;
    if (e - 953u > 130u) return scale_rare(d, chi, clo);
    const uint32_t sign = h & 0x80000000u;
    const float hi = __uint_as_float(sign | ((e - 896u) << 23) | ((h & 0xfffffu) << 3) | (l >> 29));
    // the lower 29 bits in units of 2^(e - 1023 - 52)
    const float unit = __uint_as_float(sign | ((e - 896u - 52u) << 23));
    const float lo = __uint2float_rn(l & 0x1fffffffu) * unit;
    const float p = mul(hi, chi);  // rounded by itself: r holds what the rounding leaves
    float r = fmaf(hi, chi, -p);
    r = fmaf(hi, clo, r);
    r = fmaf(lo, chi, r);
    return __fadd_rn(p, r);
}

// Raw storage <-> float64 populations for elements e in [e0, e0 + count) of the
// [s][41][nz][ny][nx] array; the float64 side is indexed by e - e0.  blockIdx.y counts the
// (sub-lattice, population) planes from the one that holds e0, so that the weight is uniform in a
// block and no element index is divided; a block covers kConvPer x 256 elements of its plane, each
// thread kConvPer of them 256 apart.
constexpr int kConvPer = 4;

template <class F>
__device__ __forceinline__ void for_plane_elements(int64_t plane, int64_t e0, int64_t count, F&& body) {
    const int64_t p = e0 / plane + blockIdx.y, first = p * plane;
    const int i = (int)(p % kQ);
    const int64_t lo = max(first, e0), hi = min(first + plane, e0 + count);
    const int64_t e = first + (int64_t)blockIdx.x * (kConvPer * 256) + threadIdx.x;
    body(i, e, lo, hi);
}

// FP64 work per element: one fused multiply-add (from storage), one subtraction (to storage); the
// conversions and the scaling are FP32 and integer operations.
template <class Codec>
__global__ void __launch_bounds__(256) k_to_f64(const typename Codec::raw_t* __restrict__ src, int64_t plane, W41 w,
                                                int64_t e0, int64_t count, double* __restrict__ f) {
    for_plane_elements(plane, e0, count, [&](int i, int64_t e, int64_t lo, int64_t hi) {
        const double wi = w.w[i], ws = wi * (1.0 / Codec::kScale);
        typename Codec::raw_t r[kConvPer];
#pragma unroll
        for (int k = 0; k < kConvPer; ++k)
            if (e + 256 * k >= lo && e + 256 * k < hi) r[k] = src[e + 256 * k];
#pragma unroll
        for (int k = 0; k < kConvPer; ++k) {
            if (e + 256 * k < lo || e + 256 * k >= hi) continue;
            if constexpr (Codec::stores_f)
                f[e + 256 * k - e0] = r[k];
            else
                f[e + 256 * k - e0] = fma(widen(Codec::value(r[k])), ws, wi);
        }
    });
}

template <class Codec>
__global__ void __launch_bounds__(256) k_from_f64(const double* __restrict__ f, int64_t plane, W41 w, int64_t e0,
                                                  int64_t count, typename Codec::raw_t* __restrict__ dst) {
    for_plane_elements(plane, e0, count, [&](int i, int64_t e, int64_t lo, int64_t hi) {
        const double wi = w.w[i];
        const float chi = w.chi[i] * (float)Codec::kScale, clo = w.clo[i] * (float)Codec::kScale;
        double v[kConvPer];
#pragma unroll
        for (int k = 0; k < kConvPer; ++k)
            if (e + 256 * k >= lo && e + 256 * k < hi) v[k] = f[e + 256 * k - e0];
#pragma unroll
        for (int k = 0; k < kConvPer; ++k) {
            if (e + 256 * k < lo || e + 256 * k >= hi) continue;
            if constexpr (Codec::stores_f)
                dst[e + 256 * k] = v[k];
            else
                dst[e + 256 * k] = Codec::to_raw(scale_to_float(v[k] - wi, chi, clo));
        }
    });
}

}  // namespace gblb
