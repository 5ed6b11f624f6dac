// hg_device.cuh -- device code of the stream-collide kernel, shared by the
// translation units that instantiate it (hg_sc_part.cu, compiled once per storage
// type, scheme and launch parity, in parallel) and by hg_kernels.cu,
// whose read-back and boundary kernels use the same lattice tables, storage
// traits and collision.  Everything here has internal linkage, so each
// translation unit owns the instantiations it makes.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

#include "hg_internal.h"

namespace hg {
namespace {

// ---- D3Q19 (rest; +x,-x,+y,-y,+z,-z; 12 diagonals in opposite pairs) ----
__host__ __device__ constexpr int CX(int i) {
    return (i == 1 || i == 7 || i == 9 || i == 11 || i == 13) ? 1
         : (i == 2 || i == 8 || i == 10 || i == 12 || i == 14) ? -1 : 0;
}
__host__ __device__ constexpr int CY(int i) {
    return (i == 3 || i == 7 || i == 10 || i == 15 || i == 17) ? 1
         : (i == 4 || i == 8 || i == 9 || i == 16 || i == 18) ? -1 : 0;
}
__host__ __device__ constexpr int CZ(int i) {
    return (i == 5 || i == 11 || i == 14 || i == 15 || i == 18) ? 1
         : (i == 6 || i == 12 || i == 13 || i == 16 || i == 17) ? -1 : 0;
}
__host__ __device__ constexpr int OPP(int i) { return i == 0 ? 0 : ((i & 1) ? i + 1 : i - 1); }
__host__ __device__ constexpr float W(int i) {
    return i == 0 ? (1.0f / 3.0f) : (i <= 6 ? (1.0f / 18.0f) : (1.0f / 36.0f));
}
__host__ __device__ constexpr double WD(int i) {
    return i == 0 ? (1.0 / 3.0) : (i <= 6 ? (1.0 / 18.0) : (1.0 / 36.0));
}

// Lattice weights in FP32 as an unevaluated sum hi + lo (hi = w rounded to FP32,
// lo = the remainder rounded to FP32): a product w x is formed as fma(hi, x, lo x),
// good to about one rounding of the product.  With w rounded once to FP32 every
// product would carry the weight's own relative error (up to 3e-8, the same sign at
// every site and step), so the FP32 equilibrium would gain or lose mass and momentum
// by that fraction in every collision -- a bias that accumulates over thousands of
// steps, where the rounding of the products themselves varies and averages out.
__host__ __device__ constexpr float WLO(int i) { return (float)(WD(i) - (double)W(i)); }
template <int I> __device__ __forceinline__ float mulw(float x) {
    return __fmaf_rn(W(I), x, __fmul_rn(WLO(I), x));
}

// ---- storage traits ----
// ld/st convert between storage and the collision variable: FP32 stores f~ and
// collides on f~; FP16/BF16 store h = f~/w (avoids subnormals) and collide on h
// directly (collide_scaled), so no per-value scaling is executed.  phys gives
// the physical deviation f~ for read-back.
template <int S> struct St;
template <> struct St<kF32> {
    using T = float;
    static constexpr bool kScaled = false;
    template <int I> static __device__ __forceinline__ float ld(T v) { return v; }
    template <int I> static __device__ __forceinline__ T st(float v) { return v; }
    template <int I> static __device__ __forceinline__ float phys(T v) { return v; }
};
template <> struct St<kF16> {
    using T = __half;
    static constexpr bool kScaled = true;
    template <int I> static __device__ __forceinline__ float ld(T v) { return __half2float(v); }
    template <int I> static __device__ __forceinline__ T st(float v) { return __float2half_rn(v); }
    template <int I> static __device__ __forceinline__ float phys(T v) { return mulw<I>(__half2float(v)); }
};
template <> struct St<kBF16> {
    using T = __nv_bfloat16;
    static constexpr bool kScaled = true;
    template <int I> static __device__ __forceinline__ float ld(T v) { return __bfloat162float(v); }
    template <int I> static __device__ __forceinline__ T st(float v) { return __float2bfloat16_rn(v); }
    template <int I> static __device__ __forceinline__ float phys(T v) { return mulw<I>(__bfloat162float(v)); }
};

template <int N> struct IC { static constexpr int v = N; };
template <int B, int E, typename F> __device__ __forceinline__ void unroll(F &&f) {
    if constexpr (B < E) {
        f(IC<B>{});
        unroll<B + 1, E>(f);
    }
}

// Iolet rules for link I of a site next to iolet k; raw = the site's own post-collision value
// leaving towards x - c_I (direction opp(I)), in the collision variable; val = the iolet's
// boundary value.  Scaled storage (h = f~/w) drops the w_I factors (w_I = w_opp(I)); its
// velocity coefficients are stored divided by w_I.
template <int I, bool SC> __device__ __forceinline__ float pressure_rule(float val, float raw) {
    return -raw + (SC ? 2.0f * val : mulw<I>(2.0f * val));  // anti-bounce-back
}
__device__ __forceinline__ float velocity_rule(float val, float coef, float raw) {
    return __fmaf_rn(val, coef, raw);  // moving wall
}

// LBGK collision in deviation form, in place on g[19]; returns (drho, u).
// Every product and sum is written with explicit rounding intrinsics, so the compiler
// cannot contract them differently in the different kernels that inline this: all
// variants produce the same bits.
#define HG_MUL __fmul_rn
#define HG_ADD __fadd_rn
#define HG_SUB __fsub_rn
#define HG_FMA __fmaf_rn

// Two FP32 values (the same quantity of two sites) in one 64-bit register pair.  sm_103a
// adds, multiplies and fuses both with one instruction, each half rounded exactly as the
// scalar instruction rounds it.  The 16-bit kernels and the FP32 kernels with a decoded
// table were bound by instruction issue, and the collision is half of their instructions.
struct F2 {
    unsigned long long v;
};
__device__ __forceinline__ F2 pk2(float a, float b) {
    F2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ float lo2(F2 x) {
    float a;
    asm("{\n\t.reg .f32 t;\n\tmov.b64 {%0, t}, %1;\n\t}" : "=f"(a) : "l"(x.v));
    return a;
}
__device__ __forceinline__ float hi2(F2 x) {
    float b;
    asm("{\n\t.reg .f32 t;\n\tmov.b64 {t, %0}, %1;\n\t}" : "=f"(b) : "l"(x.v));
    return b;
}
__device__ __forceinline__ float vadd(float a, float b) { return HG_ADD(a, b); }
__device__ __forceinline__ float vsub(float a, float b) { return HG_SUB(a, b); }
__device__ __forceinline__ float vmul(float a, float b) { return HG_MUL(a, b); }
__device__ __forceinline__ float vfma(float a, float b, float c) { return HG_FMA(a, b, c); }
__device__ __forceinline__ float vrcp(float a) { return __frcp_rn(a); }
__device__ __forceinline__ F2 vadd(F2 a, F2 b) {
    F2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ F2 vsub(F2 a, F2 b) {
    F2 r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ F2 vmul(F2 a, F2 b) {
    F2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ F2 vfma(F2 a, F2 b, F2 c) {
    F2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
    return r;
}
__device__ __forceinline__ F2 vrcp(F2 a) { return pk2(__frcp_rn(lo2(a)), __frcp_rn(hi2(a))); }
// A product that a following addition must not be fused with: ptxas contracts
// mul.rn.f32x2 + add.rn.f32x2 (as it never does the scalar pair), so the packed product is
// formed as a b + z with z = (-0, -0) that the compiler does not know (it adds nothing).
__device__ __forceinline__ float vmul_apart(float a, float b, unsigned long long) { return HG_MUL(a, b); }
__device__ __forceinline__ F2 vmul_apart(F2 a, F2 b, unsigned long long z) { return vfma(a, b, F2{z}); }
template <typename V> __device__ __forceinline__ V vset(float x);
template <> __device__ __forceinline__ float vset<float>(float x) { return x; }
template <> __device__ __forceinline__ F2 vset<F2>(float x) { return pk2(x, x); }
template <int I, typename V> __device__ __forceinline__ V vmulw(V x) {  // mulw<I>, see above
    return vfma(vset<V>(W(I)), x, vmul(vset<V>(WLO(I)), x));
}

// (drho, ux, uy, uz) of one site (V = float) or two (V = F2)
template <typename V> struct MomT {
    V drho, ux, uy, uz;
};

// SC: the scaled variable h = f~/w (16-bit storage): its moments weight h by w, its
// equilibrium h~eq_i = drho + rho (3 c.u + 4.5 (c.u)^2 - 1.5 u.u) carries no weight.
// Otherwise f~, whose equilibrium is w times that (split-weight products).
template <bool SC, typename V>
__device__ __forceinline__ MomT<V> collide_v(V g[19], float omega_, unsigned long long neg_zero2) {
    V drho, jx, jy, jz;
    const V d12 = vsub(g[1], g[2]), d34 = vsub(g[3], g[4]), d56 = vsub(g[5], g[6]);
    const V d78 = vsub(g[7], g[8]), d910 = vsub(g[9], g[10]), d1112 = vsub(g[11], g[12]);
    const V d1314 = vsub(g[13], g[14]), d1516 = vsub(g[15], g[16]), d1718 = vsub(g[17], g[18]);
    if constexpr (SC) {
        const V sa = vadd(vadd(vadd(g[1], g[2]), vadd(g[3], g[4])), vadd(g[5], g[6]));
        const V sd = vadd(vadd(vadd(vadd(g[7], g[8]), vadd(g[9], g[10])),
                               vadd(vadd(g[11], g[12]), vadd(g[13], g[14]))),
                          vadd(vadd(g[15], g[16]), vadd(g[17], g[18])));
        drho = vadd(vmulw<0>(g[0]), vadd(vmulw<1>(sa), vmulw<7>(sd)));
        const V ex = vadd(vadd(d78, d910), vadd(d1112, d1314));
        const V ey = vadd(vsub(d78, d910), vadd(d1516, d1718));
        const V ez = vadd(vsub(d1112, d1314), vsub(d1516, d1718));
        jx = vadd(vmulw<1>(d12), vmulw<7>(ex));
        jy = vadd(vmulw<1>(d34), vmulw<7>(ey));
        jz = vadd(vmulw<1>(d56), vmulw<7>(ez));
    } else {
        drho = g[0];
#pragma unroll
        for (int i = 1; i < 19; ++i) drho = vadd(drho, g[i]);
        jx = vadd(vadd(vadd(d12, d78), vadd(d910, d1112)), d1314);
        jy = vadd(vadd(vsub(vadd(d34, d78), d910), d1516), d1718);
        jz = vsub(vadd(vsub(vadd(d56, d1112), d1314), d1516), d1718);
    }
    const V omega = vset<V>(omega_);
    const V rho = vadd(vset<V>(1.0f), drho);
    const V inv = vrcp(rho);
    const V ux = vmul(jx, inv), uy = vmul(jy, inv), uz = vmul(jz, inv);
    const V usq = vfma(ux, ux, vfma(uy, uy, vmul(uz, uz)));
    const V base = vfma(vmul(vset<V>(-1.5f), rho), usq, drho);  // drho - 1.5 rho u.u
    const V r45 = vmul(vset<V>(4.5f), rho), r3 = vmul(vset<V>(3.0f), rho);
    if constexpr (SC) g[0] = vfma(omega, vsub(base, g[0]), g[0]);
    else g[0] = vfma(omega, vsub(vmulw<0>(base), g[0]), g[0]);
    auto pair = [&](auto ia, int b, V cu) {
        constexpr int a = decltype(ia)::v;
        const V q = vfma(vmul(r45, cu), cu, base);    // base + 4.5 rho cu^2
        const V c3 = vmul_apart(r3, cu, neg_zero2);
        V sym = q, asym = c3;
        if constexpr (!SC) {
            sym = vmulw<a>(q);
            asym = vmulw<a>(c3);
        }
        g[a] = vfma(omega, vsub(vadd(sym, asym), g[a]), g[a]);
        g[b] = vfma(omega, vsub(vsub(sym, asym), g[b]), g[b]);
    };
    pair(IC<1>{}, 2, ux);
    pair(IC<3>{}, 4, uy);
    pair(IC<5>{}, 6, uz);
    pair(IC<7>{}, 8, vadd(ux, uy));
    pair(IC<9>{}, 10, vsub(ux, uy));
    pair(IC<11>{}, 12, vadd(ux, uz));
    pair(IC<13>{}, 14, vsub(ux, uz));
    pair(IC<15>{}, 16, vadd(uy, uz));
    pair(IC<17>{}, 18, vsub(uy, uz));
    return {drho, ux, uy, uz};
}

template <int S> __device__ __forceinline__ float4 collide_s(float g[19], float omega) {
    const MomT<float> m = collide_v<St<S>::kScaled>(g, omega, 0);
    return make_float4(m.drho, m.ux, m.uy, m.uz);
}
__device__ __forceinline__ float4 mom_lo(const MomT<F2> &m) {
    return make_float4(lo2(m.drho), lo2(m.ux), lo2(m.uy), lo2(m.uz));
}
__device__ __forceinline__ float4 mom_hi(const MomT<F2> &m) {
    return make_float4(hi2(m.drho), hi2(m.ux), hi2(m.uy), hi2(m.uz));
}


template <typename T> __device__ __forceinline__ T ldg_nc(const T *p) { return __ldg(p); }
template <> __device__ __forceinline__ __half ldg_nc(const __half *p) {
    return __ushort_as_half(__ldg(reinterpret_cast<const unsigned short *>(p)));
}
template <> __device__ __forceinline__ __nv_bfloat16 ldg_nc(const __nv_bfloat16 *p) {
    return __ushort_as_bfloat16(__ldg(reinterpret_cast<const unsigned short *>(p)));
}

// Loads carrying an L2 prefetch-size hint (256 B): a miss fetches the whole
// 256-byte span, which neighbouring warps' gathers then hit.  ld_ro: read-only
// data (non-coherent path); ld_rw: data this kernel also writes (AA).
template <typename T> struct HintLd;
template <> struct HintLd<float> {
    static __device__ __forceinline__ float ro(const float *p) {
        float v;
        asm("ld.global.nc.L2::256B.f32 %0, [%1];" : "=f"(v) : "l"(p));
        return v;
    }
    static __device__ __forceinline__ float rw(const float *p) {
        float v;
        asm("ld.global.L2::256B.f32 %0, [%1];" : "=f"(v) : "l"(p) : "memory");
        return v;
    }
};
template <> struct HintLd<int32_t> {
    static __device__ __forceinline__ int32_t ro(const int32_t *p) {
        int32_t v;
        asm("ld.global.nc.L2::256B.s32 %0, [%1];" : "=r"(v) : "l"(p));
        return v;
    }
};
template <typename H> struct HintLd16 {
    static __device__ __forceinline__ H ro(const H *p) {
        unsigned short v;
        asm("ld.global.nc.L2::256B.b16 %0, [%1];" : "=h"(v) : "l"(p));
        return *reinterpret_cast<H *>(&v);
    }
    static __device__ __forceinline__ H rw(const H *p) {
        unsigned short v;
        asm("ld.global.L2::256B.b16 %0, [%1];" : "=h"(v) : "l"(p) : "memory");
        return *reinterpret_cast<H *>(&v);
    }
};
template <> struct HintLd<__half> : HintLd16<__half> {};
template <> struct HintLd<__nv_bfloat16> : HintLd16<__nv_bfloat16> {};

template <bool HINT, typename T> __device__ __forceinline__ T load_ro(const T *p) {
    if constexpr (HINT) return HintLd<T>::ro(p);
    else return ldg_nc(p);
}
template <bool HINT> __device__ __forceinline__ int32_t load_nbr(const int32_t *p) {
    if constexpr (HINT) return HintLd<int32_t>::ro(p);
    else return __ldg(p);
}
template <bool HINT, typename T> __device__ __forceinline__ T load_rw(const T *p) {
    if constexpr (HINT) return HintLd<T>::rw(p);
    else return *p;
}

// ---- the links of a site: the 18-row neighbour table or its run encoding ----
// The table (72 bytes per site) gives for link I (1..18) the fluid neighbour's device
// index, or for a non-fluid link the virtual index s + dd np with dd = opp(I) - I (A/B)
// or I - opp(I) (AA).
// The run encoding: a word per site (non-fluid flags, run within the chunk), the
// chunk's first run, and the run's 80-byte row, which the run's other sites also read
// (L1 hits): about 4 + 80 / run-length bytes per site.  Rows 2k+1 and 2k+2 of the
// distributions are the two directions of one opposite pair, so both places a link can
// read or write -- the neighbour's row and the own site's opposite row -- lie in one
// pair: the run's row holds for every link the element offset of the fluid place from the
// own site in the pair's first row, and a flagged link takes 0 or np instead: a select, one
// 32 x 32 + 64-bit multiply-add and the load.
// Link I's element offset from the own site in the first row of its pair (d = the run row's
// entry, w = the site's word).  Flagged: the own site in the opposite row (A/B) or the own row
// (AA, whose odd step gathers row OPP(I)).
template <int SCHEME, int I> __device__ __forceinline__ int32_t run_offset(uint32_t w, int32_t d, int32_t np) {
    constexpr bool second = SCHEME == kAB ? (I & 1) != 0 : (I & 1) == 0;
    return ((w >> (I - 1)) & 1u) ? (second ? np : 0) : d;
}
// f(IC<I>, entry) for links I = 4 K + 1 .. 4 K + 4 (up to 18) from the run row's K-th 16 bytes.
template <int K, typename F> __device__ __forceinline__ void run_links4(const int32_t *row, F &&f) {
    const int4 v = __ldg(reinterpret_cast<const int4 *>(row) + K);
    const int32_t d[4] = {v.x, v.y, v.z, v.w};
    unroll<0, (K < 4 ? 4 : 2)>([&](auto jc) {
        constexpr int J = decltype(jc)::v;
        f(IC<4 * K + J + 1>{}, d[J]);
    });
}
// Row I of the distributions at p (np values, npb bytes, per row): one multiply-add.
template <int I, typename T> __device__ __forceinline__ T *row_at(T *p, uint32_t npb) {
    using C = typename std::conditional<std::is_const<T>::value, const char, char>::type;
    return (T *)((C *)p + (uint64_t)npb * (uint32_t)I);
}
// The first row of link I's opposite pair.
template <int I, typename T> __device__ __forceinline__ T *pair_row(T *p, uint32_t npb) {
    return row_at<(I - 1) / 2 * 2 + 1>(p, npb);
}

// ---- sites next to an iolet (rare path) ----
// Neighbour table entries of non-fluid links hold a virtual index that makes
// the ordinary address formula land on the site's own opposite slot, so a wall
// needs no code at all.  Sites with a link into an iolet opening are flagged in
// `iomask`; their slot is the rank of the flag (per-32-site prefix + popcount)
// and their canonical link codes sit in io_codes[slot][18].
__device__ __forceinline__ bool site_flag(const DomDev &D, int64_t s, uint32_t &word) {
    word = __ldg(D.iomask + (s >> 5));
    return (word >> (s & 31)) & 1u;
}
__device__ __forceinline__ int site_slot(const DomDev &D, int64_t s, uint32_t word) {
    return __ldg(D.ioprefix + (s >> 5)) + __popc(word & ((1u << (s & 31)) - 1u));
}
// f(IC<I>, rule) for every iolet link of boundary slot `slot`, rule: raw value -> value.  A
// slot whose links all lead into one iolet (nearly every one) has its mask and iolet in one
// word, so its value and kind are one round of loads, where decoding the 18 codes one after
// another chained up to three loads per link.  AHEAD also loads the velocity coefficients
// ahead of the links (18 registers: for the resident kernel, whose steps wait for these).
template <int S, bool AHEAD, typename F>
__device__ __forceinline__ void each_iolet_link(const DomDev &D, const float *bcv, int slot, uint32_t word, F &&f) {
    constexpr bool SC = St<S>::kScaled;
    const float *coef = D.coef + (int64_t)slot * 18;
    if (word != kManyIolets) {
        const int k = (int)(word >> 18);
        const float val = bcv[k];
        if (D.io_kind[k] == 0) {
            unroll<1, 19>([&](auto ic) {
                constexpr int I = decltype(ic)::v;
                if ((word >> (I - 1)) & 1u) f(ic, [&](float raw) { return pressure_rule<I, SC>(val, raw); });
            });
        } else {
            float c[18];
            if constexpr (AHEAD) {
#pragma unroll
                for (int i = 0; i < 18; ++i) c[i] = __ldg(coef + i);
            }
            unroll<1, 19>([&](auto ic) {
                constexpr int I = decltype(ic)::v;
                if ((word >> (I - 1)) & 1u)
                    f(ic, [&](float raw) {
                        return velocity_rule(val, AHEAD ? c[I - 1] : __ldg(coef + (I - 1)), raw);
                    });
            });
        }
        return;
    }
    const int32_t *codes = D.io_codes + (int64_t)slot * 18;
    unroll<1, 19>([&](auto ic) {
        constexpr int I = decltype(ic)::v;
        const int32_t k = -__ldg(codes + (I - 1)) - 2;
        if (k >= 0)
            f(ic, [&](float raw) {
                return D.io_kind[k] == 0 ? pressure_rule<I, SC>(bcv[k], raw)
                                         : velocity_rule(bcv[k], __ldg(coef + (I - 1)), raw);
            });
    });
}
__device__ __forceinline__ uint32_t io_word(const DomDev &D, int slot) { return __ldg(D.io_words + slot); }
template <int S, bool AHEAD = false>
__device__ __forceinline__ void apply_iolet_links(const DomDev &D, const float *bcv, int slot, uint32_t word,
                                                  float g[19]) {
    each_iolet_link<S, AHEAD>(D, bcv, slot, word, [&](auto ic, auto rule) {
        constexpr int I = decltype(ic)::v;
        g[I] = rule(g[I]);
    });
}
// A stream-collide launch may start while the previous step's iolet update is
// still running (programmatic dependent launch): everything it reads except the
// boundary values was complete before that update began, which is a plain launch
// behind the previous step's stream-collide.  (Launched early as well, waiting here for
// that step, it would let this launch go on the strength of a wait that makes the
// step's writes visible to the update alone; it gained 1.6 us of a 36 us step at 1M sites
// and cost A/B steps of 35k sites with 200 iolets 4.5 of 12.6.)  Only the sites with
// an iolet link use the boundary values (and overwrite the moments slot the update
// reads), so only they wait here for the update to finish.  Without an
// overlapping launch the wait returns at once.
__device__ __forceinline__ void wait_for_iolet_update() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

template <int S>
__device__ __forceinline__ int iolet_fixup(const DomDev &D, int64_t s, float g[19]) {
    uint32_t word;
    if (!site_flag(D, s, word)) return -1;
    wait_for_iolet_update();
    const int slot = site_slot(D, s, word);
    apply_iolet_links<S>(D, D.bcv, slot, io_word(D, slot), g);
    return slot;
}
// The same for one half of a packed pair (HI: the second site); the caller found the flag.
template <int S, bool HI>
__device__ __forceinline__ void iolet_links_half(const DomDev &D, const float *bcv, int slot, F2 g[19]) {
    each_iolet_link<S, false>(D, bcv, slot, io_word(D, slot), [&](auto ic, auto rule) {
        constexpr int I = decltype(ic)::v;
        const float a = lo2(g[I]), b = hi2(g[I]);
        g[I] = HI ? pk2(a, rule(b)) : pk2(rule(a), b);
    });
}
template <int S>
__device__ __forceinline__ void iolet_fixup2(const DomDev &D, int64_t sa, int64_t sb, F2 g[19], int &slot_a,
                                             int &slot_b) {
    uint32_t wa, wb;
    const bool fa = site_flag(D, sa, wa), fb = site_flag(D, sb, wb);
    slot_a = slot_b = -1;
    if (fa || fb) {
        wait_for_iolet_update();
        if (fa) {
            slot_a = site_slot(D, sa, wa);
            iolet_links_half<S, false>(D, D.bcv, slot_a, g);
        }
        if (fb) {
            slot_b = site_slot(D, sb, wb);
            iolet_links_half<S, true>(D, D.bcv, slot_b, g);
        }
    }
}

template <typename T> __device__ __forceinline__ T *opaque(T *p) {
    T *q;
    asm volatile("mov.b64 %0, %1;" : "=l"(q) : "l"(p));
    return q;
}

// ---- AA even step: state G_t natural at the own site -> F_t swapped at the own site ----
// One site (the ragged end of a tile; the rest goes in pairs).
template <int S>
__device__ __forceinline__ void site_aa_even(const DomDev &D, typename St<S>::T *buf, int64_t s) {
    using Tr = St<S>;
    const int64_t np = D.np;
    float g[19];
    unroll<0, 19>([&](auto ic) {
        constexpr int I = decltype(ic)::v;
        g[I] = Tr::template ld<I>(buf[(int64_t)I * np + s]);
    });
    const int slot = iolet_fixup<S>(D, s, g);  // the odd step left raw values on iolet links
    const float4 m = collide_s<S>(g, D.omega);
    typename St<S>::T *wb = opaque(buf + s);
    unroll<0, 19>([&](auto ic) {
        constexpr int I = decltype(ic)::v;
        wb[(int64_t)OPP(I) * np] = Tr::template st<I>(g[I]);
    });
    if (slot >= 0) D.bnd[slot] = m;
}

// ---- pairs of adjacent sites: vector loads and stores, packed arithmetic ----
template <int S> struct Pair;
template <> struct Pair<kF32> {
    template <int I> static __device__ __forceinline__ void ld(const float *p, float &a, float &b) {
        const float2 v = *(const float2 *)p;
        a = v.x;
        b = v.y;
    }
    template <int I> static __device__ __forceinline__ void st(float *p, float a, float b) {
        *(float2 *)p = make_float2(a, b);
    }
};
// Two adjacent 16-bit values move as one 4-byte word and convert with the paired
// intrinsics (same round-to-nearest-even as the scalar conversions, so the bits
// are those of every other variant; fewer instructions for kernels near their
// issue limit).
template <int S16> struct Pair16;
template <> struct Pair16<kF16> {
    template <int I> static __device__ __forceinline__ void ld(const __half *p, float &a, float &b) {
        const float2 f = __half22float2(*reinterpret_cast<const __half2 *>(p));
        a = f.x;
        b = f.y;
    }
    template <int I> static __device__ __forceinline__ void st(__half *p, float a, float b) {
        *reinterpret_cast<__half2 *>(p) = __floats2half2_rn(a, b);
    }
};
template <> struct Pair16<kBF16> {
    template <int I> static __device__ __forceinline__ void ld(const __nv_bfloat16 *p, float &a, float &b) {
        const float2 f = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(p));
        a = f.x;
        b = f.y;
    }
    template <int I> static __device__ __forceinline__ void st(__nv_bfloat16 *p, float a, float b) {
        *reinterpret_cast<__nv_bfloat162 *>(p) = __floats2bfloat162_rn(a, b);
    }
};
template <> struct Pair<kF16> : Pair16<kF16> {};
template <> struct Pair<kBF16> : Pair16<kBF16> {};

template <int S, int I> __device__ __forceinline__ F2 ld_pair(const typename St<S>::T *p) {
    float a, b;
    Pair<S>::template ld<I>(p, a, b);
    return pk2(a, b);
}
template <int S, int I> __device__ __forceinline__ void st_pair(typename St<S>::T *p, F2 v) {
    Pair<S>::template st<I>(p, lo2(v), hi2(v));
}
__device__ __forceinline__ void put_moments(const DomDev &D, int slot_a, int slot_b, const MomT<F2> &m) {
    if (slot_a >= 0) D.bnd[slot_a] = mom_lo(m);
    if (slot_b >= 0) D.bnd[slot_b] = mom_hi(m);
}

// ---- A/B pull on a pair of adjacent sites (18-row table, 16-bit storage) ----
// Sites s and s+1 (s even) share one 8-byte load per neighbour-table row, one
// 4-byte load of the rest values and one 4-byte store per direction: fewer
// memory instructions per site for a kernel that runs near its issue limit
// (~10M-site tree in rows: 221 us against 252 for one site per thread).
template <int S>
__device__ __forceinline__ void site_ab_pair(const DomDev &D, const typename St<S>::T *__restrict__ src,
                                             typename St<S>::T *__restrict__ dst, int64_t s) {
    using Tr = St<S>;
    const int64_t np = D.np;
    F2 g[19];
    g[0] = ld_pair<S, 0>(src + s);
    unroll<1, 19>([&](auto ic) {
        constexpr int I = decltype(ic)::v;
        const int2 nb = __ldg(reinterpret_cast<const int2 *>(D.nbr + (int64_t)(I - 1) * np + s));
        g[I] = pk2(Tr::template ld<I>(ldg_nc(src + ((int64_t)I * np + nb.x))),
                   Tr::template ld<I>(ldg_nc(src + ((int64_t)I * np + nb.y))));
    });
    int slot_a, slot_b;
    iolet_fixup2<S>(D, s, s + 1, g, slot_a, slot_b);
    const MomT<F2> m = collide_v<Tr::kScaled>(g, D.omega, D.neg_zero2);
    typename St<S>::T *wb = opaque(dst + s);
    unroll<0, 19>([&](auto ic) {
        constexpr int I = decltype(ic)::v;
        st_pair<S, I>(wb + (int64_t)I * np, g[I]);
    });
    put_moments(D, slot_a, slot_b, m);
}

// AA even step on adjacent pairs: local, vector loads and stores of both sites.
template <int S>
__device__ __forceinline__ void site_aa_even_pair(const DomDev &D, typename St<S>::T *buf, int64_t s) {
    const int64_t np = D.np;
    F2 g[19];
    unroll<0, 19>([&](auto ic) {
        constexpr int I = decltype(ic)::v;
        g[I] = ld_pair<S, I>(buf + (int64_t)I * np + s);
    });
    int slot_a, slot_b;
    iolet_fixup2<S>(D, s, s + 1, g, slot_a, slot_b);
    const MomT<F2> m = collide_v<St<S>::kScaled>(g, D.omega, D.neg_zero2);
    typename St<S>::T *wb = opaque(buf + s);
    unroll<0, 19>([&](auto ic) {
        constexpr int I = decltype(ic)::v;
        st_pair<S, I>(wb + (int64_t)OPP(I) * np, g[I]);
    });
    put_moments(D, slot_a, slot_b, m);
}

template <int S>
__device__ __forceinline__ void tile_aa_even_pairs(const DomDev &D, const TileDev &tl) {
    using T = typename St<S>::T;
    T *buf = (T *)D.f[0];
    for (int r = 2 * threadIdx.x; r < tl.count; r += 2 * blockDim.x) {
        const int64_t s = tl.start + r;  // even: tiles start at multiples of 32
        if (r + 1 >= tl.count) site_aa_even<S>(D, buf, s);  // ragged tail: one site
        else site_aa_even_pair<S>(D, buf, s);
    }
}

// ==== one site per thread: the A/B step and the AA odd step ====================
// FP32 AA odd through the run encoding: bound by the misaligned scatter's sectors (268 us on the
// ~10M-site tree, 303 before the links were decoded as below); 40 registers, so 48 warps per SM
// hide the chain word -> run row -> gathers.
// With the 18-row table it is bound by the table's 72 bytes and the scattered sectors of
// Morton order (~10M-site tree, Morton / rows): FP32 A/B 330 / 320 us (475 before the 32-bit
// multiply-add addresses), FP16 AA odd 343 / 260 and FP32 AA odd 429 / 340, against 391 / 346
// and 471 / 428 for gathers staged by cp.async and 393 / 272 and 483 / 354 for adjacent pairs.
template <int S, int SCHEME, bool HINT> __device__ __forceinline__ float link_ld(const typename St<S>::T *p) {
    if constexpr (SCHEME == kAA) return St<S>::template ld<0>(load_rw<HINT>(p));
    else return St<S>::template ld<0>(load_ro<HINT>(p));
}
struct RunSite {
    uint32_t w;
    const int32_t *row;
};
__device__ __forceinline__ RunSite run_site(const DomDev &D, int64_t s) {
    RunSite r;
    r.w = (uint32_t)load_nbr<true>(reinterpret_cast<const int32_t *>(D.lword) + s);
    r.row = D.rdelta + (int64_t)(__ldg(D.run0 + (s >> 10)) + (int32_t)((r.w >> 18) & 1023u)) * kRunStride;
    return r;
}
// The links of a site as offsets from the own site in the first row of the link's opposite
// pair: each(f) calls f(IC<I>, offset) for I = 1..18.
template <int SCHEME> struct RunOffsets {
    RunSite r;
    int32_t np;
    template <typename F> __device__ __forceinline__ void each(F &&f) const {
        unroll<0, 5>([&](auto kc) {
            run_links4<decltype(kc)::v>(r.row, [&](auto ic, int32_t d) {
                f(ic, run_offset<SCHEME, decltype(ic)::v>(r.w, d, np));
            });
        });
    }
    __device__ __forceinline__ bool next_to_iolet(const DomDev &, int64_t) const { return r.w >> 31; }
};
template <int SCHEME, bool HINT> struct TableOffsets {
    const int32_t *p;  // entry 1 of the site
    int32_t s, np;
    template <typename F> __device__ __forceinline__ void each(F &&f) const {
        unroll<1, 19>([&](auto ic) {
            constexpr int I = decltype(ic)::v;
            constexpr bool second = SCHEME == kAB ? (I & 1) == 0 : (I & 1) != 0;  // the row gathered from
            f(ic, load_nbr<HINT>(p + (int64_t)(I - 1) * np) - s + (second ? np : 0));
        });
    }
    __device__ __forceinline__ bool next_to_iolet(const DomDev &D, int64_t at) const {
        uint32_t word;
        return site_flag(D, at, word);
    }
};
// A/B step or AA odd step of one site.  The AA scatter goes to the places the gather read
// (direction I where its opposite was read); their 18 offsets wait in shared memory, one bank
// per thread (`stash`: this thread's, a word per `stride`), instead of being decoded again.
template <int S, int SCHEME, bool HINT, typename L>
__device__ __forceinline__ void site_links(const DomDev &D, const typename St<S>::T *src, typename St<S>::T *dst,
                                           int64_t s, const L &links, int32_t *stash, int stride) {
    using Tr = St<S>;
    using T = typename Tr::T;
    const uint32_t npb = (uint32_t)D.np * sizeof(T);
    const T *p = src + s;
    float g[19];
    g[0] = link_ld<S, SCHEME, HINT>(p);
    links.each([&](auto ic, int32_t off) {
        constexpr int I = decltype(ic)::v;
        g[I] = link_ld<S, SCHEME, HINT>(pair_row<I>(p, npb) + off);
        if constexpr (SCHEME == kAA) stash[(I - 1) * stride] = off;
    });
    int slot = -1;
    if (links.next_to_iolet(D, s)) {
        wait_for_iolet_update();
        slot = site_slot(D, s, __ldg(D.iomask + (s >> 5)));
        apply_iolet_links<S>(D, D.bcv, slot, io_word(D, slot), g);
    }
    const float4 m = collide_s<S>(g, D.omega);
    int32_t *back = stash;
    if constexpr (SCHEME == kAA)
        // the address is known only once the collision has produced m: the reads cannot
        // move above it, so the 18 offsets are not live across it
        asm volatile("{\n\t.reg .f32 t;\n\tmov.f32 t, %2;\n\tmov.b64 %0, %1;\n\t}"
                     : "=l"(back) : "l"(stash), "f"(m.x) : "memory");
    T *q = opaque(dst + s);
    *q = Tr::template st<0>(g[0]);
    unroll<1, 19>([&](auto ic) {
        constexpr int I = decltype(ic)::v;
        const T v = Tr::template st<I>(g[I]);
        if constexpr (SCHEME == kAB) *row_at<I>(q, npb) = v;
        else pair_row<I>(q, npb)[back[(OPP(I) - 1) * stride]] = v;
    });
    if (slot >= 0) D.bnd[slot] = m;
}
// ---- A/B step or 16-bit AA odd step of a pair of adjacent sites, run encoding ----
// The A/B steps and the 16-bit AA odd step run near the issue limit one site per thread (420 to
// 518 instructions per site and step).  A pair (s even) shares the word load, the run row where
// the run is the same (98 % of the pairs), the rows' addresses, vector stores (A/B) and a packed
// collision: 303 instructions per site for A/B, 390 for AA odd.  Registers decide: ~10M-site
// tree, FP16 A/B at 76 / 72 / 64 / 56 registers 178 / 167 / 158 / 166 us (one site per thread
// 178), FP16 AA odd at 85 / 72 / 64 213 / 190 / 200 (197).  Bound now by the latency of the
// chain word -> row -> gathers at 28 warps per SM.
// Tried and slower: sites l and l + 32 of a warp as the pair (188-230 us); lists of all-fluid
// pairs and single sites (250 instructions per site, but their stores leave sectors half
// written: FP32 A/B 296 us); an L2 prefetch of the distributions 64K..1M sites ahead (no change
// to 20 % slower); joining the AA scatter's two stores where they meet (FP16 190 -> 211).
template <int S, int SCHEME>
__device__ __forceinline__ void site_run_pair(const DomDev &D, const typename St<S>::T *src,
                                              typename St<S>::T *dst, int64_t s, int2 *stash) {
    using Tr = St<S>;
    using T = typename Tr::T;
    const int32_t np = (int32_t)D.np;
    const uint32_t npb = (uint32_t)D.np * sizeof(T);
    const uint2 w = __ldg(reinterpret_cast<const uint2 *>(D.lword + s));
    const int32_t r0 = __ldg(D.run0 + (s >> 10));
    const int32_t *ra = D.rdelta + (int64_t)(r0 + (int32_t)((w.x >> 18) & 1023u)) * kRunStride;
    const int32_t *rb = D.rdelta + (int64_t)(r0 + (int32_t)((w.y >> 18) & 1023u)) * kRunStride;
    const bool same = ra == rb;
    const T *p = src + s;
    F2 g[19];
    g[0] = ld_pair<S, 0>(p);
    unroll<0, 5>([&](auto kc) {
        constexpr int K = decltype(kc)::v;
        const int4 va = __ldg(reinterpret_cast<const int4 *>(ra) + K);
        int4 vb = va;
        if (!same) vb = __ldg(reinterpret_cast<const int4 *>(rb) + K);
        const int32_t da[4] = {va.x, va.y, va.z, va.w}, db[4] = {vb.x, vb.y, vb.z, vb.w};
        unroll<0, (K < 4 ? 4 : 2)>([&](auto jc) {
            constexpr int J = decltype(jc)::v, I = 4 * K + J + 1;
            const T *q = pair_row<I>(p, npb);
            const int32_t oa = run_offset<SCHEME, I>(w.x, da[J], np), ob = run_offset<SCHEME, I>(w.y, db[J], np);
            const float a = link_ld<S, SCHEME, true>(q + oa);
            const float b = link_ld<S, SCHEME, true>(q + 1 + ob);
            g[I] = pk2(a, b);
            if constexpr (SCHEME == kAA) stash[(I - 1) * blockDim.x] = make_int2(oa, ob);
        });
    });
    int slot_a = -1, slot_b = -1;
    if ((w.x | w.y) >> 31) {
        wait_for_iolet_update();
        const uint32_t word = __ldg(D.iomask + (s >> 5));
        if (w.x >> 31) {
            slot_a = site_slot(D, s, word);
            iolet_links_half<S, false>(D, D.bcv, slot_a, g);
        }
        if (w.y >> 31) {
            slot_b = site_slot(D, s + 1, word);
            iolet_links_half<S, true>(D, D.bcv, slot_b, g);
        }
    }
    const MomT<F2> m = collide_v<Tr::kScaled>(g, D.omega, D.neg_zero2);
    int2 *back = stash;
    if constexpr (SCHEME == kAA)
        asm volatile("{\n\t.reg .b64 t;\n\tmov.b64 t, %2;\n\tmov.b64 %0, %1;\n\t}"
                     : "=l"(back) : "l"(stash), "l"(m.drho.v) : "memory");
    T *q = opaque(dst + s);
    st_pair<S, 0>(q, g[0]);
    unroll<1, 19>([&](auto ic) {
        constexpr int I = decltype(ic)::v;
        if constexpr (SCHEME == kAB) {
            st_pair<S, I>(row_at<I>(q, npb), g[I]);
        } else {
            const int2 o = back[(OPP(I) - 1) * blockDim.x];
            T *r = pair_row<I>(q, npb);
            r[o.x] = Tr::template st<I>(lo2(g[I]));
            r[1 + o.y] = Tr::template st<I>(hi2(g[I]));
        }
    });
    put_moments(D, slot_a, slot_b, m);
}

constexpr int64_t kWordsAhead = 196608;  // sites

// Launch bounds: the run-encoded pair forms are held to 64 (A/B) and 72 (AA odd) registers; the
// others keep what 512 threads leave them, which they use least of (40 to 76).
constexpr bool pair_runs(int s, int scheme, int par, bool runs) {
    return runs && (scheme == kAB || (par == 1 && s != kF32));
}
constexpr int sc_threads(int s, int scheme, int par, bool runs) { return pair_runs(s, scheme, par, runs) ? 128 : 512; }
constexpr int sc_blocks(int s, int scheme, int par, bool runs) {
    return pair_runs(s, scheme, par, runs) ? (scheme == kAB ? 8 : 7) : 0;
}

// The last site of an odd-sized tile.  Not inlined: the single-site body beside the pair's cost
// the pair registers (FP16 A/B 160 us against 155, FP16 AA odd 194 against 184).
template <int S, int SCHEME>
__device__ __noinline__ void tail_site(const DomDev &D, const typename St<S>::T *src, typename St<S>::T *dst,
                                       int64_t s, int32_t *stash) {
    site_links<S, SCHEME, true>(D, src, dst, s, RunOffsets<SCHEME>{run_site(D, s), (int32_t)D.np}, stash,
                                2 * (int)blockDim.x);
}

// One tile of one domain, after the prologue has located it.
// PAR is the parity of the step this launch executes: 0 = even, 1 = odd (the
// AA step kind), 2 = read from the domain's step counter per block (A/B, and AA
// batches whose domains are at different parities).  RUNS: the domain has a run
// encoding (the host launches the form only on such domains; a domain without one here is
// reported through the error word, code 2, and left untouched).
template <int S, int SCHEME, int PAR, bool RUNS>
__device__ __forceinline__ void stream_collide_tile(const DomDev &D, const TileDev &tl, bool odd, int32_t *stash) {
    using T = typename St<S>::T;
    constexpr int SPT = sc_spt(S, SCHEME, PAR, RUNS);
    if (RUNS && D.lword == nullptr) {
        if (threadIdx.x == 0) atomicExch(D.err, 2);
        return;
    }
    if (SCHEME == kAA && (PAR == 0 || (PAR == 2 && !odd))) {
        tile_aa_even_pairs<S>(D, tl);
        return;
    }
    const T *src = (const T *)D.f[SCHEME == kAA || odd ? 0 : 1];  // A/B: F_{t-1} sits in f[(t-1) & 1]
    T *dst = (T *)D.f[SCHEME == kAA || !odd ? 0 : 1];
    if constexpr (RUNS) {
        if constexpr (SCHEME == kAB) {
            // the words of a later tile into L2 (a line per thread): FP32 235 -> 231 us, FP16 158
            // -> 156 at 128K..300K sites ahead, nothing at 1.2M; AA odd loses 3 %
            const int64_t at = tl.start + kWordsAhead + 32 * (int64_t)threadIdx.x;
            if (threadIdx.x < kTile / 32 && at < D.n) asm volatile("prefetch.global.L2 [%0];" ::"l"(D.lword + at));
        }
        constexpr bool PAIRS = pair_runs(S, SCHEME, PAR, true);
        constexpr int WORDS = PAIRS ? 2 : 1;  // of shared memory per thread and link
        auto one_site = [&](int64_t s) {
            site_links<S, SCHEME, true>(D, src, dst, s, RunOffsets<SCHEME>{run_site(D, s), (int32_t)D.np},
                                        stash + WORDS * threadIdx.x, WORDS * (int)blockDim.x);
        };
        if constexpr (PAIRS) {
            const int r = 2 * threadIdx.x;  // even sites: tiles start at multiples of kTile
            if (r + 1 < tl.count) site_run_pair<S, SCHEME>(D, src, dst, tl.start + r, (int2 *)stash + threadIdx.x);
            else if (r < tl.count) tail_site<S, SCHEME>(D, src, dst, tl.start + r, stash + WORDS * threadIdx.x);
        } else {
#pragma unroll
            for (int j = 0; j < SPT; ++j) {
                const int r = j * blockDim.x + threadIdx.x;
                if (r < tl.count) one_site(tl.start + r);
            }
        }
    } else {
        // FP32 AA without the 256-byte hints: 429 us against 446 (Morton), 340 against 346 (rows)
        constexpr bool HINT = !(SCHEME == kAA && S == kF32);
        auto one_site = [&](int64_t s) {
            site_links<S, SCHEME, HINT>(D, src, dst, s,
                                        TableOffsets<SCHEME, HINT>{D.nbr + s, (int32_t)s, (int32_t)D.np},
                                        stash + threadIdx.x, (int)blockDim.x);
        };
        if constexpr (SCHEME == kAB && S != kF32) {
            const int r = 2 * threadIdx.x;  // even sites: tiles start at multiples of kTile
            if (r + 1 < tl.count) site_ab_pair<S>(D, src, dst, tl.start + r);
            else if (r < tl.count) one_site(tl.start + r);
        } else {
#pragma unroll
            for (int j = 0; j < SPT; ++j) {
                const int r = j * blockDim.x + threadIdx.x;
                if (r < tl.count) one_site(tl.start + r);
            }
        }
    }
}

// A launch that started early ends only after the one before it has ended (the last block
// waits), so that the iolet update, a plain launch after the last of a chain, follows all of it.
__device__ __forceinline__ void end_after_previous() {
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) wait_for_iolet_update();
}

// Many domains per launch: each block finds its tile in the tile table; the
// first threads copy the tile's domain descriptor into shared memory, one
// 8-byte word each, while thread 0 reads the domain's step counter.
template <int S, int SCHEME, int PAR, bool RUNS>
__global__ void __launch_bounds__(sc_threads(S, SCHEME, PAR, RUNS), sc_blocks(S, SCHEME, PAR, RUNS))
    k_stream_collide(const DomDev *__restrict__ doms, const TileDev *__restrict__ tiles,
                     const int64_t *__restrict__ steps, int off) {
    static_assert(sizeof(DomDev) % 8 == 0, "descriptor copied in 8-byte words");
    constexpr int kWords = (int)(sizeof(DomDev) / 8);
    __shared__ DomDev D;
    __shared__ int64_t t_now;
    extern __shared__ __align__(128) int32_t stash[];
    const TileDev tl = tiles[blockIdx.x];
    if (threadIdx.x < kWords)
        reinterpret_cast<uint64_t *>(&D)[threadIdx.x] =
            __ldg(reinterpret_cast<const uint64_t *>(doms + tl.dom) + threadIdx.x);
    // the step this launch executes (1-based); only its parity matters, and a
    // launch whose domains all share it gets it as a template argument
    if constexpr (PAR == 2)
        if (threadIdx.x == 0) t_now = __ldg(steps + tl.dom) + off + 1;
    __syncthreads();
    const bool odd = PAR == 2 ? (t_now & 1) != 0 : PAR == 1;
    stream_collide_tile<S, SCHEME, PAR, RUNS>(D, tl, odd, stash);
    end_after_previous();
}

// One domain per launch: the descriptor is a kernel parameter (constant bank)
// and block b takes sites [b*T, b*T + T) with T = sites per thread * blockDim, so no
// block waits on a table load or a barrier before its first neighbour-table load.
template <int S, int SCHEME, int PAR, bool RUNS>
__global__ void __launch_bounds__(sc_threads(S, SCHEME, PAR, RUNS), sc_blocks(S, SCHEME, PAR, RUNS))
    k_stream_collide_one(const __grid_constant__ DomDev D, int64_t n, int off) {
    // a launch chained after this one (the next domain of a per-domain launch
    // sequence) may be scheduled once every block here has started; kernels launched
    // without programmatic serialisation ignore the trigger
    asm volatile("griddepcontrol.launch_dependents;");
    extern __shared__ __align__(128) int32_t stash[];
    const int64_t ts = (int64_t)sc_spt(S, SCHEME, PAR, RUNS) * blockDim.x;
    TileDev tl;
    tl.dom = 0;
    tl.start = (int64_t)blockIdx.x * ts;
    tl.count = (int32_t)(n - tl.start < ts ? n - tl.start : ts);
    bool odd;
    if constexpr (PAR == 2) odd = ((__ldg(D.step) + off + 1) & 1) != 0;
    else odd = PAR == 1;
    stream_collide_tile<S, SCHEME, PAR, RUNS>(D, tl, odd, stash);
    end_after_previous();
}

template <int S, int SCHEME, int PAR, bool RUNS>
cudaError_t launch_sc(const CollideCfg &cfg, const DomDev *doms, const TileDev *tiles, int64_t n_tiles, int off,
                      const OneDomain &one, cudaStream_t st) {
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3((unsigned)n_tiles);
    lc.blockDim = dim3((unsigned)cfg.block);
    // the AA odd step's 18 offsets per thread (two sites' in the pair form)
    lc.dynamicSmemBytes = SCHEME == kAA && PAR != 0 ? (size_t)18 * 4 * (PAR == 1 ? cfg.spt : 1) * cfg.block : 0;
    lc.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    lc.attrs = at;
    lc.numAttrs = one.overlap_previous ? 1 : 0;  // start while the previous iolet update runs
    if (one.d) return cudaLaunchKernelEx(&lc, k_stream_collide_one<S, SCHEME, PAR, RUNS>, *one.d, one.n, off);
    return cudaLaunchKernelEx(&lc, k_stream_collide<S, SCHEME, PAR, RUNS>, doms, tiles, one.steps, off);
}

}  // namespace

}  // namespace hg
