// Device-side body of the fused fluid update (Eq. lbequation), shared by the
// single-simulation kernel (fluid.cu) and the batched persistent kernel
// (batch.cu).  See fluid.cu for the description of the update.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "lbib_internal.h"

namespace lbib {

// Storage of one population.  FP32 is stored as is.  FP16/BF16 store the
// deviation times 2^s with stochastic rounding: the conversion moves to the
// neighbouring representable value of larger magnitude with probability
// equal to the dropped fraction of a unit in the last place, so the stored
// value is unbiased.  Rounding to nearest would turn
// the per-step forcing increment, which is far below one unit in the last
// place of a 16-bit number once the flow has built up, into a systematic
// error.  The rounding is the hardware's (cvt.rs, which converts two FP32
// numbers into a packed pair with 32 random bits); the random bits come
// from a counter-based hash of (cell, step) stepped by a linear
// congruential generator across the directions, so results are
// reproducible.
//
// PopIO::ld reads a deviation (read-outs and reductions); Raw below is the
// step kernel's access to the stored numbers themselves.
template <typename T>
struct PopIO;

template <>
struct PopIO<float> {
    static __device__ __forceinline__ float ld(const float *p, float) { return __ldg(p); }
};
template <>
struct PopIO<__half> {
    static __device__ __forceinline__ float ld(const __half *p, float inv) { return __half2float(__ldg(p)) * inv; }
};
template <>
struct PopIO<__nv_bfloat16> {
    static __device__ __forceinline__ float ld(const __nv_bfloat16 *p, float inv) {
        return __bfloat162float(__ldg(p)) * inv;
    }
};

// 32-bit integer hash (xor-shift / multiply finaliser) for the rounding bits.
__device__ __forceinline__ uint32_t mix32(uint32_t x) {
    x ^= x >> 16;
    x *= 0x7feb352du;
    x ^= x >> 15;
    x *= 0x846ca68bu;
    x ^= x >> 16;
    return x;
}

// Where a cell (or the first cell of a pair) pulls from, as indices into a
// plane (a plane's base is the same for all threads, so an address is one
// multiply-add of a 32-bit index): the rows (y - ey, z - ez), all axes
// periodic.
struct Rows {
    uint32_t row[3][3];  // [1 + ey][1 + ez], at the cell's own x
};
__device__ __forceinline__ Rows source_rows(const SimDev &s, uint32_t f, int y, int z) {
    Rows n;
    const int ry = s.nx, rz = s.nx * s.nyf;
    const int ym = y == 0 ? (s.nyf - 1) * ry : -ry, yp = y == s.nyf - 1 ? -(s.nyf - 1) * ry : ry;
    const int zm = z == 0 ? (s.nz - 1) * rz : -rz, zp = z == s.nz - 1 ? -(s.nz - 1) * rz : rz;
    const int dy[3] = {yp, 0, ym}, dz[3] = {zp, 0, zm};
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) n.row[i][j] = f + (uint32_t)(dy[i] + dz[j]);
    return n;
}

// Two FP32 numbers to a packed pair of 16-bit numbers (lo in the low half)
// with stochastic rounding; r supplies the random bits of both.  Beyond the
// largest finite number the result saturates.
template <typename T>
struct Pack2;
template <>
struct Pack2<__half> {
    static __device__ __forceinline__ uint32_t rs(float lo, float hi, uint32_t r) {
        uint32_t d;
        asm("cvt.rs.satfinite.f16x2.f32 %0, %1, %2, %3;" : "=r"(d) : "f"(hi), "f"(lo), "r"(r));
        return d;
    }
};
template <>
struct Pack2<__nv_bfloat16> {
    static __device__ __forceinline__ uint32_t rs(float lo, float hi, uint32_t r) {
        uint32_t d;
        asm("cvt.rs.satfinite.bf16x2.f32 %0, %1, %2, %3;" : "=r"(d) : "f"(hi), "f"(lo), "r"(r));
        return d;
    }
};

template <int MODE, typename V>
__device__ __forceinline__ V ld_pop(const V *p) {
    if constexpr (MODE == MODE_MANY) return __ldcg(p);
    else return __ldg(p);
}

// Raw storage access for the step kernel: the stored number as float (the
// deviation times 2^s for FP16/BF16), and the store of two such numbers at
// two addresses, rounded together with the random bits r.
template <typename T>
struct Raw;
template <>
struct Raw<float> {
    template <int MODE>
    static __device__ __forceinline__ float ld(const float *p) { return ld_pop<MODE>(p); }
    static __device__ __forceinline__ void st2(float *p, float *q, float a, float b, uint32_t) {
        __stcs(p, a);
        __stcs(q, b);
    }
};
template <>
struct Raw<__half> {
    template <int MODE>
    static __device__ __forceinline__ float ld(const __half *p) {
        return __half2float(__ushort_as_half(ld_pop<MODE>((const unsigned short *)p)));
    }
    static __device__ __forceinline__ void st2(__half *p, __half *q, float a, float b, uint32_t r) {
        const uint32_t d = Pack2<__half>::rs(a, b, r);
        __stcs((unsigned short *)p, (unsigned short)d);
        __stcs((unsigned short *)q, (unsigned short)(d >> 16));
    }
};
template <>
struct Raw<__nv_bfloat16> {
    template <int MODE>
    static __device__ __forceinline__ float ld(const __nv_bfloat16 *p) {
        return __uint_as_float((uint32_t)ld_pop<MODE>((const unsigned short *)p) << 16);
    }
    static __device__ __forceinline__ void st2(__nv_bfloat16 *p, __nv_bfloat16 *q, float a, float b, uint32_t r) {
        const uint32_t d = Pack2<__nv_bfloat16>::rs(a, b, r);
        __stcs((unsigned short *)p, (unsigned short)d);
        __stcs((unsigned short *)q, (unsigned short)(d >> 16));
    }
};

// The cell from which population Q of a cell arrives (xm, xp: steps to x - 1
// and x + 1, periodic; walls and obstacles not considered).
template <int Q>
__device__ __forceinline__ uint32_t source_cell(const Rows &n, int xm, int xp) {
    constexpr int ex = d3q19_ex(Q), ey = d3q19_ey(Q), ez = d3q19_ez(Q);
    uint32_t g = n.row[1 + ey][1 + ez];
    if constexpr (ex == 1) g += (uint32_t)xm;
    if constexpr (ex == -1) g += (uint32_t)xp;
    return g;
}

// Pull the (raw) population of direction Q arriving at a cell.
template <typename T, int Q, int MODE>
__device__ __forceinline__ float pull(const T *__restrict__ src, size_t nfp, const Rows &n, int xm, int xp) {
    return Raw<T>::template ld<MODE>(src + (size_t)Q * nfp + source_cell<Q>(n, xm, xp));
}

// Bounce-back at obstacles: a population coming from an obstacle cell is the
// cell's own opposite one.  As at the walls, the pulls already on the way are
// replaced, and only warps with a cell next to an obstacle (near bits) come
// here.  With the 18 bits of the sources asked for before each pull, the
// kernel waited for them one after the other (fluid steps among posts:
// 199x50x30 FP16 20.5 -> 12.3 us, 256x128x128 FP16 211 -> 98, FP32 160 -> 110).
template <typename T, int MODE>
__device__ __forceinline__ void bounce_obstacles(const SimDev &s, const T *__restrict__ src, size_t nfp, uint32_t f,
                                                 const Rows &n, int xm, int xp, float (&h)[NQ]) {
    uint32_t from = 0u;
#define LBIB_SOURCE(q) from |= (uint32_t)solid_bit(s, (int)source_cell<q>(n, xm, xp)) << q;
    LBIB_SOURCE(1) LBIB_SOURCE(2) LBIB_SOURCE(3) LBIB_SOURCE(4) LBIB_SOURCE(5) LBIB_SOURCE(6) LBIB_SOURCE(7)
    LBIB_SOURCE(8) LBIB_SOURCE(9) LBIB_SOURCE(10) LBIB_SOURCE(11) LBIB_SOURCE(12) LBIB_SOURCE(13) LBIB_SOURCE(14)
    LBIB_SOURCE(15) LBIB_SOURCE(16) LBIB_SOURCE(17) LBIB_SOURCE(18)
#undef LBIB_SOURCE
#pragma unroll
    for (int q = 1; q < NQ; ++q)
        if ((from >> q) & 1u) h[q] = Raw<T>::template ld<MODE>(src + (size_t)d3q19_opp(q) * nfp + f);
}

// Bounce-back at a wall row (the row below, EY = 1, or above, EY = -1, is
// solid): the populations with that ey are the cell's own opposite ones.
// Their periodic pulls, already on the way, are replaced; only warps with a
// cell of a wall row come here.
template <typename T, int EY, int MODE>
__device__ __forceinline__ void bounce(const T *__restrict__ src, size_t nfp, uint32_t f, float (&h)[NQ]) {
#pragma unroll
    for (int q = 1; q < NQ; ++q)
        if (d3q19_ey(q) == EY) h[q] = Raw<T>::template ld<MODE>(src + (size_t)d3q19_opp(q) * nfp + f);
}

// BGK + Guo update of the opposite pair (Q, Q+1) (e_{Q+1} = -e_Q, same
// weight w), from the split into the parts even and odd in e:
//   out_{Q/Q+1} = (1 - omega) h + w 2^s [A +- B],
//   A = omega (K + 4.5 rho (e.u)^2) + fpre (9 (e.u)(e.G) - 3 u.G),
//   B = 3 omega rho (e.u) + 3 fpre (e.G),   K = drho - 1.5 rho u.u,
// which is h - omega (h - h_eq) + fpre w [3 (e - u) + 9 (e.u) e].G written
// out for both directions (2^s: raw storage units).  Per cell the
// constants Kb = omega K - 3 fpre u.G and Rb = 3 omega rho are formed once;
// per weight class (wsc = w 2^s) Kc = wsc Kb, Rc = wsc Rb, R15 = 1.5 Rc
// and Gc = 3 fpre wsc G.  As 4.5 omega rho = 1.5 Rb, a pair then costs
//   w 2^s B = Rc (e.u) + e.Gc,   w 2^s A = Kc + (e.u) (R15 (e.u) + 3 e.Gc).
// A does not reuse the rounded B (A = Kc + 1.5 (e.u) (B + e.Gc) is the same
// number in exact arithmetic): that product of e.u with a rounded multiple
// of e.u has a rounding error of one sign, which drifted the total mass of
// a 512x256x256 channel with 16-bit storage by 7.6e-6 in 20,000 steps.
struct Coll {
    float ux, uy, uz, Gx, Gy, Gz, Kb, Rb;
};
struct Cls {
    float K, R, R15, gx, gy, gz;
};
struct CollK {
    float om, c1, fp3, om3;
};

// e component E (-1, 0, 1) times v without a multiply; the zero is -0.0f,
// which the compiler drops from a sum (x + -0 = x for every x), so the
// dot products and moment sums below carry only their non-zero terms.
template <int E>
__device__ __forceinline__ float eterm(float v) {
    if constexpr (E == 1) return v;
    else if constexpr (E == -1) return -v;
    else return -0.0f;
}
template <int Q>
__device__ __forceinline__ float edot(float x, float y, float z) {
    return eterm<d3q19_ex(Q)>(x) + eterm<d3q19_ey(Q)>(y) + eterm<d3q19_ez(Q)>(z);
}

// Moments sum h and sum h e from the opposite pairs: h_Q + h_{Q+1} and
// h_Q - h_{Q+1} for Q = 1, 3, ..., 17.
struct Moments {
    float r, x, y, z;
};
template <int Q>
__device__ __forceinline__ void add_pair(Moments &m, float hq, float ho) {
    const float d = hq - ho;
    m.r += hq + ho;
    m.x += eterm<d3q19_ex(Q)>(d);
    m.y += eterm<d3q19_ey(Q)>(d);
    m.z += eterm<d3q19_ez(Q)>(d);
}
__device__ __forceinline__ Moments moments19(const float (&h)[NQ]) {
    Moments m{h[0], -0.0f, -0.0f, -0.0f};
    add_pair<1>(m, h[1], h[2]);
    add_pair<3>(m, h[3], h[4]);
    add_pair<5>(m, h[5], h[6]);
    add_pair<7>(m, h[7], h[8]);
    add_pair<9>(m, h[9], h[10]);
    add_pair<11>(m, h[11], h[12]);
    add_pair<13>(m, h[13], h[14]);
    add_pair<15>(m, h[15], h[16]);
    add_pair<17>(m, h[17], h[18]);
    return m;
}

// The constants of one weight class (wsc = w 2^s).
__device__ __forceinline__ Cls make_cls(const Coll &c, const CollK &k, float wsc) {
    const float g = k.fp3 * wsc, R = wsc * c.Rb;
    return Cls{wsc * c.Kb, R, 1.5f * R, g * c.Gx, g * c.Gy, g * c.Gz};
}

// w 2^s (A + B, A - B) for the opposite pair (Q, Q+1) of one cell.
template <int Q>
__device__ __forceinline__ float2 pair_terms(const Coll &c, const Cls &w) {
    const float eu = edot<Q>(c.ux, c.uy, c.uz);
    const float eg = edot<Q>(w.gx, w.gy, w.gz);
    const float B = fmaf(w.R, eu, eg);
    const float A = fmaf(eu, fmaf(w.R15, eu, 3.0f * eg), w.K);
    return make_float2(A + B, A - B);
}

template <typename T, int Q>
__device__ __forceinline__ void collide_pair(T *__restrict__ dst, uint32_t nfp, uint32_t f, float hq, float ho,
                                             const Coll &c, const CollK &k, const Cls &w, uint32_t rnd) {
    const float2 ab = pair_terms<Q>(c, w);
    Raw<T>::st2(dst + (uint32_t)Q * nfp + f, dst + (uint32_t)(Q + 1) * nfp + f, fmaf(k.c1, hq, ab.x),
                fmaf(k.c1, ho, ab.y), rnd);
}

// Collision constants of one cell from the raw moments.
__device__ __forceinline__ Coll make_coll(const SimDev &s, const CollK &k, float sr, float sx, float sy, float sz,
                                          float Gx, float Gy, float Gz, float &rho, float &usq) {
    const float inv = s.inv_scale;
    const float drho = sr * inv;
    rho = s.rho0 + drho;
    const float irho = __fdividef(1.0f, rho);  // rho is near 1: the fast reciprocal is within 2 ulp
    Coll c;
    c.ux = fmaf(0.5f, Gx, sx * inv) * irho;
    c.uy = fmaf(0.5f, Gy, sy * inv) * irho;
    c.uz = fmaf(0.5f, Gz, sz * inv) * irho;
    c.Gx = Gx;
    c.Gy = Gy;
    c.Gz = Gz;
    usq = c.ux * c.ux + c.uy * c.uy + c.uz * c.uz;
    const float uG = c.ux * Gx + c.uy * Gy + c.uz * Gz;
    const float K = fmaf(-1.5f * rho, usq, drho);
    c.Kb = fmaf(k.om, K, -k.fp3 * uG);
    c.Rb = k.om3 * rho;
    return c;
}

__device__ __forceinline__ CollK make_collk(const SimDev &s) {
    CollK k;
    k.om = s.omega;
    k.c1 = 1.0f - s.omega;
    k.fp3 = 3.0f * s.fpre;
    k.om3 = 3.0f * s.omega;
    return k;
}

// Velocity inlet (the inflow plane of the Sec. 6 example, whose velocity is
// set before every step): the populations pulled into an inlet cell are
// replaced by the equilibrium at the cell's own density and the prescribed
// velocity, w (drho + rho (3 e.u + 4.5 (e.u)^2 - 1.5 u.u)) in deviation
// form, before the collision.  h holds raw numbers (times 2^s).
template <int Q>
__device__ __forceinline__ float inlet_eq(float drho, float rho, float usq, const float *u, float sc) {
    const float eu = edot<Q>(u[0], u[1], u[2]);
    return (float)d3q19_w(Q) * sc * (drho + rho * (3.0f * eu + 4.5f * eu * eu - 1.5f * usq));
}

__device__ __forceinline__ void inlet_cell(const SimDev &s, int x, int yl, int z, float (&h)[NQ]) {
    const int *b = s.in_box;
    if (x < b[0] || x >= b[1] || yl < b[2] || yl >= b[3] || z < b[4] || z >= b[5]) return;
    float sr = 0.f;
#pragma unroll
    for (int q = 0; q < NQ; ++q) sr += h[q];
    const float drho = sr * s.inv_scale, rho = s.rho0 + drho, sc = s.scale;
    const float *u = s.in_u;
    const float usq = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
    h[0] = inlet_eq<0>(drho, rho, usq, u, sc);
    h[1] = inlet_eq<1>(drho, rho, usq, u, sc);
    h[2] = inlet_eq<2>(drho, rho, usq, u, sc);
    h[3] = inlet_eq<3>(drho, rho, usq, u, sc);
    h[4] = inlet_eq<4>(drho, rho, usq, u, sc);
    h[5] = inlet_eq<5>(drho, rho, usq, u, sc);
    h[6] = inlet_eq<6>(drho, rho, usq, u, sc);
    h[7] = inlet_eq<7>(drho, rho, usq, u, sc);
    h[8] = inlet_eq<8>(drho, rho, usq, u, sc);
    h[9] = inlet_eq<9>(drho, rho, usq, u, sc);
    h[10] = inlet_eq<10>(drho, rho, usq, u, sc);
    h[11] = inlet_eq<11>(drho, rho, usq, u, sc);
    h[12] = inlet_eq<12>(drho, rho, usq, u, sc);
    h[13] = inlet_eq<13>(drho, rho, usq, u, sc);
    h[14] = inlet_eq<14>(drho, rho, usq, u, sc);
    h[15] = inlet_eq<15>(drho, rho, usq, u, sc);
    h[16] = inlet_eq<16>(drho, rho, usq, u, sc);
    h[17] = inlet_eq<17>(drho, rho, usq, u, sc);
    h[18] = inlet_eq<18>(drho, rho, usq, u, sc);
}

// FP32 storage: the same BGK + Guo update written as an increment,
// out = h + Delta, where every part of Delta is formed from quantities that
// are small when the cell is near equilibrium, and the only rounding at the
// scale of h is the final addition.  Per opposite pair (Q, Q+1), with
// a = (h_Q - h_Q+1)/2, m = (h_Q + h_Q+1)/2 and j = sum h e (the momentum
// of the stored deviations, without the force):
//   odd   D_o = omega (3w e.j - a) + 3w e.G        (omega/2 + fpre = 1)
//   even  D_e = omega (w (K + 4.5 rho (e.u)^2) - m) + fpre w (9 (e.u)(e.G) - 3 u.G)
//   out_Q = h_Q + (D_e + D_o),  out_Q+1 = h_Q+1 + (D_e - D_o),
// and for the rest population out_0 = h_0 + omega (w0 K - h_0) - 3 fpre w0 u.G,
// with u = (j + G/2)/rho and K = drho - 1.5 rho u.u.  The product 3w e.j
// and the subtraction of a are one FMA (a single rounding at the scale of
// the non-equilibrium part), and 3w (1/6, 1/12) is applied as an unevaluated
// FP32 pair hi + lo: FP32 rounding of 1/6 alone changes every cell's
// momentum in the same direction by 3e-8 of itself per step, which the
// driven channel integrates into a relative velocity bias ~200 times
// larger.  Likewise the force is not added into j before it is rounded:
// adding the same small G/2 to every cell's j rounds the same way in every
// cell of a binade.
struct Inc {
    float sx, sy, sz;      // j
    float ux, uy, uz;      // u
    float Gx, Gy, Gz;      // force density of this step
    float K, r45, m3uG;    // K, 4.5 rho, -3 u.G
    float om, fpre;
};

constexpr double INC_C1 = 1.0 / 6.0;   // 3 w for |e|^2 = 1
constexpr float INC_C1_HI = (float)INC_C1;
constexpr float INC_C1_LO = (float)(INC_C1 - (double)INC_C1_HI);

template <int Q>
__device__ __forceinline__ void inc_pair(float *__restrict__ dst, uint32_t nfp, uint32_t f, float hq, float ho,
                                         const Inc &c) {
    constexpr bool axis = Q < 7;  // |e|^2 = 1; else 2 (weight and 3w halved, exactly)
    constexpr float wq = axis ? (float)(1.0 / 18.0) : (float)(1.0 / 36.0);
    constexpr float chi = axis ? INC_C1_HI : 0.5f * INC_C1_HI, clo = axis ? INC_C1_LO : 0.5f * INC_C1_LO;
    const float a = 0.5f * __fsub_rn(hq, ho), m = 0.5f * __fadd_rn(hq, ho);
    const float ej = edot<Q>(c.sx, c.sy, c.sz);
    const float eu = edot<Q>(c.ux, c.uy, c.uz);
    const float eG = edot<Q>(c.Gx, c.Gy, c.Gz);
    float t = __fmaf_rn(chi, ej, -a);
    t = __fmaf_rn(clo, ej, t);
    const float Do = __fmaf_rn(c.om, t, __fmaf_rn(chi, eG, __fmul_rn(clo, eG)));
    const float Aeq = __fmaf_rn(__fmul_rn(c.r45, wq), __fmul_rn(eu, eu), __fmul_rn(wq, c.K));
    const float Fe = __fmul_rn(__fmul_rn(c.fpre, wq), __fmaf_rn(__fmul_rn(9.0f, eu), eG, c.m3uG));
    const float De = __fmaf_rn(c.om, __fsub_rn(Aeq, m), Fe);
    __stcs(dst + (uint32_t)Q * nfp + f, __fadd_rn(hq, __fadd_rn(De, Do)));
    __stcs(dst + (uint32_t)(Q + 1) * nfp + f, __fadd_rn(ho, __fsub_rn(De, Do)));
}

// The increment-form collision and store of one FP32 cell from its pulled
// populations h; returns u.u (the stability check) and sets u, rho.
__device__ __forceinline__ float collide_increment(const SimDev &s, float *__restrict__ dst, uint32_t nfp, uint32_t f,
                                                   const float (&h)[NQ], float Gx, float Gy, float Gz, float &ux,
                                                   float &uy, float &uz, float &rho) {
    const Moments mo = moments19(h);
    Inc c;
    c.om = s.omega;
    c.fpre = s.fpre;
    c.sx = mo.x;
    c.sy = mo.y;
    c.sz = mo.z;
    c.Gx = Gx;
    c.Gy = Gy;
    c.Gz = Gz;
    const float drho = mo.r;
    rho = s.rho0 + drho;
    const float irho = __fdividef(1.0f, rho);  // rho is near 1: the fast reciprocal is within 2 ulp
    ux = fmaf(0.5f, Gx, mo.x) * irho;
    uy = fmaf(0.5f, Gy, mo.y) * irho;
    uz = fmaf(0.5f, Gz, mo.z) * irho;
    c.ux = ux;
    c.uy = uy;
    c.uz = uz;
    // explicit order: the two-cells kernel's packed instructions, bit for bit
    const float usq = __fmaf_rn(uz, uz, __fmaf_rn(uy, uy, __fmul_rn(ux, ux)));
    c.m3uG = __fmul_rn(-3.0f, __fmaf_rn(uz, Gz, __fmaf_rn(uy, Gy, __fmul_rn(ux, Gx))));
    c.K = fmaf(-1.5f * rho, usq, drho);
    c.r45 = 4.5f * rho;
    constexpr float w0 = (float)(1.0 / 3.0);
    const float h0 = h[0];
    __stcs(dst + f, __fadd_rn(h0, __fmaf_rn(c.om, __fmaf_rn(w0, c.K, -h0), __fmul_rn(c.fpre * w0, c.m3uG))));
    inc_pair<1>(dst, nfp, f, h[1], h[2], c);
    inc_pair<3>(dst, nfp, f, h[3], h[4], c);
    inc_pair<5>(dst, nfp, f, h[5], h[6], c);
    inc_pair<7>(dst, nfp, f, h[7], h[8], c);
    inc_pair<9>(dst, nfp, f, h[9], h[10], c);
    inc_pair<11>(dst, nfp, f, h[11], h[12], c);
    inc_pair<13>(dst, nfp, f, h[13], h[14], c);
    inc_pair<15>(dst, nfp, f, h[15], h[16], c);
    inc_pair<17>(dst, nfp, f, h[17], h[18], c);
    return usq;
}

// BC: the variant for simulations with obstacles or a velocity inlet (the
// plain variant carries no test for either).
// The active-cell word of the warp that owns fluid cell f (blocks start at
// multiples of 32, so a warp owns exactly one word).  Read through L2: the
// object update of the same launch may set bits.
__device__ __forceinline__ uint32_t active_word(const SimDev &s, int f) {
    const int w = f >> 5;
    return (w < s.nwords) ? __ldcg(s.amask + w) : 0u;
}

// MODE_EARLY (the kernel may be launched early, programmatic dependent launch):
// the mask word is read after dep_wait(); otherwise it is `act`, read by the
// caller before the pulls.
template <typename T, bool BC, int MODE>
__device__ __forceinline__ void fluid_cell(const SimDev &s, int par, int fi, uint32_t act, uint32_t step_seed) {
    static_assert(d3q19_opp(1) == 2 && d3q19_opp(17) == 18, "directions 2k-1, 2k must be opposite");
    const T *__restrict__ src = (const T *)s.pop[par];
    T *__restrict__ dst = (T *)s.pop[par ^ 1];
    const uint32_t nfp = (uint32_t)s.nfp, f = (uint32_t)fi;
    const bool obstacle = BC && s.solid && solid_bit(s, fi), near = BC && s.solid && near_bit(s, fi);
    const uint32_t r = s.div_nx.div(f);
    const uint32_t x = f - r * (uint32_t)s.nx;
    const uint32_t z = s.div_nyf.div(r);
    const uint32_t y = r - z * (uint32_t)s.nyf;
    const Rows n = source_rows(s, f, (int)y, (int)z);
    const int xm = x == 0 ? s.nx - 1 : -1, xp = x == (uint32_t)s.nx - 1 ? 1 - s.nx : 1;

    float h[NQ];
#define LBIB_PULL(q) h[q] = pull<T, q, MODE>(src, nfp, n, xm, xp);
    LBIB_PULL(0) LBIB_PULL(1) LBIB_PULL(2) LBIB_PULL(3) LBIB_PULL(4) LBIB_PULL(5) LBIB_PULL(6)
    LBIB_PULL(7) LBIB_PULL(8) LBIB_PULL(9) LBIB_PULL(10) LBIB_PULL(11) LBIB_PULL(12) LBIB_PULL(13)
    LBIB_PULL(14) LBIB_PULL(15) LBIB_PULL(16) LBIB_PULL(17) LBIB_PULL(18)
#undef LBIB_PULL
    if (BC && __any_sync(__activemask(), obstacle || near)) {
        if (obstacle) return;  // holds no fluid
        if (near) bounce_obstacles<T, MODE>(s, src, nfp, f, n, xm, xp, h);
    }
    const bool ylo = s.walls && y == 0, yhi = s.walls && y == (uint32_t)s.nyf - 1;
    if (__any_sync(__activemask(), ylo || yhi)) {
        if (ylo) bounce<T, 1, MODE>(src, nfp, f, h);
        if (yhi) bounce<T, -1, MODE>(src, nfp, f, h);
    }

    if (BC && s.in_on) inlet_cell(s, (int)x, (int)y + s.walls, (int)z, h);
    // the populations pulled above were written by the previous fluid step;
    // the mask and the coupling buffer below by the node update of this one
    if constexpr (MODE == MODE_EARLY) {
        dep_wait();
        dep_release();
        act = active_word(s, fi);
    }
    const bool active = (act >> (fi & 31)) & 1u;

    float Gx = s.gx, Gy = s.gy, Gz = s.gz;
    // spread force of this step; clear the buffer of the next.  Most warps have
    // no active cell: a warp vote keeps this behind a branch (a plain
    // condition becomes predicated instructions that every warp issues).
    if (__any_sync(__activemask(), active) && active) {
        const float4 g = __ldcg(s.G[par] + f);
        Gx += g.x;
        Gy += g.y;
        Gz += g.z;
        s.G[par ^ 1][f] = make_float4(0.f, 0.f, 0.f, 0.f);
    }

    if constexpr (sizeof(T) == 4) {
        float ux, uy, uz, rho;
        const float usq = collide_increment(s, (float *)dst, nfp, f, h, Gx, Gy, Gz, ux, uy, uz, rho);
        if (active) s.ufield[f] = make_float4(ux, uy, uz, rho);
        if (!(usq < 0.09f)) atomicOr(s.status, ST_UNSTABLE);
        return;
    }

    // moments of the raw numbers, then back to deviations (exact: 2^-s)
    const Moments m = moments19(h);
    const CollK k = make_collk(s);
    float rho, usq;
    const Coll c = make_coll(s, k, m.r, m.x, m.y, m.z, Gx, Gy, Gz, rho, usq);
    const float sc = s.scale;
    const float wsc0 = (float)d3q19_w(0) * sc;
    const Cls w1 = make_cls(c, k, (float)d3q19_w(1) * sc);
    const Cls w2 = make_cls(c, k, (float)d3q19_w(7) * sc);

    // 32 random bits per rounded pair of populations for FP16/BF16 (one
    // step of a linear congruential generator each)
    uint32_t rng = (sizeof(T) == 2) ? mix32(f ^ step_seed) : 0u;
    auto next = [&]() -> uint32_t {
        if (sizeof(T) != 2) return 0u;
        rng = rng * 747796405u + 2891336453u;
        return rng ^ (rng >> 15);
    };
    const float out0 = fmaf(k.c1, h[0], wsc0 * c.Kb);
    if constexpr (sizeof(T) == 2) {  // the rest population alone: the high half is discarded
        const uint32_t d = Pack2<T>::rs(out0, 0.0f, next());
        __stcs((unsigned short *)(dst + f), (unsigned short)d);
    } else {
        __stcs((float *)(dst + f), out0);
    }
    collide_pair<T, 1>(dst, nfp, f, h[1], h[2], c, k, w1, next());
    collide_pair<T, 3>(dst, nfp, f, h[3], h[4], c, k, w1, next());
    collide_pair<T, 5>(dst, nfp, f, h[5], h[6], c, k, w1, next());
    collide_pair<T, 7>(dst, nfp, f, h[7], h[8], c, k, w2, next());
    collide_pair<T, 9>(dst, nfp, f, h[9], h[10], c, k, w2, next());
    collide_pair<T, 11>(dst, nfp, f, h[11], h[12], c, k, w2, next());
    collide_pair<T, 13>(dst, nfp, f, h[13], h[14], c, k, w2, next());
    collide_pair<T, 15>(dst, nfp, f, h[15], h[16], c, k, w2, next());
    collide_pair<T, 17>(dst, nfp, f, h[17], h[18], c, k, w2, next());

    if (active) s.ufield[f] = make_float4(c.ux, c.uy, c.uz, rho);
    if (!(usq < 0.09f)) atomicOr(s.status, ST_UNSTABLE);
}

// ------------------------------------------------------------------
// Two cells per thread (no obstacles, no inlet).
// A thread owns cells f and f+1 (f even; in the same row when nx is even, else
// see fluid_pair_odd).  Populations of the
// two cells sit next to each other in every plane, so the pair is read as
// one 32-bit word where the source is even (directions without an x
// component, bounce-back) and as two 16-bit words at adjacent addresses
// otherwise, and always written as one 32-bit word; the index, neighbour
// and address arithmetic and the random bits are shared by the two cells.

template <typename T>
struct Half2Bits;
template <>
struct Half2Bits<__half> {
    static __device__ __forceinline__ float lo(uint32_t u) { return __half2float(__ushort_as_half((unsigned short)u)); }
    static __device__ __forceinline__ float hi(uint32_t u) {
        return __half2float(__ushort_as_half((unsigned short)(u >> 16)));
    }
};
template <>
struct Half2Bits<__nv_bfloat16> {
    static __device__ __forceinline__ float lo(uint32_t u) { return __uint_as_float(u << 16); }
    static __device__ __forceinline__ float hi(uint32_t u) { return __uint_as_float(u & 0xffff0000u); }
};

// Blocks of 128 threads: when a membrane block shares the SM, one of five or
// six fluid blocks gives way instead of one of three.
constexpr int PAIR_THREADS = 128;
template <typename T>
constexpr int pair_blocks() {  // per SM, at 96 (FP32) and 80 registers a thread
    return sizeof(T) == 4 ? 5 : 6;
}

// A stored pair of cells: two 16-bit numbers in a word (low half: cell f), or
// two FP32 numbers; p[i], p[i + 1] (i even) or p[i], p[j].
template <typename T>
struct PairRaw {
    using type = uint32_t;
    template <int MODE>
    static __device__ __forceinline__ uint32_t ld(const T *p, uint32_t i) {
        return ld_pop<MODE>((const unsigned int *)(p + i));
    }
    template <int MODE>
    static __device__ __forceinline__ uint32_t ld(const T *p, uint32_t i, uint32_t j) {
        return (uint32_t)ld_pop<MODE>((const unsigned short *)p + i) |
               ((uint32_t)ld_pop<MODE>((const unsigned short *)p + j) << 16);
    }
};
template <>
struct PairRaw<float> {
    using type = float2;
    template <int MODE>
    static __device__ __forceinline__ float2 ld(const float *p, uint32_t i) {
        return ld_pop<MODE>((const float2 *)(p + i));
    }
    template <int MODE>
    static __device__ __forceinline__ float2 ld(const float *p, uint32_t i, uint32_t j) {
        return make_float2(ld_pop<MODE>(p + i), ld_pop<MODE>(p + j));
    }
};

// The pair of direction Q arriving at cells f, f+1 (xm, xp: steps from f to
// x - 1 and to x + 2, periodic; walls not considered).
// Marking these loads evict-first in L2 kept the velocity and force fields
// for the node update that follows (20.7 -> 18.2 us at 256x128x128) but
// slowed the kernel 6% at 512x256x256, where the x-shifted lines shared by
// neighbouring warps were evicted in between; the loads keep the default
// policy.
template <typename T, int Q, int MODE>
__device__ __forceinline__ typename PairRaw<T>::type pull2(const T *__restrict__ src, size_t nfp, const Rows &n, int xm,
                                                           int xp) {
    constexpr int ex = d3q19_ex(Q), ey = d3q19_ey(Q), ez = d3q19_ez(Q);
    const T *p = src + (size_t)Q * nfp;
    const uint32_t o = n.row[1 + ey][1 + ez];
    if constexpr (ex == 0) return PairRaw<T>::template ld<MODE>(p, o);
    else if constexpr (ex == 1) return PairRaw<T>::template ld<MODE>(p, o + (uint32_t)xm, o);  // from x - 1 and x
    else return PairRaw<T>::template ld<MODE>(p, o + 1u, o + (uint32_t)xp);                    // from x + 1 and x + 2
}

// bounce() of the pair
template <typename T, int EY, int MODE>
__device__ __forceinline__ void bounce2(const T *__restrict__ src, size_t nfp, uint32_t f,
                                        typename PairRaw<T>::type (&P)[NQ]) {
#pragma unroll
    for (int q = 1; q < NQ; ++q)
        if (d3q19_ey(q) == EY) P[q] = PairRaw<T>::template ld<MODE>(src + (size_t)d3q19_opp(q) * nfp, f);
}

// Odd nx: the pair of direction Q from any two cells, and bounce() where one or
// both of them are at the wall
template <typename T, int Q, int MODE>
__device__ __forceinline__ typename PairRaw<T>::type pull_cells(const T *__restrict__ src, size_t nfp, const Rows &na,
                                                                int xma, int xpa, const Rows &nb, int xmb, int xpb) {
    return PairRaw<T>::template ld<MODE>(src + (size_t)Q * nfp, source_cell<Q>(na, xma, xpa), source_cell<Q>(nb, xmb, xpb));
}
// last: the pair's second place is padding (see fluid_pair_odd) and takes the first cell's value
template <typename T, int EY, int MODE>
__device__ __forceinline__ void bounce_cells(const T *__restrict__ src, size_t nfp, uint32_t f, bool a, bool b, bool last,
                                             typename PairRaw<T>::type (&P)[NQ]) {
#pragma unroll
    for (int q = 1; q < NQ; ++q)
        if (d3q19_ey(q) == EY) {
            const auto own = PairRaw<T>::template ld<MODE>(src + (size_t)d3q19_opp(q) * nfp, f);
            if constexpr (sizeof(T) == 4) P[q] = make_float2(a ? own.x : P[q].x, b ? (last ? own.x : own.y) : P[q].y);
            else P[q] = __byte_perm(P[q], own, (a ? 0x0054u : 0x0010u) | (b ? (last ? 0x5400u : 0x7600u) : 0x3200u));
        }
}

// The arithmetic of the two cells runs in packed FP32 instructions (sm_100
// family: one instruction updates both cells, each component rounded as the
// scalar instruction would round it); x holds cell f, y cell f+1.
__device__ __forceinline__ float2 v2(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, v2(-1.0f), a); }  // b * -1 is exact
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }

// s + E v, E = +-1
template <int E>
__device__ __forceinline__ float2 acc2(float2 s, float2 v) {
    static_assert(E == 1 || E == -1, "unit component");
    if constexpr (E == 1) return add2(s, v);
    else return sub2(s, v);
}

// e_Q . v for a pair representative Q (odd Q: its first non-zero component
// is +1), with only the non-zero terms.
template <int Q>
__device__ __forceinline__ float2 edot2(float2 x, float2 y, float2 z) {
    constexpr int ex = d3q19_ex(Q), ey = d3q19_ey(Q), ez = d3q19_ez(Q);
    static_assert(Q % 2 == 1, "pair representative");
    if constexpr (ex != 0) {
        static_assert(ex == 1, "leading +1");
        float2 s = x;
        if constexpr (ey != 0) s = acc2<ey>(s, y);
        if constexpr (ez != 0) s = acc2<ez>(s, z);
        return s;
    } else if constexpr (ey != 0) {
        static_assert(ey == 1, "leading +1");
        if constexpr (ez != 0) return acc2<ez>(y, z);
        else return y;
    } else {
        static_assert(ez == 1, "leading +1");
        return z;
    }
}

template <typename T>
__device__ __forceinline__ float2 unpack2(uint32_t u) {
    return make_float2(Half2Bits<T>::lo(u), Half2Bits<T>::hi(u));
}

// The pair as two FP32 numbers
template <typename T>
__device__ __forceinline__ float2 pair_f32(typename PairRaw<T>::type v) {
    if constexpr (sizeof(T) == 4) return v;
    else return unpack2<T>(v);
}

struct Moments2 {
    float2 r, x, y, z;
};
// the difference h_Q - h_{Q+1} of pair Q into the momentum sums
template <int Q>
__device__ __forceinline__ void add_diff2(Moments2 &m, float2 d) {
    if constexpr (d3q19_ex(Q) != 0) m.x = acc2<d3q19_ex(Q)>(m.x, d);
    if constexpr (d3q19_ey(Q) != 0) m.y = acc2<d3q19_ey(Q)>(m.y, d);
    if constexpr (d3q19_ez(Q) != 0) m.z = acc2<d3q19_ez(Q)>(m.z, d);
}
// The moments of both cells: sum h from the pair sums, sum h e from the
// pair differences; the axis pairs (1, 3, 5) open the x, y, z sums.
template <typename T>
__device__ __forceinline__ Moments2 moments2(const typename PairRaw<T>::type (&P)[NQ]) {
    static_assert(d3q19_ex(1) == 1 && d3q19_ey(3) == 1 && d3q19_ez(5) == 1, "axis pairs 1, 3, 5");
    Moments2 m;
    float2 a = pair_f32<T>(P[1]), b = pair_f32<T>(P[2]);
    m.r = add2(pair_f32<T>(P[0]), add2(a, b));
    m.x = sub2(a, b);
    a = pair_f32<T>(P[3]), b = pair_f32<T>(P[4]);
    m.r = add2(m.r, add2(a, b));
    m.y = sub2(a, b);
    a = pair_f32<T>(P[5]), b = pair_f32<T>(P[6]);
    m.r = add2(m.r, add2(a, b));
    m.z = sub2(a, b);
#define LBIB_M2(q)                          \
    a = pair_f32<T>(P[q]), b = pair_f32<T>(P[q + 1]); \
    m.r = add2(m.r, add2(a, b));            \
    add_diff2<q>(m, sub2(a, b));
    LBIB_M2(7) LBIB_M2(9) LBIB_M2(11) LBIB_M2(13) LBIB_M2(15) LBIB_M2(17)
#undef LBIB_M2
    return m;
}

// Coll, Cls of both cells
struct Coll2 {
    float2 ux, uy, uz, Gx, Gy, Gz, Kb, Rb;
};
struct Cls2 {
    float2 K, R, R15, gx, gy, gz;
};

// OWN: in the order in which the one-cell kernel's sums are contracted
template <bool OWN>
__device__ __forceinline__ float2 dot2(float2 ax, float2 ay, float2 az, float2 bx, float2 by, float2 bz) {
    if constexpr (OWN) return fma2(az, bz, fma2(ax, bx, mul2(ay, by)));
    else return fma2(az, bz, fma2(ay, by, mul2(ax, bx)));
}
template <bool OWN>
__device__ __forceinline__ Coll2 make_coll2(const SimDev &s, const CollK &k, const Moments2 &m, float2 Gx, float2 Gy,
                                            float2 Gz, float2 &rho, float2 &usq) {
    const float2 inv = v2(s.inv_scale), half = v2(0.5f);
    const float2 drho = mul2(m.r, inv);
    rho = add2(drho, v2(s.rho0));
    // rho is near 1: the fast reciprocal is within 2 ulp
    const float2 irho = make_float2(__fdividef(1.0f, rho.x), __fdividef(1.0f, rho.y));
    Coll2 c;
    c.ux = mul2(fma2(half, Gx, mul2(m.x, inv)), irho);
    c.uy = mul2(fma2(half, Gy, mul2(m.y, inv)), irho);
    c.uz = mul2(fma2(half, Gz, mul2(m.z, inv)), irho);
    c.Gx = Gx;
    c.Gy = Gy;
    c.Gz = Gz;
    usq = dot2<OWN>(c.ux, c.uy, c.uz, c.ux, c.uy, c.uz);
    const float2 uG = dot2<OWN>(c.ux, c.uy, c.uz, Gx, Gy, Gz);
    const float2 K = fma2(mul2(v2(-1.5f), rho), usq, drho);
    c.Kb = fma2(v2(k.om), K, mul2(v2(-k.fp3), uG));
    c.Rb = mul2(v2(k.om3), rho);
    return c;
}

__device__ __forceinline__ Cls2 make_cls2(const Coll2 &c, const CollK &k, float wsc) {
    const float2 g = v2(k.fp3 * wsc), w = v2(wsc);
    const float2 R = mul2(w, c.Rb);
    return Cls2{mul2(w, c.Kb), R, mul2(v2(1.5f), R), mul2(g, c.Gx), mul2(g, c.Gy), mul2(g, c.Gz)};
}

// pair_terms for both cells
template <int Q>
__device__ __forceinline__ void pair_terms2(const Coll2 &c, const Cls2 &w, float2 &ApB, float2 &AmB) {
    const float2 eu = edot2<Q>(c.ux, c.uy, c.uz);
    const float2 eg = edot2<Q>(w.gx, w.gy, w.gz);
    const float2 B = fma2(w.R, eu, eg);
    const float2 A = fma2(eu, fma2(w.R15, eu, mul2(v2(3.0f), eg)), w.K);
    ApB = add2(A, B);
    AmB = sub2(A, B);
}

// OWN: each cell has its own random bits (rng, rng2), as in the one-cell kernel,
// which rounds the two populations of a cell together.
template <typename T, int Q, bool OWN>
__device__ __forceinline__ void collide2(uint16_t *__restrict__ dst, size_t nfp, uint32_t f, uint32_t Pq, uint32_t Po,
                                         const Coll2 &c, const CollK &k, const Cls2 &w,
                                         uint32_t &rng, uint32_t &rng2) {
    float2 ApB, AmB;
    pair_terms2<Q>(c, w, ApB, AmB);
    const float2 oq = fma2(v2(k.c1), unpack2<T>(Pq), ApB), oo = fma2(v2(k.c1), unpack2<T>(Po), AmB);
    rng = rng * 747796405u + 2891336453u;
    if constexpr (OWN) {
        rng2 = rng2 * 747796405u + 2891336453u;
        const uint32_t a = Pack2<T>::rs(oq.x, oo.x, rng ^ (rng >> 15)), b = Pack2<T>::rs(oq.y, oo.y, rng2 ^ (rng2 >> 15));
        __stcs((unsigned int *)(dst + (size_t)Q * nfp + f), __byte_perm(a, b, 0x5410));
        __stcs((unsigned int *)(dst + (size_t)(Q + 1) * nfp + f), __byte_perm(a, b, 0x7632));
        return;
    }
    const uint32_t r1 = rng ^ (rng >> 15);
    // The second store takes the same 32 bits with their halves exchanged:
    // each rounding still sees uniform bits (so stays unbiased); only
    // population q of one cell and q-bar of the other share bits, which
    // changes the variance of sums over two cells, not their mean (the
    // 16-bit Poiseuille errors were unchanged: 2.66e-4 FP16, 1.52e-3 BF16).
    const uint32_t r2 = __byte_perm(r1, 0u, 0x1032);
    __stcs((unsigned int *)(dst + (size_t)Q * nfp + f), Pack2<T>::rs(oq.x, oq.y, r1));
    __stcs((unsigned int *)(dst + (size_t)(Q + 1) * nfp + f), Pack2<T>::rs(oo.x, oo.y, r2));
}

// The increment form (struct Inc) of both FP32 cells, in packed instructions:
// the same parts per opposite pair, with the products of constants and cell
// quantities that a weight class shares formed once.
struct Inc2 {
    Moments2 m;               // j in x, y, z
    float2 ux, uy, uz, Gx, Gy, Gz, m3uG;
    float om;
};
struct IncCls2 {
    float2 r45, K;            // w (4.5 rho), w K
    float chi, clo, fw;       // 3 w as hi + lo, fpre w
};
template <int Q>
__device__ __forceinline__ void inc_pair2(float *__restrict__ dst, size_t nfp, uint32_t f, float2 hq, float2 ho,
                                          const Inc2 &c, const IncCls2 &w) {
    const float2 ej = edot2<Q>(c.m.x, c.m.y, c.m.z), eu = edot2<Q>(c.ux, c.uy, c.uz), eG = edot2<Q>(c.Gx, c.Gy, c.Gz);
    float2 t = fma2(v2(w.chi), ej, mul2(v2(-0.5f), sub2(hq, ho)));
    t = fma2(v2(w.clo), ej, t);
    const float2 Do = fma2(v2(c.om), t, fma2(v2(w.chi), eG, mul2(v2(w.clo), eG)));
    const float2 Aeq = fma2(w.r45, mul2(eu, eu), w.K);
    const float2 Fe = mul2(v2(w.fw), fma2(mul2(v2(9.0f), eu), eG, c.m3uG));
    const float2 De = fma2(v2(c.om), fma2(v2(-0.5f), add2(hq, ho), Aeq), Fe);
    __stcs((float2 *)(dst + (size_t)Q * nfp + f), add2(hq, add2(De, Do)));
    __stcs((float2 *)(dst + (size_t)(Q + 1) * nfp + f), add2(ho, sub2(De, Do)));
}

// Collision and store of the FP32 pair; sets u, rho and returns u.u.
__device__ __forceinline__ float2 collide_increment2(const SimDev &s, float *__restrict__ dst, size_t nfp, uint32_t f,
                                                     const float2 (&h)[NQ], Inc2 &c, float2 &rho) {
    c.m = moments2<float>(h);
    c.om = s.omega;
    rho = add2(v2(s.rho0), c.m.r);
    // rho is near 1: the fast reciprocal is within 2 ulp
    const float2 irho = make_float2(__fdividef(1.0f, rho.x), __fdividef(1.0f, rho.y));
    c.ux = mul2(fma2(v2(0.5f), c.Gx, c.m.x), irho);
    c.uy = mul2(fma2(v2(0.5f), c.Gy, c.m.y), irho);
    c.uz = mul2(fma2(v2(0.5f), c.Gz, c.m.z), irho);
    const float2 usq = fma2(c.uz, c.uz, fma2(c.uy, c.uy, mul2(c.ux, c.ux)));
    c.m3uG = mul2(v2(-3.0f), fma2(c.uz, c.Gz, fma2(c.uy, c.Gy, mul2(c.ux, c.Gx))));
    const float2 K = fma2(mul2(v2(-1.5f), rho), usq, c.m.r), r45 = mul2(v2(4.5f), rho);
    constexpr float w0 = (float)(1.0 / 3.0), w1 = (float)(1.0 / 18.0), w2 = (float)(1.0 / 36.0);
    __stcs((float2 *)(dst + f),
           add2(h[0], fma2(v2(c.om), fma2(v2(w0), K, mul2(v2(-1.0f), h[0])), mul2(v2(s.fpre * w0), c.m3uG))));
    {
        const IncCls2 w{mul2(r45, v2(w1)), mul2(v2(w1), K), INC_C1_HI, INC_C1_LO, s.fpre * w1};
        inc_pair2<1>(dst, nfp, f, h[1], h[2], c, w);
        inc_pair2<3>(dst, nfp, f, h[3], h[4], c, w);
        inc_pair2<5>(dst, nfp, f, h[5], h[6], c, w);
    }
    const IncCls2 w{mul2(r45, v2(w2)), mul2(v2(w2), K), 0.5f * INC_C1_HI, 0.5f * INC_C1_LO, s.fpre * w2};
    inc_pair2<7>(dst, nfp, f, h[7], h[8], c, w);
    inc_pair2<9>(dst, nfp, f, h[9], h[10], c, w);
    inc_pair2<11>(dst, nfp, f, h[11], h[12], c, w);
    inc_pair2<13>(dst, nfp, f, h[13], h[14], c, w);
    inc_pair2<15>(dst, nfp, f, h[15], h[16], c, w);
    inc_pair2<17>(dst, nfp, f, h[17], h[18], c, w);
    return usq;
}

// Collision and store of the cell pair (f, f+1) from its pulled populations
// P (packed pairs, low half: cell f).
// c: the coupling of the pair, as load_coupling returned it.
struct Coupling {
    float4 a, b;   // spread force on cells f and f + 1
    uint32_t act;  // active-cell bits of f (bit 0) and f + 1 (bit 1)
    bool any;      // of the warp
};
// The spread force of this step on the active cells of the pair; clears
// their places in the buffer of the next.  Most warps have no active cell: a
// warp vote keeps the rest behind a branch (a plain condition becomes
// predicated instructions that every warp issues).  Issuing these loads
// right after the pulls', before their first use, was no faster with objects
// (67.7 us for the 16-bit kernel at 256x128x128 with 200 cells either way)
// and slower without (59.2 against 57.6).
__device__ __forceinline__ Coupling load_coupling(const SimDev &s, int par, uint32_t f, uint32_t act) {
    Coupling c{make_float4(0.f, 0.f, 0.f, 0.f), make_float4(0.f, 0.f, 0.f, 0.f), act,
               (bool)__any_sync(__activemask(), act != 0u)};
    if (c.any) {
        if (act & 1u) c.a = __ldcg(s.G[par] + f);
        if (act & 2u) c.b = __ldcg(s.G[par] + f + 1);
        if (act & 1u) s.G[par ^ 1][f] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (act & 2u) s.G[par ^ 1][f + 1] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    return c;
}

template <typename T, bool OWN = false>
__device__ __forceinline__ void pair_update(const SimDev &s, int par, uint32_t f, const typename PairRaw<T>::type (&P)[NQ],
                                            uint32_t step_seed, const Coupling &cp) {
    const size_t nfp = (size_t)s.nfp;
    const float2 Gx = make_float2(s.gx + cp.a.x, s.gx + cp.b.x), Gy = make_float2(s.gy + cp.a.y, s.gy + cp.b.y),
                 Gz = make_float2(s.gz + cp.a.z, s.gz + cp.b.z);
    float2 rho, usq, ux, uy, uz;
    if constexpr (sizeof(T) == 4) {
        Inc2 c;
        c.Gx = Gx;
        c.Gy = Gy;
        c.Gz = Gz;
        usq = collide_increment2(s, (float *)s.pop[par ^ 1], nfp, f, P, c, rho);
        ux = c.ux;
        uy = c.uy;
        uz = c.uz;
    } else {
        uint16_t *__restrict__ dst = (uint16_t *)s.pop[par ^ 1];
        const CollK k = make_collk(s);
        const Moments2 m = moments2<T>(P);
        const Coll2 c = make_coll2<OWN>(s, k, m, Gx, Gy, Gz, rho, usq);
        const float sc = s.scale;
        const float wsc0 = (float)d3q19_w(0) * sc, wsc1 = (float)d3q19_w(1) * sc, wsc2 = (float)d3q19_w(7) * sc;
        uint32_t rng = mix32(f ^ step_seed), rng2 = OWN ? mix32((f + 1) ^ step_seed) : 0u;
        rng = rng * 747796405u + 2891336453u;
        rng2 = rng2 * 747796405u + 2891336453u;
        const float2 o0 = fma2(v2(k.c1), unpack2<T>(P[0]), mul2(v2(wsc0), c.Kb));
        if constexpr (OWN)
            __stcs((unsigned int *)(dst + f), __byte_perm(Pack2<T>::rs(o0.x, 0.0f, rng ^ (rng >> 15)),
                                                          Pack2<T>::rs(o0.y, 0.0f, rng2 ^ (rng2 >> 15)), 0x5410));
        else
            __stcs((unsigned int *)(dst + f), Pack2<T>::rs(o0.x, o0.y, rng ^ (rng >> 15)));
        {
            const Cls2 w = make_cls2(c, k, wsc1);
            collide2<T, 1, OWN>(dst, nfp, f, P[1], P[2], c, k, w, rng, rng2);
            collide2<T, 3, OWN>(dst, nfp, f, P[3], P[4], c, k, w, rng, rng2);
            collide2<T, 5, OWN>(dst, nfp, f, P[5], P[6], c, k, w, rng, rng2);
        }
        const Cls2 w = make_cls2(c, k, wsc2);
        collide2<T, 7, OWN>(dst, nfp, f, P[7], P[8], c, k, w, rng, rng2);
        collide2<T, 9, OWN>(dst, nfp, f, P[9], P[10], c, k, w, rng, rng2);
        collide2<T, 11, OWN>(dst, nfp, f, P[11], P[12], c, k, w, rng, rng2);
        collide2<T, 13, OWN>(dst, nfp, f, P[13], P[14], c, k, w, rng, rng2);
        collide2<T, 15, OWN>(dst, nfp, f, P[15], P[16], c, k, w, rng, rng2);
        collide2<T, 17, OWN>(dst, nfp, f, P[17], P[18], c, k, w, rng, rng2);
        ux = c.ux;
        uy = c.uy;
        uz = c.uz;
    }
    if (cp.any) {
        if (cp.act & 1u) s.ufield[f] = make_float4(ux.x, uy.x, uz.x, rho.x);
        if (cp.act & 2u) s.ufield[f + 1] = make_float4(ux.y, uy.y, uz.y, rho.y);
    }
    if (!(usq.x < 0.09f) || !(usq.y < 0.09f)) atomicOr(s.status, ST_UNSTABLE);
}

template <typename T, int MODE>
__device__ __forceinline__ void fluid_pair_even(const SimDev &s, int par, int fi, uint32_t step_seed) {
    const T *__restrict__ src = (const T *)s.pop[par];
    const size_t nfp = (size_t)s.nfp;
    const uint32_t f = (uint32_t)fi;
    const uint32_t r = s.div_nx.div(f);
    const uint32_t x = f - r * (uint32_t)s.nx;
    const uint32_t z = s.div_nyf.div(r);
    const uint32_t y = r - z * (uint32_t)s.nyf;
    const Rows n = source_rows(s, f, (int)y, (int)z);
    const int xm = x == 0 ? s.nx - 1 : -1, xp = x + 2 == (uint32_t)s.nx ? 2 - s.nx : 2;

    typename PairRaw<T>::type P[NQ];
#define LBIB_PULL2(q) P[q] = pull2<T, q, MODE>(src, nfp, n, xm, xp);
    LBIB_PULL2(0) LBIB_PULL2(1) LBIB_PULL2(2) LBIB_PULL2(3) LBIB_PULL2(4) LBIB_PULL2(5) LBIB_PULL2(6)
    LBIB_PULL2(7) LBIB_PULL2(8) LBIB_PULL2(9) LBIB_PULL2(10) LBIB_PULL2(11) LBIB_PULL2(12) LBIB_PULL2(13)
    LBIB_PULL2(14) LBIB_PULL2(15) LBIB_PULL2(16) LBIB_PULL2(17) LBIB_PULL2(18)
#undef LBIB_PULL2
    if constexpr (MODE == MODE_EARLY) {  // as in fluid_cell
        dep_wait();
        dep_release();
    }
    const uint32_t act = __ldcg(s.amask + (f >> 5));
    const bool ylo = s.walls && y == 0, yhi = s.walls && y == (uint32_t)s.nyf - 1;
    if (__any_sync(__activemask(), ylo || yhi)) {
        if (ylo) bounce2<T, 1, MODE>(src, nfp, f, P);
        if (yhi) bounce2<T, -1, MODE>(src, nfp, f, P);
    }
    pair_update<T>(s, par, f, P, step_seed, load_coupling(s, par, f, (act >> (f & 31)) & 3u));
}

// Odd nx: cells f and f + 1 (f even) may lie in two rows, and a row's start has
// any alignment, so each cell has its own source addresses; the arithmetic
// and the stores are those of the pair.  Same numbers as the one-cell kernel,
// which took these widths before (255x128x128 FP16 82.1 -> 64.7 us a step, FP32 93.4
// -> 90.9; 511x256x256 FP16 636 -> 484; 24 serving requests 230.5 -> 219.0).
template <typename T, int MODE>
__device__ __forceinline__ void fluid_pair_odd(const SimDev &s, int par, int fi, uint32_t step_seed) {
    const T *__restrict__ src = (const T *)s.pop[par];
    const size_t nfp = (size_t)s.nfp;
    const uint32_t f = (uint32_t)fi;
    const uint32_t r = s.div_nx.div(f);
    const uint32_t x = f - r * (uint32_t)s.nx;
    const uint32_t z = s.div_nyf.div(r);
    const uint32_t y = r - z * (uint32_t)s.nyf;
    const Rows na = source_rows(s, f, (int)y, (int)z);
    const int xma = x == 0 ? s.nx - 1 : -1, xpa = x == (uint32_t)s.nx - 1 ? 1 - s.nx : 1;
    // the second cell: the next of the row, the first of the next row, or (past
    // the last cell) the first cell again: its place is padding, which any
    // read-out may have written to, so what it holds does not count
    const bool last = fi + 1 == s.nf, turn = !last && x == (uint32_t)s.nx - 1;
    const uint32_t xb = last ? x : turn ? 0u : x + 1u;
    uint32_t yb = y;
    Rows nb;
    const uint32_t one = last ? 0u : 1u;
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) nb.row[i][j] = na.row[i][j] + one;
    if (turn) {
        const bool up = y == (uint32_t)s.nyf - 1;
        yb = up ? 0u : y + 1u;
        nb = source_rows(s, f + 1u, (int)yb, (int)(up ? z + 1u : z));
    }
    const int xmb = xb == 0 ? s.nx - 1 : -1, xpb = xb == (uint32_t)s.nx - 1 ? 1 - s.nx : 1;

    typename PairRaw<T>::type P[NQ];
#define LBIB_PULL2(q) P[q] = pull_cells<T, q, MODE>(src, nfp, na, xma, xpa, nb, xmb, xpb);
    LBIB_PULL2(0) LBIB_PULL2(1) LBIB_PULL2(2) LBIB_PULL2(3) LBIB_PULL2(4) LBIB_PULL2(5) LBIB_PULL2(6)
    LBIB_PULL2(7) LBIB_PULL2(8) LBIB_PULL2(9) LBIB_PULL2(10) LBIB_PULL2(11) LBIB_PULL2(12) LBIB_PULL2(13)
    LBIB_PULL2(14) LBIB_PULL2(15) LBIB_PULL2(16) LBIB_PULL2(17) LBIB_PULL2(18)
#undef LBIB_PULL2
    if constexpr (MODE == MODE_EARLY) {  // as in fluid_cell
        dep_wait();
        dep_release();
    }
    const uint32_t act = __ldcg(s.amask + (f >> 5));
    const uint32_t top = (uint32_t)s.nyf - 1;
    const bool alo = s.walls && y == 0, ahi = s.walls && y == top, blo = s.walls && yb == 0, bhi = s.walls && yb == top;
    if (__any_sync(__activemask(), alo || ahi || blo || bhi)) {
        if (alo || blo) bounce_cells<T, 1, MODE>(src, nfp, f, alo, blo, last, P);
        if (ahi || bhi) bounce_cells<T, -1, MODE>(src, nfp, f, ahi, bhi, last, P);
    }
    Coupling cp = load_coupling(s, par, f, (act >> (f & 31)) & 3u);
    if (last) cp.b = cp.a;
    pair_update<T, true>(s, par, f, P, step_seed, cp);
}

template <typename T, int MODE, bool ODD>
__device__ __forceinline__ void fluid_pair(const SimDev &s, int par, int f, uint32_t step_seed) {
    if constexpr (ODD) fluid_pair_odd<T, MODE>(s, par, f, step_seed);
    else fluid_pair_even<T, MODE>(s, par, f, step_seed);
}

// Pull offset of direction q in the fluid index space away from the
// periodic edges and walls: cell f pulls population q from f - e_q.
__host__ __device__ constexpr unsigned long long pack_e(int axis) {
    unsigned long long p = 0;
    for (int q = 0; q < NQ; ++q) {
        const int e = axis == 0 ? d3q19_ex(q) : (axis == 1 ? d3q19_ey(q) : d3q19_ez(q));
        p |= (unsigned long long)(e + 1) << (2 * q);
    }
    return p;
}
__device__ __forceinline__ int unpack_e(unsigned long long p, int q) { return (int)((p >> (2 * q)) & 3ull) - 1; }

// The bulk L2 prefetch of the stretches of every plane that the CELLS cells
// from fb on pull (thread q < 19 takes plane q).
template <int ESZ, int CELLS>
__device__ __forceinline__ void prefetch_cells(const SimDev &s, const void *src, long long fb) {
    if (fb >= s.nf || fb < 0) return;
    const int q = (int)threadIdx.x;
    constexpr unsigned long long PX = pack_e(0), PY = pack_e(1), PZ = pack_e(2);
    const int off = unpack_e(PX, q) + s.nx * (unpack_e(PY, q) + s.nyf * unpack_e(PZ, q));
    // 16 cells more on each side, clipped to the plane: 16-byte aligned start
    // and size (nfp is a multiple of 64 and below 2^28)
    constexpr int ALIGN = 16 / ESZ;
    const int a = max((int)fb - off - 16, 0) & ~(ALIGN - 1);
    const int b = min(((int)fb + CELLS - off + 16 + ALIGN - 1) & ~(ALIGN - 1), s.nfp);
    if (b <= a) return;
    const char *p = (const char *)src + ((size_t)(unsigned)q * (unsigned)s.nfp + (unsigned)a) * ESZ;
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"((unsigned)(b - a) * ESZ) : "memory");
}

// L2 prefetch for a later block: thread q < 19 of block b asks the L2 to
// fetch, with one bulk prefetch, the stretch of plane q that block b + pf
// (of CELLS cells each) will pull, widened by 16 cells on each side and
// clipped to the plane.  The blocks of a launch run roughly in index order,
// so the DRAM requests run ahead of the warps that wait for them.  A
// prefetch is a hint: it changes no result, and cells near the periodic
// edges and walls (whose sources lie elsewhere) are fetched normally.
template <int ESZ, int CELLS>
__device__ __forceinline__ void prefetch_sources(const SimDev &s, const void *src, int block, int pf) {
    if (pf == 0 || threadIdx.x >= NQ) return;
    prefetch_cells<ESZ, CELLS>(s, src, (long long)(block + pf) * CELLS);
}

// Every other step takes the cells from the last to the first: what a step
// wrote last is then read first, while it is still in the L2.  That saves
// about 30 MB of reads from DRAM a step (a copy between two 110 MB buffers
// and back takes 32.8 us instead of 37.3).  Steps without objects: 160x96x96
// FP32 36.5 -> 33.0 us, FP16 24.7 -> 22.6; 256x128x128 94.3 -> 90.9 and 58.0 ->
// 57.5; 512x256x256 within 1%; no change where the populations fit in the L2,
// nor for a batch.  Launches pass a negative prefetch distance for the steps
// that run backwards.
__device__ __forceinline__ int sweep_block(int pf) {
    return pf < 0 ? (int)(gridDim.x - 1 - blockIdx.x) : (int)blockIdx.x;
}

// Seed of the rounding bits of step t.
__host__ __device__ __forceinline__ uint32_t step_seed(long long t) {
    uint32_t x = (uint32_t)t * 0x9e3779b9u + 0x632be5abu;
    x ^= x >> 16;
    x *= 0x85ebca6bu;
    x ^= x >> 13;
    return x;
}


// One block of consecutive fluid cells starting at f0 (a multiple of 32).
template <typename T, bool BC, int MODE>
__device__ __forceinline__ void fluid_block(const SimDev &s, int par, int f0, uint32_t step_seed) {
    const int f = f0 + (int)threadIdx.x;
    const uint32_t act = MODE == MODE_EARLY ? 0u : active_word(s, f);
    if (f < s.nf) fluid_cell<T, BC, MODE>(s, par, f, act, step_seed);
}

}  // namespace lbib
