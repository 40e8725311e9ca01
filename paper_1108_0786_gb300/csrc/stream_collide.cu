// stream_collide.cu -- the fused D3Q19 stream + bounce-back + refill + LBGK
// update of one coupled step (Eq. 1-4 of the paper, and the moving-wall rule
// and the reconstruction of uncovered cells of Sec. 2.3).  It moves >99% of
// the bytes of a step and is bound by HBM bandwidth: per cell it reads 19
// populations and a flag byte and writes 19 populations
// (2 * 19 * sizeof(T) + 1 bytes).
//
// Two kernels write the populations of step n (pull scheme, two grids: src =
// step n-1, dst = step n):
//
//  bulk      every cell the remap did not list: f_b(x) = f~_b(x - e_b) for
//            all 19 b (f~_{-b}(x) where x - e_b lies beyond a no-slip wall,
//            Eq. 4), LBGK relaxation to the second-order equilibrium with
//            Guo's forcing, store; solid cells store deviation 0.
//  boundary  only the listed fluid cells (F_NEAR, F_SOLID_PREV or F_LINK: they
//            lie in the cubes around the bodies; the bulk kernel leaves them
//            alone, so the two kernels may run concurrently):
//              - x was solid at n-1 (uncovered): f_b = f_eq(rho_avg, u_w(x)),
//                rho_avg the mean density of the D3Q19 neighbours that are
//                fluid in both epochs (1 if none), u_w at the state of step n;
//              - otherwise per b: if the source y = x - e_b lies beyond a
//                no-slip wall, f_b = f~_{-b}(x) (Eq. 4); if y was solid at
//                n-1, f_b = f~_{-b}(x) + 6 w_b rho(x) e_b . u_w(y) with rho(x)
//                the density of x at n-1 and u_w at the state of step n-1;
//            then the same LBGK collision (sums in another order).
//
// Populations are stored as deviations delta = f - w from the rest
// equilibrium (16-bit formats: FP16 scaled by 2^10, BF16 unscaled), so the
// small velocity signal survives FP32 and 16-bit storage; the collision runs
// in FP64 for FP64 storage and in FP32 otherwise.
//
// Memory access of the bulk kernel: a thread handles V consecutive cells of a
// row, the V-cell groups of a z-plane dealt to the threads in row order; each
// population is fetched as one aligned V-wide vector, and the +-1 x shift of the
// pull is completed with a warp shuffle from the neighbouring lane (a scalar load
// at row and warp ends).  Every population byte is read once and written once.
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <algorithm>
#include <cstring>
#include <type_traits>

#include "lbm_internal.cuh"

namespace lbm {
namespace {

template <int BYTES> struct Raw;
template <> struct Raw<1> { using type = unsigned char; };
template <> struct Raw<2> { using type = unsigned short; };
template <> struct Raw<4> { using type = unsigned int; };
template <> struct Raw<8> { using type = uint2; };
template <> struct Raw<16> { using type = uint4; };

// storage codecs: deviation value <-> compute type
template <typename T> struct Codec;
template <> struct Codec<double> {
    using C = double;
    __device__ static C ld(double v, float) { return v; }
    __device__ static double st(C v, float) { return v; }
};
template <> struct Codec<float> {
    using C = float;
    __device__ static C ld(float v, float) { return v; }
    __device__ static float st(C v, float) { return v; }
};
template <> struct Codec<__half> {
    using C = float;
    __device__ static C ld(__half v, float inv_scale) { return __half2float(v) * inv_scale; }
    __device__ static __half st(C v, float scale) { return __float2half_rn(v * scale); }
};
template <> struct Codec<__nv_bfloat16> {
    using C = float;
    __device__ static C ld(__nv_bfloat16 v, float) { return __bfloat162float(v); }
    __device__ static __nv_bfloat16 st(C v, float) { return __float2bfloat16_rn(v); }
};

template <typename T, int V>
__device__ __forceinline__ void load_vec(const T *p, T (&out)[V]) {
    using R = typename Raw<sizeof(T) * V>::type;
    R r = __ldg(reinterpret_cast<const R *>(p));
    memcpy(&out, &r, sizeof(R));
}

template <typename T, int V>
__device__ __forceinline__ void store_vec(T *p, const T (&in)[V]) {
    using R = typename Raw<sizeof(T) * V>::type;
    R r;
    memcpy(&r, &in, sizeof(R));
    *reinterpret_cast<R *>(p) = r;
}

template <typename T>
__device__ __forceinline__ T shfl(T v, int delta, bool up) {
    if constexpr (sizeof(T) == 8) {
        unsigned long long b;
        memcpy(&b, &v, 8);
        b = up ? __shfl_up_sync(0xffffffffu, b, delta) : __shfl_down_sync(0xffffffffu, b, delta);
        memcpy(&v, &b, 8);
    } else {
        unsigned int b = 0;
        memcpy(&b, &v, sizeof(T));
        b = up ? __shfl_up_sync(0xffffffffu, b, delta) : __shfl_down_sync(0xffffffffu, b, delta);
        memcpy(&v, &b, sizeof(T));
    }
    return v;
}

// explicit fused multiply-adds: this file is compiled without implicit
// contraction (-fmad=false), so the bulk kernel's launch shapes, its batched form
// and the near kernel round a cell's arithmetic identically, and so do the two
// boundary kernels (whose sums run in another order than the bulk kernel's: which
// cells are listed depends on the bodies alone); the FMAs the collision wants are
// spelled out
__device__ __forceinline__ float mad(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double mad(double a, double b, double c) { return __fma_rn(a, b, c); }

// e_b . (x, y, z) over the non-zero components of e_b only, in x, y, z
// order (a zero component would still cost a multiply and an add: 0 * z is
// not 0 for every z)
template <typename R>
__device__ __forceinline__ R edot(int b, R x, R y, R z) {
    R r = 0;
    bool any = false;
    if (ex(b)) { r = ex(b) > 0 ? x : -x; any = true; }
    if (ey(b)) { const R t = ey(b) > 0 ? y : -y; r = any ? r + t : t; any = true; }
    if (ez(b)) { const R t = ez(b) > 0 ? z : -z; r = any ? r + t : t; }
    return r;
}

// LBGK collision of one cell in place (deviation form):
//   drho = sum delta, rho = 1 + drho, u = (sum e delta + g/2) / rho,
//   delta_eq_b = w_b (drho + rho (3 e.u + 4.5 (e.u)^2 - 1.5 u.u)),
//   delta~_b = delta_b + (delta_eq_b - delta_b) / tau
//              + (1 - 1/(2 tau)) w_b (3 (e_b - u) . g + 9 (e_b . u)(e_b . g)).
// In exact arithmetic the increments delta~_b - delta_b carry zero mass and
// momentum exactly g.  With FP32 storage the rounded velocity that enters the
// equilibrium would make each collision a small momentum source in every
// cell, constant in a steady flow, and the slow viscous mode of a channel
// integrates it into a ~1e-5 velocity error.  The FP32 update therefore sums
// mass and momentum of the increments (small numbers, so the sums are
// accurate) and moves the defect to the +-x, +-y, +-z pairs and the rest
// population: only the value-dependent rounding of the final additions
// remains.  FP64 keeps the plain update (collide_f64), as do the 16-bit formats, whose
// storage rounding (2^-9 .. 2^-11 relative) dwarfs this effect.
// collide_f32 is that FP32 update.  It evaluates opposite directions (b, b + 1)
// together: they share w, (e.u)^2 and e.g up to sign, so
// deq = w (base + 4.5 rho (e.u)^2 +- 3 rho e.u) saves a fifth of the
// arithmetic.
__device__ __forceinline__ void collide_f32(float (&f)[Q], const Device &dv) {
    float s = 0, jx = 0, jy = 0, jz = 0;
#pragma unroll
    for (int b = 0; b < Q; ++b) {
        s += f[b];
        if (ex(b)) jx += ex(b) > 0 ? f[b] : -f[b];
        if (ey(b)) jy += ey(b) > 0 ? f[b] : -f[b];
        if (ez(b)) jz += ez(b) > 0 ? f[b] : -f[b];
    }
    const float rho = 1.0f + s;
    const float inv = 1.0f / rho;
    // the parameters rounded once on the host (no FP64 conversion per cell)
    const float gx = dv.g_f[0], gy = dv.g_f[1], gz = dv.g_f[2];
    const float ux = mad(0.5f, gx, jx) * inv, uy = mad(0.5f, gy, jy) * inv, uz = mad(0.5f, gz, jz) * inv;
    const float usq = mad(ux, ux, mad(uy, uy, uz * uz));
    const float om = dv.omega_f, guo = dv.guo_f;
    const float ug = mad(ux, gx, mad(uy, gy, uz * gz));
    const float base = mad(-1.5f * rho, usq, s);       // deviation of f_eq without the e.u terms, over w
    float m = 0, px = 0, py = 0, pz = 0;
    // one relaxation: the increment of direction b towards deq (+ Guo's term
    // gt), summed for the conservation closure
    auto relax = [&](int b, float deq, float gt) {
        const float d = dv.forced ? mad(om, deq - f[b], gt) : om * (deq - f[b]);
        m += d;
        if (ex(b)) px += ex(b) > 0 ? d : -d;
        if (ey(b)) py += ey(b) > 0 ? d : -d;
        if (ez(b)) pz += ez(b) > 0 ? d : -d;
        f[b] += d;
    };
    {
        const float w = (float)wgt(0);
        relax(0, w * base, dv.forced ? guo * w * (-3.0f * ug) : 0.0f);
    }
#pragma unroll
    for (int b = 1; b < Q; b += 2) {
        const float w = (float)wgt(b);
        const float eu = edot(b, ux, uy, uz);
        const float a = mad(4.5f * rho * eu, eu, base);
        const float c = 3.0f * rho * eu;
        float g1 = 0, g2 = 0;
        if (dv.forced) {
            const float eg = edot(b, gx, gy, gz);
            const float sym = mad(9.0f * eu, eg, -3.0f * ug), asym = 3.0f * eg;
            g1 = guo * w * (sym + asym);
            g2 = guo * w * (sym - asym);
        }
        relax(b, w * (a + c), g1);
        relax(b + 1, w * (a - c), g2);
    }
    const float hx = 0.5f * (gx - px), hy = 0.5f * (gy - py), hz = 0.5f * (gz - pz);
    f[1] += hx; f[2] -= hx;
    f[3] += hy; f[4] -= hy;
    f[5] += hz; f[6] -= hz;
    f[0] -= m;
}

// LBGK (+ Guo) of one cell for FP64 storage, the same update written for the
// fewest FP64 instructions: an FP64 warp instruction occupies its
// sub-partition for 64 cycles here, so the FP64 bulk kernel is bound by their
// number and not by HBM.  Opposite directions share the moments' sums and
// differences and the even part of the equilibrium, the weights and omega are
// folded into per-cell factors of the two weight classes, and a population
// takes two FMAs:
//   f~ = ((1 - omega) f + a) +- C e.u,  a = omega w (drho - 1.5 rho u.u + 4.5 rho (e.u)^2),
//   C = 3 omega w rho  (+ (1 - omega/2) w (9 (e.u)(e.g) - 3 u.g +- 3 e.g) with forcing).
// 130 FP64 instructions a cell (112 at tau = 1) against 240 with each direction on
// its own: a launch on 203 x 149 x 131 cells takes 977 us (842 at tau = 1, 1337
// with a body force).  Against 64-bit-mantissa arithmetic a collision's error is
// 0.7 to 0.9 times that of the plain form for tau in 0.51 .. 2.
__device__ __forceinline__ void collide_f64(double (&f)[Q], const Device &dv) {
    double d[Q / 2];
    double s = f[0];
#pragma unroll
    for (int p = 0; p < Q / 2; ++p) {
        d[p] = f[2 * p + 1] - f[2 * p + 2];
        s += f[2 * p + 1] + f[2 * p + 2];
    }
    double jx = d[0] + ((d[3] + d[4]) + (d[5] + d[6]));
    double jy = d[1] + ((d[3] - d[4]) + (d[7] + d[8]));
    double jz = d[2] + ((d[5] - d[6]) + (d[7] - d[8]));
    const bool forced = dv.forced;
    const double gx = dv.g[0], gy = dv.g[1], gz = dv.g[2];
    if (forced) {
        jx = mad(0.5, gx, jx);
        jy = mad(0.5, gy, jy);
        jz = mad(0.5, gz, jz);
    }
    const double rho = 1.0 + s;
    const double inv = 1.0 / rho;
    const double ux = jx * inv, uy = jy * inv, uz = jz * inv;
    const double sq[3] = {ux * ux, uy * uy, uz * uz};
    const double base = mad(-1.5 * rho, (sq[0] + sq[1]) + sq[2], s);
    const double om1 = dv.om1;
    const double ug3 = forced ? -3.0 * mad(ux, gx, mad(uy, gy, uz * gz)) : 0.0;
    f[0] = mad(om1, f[0], dv.ow[0] * base);
    if (forced) f[0] = mad(dv.gw[0], ug3, f[0]);
    double b1 = dv.ow[1] * base, b2 = dv.ow[2] * base;
    if (forced) {
        b1 = mad(dv.gw[1], ug3, b1);
        b2 = mad(dv.gw[2], ug3, b2);
    }
    const double r3[2] = {3.0 * dv.ow[1] * rho, 3.0 * dv.ow[2] * rho};
    const double r45[2] = {1.5 * r3[0], 1.5 * r3[1]};
    if (om1 == 0.0 && !forced) {
        // tau = 1: the update is the equilibrium itself, the same bits without 18
        // of the FMAs (0 f + a = a; a non-finite f makes every moment so)
#pragma unroll
        for (int p = 0; p < Q / 2; ++p) {
            const int b = 2 * p + 1, wc = p < 3 ? 0 : 1;
            const double eu = edot(b, ux, uy, uz);
            const double a = mad(r45[wc], p < 3 ? sq[p] : eu * eu, wc ? b2 : b1);
            f[b] = mad(r3[wc], eu, a);
            f[b + 1] = mad(-r3[wc], eu, a);
        }
        return;
    }
#pragma unroll
    for (int p = 0; p < Q / 2; ++p) {
        const int b = 2 * p + 1, wc = p < 3 ? 0 : 1;
        const double eu = edot(b, ux, uy, uz);
        double a = mad(r45[wc], p < 3 ? sq[p] : eu * eu, wc ? b2 : b1);
        if (forced) {
            const double eg = edot(b, gx, gy, gz), gw = dv.gw[1 + wc];
            a = mad(9.0 * gw * eu, eg, a);
            const double c = mad(r3[wc], eu, 3.0 * gw * eg);
            f[b] = mad(om1, f[b], a) + c;
            f[b + 1] = mad(om1, f[b + 1], a) - c;
        } else {
            f[b] = mad(r3[wc], eu, mad(om1, f[b], a));
            f[b + 1] = mad(-r3[wc], eu, mad(om1, f[b + 1], a));
        }
    }
}

// Two FP32 values in one 64-bit register pair and the packed FP32 operations of
// sm_100 and later on them (PTX add / mul / fma .f32x2, each half rounded to
// nearest like the scalar operation): one issue slot for two cells' arithmetic.
struct F2 {
    unsigned long long v;
};
__device__ __forceinline__ F2 pack2(float lo, float hi) {
    F2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ float lo2(F2 a) { return __uint_as_float((unsigned)a.v); }
__device__ __forceinline__ float hi2(F2 a) { return __uint_as_float((unsigned)(a.v >> 32)); }

// the operations the lean collision is written in, for one cell or two
__device__ __forceinline__ float vadd(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float vsub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float vmul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float vfma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
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
template <typename R> __device__ __forceinline__ R splat(float x);
template <> __device__ __forceinline__ float splat<float>(float x) { return x; }
template <> __device__ __forceinline__ F2 splat<F2>(float x) { return pack2(x, x); }
// a times, or times and plus, a launch constant: two scalar operations on its
// place in the constant bank, which a packed one would first copy to registers
__device__ __forceinline__ float vscale(float a, float c) { return __fmul_rn(a, c); }
__device__ __forceinline__ F2 vscale(F2 a, float c) { return pack2(__fmul_rn(lo2(a), c), __fmul_rn(hi2(a), c)); }
__device__ __forceinline__ float vscale_add(float a, float c, float b) { return __fmaf_rn(a, c, b); }
__device__ __forceinline__ F2 vscale_add(F2 a, float c, F2 b) {
    return pack2(__fmaf_rn(lo2(a), c, lo2(b)), __fmaf_rn(hi2(a), c, hi2(b)));
}
__device__ __forceinline__ float vmul_apart(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ F2 vmul_apart(F2 a, F2 b) {
    return pack2(__fmul_rn(lo2(a), lo2(b)), __fmul_rn(hi2(a), hi2(b)));
}
__device__ __forceinline__ float vplus(float a, float c) { return __fadd_rn(a, c); }
__device__ __forceinline__ F2 vplus(F2 a, float c) { return pack2(__fadd_rn(lo2(a), c), __fadd_rn(hi2(a), c)); }
__device__ __forceinline__ float vrcp(float a) { return __frcp_rn(a); }
__device__ __forceinline__ F2 vrcp(F2 a) { return pack2(__frcp_rn(lo2(a)), __frcp_rn(hi2(a))); }

// e_b . (x, y, z) for odd b, whose first non-zero component is +1
template <typename R>
__device__ __forceinline__ R vdot(int b, R x, R y, R z) {
    const R first = ex(b) ? x : (ey(b) ? y : z);
    if (b < 7) return first;
    const R second = ez(b) ? z : y;
    return (ez(b) ? ez(b) : ey(b)) > 0 ? vadd(first, second) : vsub(first, second);
}

// LBGK (+ Guo) for 16-bit storage in forms with few instructions, for one cell
// (R = float) or two (R = F2) with the same bits.  Opposite directions
// (b, b + 1) are paired: the moments come from pair sums and differences.  The
// weight comes last:
//   f~_b = (1 - omega) f_b + omega w (a +- c),  c = 3 rho e.u,
//   a = drho - 1.5 rho u.u + 4.5 rho (e.u)^2
//   (+ (1 - omega/2) w (9 (e.u)(e.g) - 3 u.g +- 3 e.g) with forcing).
// With the weight folded into per-cell factors (3 omega w rho, ...) the factors'
// roundings are the same in every step and cell of a slow flow (rho has few
// values near 1), a momentum source of up to 6e-8 a step: the channel swimmer's
// displacement in BF16 was 1.25 +- 0.03 times as far from the FP64 path (64
// offsets, 4000 steps), though BF16's rounding is stochastic.  FP16 (SCALED: the
// populations are k delta, k = f16_scale, a power of two, on entry and exit)
// rounds to nearest, and in a slow flow, whose populations are a few units in the
// last place, exact results often lie half way between two FP16 values; with c
// and its sum rounded apart FP32 gives the half-way value itself and the rounding
// to even is unbiased (one rounding: 1.1 times the error of the velocity field;
// folded weights: 1.4 to 2 times).
// Use: rest(f_0), pair(f_b, f_b+1) for the nine pairs in order, solve(), then
// relax0 and relax for the populations.
template <typename R, bool SCALED>
struct Lean {
    R s, jx, jy, jz;        // sum of delta, momentum; after solve(): u in jx, jy, jz
    R base;                 // k (drho - 1.5 rho u.u)
    R kr;                   // k rho
    R ug3;                  // -3 k u.g (forcing)
    R A, C;                 // a = A (e.u)^2 + base, c = C e.u, C = 3 k rho

    __device__ __forceinline__ void rest(R f0) { s = f0; }
    __device__ __forceinline__ void pair(int p, R f1, R f2) {
        const int b = 2 * p + 1;
        s = vadd(s, vadd(f1, f2));
        const R d = vsub(f1, f2);
        if (ex(b)) jx = p == 0 ? d : vadd(jx, d);
        if (ey(b)) jy = p == 1 ? d : (ey(b) > 0 ? vadd(jy, d) : vsub(jy, d));
        if (ez(b)) jz = p == 2 ? d : (ez(b) > 0 ? vadd(jz, d) : vsub(jz, d));
    }
    __device__ __forceinline__ void solve(const Device &dv) {
        const float k = SCALED ? dv.f16_scale : 1.0f;
        const bool forced = dv.forced;
        if (forced) {
            const float kh = 0.5f * k;
            jx = vplus(jx, kh * dv.g_f[0]);
            jy = vplus(jy, kh * dv.g_f[1]);
            jz = vplus(jz, kh * dv.g_f[2]);
        }
        const float ik = SCALED ? dv.f16_inv_scale : 1.0f;
        const R rho = vplus(SCALED ? vscale(s, ik) : s, 1.0f);
        R inv = vrcp(rho);
        if (SCALED) inv = vscale(inv, ik);
        jx = vmul(jx, inv);
        jy = vmul(jy, inv);
        jz = vmul(jz, inv);
        const R usq = vfma(jx, jx, vfma(jy, jy, vmul(jz, jz)));
        kr = SCALED ? vscale(rho, k) : rho;
        base = vfma(vscale(kr, -1.5f), usq, s);
        A = vscale(kr, 4.5f);
        C = vscale(kr, 3.0f);
        if (forced)
            ug3 = vscale(vscale_add(jx, dv.g_f[0], vscale_add(jy, dv.g_f[1], vscale(jz, dv.g_f[2]))), -3.0f * k);
    }
    // TAU1: omega = 1, the old populations have the factor 0 and are not read
    template <bool TAU1 = false>
    __device__ __forceinline__ R relax0(R f0, const Device &dv) const {
        R r = vscale(base, dv.ow_f[0]);
        if (dv.forced) r = vscale_add(ug3, dv.gw_f[0], r);
        return TAU1 ? r : vscale_add(f0, dv.om1_f, r);
    }
    template <bool TAU1 = false>
    __device__ __forceinline__ void relax(int p, R &f1, R &f2, const Device &dv) const {
        const int i = 2 * p + 1, wc = p < 3 ? 1 : 2;
        const R eu = vdot(i, jx, jy, jz);
        const R a = vfma(A, vmul(eu, eu), base);
        // scalar products: the assembler fuses a packed product with the sum after it
        const R c = vmul_apart(C, eu);
        R r1, r2;
        if constexpr (SCALED) {
            r1 = vscale(vadd(a, c), dv.ow_f[wc]);
            r2 = vscale(vsub(a, c), dv.ow_f[wc]);
        } else {
            const R ow = splat<R>(dv.ow_f[wc]);
            r1 = vmul(vadd(a, c), ow);
            r2 = vmul(vsub(a, c), ow);
        }
        if (dv.forced) {
            const float k = SCALED ? dv.f16_scale : 1.0f, eg = edot(i, dv.g_f[0], dv.g_f[1], dv.g_f[2]), gw = dv.gw_f[wc];
            const R g = vscale_add(vscale(eu, 9.0f * k), eg, ug3);
            r1 = vscale_add(vplus(g, 3.0f * k * eg), gw, r1);
            r2 = vscale_add(vplus(g, -3.0f * k * eg), gw, r2);
        }
        if constexpr (TAU1) {
            f1 = r1;
            f2 = r2;
        } else if constexpr (SCALED) {
            f1 = vscale_add(f1, dv.om1_f, r1);
            f2 = vscale_add(f2, dv.om1_f, r2);
        } else {
            const R om1 = splat<R>(dv.om1_f);
            f1 = vfma(f1, om1, r1);
            f2 = vfma(f2, om1, r2);
        }
    }
};

template <bool SCALED>
__device__ __forceinline__ void collide_lean(float (&f)[Q], const Device &dv) {
    Lean<float, SCALED> c;
    c.rest(f[0]);
#pragma unroll
    for (int p = 0; p < Q / 2; ++p) c.pair(p, f[2 * p + 1], f[2 * p + 2]);
    c.solve(dv);
    f[0] = c.relax0(f[0], dv);
#pragma unroll
    for (int p = 0; p < Q / 2; ++p) c.relax(p, f[2 * p + 1], f[2 * p + 2], dv);
}

// the collision of storage type T on its values as loaded (raw_ld for 16-bit storage)
template <typename T, typename Cd>
__device__ __forceinline__ void collide(Cd (&f)[Q], const Device &dv) {
    if constexpr (std::is_same<T, double>::value) collide_f64(f, dv);
    else if constexpr (std::is_same<T, float>::value) collide_f32(f, dv);
    else collide_lean<std::is_same<T, __half>::value>(f, dv);
}

// 16-bit storage without a per-population scale: FP16 keeps k delta, so the
// stored value itself is what collide_lean<true> works on
template <typename T> __device__ __forceinline__ float raw_ld(T v);
template <> __device__ __forceinline__ float raw_ld<__half>(__half v) { return __half2float(v); }
template <> __device__ __forceinline__ float raw_ld<__nv_bfloat16>(__nv_bfloat16 v) { return __bfloat162float(v); }


// ---- stochastic rounding of BF16 storage ------------------------------------
// BF16 keeps 8 significant bits.  Rounded to nearest, a population whose
// update is below half an ulp is rounded back to the same value every step:
// slow terms are lost and the flow settles at a biased state (Guo's term in
// the channel workload adds ~2e-8 a step to populations whose ulp is ~2e-7).
// BF16 stores therefore round up with a probability equal to the fraction of
// the ulp that is dropped: the rounding error has zero mean, and the slow
// terms accumulate as they do in FP32.  The random bits come from a
// counter-based hash of (cell, step), so a cell's rounding depends neither
// on the launch shape nor on which kernel stores the cell: 8 bits for each
// population, bytes of five 32-bit words per cell.
struct Dither {
    unsigned h[5];
};

// MurmurHash3's 32-bit finalizer (Appleby): a bijective integer mixer
__device__ __forceinline__ unsigned fmix32(unsigned x) {
    x ^= x >> 16;
    x *= 0x85ebca6bu;
    x ^= x >> 13;
    x *= 0xc2b2ae35u;
    x ^= x >> 16;
    return x;
}

// the five words of a cell and step: the finalizer of a key of (cell, step),
// then four steps of a 32-bit linear congruential generator (the
// multiplier and increment of Numerical Recipes' quick generator), each
// output xor-shifted so that its low bytes carry the state's high bits
__device__ __forceinline__ Dither bf16_dither(long long c, long long t) {
    const unsigned key = (unsigned)c * 0x9E3779B1u ^ ((unsigned)t * 0x85EBCA77u + (unsigned)(t >> 32));
    Dither d;
    unsigned x = fmix32(key);
    d.h[0] = x;
#pragma unroll
    for (int k = 1; k < 5; ++k) {
        x = x * 1664525u + 1013904223u;
        d.h[k] = x ^ (x >> 15);
    }
    return d;
}

// word k of bf16_dither alone
__device__ __forceinline__ unsigned bf16_dither_word(long long c, long long t, int k) {
    unsigned x = fmix32((unsigned)c * 0x9E3779B1u ^ ((unsigned)t * 0x85EBCA77u + (unsigned)(t >> 32)));
    if (k == 0) return x;
    for (int i = 0; i < k; ++i) x = x * 1664525u + 1013904223u;
    return x ^ (x >> 15);
}

// v rounded stochastically to BF16 with byte a % 4 of word a / 4 of d, its
// bits in the upper half of the result: adding 8 random bits and half a
// step of them below the kept bits, then truncating, rounds the magnitude
// up with the probability of the dropped fraction (to 2^-9 of an ulp)
__device__ __forceinline__ unsigned bf16_sr_add(float v, unsigned word, int a) {
    const unsigned r = __byte_perm(word, 0x80u, 0x5504u | ((unsigned)(a & 3) << 4));          // byte << 8 | 0x80
    return __float_as_uint(v) + r;
}
__device__ __forceinline__ unsigned bf16_sr_word(float v, const Dither &d, int a) { return bf16_sr_add(v, d.h[a >> 2], a); }

// the same BF16 bits in the low half
__device__ __forceinline__ unsigned bf16_sr_bits(float v, const Dither &d, int a) {
    return bf16_sr_word(v, d, a) >> 16;
}

// a 16-bit population as stored: FP16 rounded to nearest, BF16 rounded
// stochastically (the dither is used only for BF16)
template <typename T> __device__ __forceinline__ T store16(float v, const Dither &d, int a);
template <> __device__ __forceinline__ __half store16<__half>(float v, const Dither &, int) {
    return __float2half_rn(v);
}
template <> __device__ __forceinline__ __nv_bfloat16 store16<__nv_bfloat16>(float v, const Dither &d, int a) {
    return __ushort_as_bfloat16((unsigned short)bf16_sr_bits(v, d, a));
}

// the dither of cell c in the step whose index *t holds (read only for BF16)
template <typename T> __device__ __forceinline__ Dither dither_for(long long c, const long long *t) {
    if constexpr (std::is_same<T, __nv_bfloat16>::value) return bf16_dither(c, *t);
    else return Dither{};
}

// The thread's V-cell group of a z-plane: the groups in row order, BULK_THREADS
// a block, so that no lane idles at the end of a row whatever nx is.  A warp's
// lanes may cross a row end, where the loads of a row's first and last cell
// take over from the shuffles.  (Blocks of 32 or 128 groups of one row left 21 %
// of the FP64 kernel's lanes idle at nx = 203, which cost 26 % of its time, and
// 22 % of the FP32 kernel's at nx = 100.)
constexpr int BULK_THREADS = 256;

__device__ __forceinline__ void plane_group(const Blk &bk, int nxq, int ny, unsigned recip, int &xq, int &y,
                                            bool &active) {
    const unsigned per_plane = (unsigned)nxq * ny;
    unsigned q = bk.x * BULK_THREADS + threadIdx.x;
    active = q < per_plane;
    q = min(q, per_plane - 1);          // inactive lanes still join the shuffles
    // q / nxq by row_recip: the truncated reciprocal loses less than q / 2^32
    // < 1, which the comparison restores
    unsigned r = __umulhi(q, recip), x = q - r * nxq;
    if (x >= (unsigned)nxq) {
        x -= nxq;
        ++r;
    }
    xq = (int)x;
    y = (int)r;
}

// No-slip walls (Eq. 4) in the bulk kernels (WALLS instances, for lattices with
// a non-periodic axis): where the source of direction b lies beyond a wall, the
// cell takes its own reversed population of step n-1, so a row on a y or z wall
// reads the reversed direction's plane at its own place, unshifted, and the
// first and last cell of a row do so on x walls.  A kernel of their own over the
// wall faces, a thread a cell, took 15 us on a 128 x 64 x 64 channel and 36 us on
// 100 x 100 x 200 cells (x walls: one 4-byte value a sector), in series with the
// boundary kernel.
struct WallRows {
    bool y0, y1, z0, z1, x;         // this row lies on that wall; the x axis has walls
    __device__ __forceinline__ bool beyond(int b) const {
        return (ey(b) > 0 && y0) || (ey(b) < 0 && y1) || (ez(b) > 0 && z0) || (ez(b) < 0 && z1);
    }
};

__device__ __forceinline__ WallRows wall_rows(const Domain &d, int y, int z) {
    return WallRows{!d.py && y == 0, !d.py && y == d.ny - 1, !d.pz && z == 0, !d.pz && z == d.nz - 1, !d.px};
}

// cells the bulk kernels write: all but the fluid cells the remap listed for
// the boundary kernel
__device__ __forceinline__ bool bulk_cell(uint8_t f) { return (f & F_SOLID) || !(f & F_LISTED); }

template <typename T, int V, bool WALLS, bool TILE = false, bool AHEAD = false>
__device__ __forceinline__ void bulk_body(const Device &dv, const StepPtrs &sp, const Blk &bk) {
    using Cd = typename Codec<T>::C;
    const Domain d = dv.dom;
    const int nxq = d.nx / V;
    int xq, y;
    bool active;
    if constexpr (TILE) {
        // one TILE_X-cell tile of a row a block (the near kernel)
        xq = bk.x * TILE_X + threadIdx.x;
        y = bk.y;
        active = xq < nxq;
        xq = min(xq, nxq - 1);          // inactive lanes still join the shuffles
    } else {
        plane_group(bk, nxq, d.ny, sp.row_recip, xq, y, active);
    }
    const int z = bk.z;
    const int lane = threadIdx.x & 31;
    const int x0 = xq * V;
    const int ym = y == 0 ? d.ny - 1 : y - 1, yp = y == d.ny - 1 ? 0 : y + 1;
    const int zm = z == 0 ? d.nz - 1 : z - 1, zp = z == d.nz - 1 ? 0 : z + 1;
    const long long C = d.C;
    const long long c0 = ((long long)z * d.ny + y) * d.nx + x0;
    const T *__restrict__ src = static_cast<const T *>(sp.src);
    T *__restrict__ dst = static_cast<T *>(sp.dst);
    const float inv_scale = dv.f16_inv_scale, scale = dv.f16_scale;

    uint8_t fl[V];
    load_vec<uint8_t, V>(sp.flags_cur + c0, fl);
    // 16-bit storage: stored values as they are (collide_lean takes FP16's scale)
    constexpr bool raw16 = sizeof(T) == 2;
    auto ld = [&](T v) -> Cd {
        if constexpr (raw16) return raw_ld<T>(v);
        else return Codec<T>::ld(v, inv_scale);
    };

    const WallRows wr = wall_rows(d, y, z);
    // offsets of the rows within a direction's plane (C < 2^31): the planes'
    // addresses are the same for all threads
    const unsigned nxu = (unsigned)d.nx;
    const unsigned rows[3][3] = {{(zm * d.ny + ym) * nxu, (zm * d.ny + y) * nxu, (zm * d.ny + yp) * nxu},
                                 {(z * d.ny + ym) * nxu, (z * d.ny + y) * nxu, (z * d.ny + yp) * nxu},
                                 {(zp * d.ny + ym) * nxu, (zp * d.ny + y) * nxu, (zp * d.ny + yp) * nxu}};
    // AHEAD: all loads before the first shuffle, the row ends' single cells
    // included: with each row end's load behind its direction's shuffle the loads
    // of several directions wait for one another (FP32, 512 x 256 x 256 cells: 762 us in
    // the then best shape, 746 us ahead; 100 x 100 x 200 with walls 69.9 and
    // 58.7 us).  Not where the registers are short or the loads do not bound:
    // the batched kernels (48 boxes of edge 48 to 96, a step: 636 us, 655 us ahead) and
    // FP64 (a pass of the ragged swarm 7153 against 7294 us).
    const bool e0 = lane == 0 || x0 == 0, e1 = lane == 31 || x0 + V == d.nx;
    auto row_of = [&](int b) -> const T * {
        if (WALLS && wr.beyond(b)) return src + (long long)opp(b) * C + rows[1][1];
        return src + (long long)b * C + rows[1 - ez(b)][1 - ey(b)];
    };
    auto left_end = [&](int b) -> T {            // pull from x - 1
        if (WALLS && wr.x && x0 == 0) return src[(long long)opp(b) * C + c0];
        return row_of(b)[x0 == 0 ? d.nx - 1 : x0 - 1];
    };
    auto right_end = [&](int b) -> T {           // pull from x + 1
        if (WALLS && wr.x && x0 + V == d.nx) return src[(long long)opp(b) * C + c0 + V - 1];
        return row_of(b)[x0 + V == d.nx ? 0 : x0 + V];
    };
    T raw[Q][V], end[Q];
    if constexpr (AHEAD) {
#pragma unroll
        for (int b = 0; b < Q; ++b) {
            load_vec<T, V>(row_of(b) + (unsigned)x0, raw[b]);
            if (ex(b) > 0 && e0) end[b] = left_end(b);
            if (ex(b) < 0 && e1) end[b] = right_end(b);
        }
    }
    Cd f[Q][V];
#pragma unroll
    for (int b = 0; b < Q; ++b) {
        const bool own = WALLS && wr.beyond(b);
        T (&A)[V] = raw[b];
        if constexpr (!AHEAD) load_vec<T, V>(row_of(b) + (unsigned)x0, A);
        if (ex(b) == 0) {
#pragma unroll
            for (int i = 0; i < V; ++i) f[b][i] = ld(A[i]);
        } else if (ex(b) > 0) {
            T left = shfl(A[V - 1], 1, true);
            if (e0) left = AHEAD ? end[b] : left_end(b);
            f[b][0] = ld(own ? A[0] : left);
#pragma unroll
            for (int i = 1; i < V; ++i) f[b][i] = ld(own ? A[i] : A[i - 1]);
        } else {
            T right = shfl(A[0], 1, false);
            if (e1) right = AHEAD ? end[b] : right_end(b);
#pragma unroll
            for (int i = 0; i < V - 1; ++i) f[b][i] = ld(own ? A[i] : A[i + 1]);
            f[b][V - 1] = ld(own ? A[V - 1] : right);
        }
    }

#pragma unroll
    for (int i = 0; i < V; ++i) {
        Cd g[Q];
#pragma unroll
        for (int b = 0; b < Q; ++b) g[b] = f[b][i];
        collide<T>(g, dv);
        const bool solid = fl[i] & F_SOLID;
        if constexpr (WALLS) {
#pragma unroll
            for (int b = 0; b < Q; ++b) f[b][i] = solid ? (Cd)0 : g[b];
        } else {
            // few warps have a solid cell: a branch instead of 19 selects a cell
            // (FP32, 512 x 256 x 256 cells: 794 -> 760 us, 24 bytes of spills for
            // 40; the WALLS instance, with more registers held, is 2 % slower so)
#pragma unroll
            for (int b = 0; b < Q; ++b) f[b][i] = g[b];
            if (solid) {
#pragma unroll
                for (int b = 0; b < Q; ++b) f[b][i] = (Cd)0;
            }
        }
    }
    // overlapped steps: a tile near a body is the near kernel's
    const bool far = !sp.far_skip || sp.far_skip[((long long)z * d.ny + y) * ((d.nx + TILE_X - 1) / TILE_X) +
                                                 x0 / TILE_X] == 0u;
    if (!active || !far) return;
    // BF16 rounds stochastically (one cell per thread for 16-bit storage here)
    static_assert(!raw16 || V == 1, "16-bit storage with several cells per thread uses bulk16_kernel");
    static_assert(TILE_X % V == 0, "a thread's cells lie in one tile");
    const Dither dz = raw16 ? dither_for<T>(c0, sp.tstep) : Dither{};
    auto st = [&](Cd v, int b) -> T {
        if constexpr (raw16) return store16<T>(v, dz, b);
        else return Codec<T>::st(v, scale);
    };
    // listed fluid cells belong to the boundary kernel, which may run
    // concurrently: leave them alone
    bool all_mine = true;
#pragma unroll
    for (int i = 0; i < V; ++i) all_mine = all_mine && bulk_cell(fl[i]);
    if (all_mine) {
#pragma unroll
        for (int b = 0; b < Q; ++b) {
            T out[V];
#pragma unroll
            for (int i = 0; i < V; ++i) out[i] = st(f[b][i], b);
            store_vec<T, V>(dst + (long long)b * C + (unsigned)c0, out);
        }
        return;
    }
#pragma unroll
    for (int b = 0; b < Q; ++b)
#pragma unroll
        for (int i = 0; i < V; ++i)
            if (bulk_cell(fl[i])) dst[(long long)b * C + c0 + i] = st(f[b][i], b);
}

// MINB == 1 leaves the register budget to the compiler (an explicit minimum
// of one block lets it spend far more registers than it needs)
template <typename T, int V, int MINB, bool WALLS>
__global__ void __launch_bounds__(BULK_THREADS, MINB == 1 ? 0 : MINB)
bulk_kernel(const Device dv, const StepPtrs sp) {
    pdl_enter();
    bulk_body<T, V, WALLS, false, sizeof(T) != 8>(dv, sp, launch_blk());
}

// a batched bulk block takes BATCH_PZ consecutive z-planes of its member:
// the member lookup at its start (a few dependent loads and barriers with
// no population traffic in flight) is paid once for all of them
constexpr int BATCH_PZ = 4;

template <typename T, int V, int MINB, bool WALLS>
__global__ void __launch_bounds__(BULK_THREADS, MINB == 1 ? 0 : MINB) bulk_batch(const Batch bt) {
    LBM_BATCH_MEMBER(bt);
    const int z0 = sbk.z * BATCH_PZ, z1 = min(z0 + BATCH_PZ, sdv.dom.nz);
    for (int z = z0; z < z1; ++z) {
        Blk pb = sbk;
        pb.z = z;
        bulk_body<T, V, WALLS>(sdv, ssp, pb);
    }
}

// the two cells of a 32-bit word of 16-bit populations (the lower address in
// the low half), widened to FP32
template <typename T> __device__ __forceinline__ F2 widen(unsigned w);
template <> __device__ __forceinline__ F2 widen<__half>(unsigned w) {
    const __half2 h = *reinterpret_cast<const __half2 *>(&w);
    const float2 f = __half22float2(h);
    return pack2(f.x, f.y);
}
template <> __device__ __forceinline__ F2 widen<__nv_bfloat16>(unsigned w) {
    return pack2(__uint_as_float(w << 16), __uint_as_float(w & 0xffff0000u));
}

// population a of two cells as a stored word: FP16 to nearest, BF16
// stochastically (the rounded bits are the upper halves of the sums)
template <typename T> __device__ __forceinline__ unsigned narrow(F2 v, const Dither &d0, const Dither &d1, int a);
template <> __device__ __forceinline__ unsigned narrow<__half>(F2 v, const Dither &, const Dither &, int) {
    const __half2 h = __floats2half2_rn(lo2(v), hi2(v));
    return *reinterpret_cast<const unsigned *>(&h);
}
template <> __device__ __forceinline__ unsigned narrow<__nv_bfloat16>(F2 v, const Dither &d0, const Dither &d1, int a) {
    return __byte_perm(bf16_sr_word(lo2(v), d0, a), bf16_sr_word(hi2(v), d1, a), 0x7632);
}

// collide the V cells in the words w of a thread (pairs 2j, 2j + 1 in word j)
template <typename T, int V>
__device__ __forceinline__ void collide_words(unsigned (&w)[Q][V / 2], const uint8_t (&fl)[V], long long c0,
                                              const Device &dv, const StepPtrs &sp) {
#pragma unroll
    for (int j = 0; j < V / 2; ++j) {
        Lean<F2, std::is_same<T, __half>::value> c;
        c.rest(widen<T>(w[0][j]));
#pragma unroll
        for (int p = 0; p < Q / 2; ++p) c.pair(p, widen<T>(w[2 * p + 1][j]), widen<T>(w[2 * p + 2][j]));
        c.solve(dv);
        // the words are opaque from here, so that the compiler widens them anew
        // instead of keeping 38 FP32 values
#pragma unroll
        for (int b = 0; b < Q; ++b) asm volatile("" : "+r"(w[b][j]));
        const Dither d0 = dither_for<T>(c0 + 2 * j, sp.tstep), d1 = dither_for<T>(c0 + 2 * j + 1, sp.tstep);
        // solid cells store 0
        const unsigned keep = (fl[2 * j] & F_SOLID ? 0u : 0xffffu) | (fl[2 * j + 1] & F_SOLID ? 0u : 0xffff0000u);
        if (dv.om1_f == 0.0f) {             // tau = 1: nothing to widen again
            w[0][j] = narrow<T>(c.template relax0<true>(c.base, dv), d0, d1, 0) & keep;
#pragma unroll
            for (int p = 0; p < Q / 2; ++p) {
                F2 f1, f2;
                c.template relax<true>(p, f1, f2, dv);
                w[2 * p + 1][j] = narrow<T>(f1, d0, d1, 2 * p + 1) & keep;
                w[2 * p + 2][j] = narrow<T>(f2, d0, d1, 2 * p + 2) & keep;
            }
            continue;
        }
        w[0][j] = narrow<T>(c.relax0(widen<T>(w[0][j]), dv), d0, d1, 0) & keep;
#pragma unroll
        for (int p = 0; p < Q / 2; ++p) {
            F2 f1 = widen<T>(w[2 * p + 1][j]), f2 = widen<T>(w[2 * p + 2][j]);
            c.relax(p, f1, f2, dv);
            w[2 * p + 1][j] = narrow<T>(f1, d0, d1, 2 * p + 1) & keep;
            w[2 * p + 2][j] = narrow<T>(f2, d0, d1, 2 * p + 2) & keep;
        }
    }
}

// store them, but for the cells of a near tile and listed ones
template <int V>
__device__ __forceinline__ void store_words(const unsigned (&w)[Q][V / 2], const uint8_t (&fl)[V], bool active, int x0,
                                            int y, int z, long long c0, const Device &dv, const StepPtrs &sp) {
    using RawV = typename Raw<2 * V>::type;
    const Domain &d = dv.dom;
    const long long C = d.C;
    unsigned short *__restrict__ dst = static_cast<unsigned short *>(sp.dst);
    // overlapped steps: a tile near a body is the near kernel's
    static_assert(TILE_X % V == 0, "a thread's cells lie in one tile");
    const bool far = !sp.far_skip || sp.far_skip[((long long)z * d.ny + y) * ((d.nx + TILE_X - 1) / TILE_X) +
                                                 x0 / TILE_X] == 0u;
    if (!active || !far) return;
    // listed fluid cells belong to the boundary kernel, which may run
    // concurrently: leave them alone
    bool all_mine = true;
#pragma unroll
    for (int i = 0; i < V; ++i) all_mine = all_mine && bulk_cell(fl[i]);
    if (all_mine) {
#pragma unroll
        for (int b = 0; b < Q; ++b) {
            RawV r;
            memcpy(&r, &w[b], sizeof(r));
            *reinterpret_cast<RawV *>(reinterpret_cast<char *>(dst + (long long)b * C) + 2u * (unsigned)c0) = r;
        }
        return;
    }
#pragma unroll
    for (int b = 0; b < Q; ++b)
#pragma unroll
        for (int i = 0; i < V; ++i)
            if (bulk_cell(fl[i]))
                dst[(long long)b * C + c0 + i] = (unsigned short)((i & 1) ? w[b][i >> 1] >> 16 : w[b][i >> 1] & 0xffffu);
}

// The bulk kernel for 16-bit storage, V (even) cells per thread.  The
// populations stay packed two to a word (the thread's cells 2j and 2j + 1
// in word j) from load to store, half the registers of widened values, so
// that more warps -- or more bytes per warp -- keep HBM requests in flight.
// A shift along x is a byte permute of adjacent words (and of one word
// shuffled from the neighbouring lane).  The two cells of a word collide
// together in packed FP32 arithmetic (Lean<F2>); the words are widened once for
// the moments and again for the relaxation, so that only one pair's populations
// are held in FP32 at a time, and at tau = 1, where they do not enter the
// relaxation, not again at all.  All loads, the row ends' single cells included,
// stand before the first shuffle: with each row end's load behind its
// direction's shuffle the loads of several directions wait for one another (four
// cells a thread, FP16: 520 us, 429 ahead).  Bound by the
// bytes in flight and, in BF16 (the rounding), by instruction issue: 512 x 256 x
// 256 cells at tau = 1 take 396 us in FP16 (6.5 TB/s) and 441 us in BF16, 429 and
// 486 us at tau = 0.8, against 449 and 542 us with a cell at a time in scalar
// arithmetic.  (Copying the sources ahead into shared memory with cp.async, two
// stages at 16 warps an SM, took 525 and 549 us.)
template <typename T, int V, bool WALLS>
__device__ __forceinline__ void bulk16_body(const Device &dv, const StepPtrs &sp, const Blk &bk) {
    static_assert(sizeof(T) == 2 && V % 2 == 0, "two 16-bit cells a word");
    constexpr int W = V / 2;
    using RawV = typename Raw<2 * V>::type;
    const Domain d = dv.dom;
    const int nxq = d.nx / V;
    int xq, y;
    bool active;
    plane_group(bk, nxq, d.ny, sp.row_recip, xq, y, active);
    const int z = bk.z;
    const int lane = threadIdx.x & 31;
    const int x0 = xq * V;
    const int ym = y == 0 ? d.ny - 1 : y - 1, yp = y == d.ny - 1 ? 0 : y + 1;
    const int zm = z == 0 ? d.nz - 1 : z - 1, zp = z == d.nz - 1 ? 0 : z + 1;
    const long long C = d.C;
    const long long c0 = ((long long)z * d.ny + y) * d.nx + x0;
    const unsigned short *__restrict__ src = static_cast<const unsigned short *>(sp.src);

    uint8_t fl[V];
    load_vec<uint8_t, V>(sp.flags_cur + c0, fl);

    const WallRows wr = wall_rows(d, y, z);
    // byte offsets of the rows within a direction's plane (2 C < 2^32): the
    // planes' addresses are the same for all threads, so an access is a uniform
    // base and a 32-bit offset
    const unsigned cy = (unsigned)z * d.ny;
    const unsigned pitch = 2u * (unsigned)d.nx;
    const unsigned rows[3][3] = {{(zm * d.ny + ym) * pitch, (zm * d.ny + y) * pitch, (zm * d.ny + yp) * pitch},
                                 {(cy + ym) * pitch, (cy + y) * pitch, (cy + yp) * pitch},
                                 {(zp * d.ny + ym) * pitch, (zp * d.ny + y) * pitch, (zp * d.ny + yp) * pitch}};
    const unsigned xl = 2u * (x0 == 0 ? d.nx - 1 : x0 - 1), xr = 2u * (x0 + V == d.nx ? 0 : x0 + V);
    unsigned w[Q][W], edge[Q];
    const bool e0 = lane == 0 || x0 == 0, e1 = lane == 31 || x0 + V == d.nx;
#pragma unroll
    for (int b = 0; b < Q; ++b) {
        const bool own = WALLS && wr.beyond(b);
        const char *plane = reinterpret_cast<const char *>(src + (long long)b * C);
        unsigned row = rows[1 - ez(b)][1 - ey(b)];
        if (own) {
            plane = reinterpret_cast<const char *>(src + (long long)opp(b) * C);
            row = rows[1][1];
        }
        const RawV r = __ldg(reinterpret_cast<const RawV *>(plane + (row + 2u * x0)));
        memcpy(&w[b], &r, sizeof(r));
        edge[b] = 0;
        if (ex(b) > 0 && e0) {
            if (WALLS && wr.x && x0 == 0) edge[b] = (unsigned)src[(long long)opp(b) * C + c0];
            else edge[b] = (unsigned)__ldg(reinterpret_cast<const unsigned short *>(plane + (row + xl)));
        }
        if (ex(b) < 0 && e1) {
            if (WALLS && wr.x && x0 + V == d.nx) edge[b] = (unsigned)src[(long long)opp(b) * C + c0 + V - 1];
            else edge[b] = (unsigned)__ldg(reinterpret_cast<const unsigned short *>(plane + (row + xr)));
        }
    }
#pragma unroll
    for (int b = 0; b < Q; ++b) {
        const bool own = WALLS && wr.beyond(b);
        if (ex(b) > 0) {                 // pull from x - 1: the left neighbour's last half-word first
            unsigned lw = __shfl_up_sync(0xffffffffu, w[b][W - 1], 1);
            if (e0) lw = edge[b] << 16;
            unsigned o[W];
#pragma unroll
            for (int j = 0; j < W; ++j) o[j] = own ? w[b][j] : __byte_perm(j ? w[b][j - 1] : lw, w[b][j], 0x5432);
#pragma unroll
            for (int j = 0; j < W; ++j) w[b][j] = o[j];
        } else if (ex(b) < 0) {          // pull from x + 1: the right neighbour's first half-word last
            unsigned rw = __shfl_down_sync(0xffffffffu, w[b][0], 1);
            if (e1) rw = edge[b];
#pragma unroll
            for (int j = 0; j < W; ++j)
                w[b][j] = own ? w[b][j] : __byte_perm(w[b][j], j + 1 < W ? w[b][j + 1 < W ? j + 1 : j] : rw, 0x5432);
        }
    }

    collide_words<T, V>(w, fl, c0, dv, sp);
    store_words<V>(w, fl, active, x0, y, z, c0, dv, sp);
}

template <typename T, int V, int MINB, bool WALLS>
__global__ void __launch_bounds__(BULK_THREADS, MINB == 1 ? 0 : MINB)
bulk16_kernel(const Device dv, const StepPtrs sp) {
    pdl_enter();
    bulk16_body<T, V, WALLS>(dv, sp, launch_blk());
}

template <typename T, int V, int MINB, bool WALLS>
__global__ void __launch_bounds__(BULK_THREADS, MINB == 1 ? 0 : MINB) bulk16_batch(const Batch bt) {
    LBM_BATCH_MEMBER(bt);
    const int z0 = sbk.z * BATCH_PZ, z1 = min(z0 + BATCH_PZ, sdv.dom.nz);
    for (int z = z0; z < z1; ++z) {
        Blk pb = sbk;
        pb.z = z;
        bulk16_body<T, V, WALLS>(sdv, ssp, pb);
    }
}

// Minimum image of a cell difference by integer compares
__device__ __forceinline__ int near_cell(int o, int n, int periodic) {
    if (!periodic) return o;
    return 2 * o > n ? o - n : (2 * o < -n ? o + n : o);
}

// V + W x (p - X) of body k's surface at lattice point p: the minimum-image
// offset is an integer difference of cells wrapped by compares minus the centre's
// position within its cell (FP32: exact to the rounding of a few-cell offset).
// g: the geometry record of the state, st: the state itself (FP64).
__device__ __forceinline__ void wall_velocity(const Domain &d, const BodyGeom &g, const BodyState &, int px, int py,
                                              int pz, float (&u)[3]) {
    const float o0 = (float)near_cell(px - g.ci[0], d.nx, d.px) - g.cf[0];
    const float o1 = (float)near_cell(py - g.ci[1], d.ny, d.py) - g.cf[1];
    const float o2 = (float)near_cell(pz - g.ci[2], d.nz, d.pz) - g.cf[2];
    u[0] = g.v[0] + (g.w[1] * o2 - g.w[2] * o1);
    u[1] = g.v[1] + (g.w[2] * o0 - g.w[0] * o2);
    u[2] = g.v[2] + (g.w[0] * o1 - g.w[1] * o0);
}
__device__ __forceinline__ void wall_velocity(const Domain &d, const BodyGeom &g, const BodyState &st, int px, int py,
                                              int pz, double (&u)[3]) {
    const double o0 = near_cell(px - g.ci[0], d.nx, d.px) - g.cfd[0];
    const double o1 = near_cell(py - g.ci[1], d.ny, d.py) - g.cfd[1];
    const double o2 = near_cell(pz - g.ci[2], d.nz, d.pz) - g.cfd[2];
    u[0] = st.V[0] + mad(st.W[1], o2, -(st.W[2] * o1));
    u[1] = st.V[1] + mad(st.W[2], o0, -(st.W[0] * o2));
    u[2] = st.V[2] + mad(st.W[0], o1, -(st.W[1] * o0));
}

// direction components by lane, from bit masks of the directions with + and -
constexpr unsigned component_mask(int axis, int sign) {
    unsigned m = 0;
    for (int b = 0; b < Q; ++b)
        if ((axis == 0 ? ex(b) : (axis == 1 ? ey(b) : ez(b))) == sign) m |= 1u << b;
    return m;
}
__device__ __forceinline__ int lane_component(int axis, int b) {
    constexpr unsigned P[3] = {component_mask(0, 1), component_mask(1, 1), component_mask(2, 1)};
    constexpr unsigned N[3] = {component_mask(0, -1), component_mask(1, -1), component_mask(2, -1)};
    const unsigned p = axis == 0 ? P[0] : (axis == 1 ? P[1] : P[2]), n = axis == 0 ? N[0] : (axis == 1 ? N[1] : N[2]);
    return (int)((p >> b) & 1u) - (int)((n >> b) & 1u);
}
template <typename R> __device__ __forceinline__ R signed_by(int e, R v) { return e > 0 ? v : (e < 0 ? -v : (R)0); }

// Sum and momentum of a cell whose population b lane b holds (0 on the lanes
// past the last direction): 8 lanes form each of the four sums, three values a
// lane and three butterfly steps, so that all four take five additions (FP64: a
// warp's addition costs the same whatever the lanes do).  sg: the lane's three
// factors (lane_factors).
template <typename R> struct Moments { R s, x, y, z; };
struct LaneFactors { int a, b, c; };
__device__ __forceinline__ LaneFactors lane_factors(int lane) {
    const int i = lane & 7, q = lane >> 3;
    if (q == 0) return LaneFactors{1, 1, 1};
    return LaneFactors{lane_component(q - 1, i), lane_component(q - 1, i + 8), lane_component(q - 1, i + 16)};
}
template <typename R>
__device__ __forceinline__ Moments<R> lane_moments(R f, int lane, const LaneFactors &sg) {
    constexpr unsigned FULL = 0xffffffffu;
    const int i = lane & 7;
    const R a = __shfl_sync(FULL, f, i), b = __shfl_sync(FULL, f, i + 8), c = __shfl_sync(FULL, f, i + 16);
    R v = (signed_by(sg.a, a) + signed_by(sg.b, b)) + signed_by(sg.c, c);
    v += __shfl_xor_sync(FULL, v, 1);
    v += __shfl_xor_sync(FULL, v, 2);
    v += __shfl_xor_sync(FULL, v, 4);
    return Moments<R>{__shfl_sync(FULL, v, 0), __shfl_sync(FULL, v, 8), __shfl_sync(FULL, v, 16), __shfl_sync(FULL, v, 24)};
}
template <typename R> __device__ __forceinline__ R lane_sum(R v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// LBGK (+ Guo) of a listed cell from the moments of its populations, in the forms
// of the bulk kernels but for the order of the sums; boundary_warp and
// boundary_cell share it, so that a cell gets the same value from either
template <typename Cd> struct Listed { Cd gx, gy, gz, rho, ux, uy, uz, base, ug; };
template <typename Cd>
__device__ __forceinline__ Listed<Cd> listed_cell(const Device &dv, const Moments<Cd> &mo) {
    const bool f32 = sizeof(Cd) == 4;
    Listed<Cd> c;
    c.gx = f32 ? (Cd)dv.g_f[0] : (Cd)dv.g[0];
    c.gy = f32 ? (Cd)dv.g_f[1] : (Cd)dv.g[1];
    c.gz = f32 ? (Cd)dv.g_f[2] : (Cd)dv.g[2];
    c.rho = (Cd)1 + mo.s;
    const Cd inv = (Cd)1 / c.rho;
    c.ux = mad((Cd)0.5, c.gx, mo.x) * inv;
    c.uy = mad((Cd)0.5, c.gy, mo.y) * inv;
    c.uz = mad((Cd)0.5, c.gz, mo.z) * inv;
    const Cd usq = mad(c.ux, c.ux, mad(c.uy, c.uy, c.uz * c.uz));
    c.base = mad((Cd)(-1.5) * c.rho, usq, mo.s);
    c.ug = dv.forced ? mad(c.ux, c.gx, mad(c.uy, c.gy, c.uz * c.gz)) : (Cd)0;
    return c;
}
// population f of weight w (class wc) relaxed, FP32: its increment
template <typename T, typename Cd>
__device__ __forceinline__ Cd listed_relax(const Device &dv, const Listed<Cd> &c, Cd f, Cd w, int wc, Cd eu, Cd eg) {
    if constexpr (sizeof(T) == 2) {
        // the weight last, as the bulk kernel's FP16 form (Lean)
        Cd r = dv.ow_f[wc] * (mad((Cd)4.5 * c.rho, eu * eu, c.base) + (Cd)3 * c.rho * eu);
        if (dv.forced) r = mad(dv.gw_f[wc], mad((Cd)9 * eu, eg, (Cd)(-3) * c.ug) + (Cd)3 * eg, r);
        return mad(dv.om1_f, f, r);
    } else {
        const bool f32 = sizeof(Cd) == 4;
        const Cd deq = w * mad(c.rho, mad((Cd)4.5 * eu, eu, (Cd)3 * eu), c.base);
        Cd gt = 0;
        if (dv.forced)
            gt = (f32 ? (Cd)dv.guo_f : (Cd)(1.0 - 0.5 * dv.omega)) * w * mad((Cd)9 * eu, eg, (Cd)3 * (eg - c.ug));
        const Cd om = f32 ? (Cd)dv.omega_f : (Cd)dv.omega;
        if constexpr (std::is_same<T, float>::value) return mad(om, deq - f, gt);
        else return dv.forced ? mad(om, deq - f, f) + gt : mad(om, deq - f, f);
    }
}

// The cells the remap listed (fluid with a flag of F_LISTED): refill,
// bounce-back at walls and moving obstacles, then LBGK, a warp a cell with lane b
// the direction b: the 19 pulls, wall velocities and relaxations run side by side
// and the cell's sums by shuffles.  Latency-bound (some hundred cells a body): a
// thread a cell walked ~250 dependent operations, in FP64 at 64 issue cycles
// each.  (32^3 swimmer in FP64, a step: 93 -> 50 us, the kernel 70 us of it
// before; 48^3 in FP32 with the body read: 69 -> 62 us a step.)
constexpr int BOUNDARY_WARPS = 8;

// a lane's direction
struct LaneDir {
    bool act;                       // lanes past the last direction hold none
    int b, x, y, z, ob;             // direction, its components, its reverse
    LaneFactors sg;
};
__device__ __forceinline__ LaneDir lane_dir(int lane) {
    LaneDir l;
    l.act = lane < Q;
    l.b = l.act ? lane : 0;
    l.x = lane_component(0, l.b);
    l.y = lane_component(1, l.b);
    l.z = lane_component(2, l.b);
    l.ob = l.b == 0 ? 0 : ((l.b & 1) ? l.b + 1 : l.b - 1);
    l.sg = lane_factors(lane);
    return l;
}

// listed cell cl by one warp
template <typename T>
__device__ __forceinline__ void boundary_warp(const Device &dv, const StepPtrs &sp, unsigned cl, int lane, const LaneDir &ld) {
    using Cd = typename Codec<T>::C;
    constexpr unsigned FULL = 0xffffffffu;
    const Domain &d = dv.dom;
    const bool act = ld.act;
    const int b = ld.b, bx = ld.x, by = ld.y, bz = ld.z;
    const Cd w = b == 0 ? (Cd)wgt(0) : (b < 7 ? (Cd)wgt(1) : (Cd)wgt(7));
    const long long C = d.C;
    const T *__restrict__ src = static_cast<const T *>(sp.src);
    T *__restrict__ dst = static_cast<T *>(sp.dst);
    const float s = dv.f16_inv_scale;
    const unsigned nxu = (unsigned)d.nx, nyu = (unsigned)d.ny;      // C < 2^31: 32-bit division
    const unsigned row = cl / nxu, zu = row / nyu;
    const int x = (int)(cl - row * nxu), y = (int)(row - zu * nyu), z = (int)zu;
    const uint8_t fc = sp.flags_cur[cl];
    Cd f = 0;
    if (fc & F_SOLID_PREV) {
        // uncovered cell: f = f_eq(rho_avg, u_w(x)) with the state of step n;
        // rho_avg over the D3Q19 neighbours fluid in both epochs (1 if none),
        // as deviations (small numbers: no 1 + drho is rounded), lane a the
        // neighbour x + e_a
        const int nx_ = x + bx, ny_ = y + by, nz_ = z + bz;
        const bool in = act && b > 0 &&
                        !((!d.px && (nx_ < 0 || nx_ >= d.nx)) || (!d.py && (ny_ < 0 || ny_ >= d.ny)) ||
                          (!d.pz && (nz_ < 0 || nz_ >= d.nz)));
        const long long nc = ((long long)wrap_axis(nz_, d.nz) * d.ny + wrap_axis(ny_, d.ny)) * d.nx +
                             wrap_axis(nx_, d.nx);
        Cd drho = 0;
#pragma unroll
        for (int q = 0; q < Q; ++q) drho += Codec<T>::ld(src[q * C + nc], s);
        const bool ok = in && !(sp.flags_cur[nc] & (F_SOLID | F_SOLID_PREV));
        const int cnt = __popc(__ballot_sync(FULL, ok));
        const Cd sum = lane_sum(ok ? drho : (Cd)0);
        drho = cnt ? sum / (Cd)cnt : (Cd)0;
        const Cd rho = (Cd)1 + drho;
        const int k = sp.bid_prev[cl];
        Cd u[3] = {0, 0, 0};
        if (k != NO_BODY) wall_velocity(d, dv.geom[sp.parity * dv.nb + k], sp.body_cur[k], x, y, z, u);
        const Cd uu = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
        const Cd eu = signed_by(bx, u[0]) + signed_by(by, u[1]) + signed_by(bz, u[2]);
        f = w * drho + w * rho * ((Cd)3 * eu + (Cd)4.5 * eu * eu - (Cd)1.5 * uu);
        if (!act) f = 0;
    } else {
        // bounce-back at walls (Eq. 4) and at obstacles of step n-1
        const int sx = x - bx, sy = y - by, sz = z - bz;
        const bool wall = (!d.px && (sx < 0 || sx >= d.nx)) || (!d.py && (sy < 0 || sy >= d.ny)) ||
                          (!d.pz && (sz < 0 || sz >= d.nz));
        const long long sc = ((long long)wrap_axis(sz, d.nz) * d.ny + wrap_axis(sy, d.ny)) * d.nx +
                             wrap_axis(sx, d.nx);
        const uint8_t fp = sp.flags_prev[sc];
        const int k = sp.bid_prev[sc];
        const Cd own = act ? Codec<T>::ld(src[(long long)b * C + cl], s) : (Cd)0;
        const Cd pulled = Codec<T>::ld(src[(long long)b * C + sc], s);
        const Cd rho_x = (Cd)1 + lane_sum(own);
        const Cd own_opp = __shfl_sync(FULL, own, ld.ob);
        f = pulled;
        if (wall) {
            f = own_opp;                                                 // Eq. 4
        } else if (fp & F_SOLID) {
            Cd u[3] = {0, 0, 0};
            if (k != NO_BODY) wall_velocity(d, dv.geom[(sp.parity ^ 1) * dv.nb + k], sp.body_prev[k], sx, sy, sz, u);
            const Cd eu = signed_by(bx, u[0]) + signed_by(by, u[1]) + signed_by(bz, u[2]);
            f = own_opp + (Cd)6 * w * rho_x * eu;                        // moving wall
        }
        if (!act) f = 0;
    }
    const Moments<Cd> mo = lane_moments(f, lane, ld.sg);
    if constexpr (sizeof(T) != 8)
        if (lane == 0) dv.rho_near[cl] = mo.s;      // rho - 1 for the momentum exchange
    const Listed<Cd> c = listed_cell(dv, mo);
    const Cd eu = signed_by(bx, c.ux) + signed_by(by, c.uy) + signed_by(bz, c.uz);
    const Cd eg = dv.forced ? signed_by(bx, c.gx) + signed_by(by, c.gy) + signed_by(bz, c.gz) : (Cd)0;
    const Cd v = listed_relax<T>(dv, c, f, w, b == 0 ? 0 : (b < 7 ? 1 : 2), eu, eg);
    if constexpr (std::is_same<T, float>::value) {
        // the increments' mass and momentum are moved to 0 and g (collide_f32)
        const Moments<Cd> dm = lane_moments(act ? v : (Cd)0, lane, ld.sg);
        f += v;
        if (b == 0) f -= dm.s;
        else if (b < 7)
            f += (Cd)0.5 * (signed_by(bx, c.gx - dm.x) + signed_by(by, c.gy - dm.y) + signed_by(bz, c.gz - dm.z));
    } else {
        f = v;
    }
    if (act) {
        T out;
        if constexpr (std::is_same<T, __nv_bfloat16>::value) {
            out = __ushort_as_bfloat16((unsigned short)(bf16_sr_add(f, bf16_dither_word(cl, *sp.tstep, b >> 2), b) >> 16));
        } else {
            out = Codec<T>::st(f, dv.f16_scale);
        }
        dst[(long long)b * C + cl] = out;
    }
}

template <typename T>
__device__ __forceinline__ void boundary_body(const Device &dv, const StepPtrs &sp, const Blk &bk) {
    const int lane = threadIdx.x & 31;
    // the count may pass the capacity after an overflow (reported as an error): never read past it
    const int listed = (int)min((long long)*dv.bcount, dv.blist_cap);
    int l = bk.x * BOUNDARY_WARPS + (threadIdx.x >> 5);
    if (l >= listed) return;
    const LaneDir ld = lane_dir(lane);
    for (; l < listed; l += bk.gx * BOUNDARY_WARPS) boundary_warp<T>(dv, sp, dv.blist[l], lane, ld);
}

// lane_sum and lane_moments of the populations of one thread, in their order
template <typename R> __device__ __forceinline__ R tree_sum(const R (&v)[Q]) {
    R a[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) a[i] = i + 16 < Q ? v[i] + v[i + 16] : v[i];
#pragma unroll
    for (int o = 8; o > 0; o >>= 1)
#pragma unroll
        for (int i = 0; i < o; ++i) a[i] = a[i] + a[i + o];
    return a[0];
}
template <typename R> __device__ __forceinline__ Moments<R> tree_moments(const R (&f)[Q]) {
    R out[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        R p[8];
        bool any[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            any[i] = false;
            p[i] = 0;
#pragma unroll
            for (int b = i; b < Q; b += 8) {
                const int e = q == 0 ? 1 : (q == 1 ? ex(b) : (q == 2 ? ey(b) : ez(b)));
                if (e == 0) continue;
                const R v = e > 0 ? f[b] : -f[b];
                p[i] = any[i] ? p[i] + v : v;
                any[i] = true;
            }
        }
#pragma unroll
        for (int o = 1; o < 8; o <<= 1)
#pragma unroll
            for (int i = 0; i < 8; i += 2 * o) {
                if (any[i] && any[i + o]) p[i] = p[i] + p[i + o];
                else if (any[i + o]) p[i] = p[i + o];
                any[i] = any[i] || any[i + o];
            }
        out[q] = p[0];
    }
    return Moments<R>{out[0], out[1], out[2], out[3]};
}

// Listed cell cl (not uncovered) by one thread: boundary_warp's operations in its
// order, without the additions of zeros, so the same value.
template <typename T>
__device__ __forceinline__ void boundary_cell(const Device &dv, const StepPtrs &sp, unsigned cl) {
    using Cd = typename Codec<T>::C;
    const Domain &d = dv.dom;
    const long long C = d.C;
    const T *__restrict__ src = static_cast<const T *>(sp.src);
    T *__restrict__ dst = static_cast<T *>(sp.dst);
    const float s = dv.f16_inv_scale;
    const unsigned nxu = (unsigned)d.nx, nyu = (unsigned)d.ny;
    const unsigned row = cl / nxu, zu = row / nyu;
    const int x = (int)(cl - row * nxu), y = (int)(row - zu * nyu), z = (int)zu;
    // the source of a direction with component e: [1 - e]
    const int xs[3] = {x == 0 ? d.nx - 1 : x - 1, x, x == d.nx - 1 ? 0 : x + 1};
    const int ys[3] = {y == 0 ? d.ny - 1 : y - 1, y, y == d.ny - 1 ? 0 : y + 1};
    const int zs[3] = {z == 0 ? d.nz - 1 : z - 1, z, z == d.nz - 1 ? 0 : z + 1};
    const bool xw[3] = {!d.px && x == 0, false, !d.px && x == d.nx - 1}, yw[3] = {!d.py && y == 0, false, !d.py && y == d.ny - 1},
               zw[3] = {!d.pz && z == 0, false, !d.pz && z == d.nz - 1};
    auto source = [&](int b) { return ((unsigned)zs[1 - ez(b)] * nyu + ys[1 - ey(b)]) * nxu + xs[1 - ex(b)]; };
    auto beyond = [&](int b) { return xw[1 - ex(b)] || yw[1 - ey(b)] || zw[1 - ez(b)]; };
    Cd f[Q];
    unsigned walls = 0, solid = 0;
#pragma unroll
    for (int b = 0; b < Q; ++b) {
        const unsigned sc = source(b);
        f[b] = Codec<T>::ld(src[(long long)b * C + sc], s);
        if (b > 0 && beyond(b)) walls |= 1u << b;
        else if (sp.flags_prev[sc] & F_SOLID) solid |= 1u << b;
    }
    if (walls | solid) {
        Cd own[Q];
#pragma unroll
        for (int b = 0; b < Q; ++b) own[b] = Codec<T>::ld(src[(long long)b * C + cl], s);
        const Cd rho_x = (Cd)1 + tree_sum(own);
#pragma unroll
        for (int b = 0; b < Q; ++b) {
            if (walls >> b & 1u) {
                f[b] = own[opp(b)];                                      // Eq. 4
            } else if (solid >> b & 1u) {
                const int k = sp.bid_prev[source(b)];
                Cd u[3] = {0, 0, 0};
                if (k != NO_BODY)
                    wall_velocity(d, dv.geom[(sp.parity ^ 1) * dv.nb + k], sp.body_prev[k], x - ex(b), y - ey(b), z - ez(b), u);
                const Cd w = (Cd)wgt(b);
                f[b] = own[opp(b)] + (Cd)6 * w * rho_x * edot(b, u[0], u[1], u[2]);      // moving wall
            }
        }
    }
    const Moments<Cd> mo = tree_moments(f);
    if constexpr (sizeof(T) != 8) dv.rho_near[cl] = mo.s;
    const Listed<Cd> c = listed_cell(dv, mo);
    Cd v[Q];
#pragma unroll
    for (int b = 0; b < Q; ++b)
        v[b] = listed_relax<T>(dv, c, f[b], (Cd)wgt(b), b == 0 ? 0 : (b < 7 ? 1 : 2), edot(b, c.ux, c.uy, c.uz),
                               dv.forced ? edot(b, c.gx, c.gy, c.gz) : (Cd)0);
    if constexpr (std::is_same<T, float>::value) {
        const Moments<Cd> dm = tree_moments(v);
#pragma unroll
        for (int b = 0; b < Q; ++b) {
            v[b] = f[b] + v[b];
            if (b == 0) v[b] -= dm.s;
            else if (b < 7) v[b] += (Cd)0.5 * edot(b, c.gx - dm.x, c.gy - dm.y, c.gz - dm.z);
        }
    }
    const Dither dz = dither_for<T>(cl, sp.tstep);
#pragma unroll
    for (int b = 0; b < Q; ++b) {
        T out;
        if constexpr (std::is_same<T, __nv_bfloat16>::value) out = store16<T>(v[b], dz, b);
        else out = Codec<T>::st(v[b], dv.f16_scale);
        dst[(long long)b * C + cl] = out;
    }
}

// The boundary kernel of long lists: a thread a cell, the uncovered cells (few)
// by their warp.  A warp a cell keeps a short list's latency low, but costs
// instruction issue (FP64: its pipe) for 32 lanes and a cell at a time.
constexpr int BOUNDARY_THREADS = 128;

template <typename T>
__device__ __forceinline__ void boundary_cells_body(const Device &dv, const StepPtrs &sp, const Blk &bk) {
    constexpr unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const int listed = (int)min((long long)*dv.bcount, dv.blist_cap);
    const LaneDir ld = lane_dir(lane);
    for (long long l0 = (long long)bk.x * BOUNDARY_THREADS + (threadIdx.x & ~31u); l0 < listed;
         l0 += (long long)bk.gx * BOUNDARY_THREADS) {
        const bool have = l0 + lane < listed;
        const unsigned cl = have ? dv.blist[l0 + lane] : 0u;
        const bool uncovered = have && (sp.flags_cur[cl] & F_SOLID_PREV);
        unsigned rest = __ballot_sync(FULL, uncovered);
        if (have && !uncovered) boundary_cell<T>(dv, sp, cl);
        __syncwarp();
        for (; rest; rest &= rest - 1) boundary_warp<T>(dv, sp, __shfl_sync(FULL, cl, __ffs(rest) - 1), lane, ld);
    }
}

// grid of the boundary kernels: a warp or a thread for each cell of the expected
// list and an eighth to spare, at most what the SMs hold at once (a warp a cell)
// or about four waves; longer lists take turns
int sm_count();
int boundary_blocks(const Device &dv, bool by_cell) {
    const long long cells = dv.shell + dv.shell / 8, per = by_cell ? BOUNDARY_THREADS : BOUNDARY_WARPS;
    return (int)std::min<long long>(std::max<long long>((cells + per - 1) / per, 1), (by_cell ? 16LL : 4LL) * sm_count());
}

template <typename T>
__global__ void __launch_bounds__(32 * BOUNDARY_WARPS) boundary_kernel(const Device dv, const StepPtrs sp) {
    boundary_body<T>(dv, sp, launch_blk());
}

template <typename T>
__global__ void __launch_bounds__(32 * BOUNDARY_WARPS) boundary_batch(const Batch bt) {
    LBM_BATCH_MEMBER(bt);
    boundary_body<T>(sdv, ssp, sbk);
}

template <typename T>
__global__ void __launch_bounds__(BOUNDARY_THREADS) boundary_cells_kernel(const Device dv, const StepPtrs sp) {
    boundary_cells_body<T>(dv, sp, launch_blk());
}

template <typename T>
__global__ void __launch_bounds__(BOUNDARY_THREADS) boundary_cells_batch(const Batch bt) {
    LBM_BATCH_MEMBER(bt);
    boundary_cells_body<T>(sdv, ssp, sbk);
}

// ---- TMA row-staged variant ---------------------------------------------------
//
// Persistent blocks walk the x-rows (y, z) of the lattice (row r = blockIdx.x
// + i gridDim.x).  For each row one thread issues 20 bulk copies
// (cp.async.bulk, completed on an mbarrier with the byte count): the 19
// source rows, direction b from the neighbour row (y - ey_b, z - ez_b) of
// plane b, and the row's flag bytes, into one of NSTAGE shared-memory stages;
// NSTAGE rows are in flight.  The threads then pull f_b(x) = row_b[x - ex_b]
// from shared memory, collide with the same code as the register variant
// and store -- the same arithmetic, the same bits.  Every wait on an
// mbarrier is bounded: past the limit the block records ST_TIMEOUT, waits
// (bounded again) for its copies in flight and returns.

__device__ __forceinline__ unsigned smem_u32(const void *p) { return (unsigned)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t *bar, unsigned count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, unsigned bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, unsigned parity) {
    unsigned ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.b32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// bulk copy global -> shared of `bytes` (a multiple of 16, both addresses
// 16-byte aligned), completing `bytes` transactions on bar
__device__ __forceinline__ void bulk_copy(void *dst, const void *src, unsigned bytes, uint64_t *bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     smem_u32(dst)),
                 "l"(src), "r"(bytes), "r"(smem_u32(bar))
                 : "memory");
}

constexpr int TMA_THREADS = 256;
constexpr long long TMA_WAIT_CYCLES = 1LL << 31;     // ~1 s of SM clock before a block gives up
constexpr long long TMA_EXPIRE_CYCLES = 1LL << 16;   // the bound of the expired-wait check (~30 us)
constexpr int TMA_HEADER = 128;                      // mbarriers, ahead of the stages

__host__ __device__ constexpr size_t tma_stage_bytes(int nx, int elem) { return (size_t)Q * nx * elem + (size_t)nx; }

template <typename T, int NSTAGE, int MINB, int ROWS, bool WALLS>
__global__ void __launch_bounds__(TMA_THREADS, MINB) bulk_tma_kernel(const Device dv, const StepPtrs sp) {
    pdl_enter();
    using Cd = typename Codec<T>::C;
    static_assert((NSTAGE + 1) * sizeof(uint64_t) <= TMA_HEADER, "the mbarriers fit the header");
    extern __shared__ __align__(128) unsigned char smem[];
    const Domain d = dv.dom;
    const int nx = d.nx;
    const unsigned row_bytes = (unsigned)(nx * sizeof(T));
    const unsigned flag_off = Q * row_bytes;
    const unsigned row_stage = (unsigned)tma_stage_bytes(nx, sizeof(T));     // one x-row's sources + flags
    const unsigned stage_bytes = ROWS * row_stage;
    uint64_t *bar = reinterpret_cast<uint64_t *>(smem);
    unsigned char *stages = smem + TMA_HEADER;
    const long long rows = (long long)d.ny * d.nz;
    const long long first = blockIdx.x;
    const long long nmine = rows > first ? (rows - 1 - first) / gridDim.x + 1 : 0;
    const long long ngroups = (nmine + ROWS - 1) / ROWS;     // a stage holds ROWS of this block's rows
    const T *__restrict__ src = static_cast<const T *>(sp.src);
    T *__restrict__ dst = static_cast<T *>(sp.dst);
    const long long C = d.C;
    const float inv_scale = dv.f16_inv_scale, scale = dv.f16_scale;
    const int ntx = (nx + TILE_X - 1) / TILE_X;

    if (threadIdx.x == 0) {
        // bar[NSTAGE] is never arrived at: with dv.expire_waits the first
        // wait of every block is on it, so that its bounded wait runs out
        for (int st = 0; st <= NSTAGE; ++st) mbar_init(&bar[st], 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    auto issue = [&](long long g) {          // thread 0: rows of group g into stage g % NSTAGE
        const int st = (int)(g % NSTAGE);
        const int nr = (int)min((long long)ROWS, nmine - g * ROWS);
        unsigned char *buf0 = stages + (size_t)st * stage_bytes;
        mbar_expect_tx(&bar[st], nr * row_stage);
        for (int rr = 0; rr < nr; ++rr) {
            const long long r = first + (g * ROWS + rr) * gridDim.x;
            const int y = (int)(r % d.ny), z = (int)(r / d.ny);
            unsigned char *buf = buf0 + (size_t)rr * row_stage;
#pragma unroll
            for (int b = 0; b < Q; ++b) {
                const int ys = wrap_axis(y - ey(b), d.ny), zs = wrap_axis(z - ez(b), d.nz);
                const T *from = WALLS && wall_rows(d, y, z).beyond(b)      // Eq. 4: the row's own reversed populations
                                    ? src + (long long)opp(b) * C + r * nx
                                    : src + (long long)b * C + ((long long)zs * d.ny + ys) * nx;
                bulk_copy(buf + b * row_bytes, from, row_bytes, &bar[st]);
            }
            bulk_copy(buf + flag_off, sp.flags_cur + r * nx, (unsigned)nx, &bar[st]);
        }
    };
    if (threadIdx.x == 0)
        for (long long g = 0; g < ngroups && g < NSTAGE; ++g) issue(g);

    long long g = 0;
    bool ok = true;
    for (; g < ngroups; ++g) {
        const int st = (int)(g % NSTAGE);
        const unsigned parity = (unsigned)((g / NSTAGE) & 1);
        const long long t0 = clock64();
        bool ready = false;
        if (dv.expire_waits && g == 0) {
            while (!(ready = mbar_try_wait(&bar[NSTAGE], 0)) && clock64() - t0 < TMA_EXPIRE_CYCLES) {
            }
        } else {
            while (!(ready = mbar_try_wait(&bar[st], parity)) && clock64() - t0 < TMA_WAIT_CYCLES) {
            }
        }
        ok = __syncthreads_and(ready);
        if (!ok) break;
        const int nr = (int)min((long long)ROWS, nmine - g * ROWS);
        for (int rr = 0; rr < nr; ++rr) {
            const unsigned char *buf = stages + (size_t)st * stage_bytes + (size_t)rr * row_stage;
            const T *rowb = reinterpret_cast<const T *>(buf);
            const uint8_t *fl = buf + flag_off;
            const long long r = first + (g * ROWS + rr) * gridDim.x;
            const long long c0 = r * nx;
            const WallRows wr = wall_rows(d, (int)(r % d.ny), (int)(r / d.ny));
            for (int x = threadIdx.x; x < nx; x += TMA_THREADS) {
                const uint8_t f8 = fl[x];
                if (!bulk_cell(f8)) continue;                  // the boundary kernel's cell
                if (sp.far_skip && sp.far_skip[r * ntx + x / TILE_X]) continue;    // the near kernel's
                if (f8 & F_SOLID) {
#pragma unroll
                    for (int b = 0; b < Q; ++b) dst[(long long)b * C + c0 + x] = Codec<T>::st((Cd)0, scale);
                    continue;
                }
                Cd f[Q];
#pragma unroll
                for (int b = 0; b < Q; ++b) {
                    int xs = x - ex(b);
                    const bool out = xs < 0 || xs >= nx;
                    xs = xs < 0 ? xs + nx : (xs >= nx ? xs - nx : xs);
                    if (WALLS && wr.beyond(b)) xs = x;
                    T v = rowb[b * nx + xs];
                    if (WALLS && out && wr.x) v = src[(long long)opp(b) * C + c0 + x];
                    if constexpr (sizeof(T) == 2) f[b] = raw_ld<T>(v);
                    else f[b] = Codec<T>::ld(v, inv_scale);
                }
                collide<T>(f, dv);
                if constexpr (sizeof(T) == 2) {
                    const Dither dz = dither_for<T>(c0 + x, sp.tstep);
#pragma unroll
                    for (int b = 0; b < Q; ++b) dst[(long long)b * C + c0 + x] = store16<T>(f[b], dz, b);
                } else {
#pragma unroll
                    for (int b = 0; b < Q; ++b) dst[(long long)b * C + c0 + x] = Codec<T>::st(f[b], scale);
                }
            }
        }
        __syncthreads();                         // stage st is free again
        if (threadIdx.x == 0 && g + NSTAGE < ngroups) {
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            issue(g + NSTAGE);
        }
    }
    if (!ok && threadIdx.x == 0) {
        atomicOr(dv.status, ST_TIMEOUT);
        // the copies still in flight target this block's shared memory
        for (long long j = g; j < ngroups && j < g + NSTAGE; ++j) {
            const long long t0 = clock64();
            while (!mbar_try_wait(&bar[j % NSTAGE], (unsigned)((j / NSTAGE) & 1)) &&
                   clock64() - t0 < TMA_WAIT_CYCLES) {
            }
        }
    }
}

template <typename T, int NSTAGE, int PER_SM, int ROWS = 1>
size_t tma_smem_bytes(int nx) { return TMA_HEADER + (size_t)NSTAGE * ROWS * tma_stage_bytes(nx, sizeof(T)); }

int sm_count() {
    static int n = 0;
    if (!n) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
        if (n <= 0) n = 1;
    }
    return n;
}

template <typename T, int NSTAGE, int PER_SM, int ROWS = 1>
void launch_tma(const Device &dv, const StepPtrs &sp, cudaStream_t s) {
    const size_t bytes = tma_smem_bytes<T, NSTAGE, PER_SM, ROWS>(dv.dom.nx);
    const long long rows = (long long)dv.dom.ny * dv.dom.nz;
    const long long grid = std::min<long long>(rows, (long long)sm_count() * PER_SM);
    const bool walls = !(dv.dom.px && dv.dom.py && dv.dom.pz);
    launch_kernel(dv.pdl != 0, walls ? bulk_tma_kernel<T, NSTAGE, PER_SM, ROWS, true>
                                     : bulk_tma_kernel<T, NSTAGE, PER_SM, ROWS, false>,
                  dim3((unsigned)grid), dim3(TMA_THREADS), bytes, s, dv, sp);
}

template <typename T, int NSTAGE, int PER_SM, int ROWS = 1>
bool tma_fits(int nx) {
    return nx % 16 == 0 && tma_smem_bytes<T, NSTAGE, PER_SM, ROWS>(nx) * PER_SM <= 227u * 1024u;
}

template <typename T, int NSTAGE, int PER_SM, int ROWS = 1>
void tma_prepare() {
    for (auto k : {bulk_tma_kernel<T, NSTAGE, PER_SM, ROWS, true>, bulk_tma_kernel<T, NSTAGE, PER_SM, ROWS, false>})
        cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
}

// launch shapes: V cells per thread in blocks of BULK_THREADS; MINB > 1 caps
// the registers so that MINB blocks fit an SM.  16-bit storage with an even V
// takes the packed kernel.
template <typename T, int V, int MINB>
void launch_shape(const Device &dv, const StepPtrs &ptrs, cudaStream_t s) {
    const Domain &d = dv.dom;
    StepPtrs sp = ptrs;
    sp.row_recip = row_recip(d.nx / V);
    const long long per_plane = (long long)(d.nx / V) * d.ny;
    const dim3 grid((unsigned)((per_plane + BULK_THREADS - 1) / BULK_THREADS), 1, d.nz);
    const bool walls = !(d.px && d.py && d.pz);
    if constexpr (sizeof(T) == 2 && V % 2 == 0)
        launch_kernel(dv.pdl != 0, walls ? bulk16_kernel<T, V, MINB, true> : bulk16_kernel<T, V, MINB, false>, grid,
                      dim3(BULK_THREADS), 0, s, dv, sp);
    else
        launch_kernel(dv.pdl != 0, walls ? bulk_kernel<T, V, MINB, true> : bulk_kernel<T, V, MINB, false>, grid,
                      dim3(BULK_THREADS), 0, s, dv, sp);
}

using Launcher = void (*)(const Device &, const StepPtrs &, cudaStream_t);
struct Variant {
    int precision, vec, minb;       // vec -1: TMA row-staged, minb = resident blocks per SM
    Launcher fn;
    bool (*fits)(int nx);           // staged variants: shared memory and alignment for this nx
};

// the compiled variants of the bulk kernel; the first entry of a precision
// and width is its default (FP32, two cells: without a register cap 746 us on
// 512 x 256 x 256 cells, 96 us on 204 x 148 x 132, 59 us on 100 x 100 x 200 with
// walls and 19.6 us on 128 x 64 x 64, against 830, 108, 66 and 20.3 us capped for
// 4 blocks an SM)
const Variant kVariants[] = {
    {0, 1, 1, launch_shape<double, 1, 1>},
    {0, 2, 1, launch_shape<double, 2, 1>},
    {1, 2, 1, launch_shape<float, 2, 1>},
    {1, 2, 4, launch_shape<float, 2, 4>},
    {1, 1, 1, launch_shape<float, 1, 1>},
    {1, 4, 1, launch_shape<float, 4, 1>},
    {2, 4, 2, launch_shape<__half, 4, 2>},
    {2, 4, 1, launch_shape<__half, 4, 1>},
    {2, 4, 3, launch_shape<__half, 4, 3>},
    {2, 8, 2, launch_shape<__half, 8, 2>},
    {2, 8, 1, launch_shape<__half, 8, 1>},
    {2, 2, 1, launch_shape<__half, 2, 1>},
    {2, 2, 4, launch_shape<__half, 2, 4>},
    {2, 1, 1, launch_shape<__half, 1, 1>},
    {3, 4, 2, launch_shape<__nv_bfloat16, 4, 2>},
    {3, 4, 1, launch_shape<__nv_bfloat16, 4, 1>},
    {3, 4, 3, launch_shape<__nv_bfloat16, 4, 3>},
    {3, 8, 2, launch_shape<__nv_bfloat16, 8, 2>},
    {3, 8, 1, launch_shape<__nv_bfloat16, 8, 1>},
    {3, 2, 1, launch_shape<__nv_bfloat16, 2, 1>},
    {3, 2, 4, launch_shape<__nv_bfloat16, 2, 4>},
    {3, 1, 1, launch_shape<__nv_bfloat16, 1, 1>},
    {0, -1, 1, launch_tma<double, 2, 1>, tma_fits<double, 2, 1>},
    {1, -1, 1, launch_tma<float, 4, 1>, tma_fits<float, 4, 1>},
    {1, -1, 2, launch_tma<float, 2, 2>, tma_fits<float, 2, 2>},
    {2, -1, 2, launch_tma<__half, 2, 2, 2>, tma_fits<__half, 2, 2, 2>},
    {2, -1, 3, launch_tma<__half, 2, 3>, tma_fits<__half, 2, 3>},
    {2, -1, 4, launch_tma<__half, 2, 4>, tma_fits<__half, 2, 4>},
    {3, -1, 2, launch_tma<__nv_bfloat16, 2, 2, 2>, tma_fits<__nv_bfloat16, 2, 2, 2>},
    {3, -1, 3, launch_tma<__nv_bfloat16, 2, 3>, tma_fits<__nv_bfloat16, 2, 3>},
    {3, -1, 4, launch_tma<__nv_bfloat16, 2, 4>, tma_fits<__nv_bfloat16, 2, 4>},
};
const Variant *find_variant(int precision, int vec, int minb) {
    const Variant *first = nullptr;
    for (const Variant &v : kVariants) {
        if (v.precision != precision || v.vec != vec) continue;
        if (!first) first = &v;
        if (minb == 0 || v.minb == minb) return minb == 0 ? first : &v;
    }
    return nullptr;
}

template <typename T>
void launch_boundary(const Device &dv, const StepPtrs &sp, cudaStream_t s) {
    // the list's length is on the device: blocks past it return at once
    if (boundary_by_cell(dv.precision, dv.shell))
        boundary_cells_kernel<T><<<boundary_blocks(dv, true), BOUNDARY_THREADS, 0, s>>>(dv, sp);
    else
        boundary_kernel<T><<<boundary_blocks(dv, false), 32 * BOUNDARY_WARPS, 0, s>>>(dv, sp);
}

}  // namespace

// The two kernels take the same time at lists of about 5,000 cells in FP64 (33 us)
// and 10,000 to 17,000 in the other types (16 to 18 us); past that a warp a cell
// falls behind (spheres of radius 4 and 8 in 192^3 cells, a warp and a thread a
// cell: 10,291 cells FP64 53 and 33 us, FP32 16.3 and 17.8; 34,720 cells 151 and
// 52, 34.7 and 20.4, FP16 28.0 and 18.3; 367,462 cells 1503 and 375, 283 and 114,
// 220 and 90 us).
bool boundary_by_cell(int precision, long long shell) { return shell >= (precision == 0 ? 6000 : 15000); }

bool valid_vector_width(const Device &dv, int v) {
    if (v == -1) {
        const Variant *x = find_variant(dv.precision, -1, 0);
        return x && x->fits(dv.dom.nx);
    }
    return v >= 1 && dv.dom.nx % v == 0 && find_variant(dv.precision, v, 0) != nullptr;
}

bool valid_variant(const Device &dv, int v, int minb) {
    if (!valid_vector_width(dv, v)) return false;
    const Variant *x = find_variant(dv.precision, v, minb);
    return x && (!x->fits || x->fits(dv.dom.nx));
}

void prepare_bulk_variants() {
    static bool done = false;
    if (done) return;
    tma_prepare<double, 2, 1>();
    tma_prepare<float, 4, 1>();
    tma_prepare<float, 2, 2>();
    tma_prepare<__half, 2, 2, 2>();
    tma_prepare<__half, 2, 3>();
    tma_prepare<__half, 2, 4>();
    tma_prepare<__nv_bfloat16, 2, 2, 2>();
    tma_prepare<__nv_bfloat16, 2, 3>();
    tma_prepare<__nv_bfloat16, 2, 4>();
    done = true;
}

// 16-bit storage takes 8 cells a thread (2 blocks an SM, the most bytes in flight)
// where that leaves five or more waves of blocks, else 4 (FP16 396 against
// 429 us on 512 x 256 x 256 cells, 58.9 against 61.7 us on 256 x 128 x 128, level on
// 160 x 128 x 128, 19.8 against 19.4 us on 128 x 96 x 96; BF16 448 against 476,
// 68.3 against 68.5, 48.4 against 47.1 and 23.1 against 22.0 us; 3 blocks an SM
// of 4 cells spill: FP16 494 us).
int default_vector_width(const Device &dv) {
    const bool wide = dv.precision >= 2 && dv.minb == 0 && dv.dom.C >= 5LL * 2 * sm_count() * BULK_THREADS * 8;
    const int pref = dv.precision == 0 ? 1 : (dv.precision == 1 ? 2 : (wide ? 8 : 4));
    for (int v = pref; v > 1; v >>= 1)
        if (dv.dom.nx % v == 0) return v;
    return 1;
}

int list_variants(const Device &dv, int *vec, int *minb, int max) {
    int n = 0;
    for (const Variant &v : kVariants)
        if (v.precision == dv.precision && (v.fits ? v.fits(dv.dom.nx) : dv.dom.nx % v.vec == 0) && n < max) {
            vec[n] = v.vec;
            minb[n] = v.minb;
            ++n;
        }
    return n;
}

void launch_stream_collide(const Device &dv, const StepPtrs &sp, cudaStream_t s) {
    const Variant *v = find_variant(dv.precision, dv.vec, dv.minb);
    if (!v) v = find_variant(dv.precision, 1, 0);
    v->fn(dv, sp, s);
}

void launch_boundary_fix(const Device &dv, const StepPtrs &sp, cudaStream_t s) {
    switch (dv.precision) {
    case 0: launch_boundary<double>(dv, sp, s); break;
    case 1: launch_boundary<float>(dv, sp, s); break;
    case 2: launch_boundary<__half>(dv, sp, s); break;
    default: launch_boundary<__nv_bfloat16>(dv, sp, s); break;
    }
}

// ---- overlapped steps: the near tiles -----------------------------------------

namespace {

// one listed near tile of the step a block (TILE_X threads, one cell each):
// the bulk kernel's arithmetic on the cells that are not listed
// (the same bits as any launch shape of it)
template <typename T>
__global__ void __launch_bounds__(TILE_X) near_bulk_kernel(const Device dv, const StepPtrs sp) {
    if ((int)blockIdx.x >= dv.near_count[sp.parity]) return;
    const int t = dv.near_list[sp.parity][blockIdx.x];
    const int ntx = (dv.dom.nx + TILE_X - 1) / TILE_X;
    const int row = t / ntx;
    const Blk bk{t % ntx, row % dv.dom.ny, row / dv.dom.ny, ntx, dv.dom.ny, dv.dom.nz};
    StepPtrs own = sp;
    own.far_skip = nullptr;
    bulk_body<T, 1, true, true>(dv, own, bk);
}

}  // namespace

void launch_near_bulk(const Device &dv, const StepPtrs &sp, cudaStream_t s) {
    const unsigned blocks = (unsigned)dv.near_cap;
    switch (dv.precision) {
    case 0: near_bulk_kernel<double><<<blocks, TILE_X, 0, s>>>(dv, sp); break;
    case 1: near_bulk_kernel<float><<<blocks, TILE_X, 0, s>>>(dv, sp); break;
    case 2: near_bulk_kernel<__half><<<blocks, TILE_X, 0, s>>>(dv, sp); break;
    default: near_bulk_kernel<__nv_bfloat16><<<blocks, TILE_X, 0, s>>>(dv, sp); break;
    }
}

// ---- batched launches (ensembles) ------------------------------------------

namespace {

template <typename T, int V, int MINB = 1>
void bulk_batch_launch(const Batch &bt, unsigned blocks, bool walls, cudaStream_t s) {
    if constexpr (sizeof(T) == 2 && V % 2 == 0) {
        if (walls) bulk16_batch<T, V, MINB, true><<<blocks, BULK_THREADS, 0, s>>>(bt);
        else bulk16_batch<T, V, MINB, false><<<blocks, BULK_THREADS, 0, s>>>(bt);
    } else {
        if (walls) bulk_batch<T, V, MINB, true><<<blocks, BULK_THREADS, 0, s>>>(bt);
        else bulk_batch<T, V, MINB, false><<<blocks, BULK_THREADS, 0, s>>>(bt);
    }
}

struct BatchShape {
    int precision, vec;
    void (*fn)(const Batch &, unsigned, bool, cudaStream_t);
};

// per precision, index 0 and 1 are one and two cells a thread (the
// untuned choice is 1, else 0), two cells with the registers capped for 3
// resident blocks an SM in FP32 (the compiler's own choice leaves room for
// two); the shapes after them cap the registers for 3 or 4 resident blocks
// (those that spill little at the cap)
const BatchShape kBatchShapes[] = {
    {0, 1, bulk_batch_launch<double, 1>},  {0, 2, bulk_batch_launch<double, 2>},
    {1, 1, bulk_batch_launch<float, 1>},   {1, 2, bulk_batch_launch<float, 2, 3>},
    {1, 4, bulk_batch_launch<float, 4>},   {1, 2, bulk_batch_launch<float, 2, 4>},
    {2, 1, bulk_batch_launch<__half, 1>},  {2, 2, bulk_batch_launch<__half, 2>},
    {2, 4, bulk_batch_launch<__half, 4>},  {2, 2, bulk_batch_launch<__half, 2, 4>},
    {2, 4, bulk_batch_launch<__half, 4, 3>},
    {3, 1, bulk_batch_launch<__nv_bfloat16, 1>}, {3, 2, bulk_batch_launch<__nv_bfloat16, 2>},
    {3, 4, bulk_batch_launch<__nv_bfloat16, 4>}, {3, 2, bulk_batch_launch<__nv_bfloat16, 2, 4>},
    {3, 4, bulk_batch_launch<__nv_bfloat16, 4, 3>},
};

const BatchShape *batch_shape(int precision, int i) {
    for (const BatchShape &b : kBatchShapes)
        if (b.precision == precision && i-- == 0) return &b;
    return nullptr;
}

}  // namespace

int batch_bulk_shape(int precision, int i) {
    const BatchShape *b = batch_shape(precision, i);
    return b ? b->vec : 0;
}

void batch_grid_cells(const Device &dv, int k, int variant, bool by_cell, int g[3]) {
    g[0] = g[1] = g[2] = 0;
    const Domain &d = dv.dom;
    if (k == BK_BOUNDARY && dv.nb > 0) {
        g[0] = boundary_blocks(dv, by_cell);
        g[1] = g[2] = 1;
    } else if (k == BK_BULK) {
        const BatchShape *b = batch_shape(dv.precision, variant);
        if (!b || d.nx % b->vec) return;
        // a z-plane's V-cell groups in row order (no lanes idle at row ends),
        // BATCH_PZ planes a block
        g[0] = (int)(((long long)(d.nx / b->vec) * d.ny + BULK_THREADS - 1) / BULK_THREADS);
        g[1] = 1;
        g[2] = (d.nz + BATCH_PZ - 1) / BATCH_PZ;
    }
}

template <typename T>
static void launch_boundary_batch(const Batch &bt, unsigned blocks, bool by_cell, cudaStream_t s) {
    if (by_cell) boundary_cells_batch<T><<<blocks, BOUNDARY_THREADS, 0, s>>>(bt);
    else boundary_batch<T><<<blocks, 32 * BOUNDARY_WARPS, 0, s>>>(bt);
}

void launch_batch_cells(int k, int variant, const Batch &bt, unsigned blocks, int precision, bool walls, bool by_cell,
                        cudaStream_t s) {
    if (blocks == 0) return;
    if (k == BK_BULK) {
        const BatchShape *b = batch_shape(precision, variant);
        if (b) b->fn(bt, blocks, walls, s);
        return;
    }
    switch (precision) {
    case 0: launch_boundary_batch<double>(bt, blocks, by_cell, s); break;
    case 1: launch_boundary_batch<float>(bt, blocks, by_cell, s); break;
    case 2: launch_boundary_batch<__half>(bt, blocks, by_cell, s); break;
    default: launch_boundary_batch<__nv_bfloat16>(bt, blocks, by_cell, s); break;
    }
}

}  // namespace lbm
