// collide_fix.cuh -- BGK collision of the FP64 store in 64-bit fixed point
// (arXiv:2006.12910 Sec. 2, Eqs. e.LB1, e.LB2).
//
// Why: FP64 instructions issue at about 2 lanes per clock and SM on this part,
// 64 times slower than integer ones, and the collision's 70 of them per node
// kept the FP64 pipe 87 % busy: 281 us for 2048x1024 nodes whose 302 MB take 45 us
// at the copy rate.  The populations of one node are numbers of one scale (a
// few per cent of rho0 up to rho0), so 64-bit integers in units of 2^-s with
// rho0 2^s in [2^60, 2^61) hold them with more digits than FP64 does: an addition
// is exact, a product of two such numbers is good to 1.3 units (three 32 x 32 ->
// 64-bit multiplies), where FP64 rounds the density to 2^8 units and the
// populations to 2^2 .. 2^6.  About 700 integer instructions a node: 281 -> 70 us
// a step at 2048x1024 (64 % issue, ALU pipe 63 %; 32 warps of 64 registers per
// SM, one node a lane; two nodes a lane held 12 warps and took 92 us), 256x64
// 7.75 -> 3.0 us.  One collision is off by 1.16e-17 rho0 rms a population, FP64
// arithmetic by 2.1e-17 (exact rational arithmetic as the measure).
//
// A node outside the range of the format is left to the FP64 collision: a
// population not in [2^52, 1.5 x 2^60) units before or [2^52, 2^62) after, a
// density not in [1.0625 x 2^59, 2^62), a momentum component of 2^59 or more
// (negative or vanishing populations, speeds of the order of the lattice
// speed, NaN).  Within these bounds no intermediate passes 2^63: the density sum
// is below 13.5 x 2^60 (a wrapped sign fails its check), the equilibria lie in
// (-0.39, 1.78) x 2^60, so the differences the relaxation shifts by two bits stay
// below 1.89 x 2^60.
#pragma once
#include "lbm_dev.cuh"

namespace lbmk {

// A 64-bit integer as hi * 2^32 + lo with lo in [-2^31, 2^31): every partial
// product is then a signed 32 x 32 multiply.
struct Halves {
    int32_t h, l;
};
__device__ __forceinline__ Halves halves(int64_t x) {
    const uint32_t l = (uint32_t)x;
    return Halves{(int32_t)(x >> 32) + (int32_t)(l >> 31), (int32_t)l};
}
__host__ __device__ constexpr Halves halves_of(int64_t x) {
    return Halves{(int32_t)((x >> 32) + (int64_t)(((uint64_t)x >> 31) & 1u)), (int32_t)(uint32_t)((uint64_t)x & 0xffffffffu)};
}
// c + x y / 2^64, rounded (without the product of the low halves, at most a
// quarter of a unit): three multiply-adds that accumulate 64 bits.
__device__ __forceinline__ int64_t mulhi(Halves x, Halves y, int64_t c = 0) {
    int64_t r;
    asm("{\n\t.reg .s64 m;\n\t"
        "mad.wide.s32 m, %1, %4, %6;\n\t"
        "mad.wide.s32 m, %2, %3, m;\n\t"
        "shr.s64 m, m, 32;\n\t"
        "add.s64 m, m, %5;\n\t"
        "mad.wide.s32 %0, %2, %4, m;\n\t}"
        : "=l"(r)
        : "r"(x.l), "r"(x.h), "r"(y.l), "r"(y.h), "l"(c), "l"(0x80000000ll));
    return r;
}

// Double -> units, exact; t collects the range check (unsigned maximum), from
// 2^52 units, the shift 0, to 1.5 x 2^60.
constexpr uint32_t FIX_RANGE = (8u << 20) + 0x80000u;
__device__ __forceinline__ int64_t to_fix(double f, int32_t e0, uint32_t& t) {
    const uint32_t h = (uint32_t)__double2hiint(f), l = (uint32_t)__double2loint(f);
    t = max(t, h - ((uint32_t)(e0 - 11) << 20));
    const uint32_t k = (h >> 20) - (uint32_t)(e0 - 11), m = (h & 0xFFFFFu) | 0x100000u;
    return (int64_t)(((uint64_t)__funnelshift_l(l, m, k) << 32) | (l << (k & 31u)));
}
// Units -> nearest double; t collects the range check, from 2^52 to 2^62.
__device__ __forceinline__ double from_fix(int64_t x, int32_t e0, uint32_t& t) {
    const uint32_t h = (uint32_t)((uint64_t)x >> 32);
    t = max(t, h - 0x100000u);
    const uint32_t p = 31u - (uint32_t)__clz((int)h), q = (p - 20u) & 31u;  // bits beyond the 53 kept
    const uint64_t r = (uint64_t)x + ((1u << q) >> 1);
    const uint32_t rh = (uint32_t)(r >> 32), rl = (uint32_t)r;
    return __hiloint2double((int)((rh >> q) + ((p + (uint32_t)e0 - 32u) << 20)), (int)__funnelshift_r(rl, rh, q));
}

// One node: f the pre-collision populations, out the post-collision ones when it
// returns true; false when the node is out of range.
__device__ __forceinline__ bool collide_fix(const double (&f)[9], double (&out)[9], const FixPrm& P) {
    uint32_t t = 0;
    int64_t g[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) g[i] = to_fix(f[i], P.e0, t);
    bool ok = t < FIX_RANGE;
    const int64_t a = g[1] + g[5] + g[8], b = g[3] + g[6] + g[7];
    const int64_t c = g[2] + g[5] + g[6], d = g[4] + g[7] + g[8];
    const int64_t rho = g[0] + g[2] + g[4] + a + b;
    int64_t mx = a - b, my = c - d;
    if (P.forced) {  // rho u = sum f e + tau rho g
        const Halves rh = halves(rho);
        mx = mulhi(rh, Halves{P.gxh, P.gxl}, mx);
        my = mulhi(rh, Halves{P.gyh, P.gyl}, my);
    }
    const uint32_t rhi = (uint32_t)((uint64_t)rho >> 32);
    ok = ok && rhi - 0x08800000u < 0x40000000u - 0x08800000u && (uint32_t)(mx >> 32) + 0x07FFFFF0u < 0x0FFFFFE0u &&
         (uint32_t)(my >> 32) + 0x07FFFFF0u < 0x0FFFFFE0u;
    // y = 2^62 / rho in units of 2^-60: y0, the hardware's FP32 reciprocal of the
    // leading 32 bits, is off by e = 1 - rho y0 (below 2^-21); 1 / rho is y0 times
    // the geometric series 1 / (1 - e), here 1 + e + e^2 (e^3 < 2^-63)
    const uint32_t y0 = __float2uint_rz(rcp_rho<float>((float)rhi) * 288230376151711744.0f);  // 2^58
    const int64_t e = (1ll << 60) - (int64_t)((((uint64_t)rhi * y0) << 2) + (((uint64_t)(uint32_t)rho * y0) >> 30));
    const int32_t eh = (int32_t)(e >> 16);
    const int64_t s = e + (int64_t)(((uint64_t)((int64_t)eh * eh)) >> 28);
    const int64_t y = ((int64_t)y0 << 32) + (int64_t)(((uint64_t)y0 * (uint32_t)s) >> 28) +
                      (int64_t)(int32_t)y0 * ((int32_t)(s >> 32) * 16);
    const Halves yh = halves(y), nx = halves(mx << 4), ny = halves(my << 4);
    const Halves ux = halves(mulhi(nx, yh)), uy = halves(mulhi(ny, yh));  // units of 2^-62
    // 4 m_a m_b / rho
    const int64_t qx = mulhi(nx, ux), qy = mulhi(ny, uy), qc = mulhi(nx, uy);
    const int64_t qs = qx + qy;
    // 1/9 and 3 x 1/9 as the FP64 weights are (2^64 of them), so that the
    // populations of a node sum to what FP64 weights make of its density
    constexpr Halves ninth = halves_of(0x1C71C71C71C71C00ll), third = halves_of(0x5555555555555400ll);
    const int64_t t9 = mulhi(halves(rho - (qs >> 2) - (qs >> 3)), ninth);  // (rho - 3/2 rho u.u) / 9
    const int64_t mx3 = mulhi(halves(mx), third), my3 = mulhi(halves(my), third);
    const int64_t hx = t9 + (qx >> 3), hy = t9 + (qy >> 3);  // omega_1 rho (1 + 9/2 u_a^2 - 3/2 u.u)
    const int64_t hd = (t9 >> 2) + (qs >> 5), hc = qc >> 4;
    const int64_t hp = hd + hc, hm = hd - hc, kp = (mx3 + my3) >> 2, km = (my3 - mx3) >> 2;
    const int64_t eq[9] = {t9 << 2, hx + mx3, hy + my3, hx - mx3, hy - my3, hp + kp, hm + km, hp - kp, hm - km};
    t = 0;
#pragma unroll
    for (int i = 0; i < 9; ++i)
        out[i] = from_fix(mulhi(halves((eq[i] - g[i]) << 2), Halves{P.wh, P.wl}, g[i]), P.e0, t);
    return ok && t < 0x40000000u - 0x100000u;
}

// The FP64 collision of a node collide_fix left (rare, so out of line).
static __device__ __noinline__ bool collide_f64(const DomDev& D, double* f) {
    double n9[9];
    const double none[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
#pragma unroll
    for (int i = 0; i < 9; ++i) n9[i] = f[i];
    const HotPrm<double> H = load_hot<double>(D);
    const double rho = collide_nodes<double, false, false, false>(n9, H, ExtPrm<double>{}, none, 0.0);
#pragma unroll
    for (int i = 0; i < 9; ++i) f[i] = n9[i];
    return rho_ok(rho);
}

}  // namespace lbmk
