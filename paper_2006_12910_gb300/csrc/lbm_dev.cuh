// lbm_dev.cuh -- device building blocks of the GB300 D2Q9 library: lattice
// constants, population storage kinds, the Philox4x32-10 generator and the
// per-node collision (arXiv:2006.12910 Secs. 2, 4, 5).
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "lbm_types.h"

namespace lbmk {

// ---------------------------------------------------------------------------
// D2Q9 lattice, Sec. 2: e0=(0,0); e1..e4 = (1,0),(0,1),(-1,0),(0,-1);
// e5..e8 = (1,1),(-1,1),(-1,-1),(1,-1); weights 4/9, 1/9, 1/36; c_s^2 = 1/3.
// Written as constexpr functions so fully unrolled loops fold them away.
// ---------------------------------------------------------------------------
__host__ __device__ constexpr int cx(int i) { return (i == 1 || i == 5 || i == 8) ? 1 : ((i == 3 || i == 6 || i == 7) ? -1 : 0); }
__host__ __device__ constexpr int cy(int i) { return (i == 2 || i == 5 || i == 6) ? 1 : ((i == 4 || i == 7 || i == 8) ? -1 : 0); }
__host__ __device__ constexpr int opp(int i) { return i == 0 ? 0 : (i <= 4 ? ((i + 1) % 4) + 1 : ((i - 3) % 4) + 5); }
__host__ __device__ constexpr double wgt(int i) { return i == 0 ? 4.0 / 9.0 : (i <= 4 ? 1.0 / 9.0 : 1.0 / 36.0); }

// Table 1 mode vectors e_ki (k = 3..8) for direction i, with |e_i|^2 = e2.
__host__ __device__ constexpr double mode_vec(int k, int i) {
    return k == 3 ? 3.0 * (cx(i) * cx(i) + cy(i) * cy(i)) - 2.0
         : k == 4 ? 2.0 * cx(i) * cx(i) - (cx(i) * cx(i) + cy(i) * cy(i))
         : k == 5 ? 1.0 * cx(i) * cy(i)
         : k == 6 ? (3.0 * (cx(i) * cx(i) + cy(i) * cy(i)) - 4.0) * cx(i)
         : k == 7 ? (3.0 * (cx(i) * cx(i) + cy(i) * cy(i)) - 4.0) * cy(i)
         : 9.0 * (cx(i) * cx(i) + cy(i) * cy(i)) * (cx(i) * cx(i) + cy(i) * cy(i))
               - 15.0 * (cx(i) * cx(i) + cy(i) * cy(i)) + 2.0;
}
// 1/sqrt(w_k) for the Table 1 lengths w_3..w_8 = 4, 4/9, 1/9, 2/3, 2/3, 16.
__host__ __device__ constexpr double inv_sqrt_wk(int k) {
    return k == 3 ? 0.5 : k == 4 ? 1.5 : k == 5 ? 3.0 : (k == 6 || k == 7) ? 1.2247448713915890491 : 0.25;
}
// Noise weight of mode k in direction i: omega_i chi_ki = omega_i e_ki / sqrt(w_k) (Eq. NP2).
__host__ __device__ constexpr double noise_coef(int i, int k) { return wgt(i) * mode_vec(k, i) * inv_sqrt_wk(k); }

// ---------------------------------------------------------------------------
// Arithmetic of the collision on W = double, float or float2 (two nodes at
// once in the packed FP32 instructions of this architecture).  Every
// multiply-add is written out, so that a node's result is the same bits
// whichever kernel, and whichever form, computes it.
// ---------------------------------------------------------------------------
__device__ __forceinline__ double vadd(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ double vsub(double a, double b) { return __dsub_rn(a, b); }
__device__ __forceinline__ double vmul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ double vfma(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ float vadd(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float vsub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float vmul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float vfma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ float2 vadd(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 vmul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 vfma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 vsub(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.0f, -1.0f), a); }
// Components of W, and the same value in all of them.
template <class W> struct Vec;
template <> struct Vec<double> {
    typedef double A;
    static constexpr int N = 1;
    static __device__ __forceinline__ double all(double x) { return x; }
    static __device__ __forceinline__ double get(const double& w, int) { return w; }
    static __device__ __forceinline__ void set(double& w, int, double x) { w = x; }
};
template <> struct Vec<float> {
    typedef float A;
    static constexpr int N = 1;
    static __device__ __forceinline__ float all(float x) { return x; }
    static __device__ __forceinline__ float get(const float& w, int) { return w; }
    static __device__ __forceinline__ void set(float& w, int, float x) { w = x; }
};
template <> struct Vec<float2> {
    typedef float A;
    static constexpr int N = 2;
    static __device__ __forceinline__ float2 all(float x) { return make_float2(x, x); }
    static __device__ __forceinline__ float get(const float2& w, int k) { return k ? w.y : w.x; }
    static __device__ __forceinline__ void set(float2& w, int k, float x) {
        if (k) w.y = x;
        else w.x = x;
    }
};

// ---------------------------------------------------------------------------
// Population storage kinds.  V = consecutive nodes of one row a lane owns in
// the register stream-collide kernel (one load or store of V*sizeof(T) = 8 or 16
// bytes per plane).  MINB / MINB_EXT: CTAs of 128 threads the
// register kernel asks to keep resident per SM (plain BGK / with noise or
// the power law), which caps its registers per thread.
// ---------------------------------------------------------------------------
// FP64: one node a lane.  The pull needs no edge elements then, and the
// fixed-point collision of a node leaves room for more warps.
struct StF64 {
    typedef double T; typedef double A;
    static constexpr int V = 1; static constexpr bool SHIFT = false; static constexpr bool SCALED = false;
    static constexpr int KIND = 0;
    static constexpr int MINB = 8, MINB_EXT = 4;
};
struct StF32 {
    typedef float T; typedef float A;
    static constexpr int V = 4; static constexpr bool SHIFT = false; static constexpr bool SCALED = false;
    static constexpr int KIND = 1;
    static constexpr int MINB = 5, MINB_EXT = 4;
};
struct StF32S {
    typedef float T; typedef float A;
    static constexpr int V = 4; static constexpr bool SHIFT = true; static constexpr bool SCALED = false;
    static constexpr int KIND = 2;
    static constexpr int MINB = 5, MINB_EXT = 4;
};
// Half-precision kinds take 8-byte vectors (4 nodes per lane): the register
// footprint of an FP32 lane, so five CTAs fit per SM.
struct StF16S {
    typedef __half T; typedef float A;
    static constexpr int V = 4; static constexpr bool SHIFT = true; static constexpr bool SCALED = true;
    static constexpr int KIND = 3;
    static constexpr int MINB = 5, MINB_EXT = 4;
};
struct StBF16S {
    typedef __nv_bfloat16 T; typedef float A;
    static constexpr int V = 4; static constexpr bool SHIFT = true; static constexpr bool SCALED = true;
    static constexpr int KIND = 4;
    static constexpr int MINB = 5, MINB_EXT = 4;
};

__device__ __forceinline__ double to_a(double v, double) { return v; }
__device__ __forceinline__ float to_a(float v, float) { return v; }
__device__ __forceinline__ float to_a(__half v, float inv) { return __half2float(v) * inv; }
__device__ __forceinline__ float to_a(__nv_bfloat16 v, float inv) { return __bfloat162float(v) * inv; }
__device__ __forceinline__ void from_a(double v, double, double& o) { o = v; }
__device__ __forceinline__ void from_a(float v, float, float& o) { o = v; }
__device__ __forceinline__ void from_a(float v, float s, __half& o) { o = __float2half_rn(v * s); }
__device__ __forceinline__ void from_a(float v, float s, __nv_bfloat16& o) { o = __float2bfloat16_rn(v * s); }

template <int B> struct VecOf;
template <> struct VecOf<8> { typedef uint2 type; };
template <> struct VecOf<16> { typedef uint4 type; };
__device__ __forceinline__ uint32_t pack2(float a, float b, __half) {
    const __half2 h = __floats2half2_rn(a, b);
    return *reinterpret_cast<const uint32_t*>(&h);
}
__device__ __forceinline__ uint32_t pack2(float a, float b, __nv_bfloat16) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<const uint32_t*>(&h);
}
// A load of populations.  Not through the read-only path (__ldg, ld.global.nc):
// that one is for memory nobody writes while the grid lives, and a programmatic
// dependent is resident while the launch before it still writes the arena.
// Volatile, so that it stays behind the wait for that launch; it is written as
// instructions because that constrains the code around it least (us a step with
// __ldg / plain dereferences / these: porous 2048x1024 33.5 / 33.9 / 32.8, with
// noise and tau* 56.8 / 58.4 / 56.6, 4096x2048 without particles 105.2 / 105.8 / 102.4).
__device__ __forceinline__ void load_pop(uint4& v, const void* p) {
    asm volatile("ld.global.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
}
__device__ __forceinline__ void load_pop(uint2& v, const void* p) {
    asm volatile("ld.global.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "l"(p));
}
__device__ __forceinline__ void load_pop(double& v, const void* p) {
    asm volatile("ld.global.f64 %0, [%1];" : "=d"(v) : "l"(p));
}
__device__ __forceinline__ void load_pop(float& v, const void* p) {
    asm volatile("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(p));
}
__device__ __forceinline__ void load_pop(__half& v, const void* p) {
    uint16_t u;
    asm volatile("ld.global.u16 %0, [%1];" : "=h"(u) : "l"(p));
    v = __ushort_as_half(u);
}
__device__ __forceinline__ void load_pop(__nv_bfloat16& v, const void* p) {
    uint16_t u;
    asm volatile("ld.global.u16 %0, [%1];" : "=h"(u) : "l"(p));
    v = __ushort_as_bfloat16(u);
}
// The same past the L1, for data read once (the moments of 2048x1024 nodes in FP32,
// launches back to back: 17.6 us, 19.3 through the L1, 17.6 with __ldg).
__device__ __forceinline__ void load_once(uint4& v, const void* p) {
    asm volatile("ld.global.cg.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
}
__device__ __forceinline__ void load_once(uint2& v, const void* p) {
    asm volatile("ld.global.cg.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "l"(p));
}
// Vector load of NV consecutive elements: one 8- or 16-byte access.
template <class S, int NV>
__device__ __forceinline__ void load_vec(const typename S::T* p, typename S::A (&out)[NV], typename S::A inv) {
    typedef typename VecOf<NV * sizeof(typename S::T)>::type VT;
    union { VT u; typename S::T t[NV]; } r;
    load_once(r.u, p);
#pragma unroll
    for (int k = 0; k < NV; ++k) out[k] = to_a(r.t[k], inv);
}
// A chunk as the collision takes it: V / Vec<W>::N vectors W (half-precision
// kinds in their scaled units), one 8- or 16-byte load or store.
template <class S> struct ChunkOf { typedef float2 W; static constexpr int N = S::V / 2; };
template <> struct ChunkOf<StF64> { typedef double W; static constexpr int N = StF64::V; };
template <class S>
struct Chunk {  // as loaded; get() converts
    typedef typename VecOf<S::V * sizeof(typename S::T)>::type VT;
    union { VT u; typename S::T t[S::V]; };
    __device__ __forceinline__ Chunk() {}
    __device__ __forceinline__ void load(const void* p) { load_pop(u, p); }
    __device__ __forceinline__ void load_shared(const void* p) { u = *static_cast<const VT*>(p); }
    __device__ __forceinline__ void get(typename ChunkOf<S>::W (&v)[ChunkOf<S>::N]) const {
        constexpr int N = Vec<typename ChunkOf<S>::W>::N;
#pragma unroll
        for (int k = 0; k < S::V; ++k)
            Vec<typename ChunkOf<S>::W>::set(v[k / N], k % N, to_a(t[k], (typename S::A)1));
    }
};
template <class S>
__device__ __forceinline__ void store_chunk(void* p, const typename ChunkOf<S>::W (&v)[ChunkOf<S>::N]) {
    if constexpr (sizeof(typename S::T) == 8) *static_cast<double*>(p) = v[0];
    else if constexpr (sizeof(typename S::T) == 4) *static_cast<float4*>(p) = make_float4(v[0].x, v[0].y, v[1].x, v[1].y);
    else *static_cast<uint2*>(p) = make_uint2(pack2(v[0].x, v[0].y, typename S::T()), pack2(v[1].x, v[1].y, typename S::T()));
}
// One element, by a plain dereference: in the rare branches that use it the
// volatile form costs the loops around them registers (noise and tau* 59.6 us).
template <class S>
__device__ __forceinline__ typename S::A load_one(const typename S::T* p, typename S::A inv) {
    return to_a(*p, inv);
}

// ---------------------------------------------------------------------------
// Noise of Sec. 4: counter-based random numbers, uniforms, normal deviates.
// ---------------------------------------------------------------------------
// Uniform in (0,1) from the top 23 bits, ((x >> 9) + 1/2) / 2^23, exact in FP64
// and FP32.  FP32: the 23 bits as the mantissa of a number in [1, 2) (one
// funnel shift), minus 1, plus 2^-24 -- both steps exact, so this is the same
// value with no integer to float conversion.
__device__ __forceinline__ float mant23(uint32_t x) { return __uint_as_float(__funnelshift_r(x, 0x7Fu, 9)); }
__device__ __forceinline__ double uni23d(uint32_t x) { return ((double)(x >> 9) + 0.5) * 1.1920928955078125e-07; }

// Theta_3..Theta_8 of Eq. NP2 for one node: counter (node, step, draw, domain).
// Philox4x32-10 (Salmon, Moraes, Dror & Shaw, SC'11): ten rounds of two
// 32x32 -> 64-bit multiplies, key bumped by the Weyl constants between rounds.
// The two draws of one node (counter words 2 = 0 and 1) run with their rounds
// interleaved, so that they share the key schedule (and the first round's
// products, which the compiler finds).
__device__ __forceinline__ void philox4x32_10_x2(uint4& a, uint4& b, uint32_t k0, uint32_t k1) {
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        if (r) { k0 += 0x9E3779B9u; k1 += 0xBB67AE85u; }
        const uint64_t a0 = (uint64_t)a.x * 0xD2511F53u, a1 = (uint64_t)a.z * 0xCD9E8D57u;
        const uint64_t b0 = (uint64_t)b.x * 0xD2511F53u, b1 = (uint64_t)b.z * 0xCD9E8D57u;
        a = make_uint4((uint32_t)(a1 >> 32) ^ a.y ^ k0, (uint32_t)a1, (uint32_t)(a0 >> 32) ^ a.w ^ k1, (uint32_t)a0);
        b = make_uint4((uint32_t)(b1 >> 32) ^ b.y ^ k0, (uint32_t)b1, (uint32_t)(b0 >> 32) ^ b.w ^ k1, (uint32_t)b0);
    }
}

// Reciprocal square root by the hardware approximation (FP32, x > 0; relative
// error at most 2^-22.9).
__device__ __forceinline__ float rsqrt_hw(float x) {
    float y;
    asm("rsqrt.approx.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Square root by Heron's method, r + (x - r^2) / (2 r) from r = x y with
// y ~ 1 / sqrt(x) above, which also stands for 1 / r.  If r is off by e
// (below 2^-22.3 of it) and y by n, the step leaves e^2 / 2 + e n < 2^-44 and its
// own rounding: relative error at most 2^-24 (1 + 2^-20) for x in [2^-100, 2^100];
// checked against FP64 on every mantissa.  0 where x is not positive.
// sqrtf, good to 2^-24, tests its argument for ranges that cannot occur here:
// with it the noise of 96 domains takes 188 us a step against 169, and is off by
// the same 1.824e-7 of its rms.
template <class W>
__device__ __forceinline__ W sqrt_heron(W x) {
    typedef Vec<W> K;
    W y;
#pragma unroll
    for (int k = 0; k < K::N; ++k) K::set(y, k, K::get(x, k) > 0.0f ? rsqrt_hw(K::get(x, k)) : 0.0f);
    const W r = vmul(x, y);
    return vfma(vfma(vmul(K::all(-1.0f), r), r, x), vmul(K::all(0.5f), y), r);
}
// -sqrt(-nx) for nx < 0, y ~ 1 / sqrt(-nx): the same step (the signs fall into place).
template <class W>
__device__ __forceinline__ W neg_sqrt(W nx, W y) {
    const W q = vmul(nx, y);
    return vfma(vfma(q, q, nx), vmul(Vec<W>::all(0.5f), y), q);
}
// 2 ln u of the uniform with mantissa bits m in [1, 2) as above: u = 2^e (1 + f)
// with 1 + f in [sqrt(1/2), sqrt 2), ln(1 + f) = f + f^2 (f p(f) - 1/2), p the
// degree-7 minimax polynomial of (ln(1 + f) - f + f^2 / 2) / f^3 on that interval
// with weight f^2 (Remez exchange).  Checked on the CPU for all 2^23 values:
// relative error of ln u at most 1.37 x 2^-24.  The noise variant is bound by
// arithmetic: in packed pairs this and the square root below take half the
// instructions of logf and sqrtf (2048x1024 shifted FP32 with noise: 37.5 ->
// 28.7 us a step, 1,803 -> 1,230 instructions an item with the packed
// collision).  Against 64 bits the noise of one node is off by 1.620e-7 of its
// rms (1.625e-7 with logf and sqrtf), set by the hardware sine and cosine.
template <class W>
__device__ __forceinline__ W two_ln_uniform(W m) {
    typedef Vec<W> K;
    const W u = vadd(vadd(m, K::all(-1.0f)), K::all(5.9604644775390625e-08f));
    W r, e;
#pragma unroll
    for (int k = 0; k < K::N; ++k) {
        const uint32_t i = __float_as_uint(K::get(u, k));
        const uint32_t t = (i + (64u << 23) - 0x3F3504F3u) >> 23;  // e + 64 (0x3F3504F3: sqrt(1/2))
        K::set(r, k, __uint_as_float(i + ((64u - t) << 23)));
        K::set(e, k, __uint_as_float(0x4B000000u + t));  // 2^23 + 64 + e
    }
    const W f = vadd(r, K::all(-1.0f)), ef = vadd(e, K::all(-8388672.0f));
    W p = K::all(-0.07859606295824051f);
    p = vfma(p, f, K::all(0.12881644070148468f));
    p = vfma(p, f, K::all(-0.13128754496574402f));
    p = vfma(p, f, K::all(0.14181192219257355f));
    p = vfma(p, f, K::all(-0.16624553501605988f));
    p = vfma(p, f, K::all(0.2000228613615036f));
    p = vfma(p, f, K::all(-0.25000810623168945f));
    p = vfma(p, f, K::all(0.33333316445350647f));
    const W l = vfma(ef, K::all(0.693147180559945309f), vfma(vmul(f, f), vfma(p, f, K::all(-0.5f)), f));
    return vadd(l, l);
}

// Box-Muller pair of the uniforms a, b given by their mantissas: radius
// sqrt(-2 ln a), the angle
// 2 pi b taken as pi + 2 pi (b - 1/2) with b - 1/2 exact, so the hardware sine /
// cosine work inside [-pi, pi] (absolute error about 4e-7, far inside the noise
// tolerance).
template <class W>
__device__ __forceinline__ void box_muller(W ma, W mb, W& z0, W& z1) {
    typedef Vec<W> K;
    const W nx = two_ln_uniform(ma);  // -x, x = r^2
    const W ang = vmul(vadd(vadd(mb, K::all(-1.5f)), K::all(5.9604644775390625e-08f)), K::all(6.28318530717958647692f));
    W y, s, c;
#pragma unroll
    for (int k = 0; k < K::N; ++k) {
        K::set(y, k, rsqrt_hw(-K::get(nx, k)));
        float sk, ck;
        __sincosf(K::get(ang, k), &sk, &ck);
        K::set(s, k, sk);
        K::set(c, k, ck);
    }
    const W nr = neg_sqrt(nx, y);
    z0 = vmul(nr, c);
    z1 = vmul(nr, s);
}
__device__ __forceinline__ void box_muller(double a, double b, double& z0, double& z1) {
    const double r = sqrt(-2.0 * log(a));
    double s, c;
    sincospi(2.0 * b, &s, &c);
    z0 = r * c;
    z1 = r * s;
}

// The six normals of the nodes of W, the first with index `node`.
template <class W>
__device__ __forceinline__ void thetas(uint32_t node, uint32_t step, uint32_t dom_id, uint64_t seed, W (&th)[6]) {
    typedef Vec<W> K;
    uint4 r0[K::N], r1[K::N];
#pragma unroll
    for (int k = 0; k < K::N; ++k) {
        r0[k] = make_uint4(node + k, step, 0u, dom_id);
        r1[k] = make_uint4(node + k, step, 1u, dom_id);
        philox4x32_10_x2(r0[k], r1[k], (uint32_t)seed, (uint32_t)(seed >> 32));
    }
    if constexpr (sizeof(typename K::A) == 8) {
        box_muller(uni23d(r0[0].x), uni23d(r0[0].y), th[0], th[1]);
        box_muller(uni23d(r0[0].z), uni23d(r0[0].w), th[2], th[3]);
        box_muller(uni23d(r1[0].x), uni23d(r1[0].y), th[4], th[5]);
    } else {
        W m[6];
#pragma unroll
        for (int k = 0; k < K::N; ++k) {
            const uint32_t x[6] = {r0[k].x, r0[k].y, r0[k].z, r0[k].w, r1[k].x, r1[k].y};
#pragma unroll
            for (int j = 0; j < 6; ++j) K::set(m[j], k, mant23(x[j]));
        }
#pragma unroll
        for (int j = 0; j < 6; j += 2) box_muller(m[j], m[j + 1], th[j], th[j + 1]);
    }
}

// Noise of Eq. NP2 added to the populations: f_i += amp omega_i sum_k chi_ki
// Theta_k, with the sums over the modes that have equal weights on a class of
// directions taken once (33 operations; 47 written out mode by mode).
template <class W>
__device__ __forceinline__ void add_noise(W (&f)[9], W amp, const W (&th)[6]) {
    typedef Vec<W> K;
    typedef typename K::A A;
    static_assert(noise_coef(1, 3) == noise_coef(5, 3) && noise_coef(2, 4) == -noise_coef(1, 4) &&
                      noise_coef(6, 5) == -noise_coef(5, 5) && noise_coef(2, 8) == noise_coef(1, 8) &&
                      noise_coef(6, 8) == noise_coef(5, 8) && noise_coef(2, 7) == noise_coef(1, 6) &&
                      noise_coef(5, 7) == noise_coef(5, 6), "Table 1 weights of the directions of one class");
    W t[6];
#pragma unroll
    for (int k = 0; k < 6; ++k) t[k] = vmul(amp, th[k]);
    f[0] = vfma(K::all((A)noise_coef(0, 8)), t[5], vfma(K::all((A)noise_coef(0, 3)), t[0], f[0]));
    const W s3 = vmul(K::all((A)noise_coef(1, 3)), t[0]);
    const W ax = vfma(K::all((A)noise_coef(1, 8)), t[5], s3), dg = vfma(K::all((A)noise_coef(5, 8)), t[5], s3);
    const W p = vfma(K::all((A)noise_coef(1, 4)), t[1], ax), q = vfma(K::all((A)noise_coef(2, 4)), t[1], ax);
    const W d = vfma(K::all((A)noise_coef(5, 5)), t[2], dg), g = vfma(K::all((A)noise_coef(6, 5)), t[2], dg);
    f[1] = vadd(f[1], vfma(K::all((A)noise_coef(1, 6)), t[3], p));
    f[3] = vadd(f[3], vfma(K::all((A)noise_coef(3, 6)), t[3], p));
    f[2] = vadd(f[2], vfma(K::all((A)noise_coef(2, 7)), t[4], q));
    f[4] = vadd(f[4], vfma(K::all((A)noise_coef(4, 7)), t[4], q));
    const W e = vadd(t[3], t[4]), h = vsub(t[3], t[4]);
    f[5] = vadd(f[5], vfma(K::all((A)noise_coef(5, 6)), e, d));
    f[7] = vadd(f[7], vfma(K::all((A)noise_coef(7, 6)), e, d));
    f[8] = vadd(f[8], vfma(K::all((A)noise_coef(8, 6)), h, g));
    f[6] = vadd(f[6], vfma(K::all((A)noise_coef(6, 6)), h, g));
}

// ---------------------------------------------------------------------------
// Per-domain parameters in the arithmetic type (no FP64 <-> FP32 conversion in
// the collision).  HotPrm (lbm_types.h) holds what every node needs and is
// read with 16-byte loads; ExtPrm holds what only the power-law, noise or
// Zou-He nodes need and is read only by those variants.
// ---------------------------------------------------------------------------
template <typename A> __device__ __forceinline__ HotPrm<A> load_hot(const DomDev& D);
template <> __device__ __forceinline__ HotPrm<float> load_hot<float>(const DomDev& D) {
    const float4* p = reinterpret_cast<const float4*>(&D.hot_f);
    const float4 a = __ldg(p), b = __ldg(p + 1);
    HotPrm<float> H;
    H.omega = a.x; H.om = a.y; H.tgx = a.z; H.tgy = a.w;
    H.rho0 = b.x; H.scale = b.y; H.inv_scale = b.z; H.pad = b.w;
    return H;
}
// The same from a descriptor held in the launch parameters.
template <typename A> __device__ __forceinline__ HotPrm<A> param_hot(const DomDev& D);
template <> __device__ __forceinline__ HotPrm<float> param_hot<float>(const DomDev& D) { return D.hot_f; }
template <> __device__ __forceinline__ HotPrm<double> param_hot<double>(const DomDev& D) { return D.hot_d; }
template <> __device__ __forceinline__ HotPrm<double> load_hot<double>(const DomDev& D) {
    const double2* p = reinterpret_cast<const double2*>(&D.hot_d);
    const double2 a = __ldg(p), b = __ldg(p + 1), c = __ldg(p + 2), d = __ldg(p + 3);
    HotPrm<double> H;
    H.omega = a.x; H.om = a.y; H.tgx = b.x; H.tgy = b.y;
    H.rho0 = c.x; H.scale = c.y; H.inv_scale = d.x; H.pad = d.y;
    return H;
}

__device__ __forceinline__ FixPrm load_fix(const DomDev& D) {
    const int4* p = reinterpret_cast<const int4*>(&D.fix);
    const int4 a = __ldg(p), b = __ldg(p + 1), c = __ldg(p + 2);
    return FixPrm{a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w, c.x, c.y, c.z, c.w};
}

template <typename A>
struct ExtPrm {
    A gx, gy, kT, var, var_lo, xi, n, tmin, tmax, tmin_pow, tmax_pow;
    int n_is_one;
    uint32_t dom_id;
    uint64_t seed;
};
template <typename A, bool NOISE, bool PL>
__device__ __forceinline__ ExtPrm<A> load_ext(const DomDev& D) {
    ExtPrm<A> X{};
    const bool f = sizeof(A) == 4;
    if (PL) {
        X.gx = (A)(f ? D.gx_f : D.gx); X.gy = (A)(f ? D.gy_f : D.gy);
        X.xi = (A)(f ? D.xi_pl_f : D.xi_pl); X.n = (A)(f ? D.n_pl_f : D.n_pl);
        X.tmin = (A)(f ? D.tau_min_f : D.tau_min); X.tmax = (A)(f ? D.tau_max_f : D.tau_max);
        X.tmin_pow = (A)(f ? D.tmin_pow_f : D.tmin_pow); X.tmax_pow = (A)(f ? D.tmax_pow_f : D.tmax_pow);
        X.n_is_one = D.n_is_one;
    }
    if (NOISE) {
        X.kT = (A)(f ? D.kT_f : D.kT);
        X.var = (A)(f ? D.var_f : D.var);  // PL: 3 kT alone
        X.var_lo = (A)(f ? D.var_lo_f : 0.0);
        X.dom_id = D.domain_id;
        X.seed = D.seed;
    }
    return X;
}

// Reciprocal of the density: FP32 takes the hardware approximation (relative
// error below 2^-22, far inside the FP32 path's tolerance); FP64 divides.
template <typename A> __device__ __forceinline__ A rcp_rho(A r);
template <> __device__ __forceinline__ float rcp_rho<float>(float r) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(r));
    return y;
}
template <> __device__ __forceinline__ double rcp_rho<double>(double r) { return 1.0 / r; }

// ---------------------------------------------------------------------------
// Power-law relaxation time, Sec. 5.  The shear rate of Eq. nn2 with Pi_D of
// Eq. nn3 taken from the Chapman-Enskog strain -Pi_neq / (2 rho c_s^2 tau) is
// A / tau, A = 3 sqrt|Pi_xy^2 - Pi_xx Pi_yy| / rho; nu* = xi (A/tau)^(n-1)
// (nn4, kappa = 2^(n-1)) and tau = 1/2 + 3 nu*.  g(t) = t - 1/2 - c t^(1-n),
// c = 3 xi A^(n-1), is convex for n < 1 and concave for n > 1, so Newton from
// the bracket end where g > 0 (n < 1) or g < 0 (n > 1) converges monotonically.
// ---------------------------------------------------------------------------
// FP64: one node, exact operations, converged to 10^-15.
__device__ __forceinline__ double solve_tau_f64(double astr, const ExtPrm<double>& P) {
    const double n = P.n, tmin = P.tmin, tmax = P.tmax;
    if (P.n_is_one) {
        const double t = 0.5 + 3.0 * P.xi;
        return t < tmin ? tmin : (t > tmax ? tmax : t);
    }
    if (!(astr > 0.0)) return n < 1.0 ? tmax : tmin;
    const double om = 1.0 - n;
    const double c = 3.0 * P.xi * exp2((n - 1.0) * log2(astr));
    if (tmin - 0.5 - c * P.tmin_pow >= 0.0) return tmin;
    if (tmax - 0.5 - c * P.tmax_pow <= 0.0) return tmax;
    double t = n < 1.0 ? tmax : tmin;
#pragma unroll 1
    for (int it = 0; it < 60; ++it) {
        const double p = exp2(om * log2(t));
        const double g = t - 0.5 - c * p;
        const double dg = 1.0 - c * om * p / t;
        double tn = t - g / dg;
        tn = tn < tmin ? tmin : (tn > tmax ? tmax : tn);
        const double dt = tn - t;
        t = tn;
        if (fabs(dt) <= 1e-15 * t) break;
    }
    return t;
}
template <int NN>
__device__ __forceinline__ void solve_taus(const double (&astr)[NN], const ExtPrm<double>& P, double (&tau)[NN]) {
#pragma unroll
    for (int k = 0; k < NN; ++k) tau[k] = solve_tau_f64(astr[k], P);
}

// FP32: the hardware base-2 logarithm (x > 0 here: a strain or a relaxation
// time).
__device__ __forceinline__ float pow_f32(float x, float e) { return exp2f(e * __log2f(x)); }

// FP32: the same iteration on NN nodes in step, with the fast division and to
// 2 10^-7, so that their logarithms, exponentials and divisions overlap and a
// warp runs as many iterations as its slowest node needs once, not node after
// node (power law n = 0.75, 2048x1024 shifted FP32: 36.4 -> 30.8 us a step).  A
// node's values do not depend on the others in step with it; where the strain
// is small a last-place difference of tau* grows by 10^3 within 100 steps, so
// the order of its roundings is kept.  (Newton from a near start, three
// evaluations a node, took 27.0 us and lost that.)
template <int NN>
__device__ __forceinline__ void solve_taus(const float (&astr)[NN], const ExtPrm<float>& P, float (&tau)[NN]) {
    const float n = P.n, tmin = P.tmin, tmax = P.tmax, om = 1.0f - n;
    float c[NN];
    bool open[NN], any = false;
#pragma unroll
    for (int k = 0; k < NN; ++k) {
        c[k] = __fmul_rn(3.0f * P.xi, pow_f32(astr[k], n - 1.0f));
        const bool low = astr[k] > 0.0f ? tmin - 0.5f - c[k] * P.tmin_pow >= 0.0f : n >= 1.0f;
        const bool high = astr[k] > 0.0f ? tmax - 0.5f - c[k] * P.tmax_pow <= 0.0f : n < 1.0f;
        if (P.n_is_one) tau[k] = fminf(fmaxf(0.5f + 3.0f * P.xi, tmin), tmax);
        else tau[k] = low ? tmin : (high ? tmax : (n < 1.0f ? tmax : tmin));
        open[k] = !P.n_is_one && !low && !high;
        any |= open[k];
    }
#pragma unroll 1
    for (int it = 0; any && it < 60; ++it) {
        any = false;
        float p[NN];
#pragma unroll
        for (int k = 0; k < NN; ++k) p[k] = pow_f32(tau[k], om);
#pragma unroll
        for (int k = 0; k < NN; ++k) {
            const float t = tau[k];
            const float g = __fmaf_rn(-c[k], p[k], t - 0.5f);
            const float dg = 1.0f - __fdividef(__fmul_rn(__fmul_rn(c[k], om), p[k]), t);
            const float tn = fminf(fmaxf(t - __fdividef(g, dg), tmin), tmax);
            if (open[k]) {
                tau[k] = tn;
                open[k] = !(fabsf(tn - t) <= 2e-7f * t);
                any |= open[k];
            }
        }
    }
}

// ---------------------------------------------------------------------------
// Collision of one node (Eq. e.LB1 right-hand side, Eq. e.LB2 equilibrium,
// rho u = sum f e + tau rho g, optional tau* of Eq. nn5 and noise of NP1-NP2).
// f holds the pre-collision populations, shifted by omega_i rho0 when SHIFT;
// on return it holds the post-collision values in the same units.
// Arranged for few operations, with omega = 1/tau and
// p_i = 3 e.u + 9/2 (e.u)^2 - 3/2 u.u; the pair (i, opp(i)) shares
// 9/2 (e.u)^2 - 3/2 u.u and 3 e.u.  Shifted stores (values f - w_i rho0, of
// the size of the non-equilibrium part) relax as
//   f_i' = (1 - omega) f_i + w_i (B + R p_i),  R = omega rho, B = omega (rho - rho0);
// unshifted stores (values ~ w_i) keep the difference form
//   f_i' = f_i + omega (w_i rho (1 + p_i) - f_i),
// whose rounding error stays at the scale of f_i rather than of omega f_i.
// Returns false when rho is not a positive finite number.
// ---------------------------------------------------------------------------
// RI, RO: which product of om f + w h is rounded first, om f or (false) w h, for
// fi and fo.
template <class W, bool SHIFT, bool RI, bool RO>
__device__ __forceinline__ void relax_pair(W& fi, W& fo, W e, typename Vec<W>::A w, W nusq, W R, W R3, W nR3, W B, W om,
                                           W nomega) {
    typedef Vec<W> K;
    typedef typename K::A A;
    const W q = vfma(vmul(K::all((A)4.5), e), e, nusq);
    const W h = vfma(R, q, B);
    const W hp = vfma(R3, e, h), hm = vfma(nR3, e, h);
    if (SHIFT) {
        fi = RI ? vfma(K::all(w), hp, vmul(om, fi)) : vfma(om, fi, vmul(K::all(w), hp));
        fo = RO ? vfma(K::all(w), hm, vmul(om, fo)) : vfma(om, fo, vmul(K::all(w), hm));
    } else {  // here R = rho, R3 = 3 rho, B = rho
        fi = vfma(nomega, vfma(K::all(-w), hp, fi), fi);
        fo = vfma(nomega, vfma(K::all(-w), hm, fo), fo);
    }
}

// True when rho is a positive finite number (below 1e30), from its bits: the
// FP64 pipe is the scarce one.
__device__ __forceinline__ bool rho_ok(float rho) { return __float_as_uint(rho) - 1u < 0x7149F2CAu - 1u; }  // 1e30f
__device__ __forceinline__ bool rho_ok(double rho) {
    return (unsigned long long)__double_as_longlong(rho) - 1ull < 0x46293E5939A08CEAull - 1ull;  // 1e30
}

// The strain A = 3 sqrt|Pi_xy^2 - Pi_xx Pi_yy| / rho of the nodes of W, from
// populations as collide_nodes takes them.
template <class W, bool SHIFT, bool SC>
__device__ __forceinline__ W strain(const W (&f)[9], const HotPrm<typename Vec<W>::A>& H) {
    typedef Vec<W> K;
    typedef typename K::A A;
    const W a = vadd(vadd(f[1], f[5]), f[8]), b = vadd(vadd(f[3], f[6]), f[7]);
    const W c = vadd(vadd(f[2], f[5]), f[6]), d = vadd(vadd(f[4], f[7]), f[8]);
    W s = vadd(vadd(f[0], vadd(f[2], f[4])), vadd(a, b)), jx = vsub(a, b), jy = vsub(c, d);
    W ab = vadd(a, b), cd = vadd(c, d), sxy = vsub(vadd(f[5], f[7]), vadd(f[6], f[8]));
    if (SC) {  // unscaled
        const W u1 = K::all(H.inv_scale);
        s = vmul(s, u1);
        jx = vmul(jx, u1);
        jy = vmul(jy, u1);
        ab = vmul(ab, u1);
        cd = vmul(cd, u1);
        sxy = vmul(sxy, u1);
    }
    const W rho = SHIFT ? vadd(K::all(H.rho0), s) : s;
    W irho, r;
#pragma unroll
    for (int k = 0; k < K::N; ++k) K::set(irho, k, rcp_rho<A>(K::get(rho, k)));
    const W njr = vmul(irho, K::all((A)-1)), third = K::all((A)(-1.0 / 3.0));  // s: rho, or rho - rho0 of shifted values
    const W pxx = vfma(vmul(jx, jx), njr, vfma(s, third, ab));
    const W pyy = vfma(vmul(jy, jy), njr, vfma(s, third, cd));
    const W pxy = vfma(vmul(jx, jy), njr, sxy);
    const W det = vfma(pxy, pxy, vmul(vmul(K::all((A)-1), pxx), pyy));
#pragma unroll
    for (int k = 0; k < K::N; ++k) K::set(r, k, (A)3 * sqrt(fabs(K::get(det, k))) * K::get(irho, k));
    return r;
}

// SC (shifted stores only): f holds (f - w_i rho0) * s in the store's scaled
// units, s = H.scale, and so does the result; the moments are unscaled once
// per node (exact: s is a power of two) instead of every population.  The
// components of W are nodes, th their normals (NOISE and X.kT > 0: thetas()),
// tau their relaxation times (PL: solve_taus() of strain()); returns their
// densities.
template <class W, bool SHIFT, bool NOISE, bool PL, bool SC = false>
__device__ __forceinline__ W collide_nodes(W (&f)[9], const HotPrm<typename Vec<W>::A>& H,
                                           const ExtPrm<typename Vec<W>::A>& X, const W (&th)[6], W tau) {
    static_assert(!SC || SHIFT, "scaled units are those of the shifted stores");
    typedef Vec<W> K;
    typedef typename K::A A;
    const W a = vadd(vadd(f[1], f[5]), f[8]);  // e_x > 0
    const W b = vadd(vadd(f[3], f[6]), f[7]);  // e_x < 0
    const W c = vadd(vadd(f[2], f[5]), f[6]);  // e_y > 0
    const W d = vadd(vadd(f[4], f[7]), f[8]);  // e_y < 0
    const W s_ = vadd(vadd(f[0], vadd(f[2], f[4])), vadd(a, b));
    const W jx_ = vsub(a, b), jy_ = vsub(c, d);
    // unscaled moments (SC: one multiply each by the power of two 1/s)
    const W u1 = K::all(H.inv_scale);
    const W s = SC ? vmul(s_, u1) : s_;
    const W jx = SC ? vmul(jx_, u1) : jx_, jy = SC ? vmul(jy_, u1) : jy_;
    const W rho = SHIFT ? vadd(K::all(H.rho0), s) : s;
    W irho;
#pragma unroll
    for (int k = 0; k < K::N; ++k) K::set(irho, k, rcp_rho<A>(K::get(rho, k)));
    W omega = K::all(H.omega), om = K::all(H.om), tgx = K::all(H.tgx), tgy = K::all(H.tgy);
    if (PL) {
#pragma unroll
        for (int k = 0; k < K::N; ++k) K::set(omega, k, (A)1 / K::get(tau, k));
        om = vsub(K::all((A)1), omega);
        tgx = vmul(tau, K::all(X.gx));
        tgy = vmul(tau, K::all(X.gy));
    }
    const W ux = vmul(vfma(rho, tgx, jx), irho);
    const W uy = vmul(vfma(rho, tgy, jy), irho);
    const W nusq = vmul(K::all((A)-1.5), vfma(ux, ux, vmul(uy, uy)));
    // in the units of f (SC: times s)
    const W R = SHIFT ? (SC ? vmul(vmul(omega, rho), K::all(H.scale)) : vmul(omega, rho)) : rho;
    const W B = SHIFT ? vmul(omega, SC ? s_ : s) : rho;
    const W R3 = vmul(K::all((A)3), R), nR3 = vmul(K::all((A)-3), R);
    const W nomega = vmul(K::all((A)-1), omega);
    const W h0 = vfma(R, nusq, B);
    if (SHIFT) f[0] = vfma(om, f[0], vmul(K::all((A)wgt(0)), h0));
    else f[0] = vfma(nomega, vfma(K::all(-(A)wgt(0)), h0, f[0]), f[0]);
    relax_pair<W, SHIFT, false, false>(f[1], f[3], ux, (A)wgt(1), nusq, R, R3, nR3, B, om, nomega);
    relax_pair<W, SHIFT, false, false>(f[2], f[4], uy, (A)wgt(2), nusq, R, R3, nR3, B, om, nomega);
    relax_pair<W, SHIFT, false, PL>(f[5], f[7], vadd(ux, uy), (A)wgt(5), nusq, R, R3, nR3, B, om, nomega);
    // The orders of the roundings are those the code had before it was packed:
    // the half-precision stores turn any other into differences of an ulp of
    // theirs, and tau* of shear-thinning fluids amplifies those of the strain.
    relax_pair<W, SHIFT, !NOISE || PL, !NOISE || PL>(f[6], f[8], vsub(uy, ux), (A)wgt(6), nusq, R, R3, nR3, B, om, nomega);
    if (NOISE) {
        if (X.kT > (A)0) {
            W amp;
            // var = 3 kT omega (2 - omega), as a pair hi + lo where omega is a constant
            W x;
            if (PL) x = vmul(rho, vmul(vmul(omega, vsub(K::all((A)2), omega)), K::all(X.var)));
            else x = vfma(rho, K::all(X.var), vmul(rho, K::all(X.var_lo)));
            if constexpr (sizeof(A) == 8) {
                amp = sqrt(x);
            } else {
                amp = sqrt_heron(x);  // 0 where x is not positive: no noise there
            }
            if (SC) amp = vmul(amp, K::all(H.scale));
            add_noise(f, amp, th);
        }
    }
    return rho;
}
// Zou-He density column (Zou & He 1997).  side 0: inlet at x = 0, the
// populations 1, 5, 8 enter from outside; side 1: outlet at x = nx-1, the
// populations 3, 6, 7 enter.  d_b is the prescribed density in the units of
// the stored values (rho_b - rho0 when SHIFT, rho_b otherwise); the shifts of
// the paired populations are equal.
template <typename A>
__device__ __forceinline__ A zou_he_excess(const DomDev& D, int side) {
    if (sizeof(A) == 4) return (A)(side == 0 ? D.drho_in_f : D.drho_out_f);
    return (A)(side == 0 ? D.drho_in : D.drho_out);
}
template <typename A>
__device__ __forceinline__ void zou_he(A f[9], int side, A d_b) {
    if (side == 0) {
        const A ru = d_b - (f[0] + f[2] + f[4] + (A)2 * (f[3] + f[6] + f[7]));
        f[1] = f[3] + (A)(2.0 / 3.0) * ru;
        f[5] = f[7] - (A)0.5 * (f[2] - f[4]) + (A)(1.0 / 6.0) * ru;
        f[8] = f[6] + (A)0.5 * (f[2] - f[4]) + (A)(1.0 / 6.0) * ru;
    } else {
        const A ru = (f[0] + f[2] + f[4] + (A)2 * (f[1] + f[5] + f[8])) - d_b;
        f[3] = f[1] - (A)(2.0 / 3.0) * ru;
        f[7] = f[5] + (A)0.5 * (f[2] - f[4]) - (A)(1.0 / 6.0) * ru;
        f[6] = f[8] - (A)0.5 * (f[2] - f[4]) - (A)(1.0 / 6.0) * ru;
    }
}

}  // namespace lbmk
