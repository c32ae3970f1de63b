// Device math of the probe data structure: octahedral map, bilinear texel
// filtering of bordered tiles, probe addressing and the biased 8-probe query.
// Used by the query kernel and by hit shading in the update (the previous
// frame's probes give the indirect term).
#pragma once

#include <cuda_fp16.h>

#include "ddgi_internal.h"
#include "pdl.cuh"

namespace ddgi {

__device__ __forceinline__ float3 f3(float x, float y, float z) { return make_float3(x, y, z); }
__device__ __forceinline__ float3 operator+(float3 a, float3 b) { return f3(a.x + b.x, a.y + b.y, a.z + b.z); }
__device__ __forceinline__ float3 operator-(float3 a, float3 b) { return f3(a.x - b.x, a.y - b.y, a.z - b.z); }
__device__ __forceinline__ float3 operator*(float s, float3 a) { return f3(s * a.x, s * a.y, s * a.z); }
__device__ __forceinline__ float dot(float3 a, float3 b) { return a.x * b.x + a.y * b.y + a.z * b.z; }
__device__ __forceinline__ float3 cross(float3 a, float3 b) {
    return f3(a.y * b.z - a.z * b.y, a.z * b.x - a.x * b.z, a.x * b.y - a.y * b.x);
}
__device__ __forceinline__ float length(float3 a) { return sqrtf(dot(a, a)); }
__device__ __forceinline__ float sgnnz(float x) { return x >= 0.0f ? 1.0f : -1.0f; }

// Octahedral encode (Cigolle et al. 2014): v / |v|_1, lower hemisphere folded.
__device__ __forceinline__ float2 oct_encode(float3 v) {
    float l1 = fabsf(v.x) + fabsf(v.y) + fabsf(v.z);
    float px = v.x / l1, py = v.y / l1;
    if (v.z < 0.0f) {
        float qx = (1.0f - fabsf(py)) * sgnnz(px);
        float qy = (1.0f - fabsf(px)) * sgnnz(py);
        px = qx;
        py = qy;
    }
    return make_float2(px, py);
}

// The same map with the hardware reciprocal (__fdividef, about 2 ulp) for
// the per-probe lookups of the query, where IEEE division dominated.
__device__ __forceinline__ float2 oct_encode_fast(float3 v) {
    float inv = __fdividef(1.0f, fabsf(v.x) + fabsf(v.y) + fabsf(v.z));
    float px = v.x * inv, py = v.y * inv;
    if (v.z < 0.0f) {
        float qx = (1.0f - fabsf(py)) * sgnnz(px);
        float qy = (1.0f - fabsf(px)) * sgnnz(py);
        px = qx;
        py = qy;
    }
    return make_float2(px, py);
}

// Probe grid addressing: logical (i,j,k) of the window is stored at
// ((i+shift) mod count, ...); the tracking window moves `shift`, which a
// VolView holds reduced to [0, count).
__device__ __forceinline__ int wrap(int a, int m) { int r = a % m; return r < 0 ? r + m : r; }
// (a + s) mod m and (a - s) mod m for a, s in [0, m)
__device__ __forceinline__ int wrap_add(int a, int s, int m) { int r = a + s; return r >= m ? r - m : r; }
__device__ __forceinline__ int wrap_sub(int a, int s, int m) { int r = a - s; return r < 0 ? r + m : r; }

__device__ __forceinline__ float3 probe_pos_logical(const VolView& v, int i, int j, int k) {
    return f3(v.origin.x + (float)i * v.spacing.x, v.origin.y + (float)j * v.spacing.y,
              v.origin.z + (float)k * v.spacing.z);
}

// World position of physical probe p: its grid point plus its offset (Sec. 5).
__device__ __forceinline__ float3 probe_pos_phys(const VolView& v, int p) {
    const int q = (int)fast_div((uint32_t)p, v.div_x);   // p / counts.x
    const int c = (int)fast_div((uint32_t)p, v.div_xy);  // p / (counts.x counts.y)
    const int a = p - q * v.counts.x;
    const int b = q - c * v.counts.y;
    float3 x = probe_pos_logical(v, wrap_sub(a, v.shift.x, v.counts.x), wrap_sub(b, v.shift.y, v.counts.y),
                                 wrap_sub(c, v.shift.z, v.counts.z));
    if (v.offsets) {
        const float4 o = v.offsets[p];
        x = f3(x.x + o.x, x.y + o.y, x.z + o.z);
    }
    return x;
}

// Traced, blended and used by the query: vigilant probes and sleeping probes
// woken by a dynamic object (Sec. 6.3).
__device__ __forceinline__ bool state_active(uint8_t s) {
    return s == DDGI_STATE_NEWLY_VIGILANT || s == DDGI_STATE_VIGILANT || s == DDGI_STATE_NEWLY_AWAKE ||
           s == DDGI_STATE_AWAKE;
}
// First update after becoming active: blended with hysteresis 0.
__device__ __forceinline__ bool state_newly(uint8_t s) {
    return s == DDGI_STATE_NEWLY_VIGILANT || s == DDGI_STATE_NEWLY_AWAKE;
}
// The state after a probe's update.
__device__ __forceinline__ uint8_t state_advanced(uint8_t s) {
    return s == DDGI_STATE_NEWLY_VIGILANT ? (uint8_t)DDGI_STATE_VIGILANT
                                          : (s == DDGI_STATE_NEWLY_AWAKE ? (uint8_t)DDGI_STATE_AWAKE : s);
}

// Bilinear footprint in a bordered tile of n interior texels: the octahedral
// coordinate [-1,1] spans texel positions [1, n+1]; texel k has its centre at k+0.5.
// Two floats in one 64-bit register pair, for the packed FP32 pair
// arithmetic of sm_100 and later (sub / mul / fma .rn.f32x2: each half
// rounded exactly as the scalar instruction would).
__device__ __forceinline__ uint64_t f2_pack(float lo, float hi) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void f2_unpack(uint64_t v, float& lo, float& hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ uint64_t f2_sub(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ uint64_t f2_mul(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
// a * b + c, each half one fused multiply-add (as fmaf)
__device__ __forceinline__ uint64_t f2_fma(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

struct Footprint {
    int x0, y0;
    float tx, ty;
};

__device__ __forceinline__ Footprint footprint(float2 u, int n) {
    float sx = 1.0f + (u.x + 1.0f) * 0.5f * (float)n - 0.5f;
    float sy = 1.0f + (u.y + 1.0f) * 0.5f * (float)n - 0.5f;
    float fx = floorf(sx), fy = floorf(sy);
    int x0 = (int)fx, y0 = (int)fy;
    x0 = min(max(x0, 0), n);
    y0 = min(max(y0, 0), n);
    Footprint f;
    f.x0 = x0;
    f.y0 = y0;
    f.tx = sx - (float)x0;
    f.ty = sy - (float)y0;
    return f;
}

// The same footprint, value for value, in the specialised queries, whose
// instruction issue bounds them: the floor by adding 2^23 rounded down (texel
// positions lie in [0.5, n + 0.5], n <= 64, so the sum's low bits are the
// texel) instead of conversions and clamps.  The one clamp left keeps a NaN
// position (a point on a probe: no direction) inside the tile.
__device__ __forceinline__ Footprint footprint_issue(float2 u, int n) {
    const float sx = 1.0f + (u.x + 1.0f) * 0.5f * (float)n - 0.5f;
    const float sy = 1.0f + (u.y + 1.0f) * 0.5f * (float)n - 0.5f;
    const float kx = __fadd_rd(sx, 8388608.0f), ky = __fadd_rd(sy, 8388608.0f);
    Footprint f;
    f.x0 = min(__float_as_int(kx) & 0x7f, n);
    f.y0 = min(__float_as_int(ky) & 0x7f, n);
    f.tx = sx - (kx - 8388608.0f);
    f.ty = sy - (ky - 8388608.0f);
    return f;
}

// ---- texel storage formats -------------------------------------------------
// Irradiance FP32: 4 floats per texel (rgb + an unused 0), one 16-byte load.
// FP16: 4 halves (rgb + pad).
// RGB9E5: one 32-bit word, 9-bit mantissas with a shared 5-bit exponent
// (bias 15), as in the OpenGL EXT_texture_shared_exponent specification.

__device__ __forceinline__ float3 rgb9e5_decode(uint32_t w) {
    const float s = __int_as_float(((int)(w >> 27) - 15 - 9 + 127) << 23);   // 2^(e - 15 - 9)
    return f3((float)(w & 511u) * s, (float)((w >> 9) & 511u) * s, (float)((w >> 18) & 511u) * s);
}

__device__ __forceinline__ uint32_t rgb9e5_encode(float3 c) {
    const float kMax = 65408.0f;   // (511/512) * 2^16
    float r = fminf(fmaxf(c.x, 0.0f), kMax);
    float g = fminf(fmaxf(c.y, 0.0f), kMax);
    float b = fminf(fmaxf(c.z, 0.0f), kMax);
    float mx = fmaxf(r, fmaxf(g, b));
    if (!(mx > 0.0f)) return 0u;
    // exponent such that mx / 2^(e-15-9) < 512, e >= 0
    int ex;
    frexpf(mx, &ex);                       // mx = m * 2^ex, m in [0.5, 1)
    int e = max(-16, ex - 1) + 1 + 15;     // shared exponent (biased)
    if (e < 0) e = 0;
    float s = ldexpf(1.0f, -(e - 15 - 9));
    int mmax = (int)floorf(mx * s + 0.5f);
    if (mmax == 512) { e += 1; s *= 0.5f; }
    if (e > 31) e = 31;
    uint32_t ir = (uint32_t)min(511, (int)floorf(r * s + 0.5f));
    uint32_t ig = (uint32_t)min(511, (int)floorf(g * s + 0.5f));
    uint32_t ib = (uint32_t)min(511, (int)floorf(b * s + 0.5f));
    return ir | (ig << 9) | (ib << 18) | ((uint32_t)e << 27);
}

// NC = true reads through the non-coherent (read-only) path: only for
// kernels that do not write the atlas.
template <bool NC>
__device__ __forceinline__ float ld(const float* p) { if (NC) return __ldg(p); else return *p; }
template <bool NC>
__device__ __forceinline__ uint32_t ld(const uint32_t* p) { if (NC) return __ldg(p); else return *p; }
template <bool NC>
__device__ __forceinline__ uint2 ld(const uint2* p) { if (NC) return __ldg(p); else return *p; }
template <bool NC>
__device__ __forceinline__ float2 ld(const float2* p) { if (NC) return __ldg(p); else return *p; }
template <bool NC>
__device__ __forceinline__ float4 ld(const float4* p) { if (NC) return __ldg(p); else return *p; }

template <bool NC = true>
__device__ __forceinline__ float3 load_irr(const VolView& v, int p, int x, int y) {
    int64_t t = (int64_t)p * v.irr_tile + (int64_t)y * (v.irr_n + 2) + x;
    if (v.irr_format == DDGI_IRR_FP32) {
        const float4 a = ld<NC>((const float4*)v.irr + t);
        return f3(a.x, a.y, a.z);
    } else if (v.irr_format == DDGI_IRR_FP16) {
        uint2 w = ld<NC>((const uint2*)v.irr + t);
        __half2 h0 = *reinterpret_cast<__half2*>(&w.x);
        __half2 h1 = *reinterpret_cast<__half2*>(&w.y);
        float2 a = __half22float2(h0);
        return f3(a.x, a.y, __low2float(h1));
    } else {
        // (ldexpf: with the power's bits written out as above, the queries that
        // choose the format here took 160 us for 1920 x 1080 points, 156 so)
        const uint32_t w = ld<NC>((const uint32_t*)v.irr + t);
        const float s = ldexpf(1.0f, (int)(w >> 27) - 15 - 9);
        return f3((float)(w & 511u) * s, (float)((w >> 9) & 511u) * s, (float)((w >> 18) & 511u) * s);
    }
}

__device__ __forceinline__ void store_irr(const VolView& v, int p, int x, int y, float3 c) {
    int64_t t = (int64_t)p * v.irr_tile + (int64_t)y * (v.irr_n + 2) + x;
    if (v.irr_format == DDGI_IRR_FP32) {
        ((float4*)v.irr)[t] = make_float4(c.x, c.y, c.z, 0.0f);
    } else if (v.irr_format == DDGI_IRR_FP16) {
        __half2 h0 = __floats2half2_rn(c.x, c.y);
        __half2 h1 = __floats2half2_rn(c.z, 0.0f);
        uint2 w;
        w.x = *reinterpret_cast<uint32_t*>(&h0);
        w.y = *reinterpret_cast<uint32_t*>(&h1);
        ((uint2*)v.irr)[t] = w;
    } else {
        ((uint32_t*)v.irr)[t] = rgb9e5_encode(c);
    }
}

template <bool NC = true>
__device__ __forceinline__ float2 load_dist(const VolView& v, int p, int x, int y) {
    int64_t t = (int64_t)p * v.dist_tile + (int64_t)y * (v.dist_n + 2) + x;
    if (v.dist_format == DDGI_DIST_FP32) {
        return ld<NC>((const float2*)v.dist + t);
    } else {
        uint32_t w = ld<NC>((const uint32_t*)v.dist + t);
        return __half22float2(*reinterpret_cast<__half2*>(&w));
    }
}

__device__ __forceinline__ void store_dist(const VolView& v, int p, int x, int y, float2 m) {
    int64_t t = (int64_t)p * v.dist_tile + (int64_t)y * (v.dist_n + 2) + x;
    if (v.dist_format == DDGI_DIST_FP32) {
        ((float2*)v.dist)[t] = m;
    } else {
        __half2 h = __floats2half2_rn(m.x, m.y);
        ((uint32_t*)v.dist)[t] = *reinterpret_cast<uint32_t*>(&h);
    }
}

// Bilinear samples at a footprint: one storage-format dispatch per sample,
// then the four taps (rows y0, y0 + 1 of the bordered tile).
struct Bilerp {
    float w00, w10, w01, w11;
};

__device__ __forceinline__ Bilerp bilerp_weights(const Footprint& f) {
    Bilerp b;
    b.w00 = (1.0f - f.tx) * (1.0f - f.ty);
    b.w10 = f.tx * (1.0f - f.ty);
    b.w01 = (1.0f - f.tx) * f.ty;
    b.w11 = f.tx * f.ty;
    return b;
}

__device__ __forceinline__ float3 bilerp3(const Bilerp& w, float3 a, float3 b, float3 c, float3 d) {
    return f3(w.w00 * a.x + w.w10 * b.x + w.w01 * c.x + w.w11 * d.x,
              w.w00 * a.y + w.w10 * b.y + w.w01 * c.y + w.w11 * d.y,
              w.w00 * a.z + w.w10 * b.z + w.w01 * c.z + w.w11 * d.z);
}

// Irradiance at a footprint whose bilinear weights are already known (the
// query reads every cage probe at the same footprint).
__device__ __forceinline__ float3 sample_irr_at(const VolView& v, int p, const Footprint& f, const Bilerp& w) {
    const int row = v.irr_n + 2;
    const int64_t t = (int64_t)p * v.irr_tile + (int64_t)f.y0 * row + f.x0;
    if (v.irr_format == DDGI_IRR_FP32) {
        const float4* a = (const float4*)v.irr + t;
        const float4 q00 = __ldg(a), q10 = __ldg(a + 1), q01 = __ldg(a + row), q11 = __ldg(a + row + 1);
        return bilerp3(w, f3(q00.x, q00.y, q00.z), f3(q10.x, q10.y, q10.z), f3(q01.x, q01.y, q01.z),
                       f3(q11.x, q11.y, q11.z));
    }
    return bilerp3(w, load_irr(v, p, f.x0, f.y0), load_irr(v, p, f.x0 + 1, f.y0), load_irr(v, p, f.x0, f.y0 + 1),
                   load_irr(v, p, f.x0 + 1, f.y0 + 1));
}

__device__ __forceinline__ float2 sample_dist_at(const VolView& v, int p, const Footprint& f) {
    const int row = v.dist_n + 2;
    float2 a, b, c, d;
    if (v.dist_format == DDGI_DIST_FP32) {
        const float2* q = (const float2*)v.dist + (int64_t)p * v.dist_tile + (int64_t)f.y0 * row + f.x0;
        a = __ldg(q);
        b = __ldg(q + 1);
        c = __ldg(q + row);
        d = __ldg(q + row + 1);
    } else {
        a = load_dist(v, p, f.x0, f.y0);
        b = load_dist(v, p, f.x0 + 1, f.y0);
        c = load_dist(v, p, f.x0, f.y0 + 1);
        d = load_dist(v, p, f.x0 + 1, f.y0 + 1);
    }
    float w00 = (1.0f - f.tx) * (1.0f - f.ty), w10 = f.tx * (1.0f - f.ty);
    float w01 = (1.0f - f.tx) * f.ty, w11 = f.tx * f.ty;
    return make_float2(w00 * a.x + w10 * b.x + w01 * c.x + w11 * d.x,
                       w00 * a.y + w10 * b.y + w01 * c.y + w11 * d.y);
}

// x^(gamma/2) on the gamma-encoded value (gamma = 5: x^2 sqrt(x)), sqrt(x) as
// x * rsqrt(x) (hardware reciprocal square root, about 2 ulp).
__device__ __forceinline__ float gamma_decode_half(float e, float half_gamma) {
    e = fmaxf(e, 0.0f);
    const float sq = e > 0.0f ? e * rsqrtf(e) : 0.0f;
    if (half_gamma == 2.5f) return e * e * sq;
    if (half_gamma == 0.5f) return sq;
    return powf(e, half_gamma);
}


// a - b for FP32 a, b as the unevaluated sum hi + lo, exactly (Knuth's
// TwoSum applied to a and -b, round-to-nearest); the intrinsics keep each
// step as written.
__device__ __forceinline__ void two_diff(float a, float b, float& hi, float& lo) {
    hi = __fsub_rn(a, b);
    const float bb = __fsub_rn(hi, a);
    lo = __fadd_rn(__fsub_rn(a, __fsub_rn(hi, bb)), __fsub_rn(-b, bb));
}

// A query point in the volume's own frame: x - origin = hi + lo exactly, and
// lb = lo + the self-shadow bias vector (Sec. 4.1), so the biased point is
// origin + hi + lb.  Probe-to-point vectors formed from these carry rounding
// errors relative to their own length, not to |x|: far from the world
// origin, 2^-24 |x| approaches the standard deviation the Chebyshev test
// divides by, and the weight then follows the rounding of x instead of x.
struct LocalPoint {
    float3 hi, lo, lb;
};

__device__ __forceinline__ LocalPoint local_point(const VolView& v, float3 x, float3 n, float3 wo) {
    const float k = 0.75f * v.min_spacing * v.bias;
    LocalPoint q;
    two_diff(x.x, v.origin.x, q.hi.x, q.lo.x);
    two_diff(x.y, v.origin.y, q.hi.y, q.lo.y);
    two_diff(x.z, v.origin.z, q.hi.z, q.lo.z);
    q.lb = f3(q.lo.x + (0.2f * n.x + 0.8f * wo.x) * k, q.lo.y + (0.2f * n.y + 0.8f * wo.y) * k,
              q.lo.z + (0.2f * n.z + 0.8f * wo.z) * k);
    return q;
}

// x - x_p for the grid point (i, j, k) of the cage: the high part of the
// difference (one rounding, relative to |x - x_p|); add q.lo for the
// unbiased point, q.lb for the biased one.
__device__ __forceinline__ float3 local_to_probe(const VolView& v, const LocalPoint& q, int i, int j, int k) {
    return f3(q.hi.x - (float)i * v.spacing.x, q.hi.y - (float)j * v.spacing.y, q.hi.z - (float)k * v.spacing.z);
}

// x^2.5 of a red / green pair of gamma-encoded values (gamma 5): e^2 times
// e * rsqrt(e), the squares and products as packed FP32 pairs.  The floor
// 1e-30 stands in for the zero test of gamma_decode_half: below it both
// give 0 in FP32 (x^2.5 < 1e-75), above it they are the same operations.
__device__ __forceinline__ uint64_t gamma_decode_g5_pair(float er, float eg) {
    er = fmaxf(er, 1e-30f);
    eg = fmaxf(eg, 1e-30f);
    const uint64_t E = f2_pack(er, eg);
    const uint64_t S = f2_mul(E, f2_pack(rsqrtf(er), rsqrtf(eg)));
    return f2_mul(f2_mul(E, E), S);
}

// What a specialised query form fixes at compile time (query_form).
template <int FORM>
struct QueryForm {
    static constexpr bool kHalf =                            // FP16 atlases
        FORM == kQueryHalf || FORM == kQueryHalfGamma1 || FORM == kQueryHalfAny;
    static constexpr bool kE5 =                              // RGB9E5 irradiance
        FORM == kQueryE5 || FORM == kQueryE5Gamma1 || FORM == kQueryE5Any;
    static constexpr bool kGamma1 =                          // gamma 1,
        FORM == kQueryGamma1 || FORM == kQueryHalfGamma1 || FORM == kQueryE5Gamma1;
    static constexpr bool kAnyGamma =                        // or the view's (else 5)
        FORM == kQueryFp32Any || FORM == kQueryHalfAny || FORM == kQueryE5Any;
    static constexpr bool kMoved = FORM == kQueryMoved;      // probe offsets
};

// The four taps of a probe's irradiance tile at a footprint, bilinearly
// weighted: red and green as a packed pair, blue.
template <int FORM>
__device__ __forceinline__ uint64_t irr_taps(const VolView& v, int p, const Footprint& f, const Bilerp& w, float& eb) {
    const int row = v.irr_n + 2;
    const int64_t t = (int64_t)p * v.irr_tile + ((int64_t)f.y0 * row + f.x0);
    float3 q00, q10, q01, q11;
    if constexpr (FORM == kQueryGeneral) {
        const float3 e = sample_irr_at(v, p, f, w);
        eb = e.z;
        return f2_pack(e.x, e.y);
    } else if constexpr (QueryForm<FORM>::kHalf) {
        const uint2* a = (const uint2*)v.irr + t;
        const uint2 h[4] = {__ldg(a), __ldg(a + 1), __ldg(a + row), __ldg(a + row + 1)};
        float3* o[4] = {&q00, &q10, &q01, &q11};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const float2 rg = __half22float2(*reinterpret_cast<const __half2*>(&h[k].x));
            *o[k] = f3(rg.x, rg.y, __low2float(*reinterpret_cast<const __half2*>(&h[k].y)));
        }
    } else if constexpr (QueryForm<FORM>::kE5) {
        const uint32_t* a = (const uint32_t*)v.irr + t;
        const uint32_t h00 = __ldg(a), h10 = __ldg(a + 1), h01 = __ldg(a + row), h11 = __ldg(a + row + 1);
        q00 = rgb9e5_decode(h00);
        q10 = rgb9e5_decode(h10);
        q01 = rgb9e5_decode(h01);
        q11 = rgb9e5_decode(h11);
    } else {
        const float4* a = (const float4*)v.irr + t;
        const float4 f00 = __ldg(a), f10 = __ldg(a + 1), f01 = __ldg(a + row), f11 = __ldg(a + row + 1);
        q00 = f3(f00.x, f00.y, f00.z);
        q10 = f3(f10.x, f10.y, f10.z);
        q01 = f3(f01.x, f01.y, f01.z);
        q11 = f3(f11.x, f11.y, f11.z);
    }
    uint64_t rg = f2_mul(f2_pack(w.w00, w.w00), f2_pack(q00.x, q00.y));
    rg = f2_fma(f2_pack(w.w10, w.w10), f2_pack(q10.x, q10.y), rg);
    rg = f2_fma(f2_pack(w.w01, w.w01), f2_pack(q01.x, q01.y), rg);
    rg = f2_fma(f2_pack(w.w11, w.w11), f2_pack(q11.x, q11.y), rg);
    eb = w.w00 * q00.z + w.w10 * q10.z + w.w01 * q01.z + w.w11 * q11.z;
    return rg;
}

// A Chebyshev weight is the ratio of a variance, the difference of two moments,
// to that and the squared distance beyond the mean.  Where both are small the
// last bits of the moments and of the distance decide it (the other order moves
// single points near an occluder by 0.3 %), so their sums are written out as
// fused operations in one order for each form.  They begin with the first product,
// as the general form's plain expressions are compiled; with the second in FP32
// gamma 5 queries of a volume's or a cascade's points and hits, as those expressions
// were compiled for them alone (in cascades the distance stays the plain
// expression).  The allocation-free update has the first order by a form of its
// own (kQueryFp32First): the second was 1.04 times as far from 64 bits over 99
// volumes, 3.5 times in one of them.  For a cascade's query either is as far (3.2e-7
// to 6.4e-7 rms over six rooms).
template <int FORM, bool ADJOINT>
struct SumOrder {
    static constexpr bool kFirst = ADJOINT || FORM != kQueryFp32;
};

// The distance moments of a form's atlas at a footprint as packed (mean, mean
// square) pairs.
template <int FORM, bool ADJOINT = false>
__device__ __forceinline__ float2 dist_taps(const VolView& v, int p, const Footprint& f) {
    if constexpr (FORM == kQueryGeneral) return sample_dist_at(v, p, f);
    const int row = v.dist_n + 2;
    const int64_t t = (int64_t)p * v.dist_tile + (int64_t)f.y0 * row + f.x0;
    uint64_t a, b, c, d;
    if constexpr (QueryForm<FORM>::kHalf) {
        const uint32_t* q = (const uint32_t*)v.dist + t;
        const uint32_t h[4] = {__ldg(q), __ldg(q + 1), __ldg(q + row), __ldg(q + row + 1)};
        uint64_t* o[4] = {&a, &b, &c, &d};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const float2 m = __half22float2(*reinterpret_cast<const __half2*>(&h[k]));
            *o[k] = f2_pack(m.x, m.y);
        }
    } else {
        const unsigned long long* q = (const unsigned long long*)v.dist + t;
        a = __ldg(q);
        b = __ldg(q + 1);
        c = __ldg(q + row);
        d = __ldg(q + row + 1);
    }
    const Bilerp w = bilerp_weights(f);
    const uint64_t W00 = f2_pack(w.w00, w.w00), W10 = f2_pack(w.w10, w.w10);
    uint64_t m = SumOrder<FORM, ADJOINT>::kFirst ? f2_fma(W10, b, f2_mul(W00, a)) : f2_fma(W00, a, f2_mul(W10, b));
    m = f2_fma(f2_pack(w.w01, w.w01), c, m);
    m = f2_fma(f2_pack(w.w11, w.w11), d, m);
    float2 r;
    f2_unpack(m, r.x, r.y);
    return r;
}

// The eight-probe cage of a biased point: its base cell and, per axis, the
// fraction and the two planes' physical index, x - x_p (high part) and
// trilinear factor, so that a corner's values are registers.
struct Cage {
    int base[3];
    int px[2], py[2], pz[2];
    float ax[2], ay[2], az[2];
    float tx[2], ty[2], tz[2];
    // Corner c's trilinear factor.  A point on a grid plane or beyond the
    // grid has its fraction clamped to 0 or 1, so that half, three quarters
    // or seven eighths of its cage weigh exactly 0 and need no lookup.
    __device__ __forceinline__ float trilinear(int c) const { return side(tx, c & 1) * side(ty, c & 2) * side(tz, c & 4); }
    __device__ __forceinline__ int probe(const VolView& v, int c) const {
        return side(px, c & 1) + v.counts.x * (side(py, c & 2) + v.counts.y * side(pz, c & 4));
    }
    // x - x_p (high part) to corner c's grid point
    __device__ __forceinline__ float3 to_grid(int c) const { return f3(side(ax, c & 1), side(ay, c & 2), side(az, c & 4)); }
    // an element by selection, so that the pairs stay in registers for any c
    template <typename T>
    static __device__ __forceinline__ T side(const T (&pair)[2], int upper) { return upper ? pair[1] : pair[0]; }
};

__device__ __forceinline__ Cage cage_of(const VolView& v, const LocalPoint& q) {
    Cage k;
    const float g[3] = {(q.hi.x + q.lb.x) / v.spacing.x, (q.hi.y + q.lb.y) / v.spacing.y,
                        (q.hi.z + q.lb.z) / v.spacing.z};
    const int cnt[3] = {v.counts.x, v.counts.y, v.counts.z};
    float fr[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        float b = floorf(g[a]);
        b = fminf(fmaxf(b, 0.0f), (float)(cnt[a] - 2));
        k.base[a] = (int)b;
        fr[a] = fminf(fmaxf(g[a] - b, 0.0f), 1.0f);
    }
#pragma unroll
    for (int o = 0; o < 2; ++o) {
        k.px[o] = wrap_add(k.base[0] + o, v.shift.x, cnt[0]);
        k.py[o] = wrap_add(k.base[1] + o, v.shift.y, cnt[1]);
        k.pz[o] = wrap_add(k.base[2] + o, v.shift.z, cnt[2]);
        k.ax[o] = q.hi.x - (float)(k.base[0] + o) * v.spacing.x;
        k.ay[o] = q.hi.y - (float)(k.base[1] + o) * v.spacing.y;
        k.az[o] = q.hi.z - (float)(k.base[2] + o) * v.spacing.z;
        k.tx[o] = o ? fr[0] : 1.0f - fr[0];
        k.ty[o] = o ? fr[1] : 1.0f - fr[1];
        k.tz[o] = o ? fr[2] : 1.0f - fr[2];
    }
    return k;
}

// Weight of cage corner c (probe p) in a form's query: trilinear, backface
// and Chebyshev factors, floored (query_M_look).  Where a Chebyshev weight is
// near the depth it tests, the last bits of the distance and of the lookup
// decide it, and hit shading carries them into the atlas and every later
// frame: the operations are those of the general form.  BRANCH keeps the
// general form's branches, which the cascade kernels are faster with (2567 us a
// frame against 2580); a single volume's are slower (city frame with FP16
// atlases 504 us against 498).  IEEE: the distance and the lookup's
// coordinates by rounded square root and division (the adjoint, where one
// point's weight can be a whole texel's gradient).  The backface cosine, the
// Chebyshev ratio and the adjoint's decode (decode_slope) use the hardware's
// reciprocals there too, about 2 ulp each: rounded as well they were no closer to 64
// bits (texel gradients of 1280 x 720 points 3.0e-5 rms, 2.7e-5 as it is, the
// same over fifteen drawn cases) and took 267 us for 1920 x 1080 points
// instead of 234.
template <int FORM, bool IEEE = false, bool BRANCH = false>
__device__ __forceinline__ float corner_weight(const VolView& v, const LocalPoint& q, const Cage& k, int c, int p,
                                               float3 n) {
    float3 a = k.to_grid(c);
    if (QueryForm<FORM>::kMoved || (FORM == kQueryGeneral && v.offsets)) {
        const float4 po = __ldg(v.offsets + p);   // the probe's own (moved) position; the cage stays on the grid
        a = f3(a.x - po.x, a.y - po.y, a.z - po.z);
    }
    const float wt = k.trilinear(c);
    const float3 dp = f3(-(a.x + q.lo.x), -(a.y + q.lo.y), -(a.z + q.lo.z));   // probe - x
    const float dd = dot(dp, dp);
    const float cw = dd > 0.0f ? dot(n, dp) * rsqrtf(dd) : 1.0f;
    const float hb = (1.0f + cw) * 0.5f;
    const float wb = hb * hb + 0.2f;
    const float3 pv = a + q.lb;                                                // biased point - probe
    const float xy = SumOrder<FORM, IEEE>::kFirst ? __fmaf_rn(pv.y, pv.y, __fmul_rn(pv.x, pv.x))
                                                  : __fmaf_rn(pv.x, pv.x, __fmul_rn(pv.y, pv.y));
    const float rr = BRANCH ? dot(pv, pv) : __fmaf_rn(pv.z, pv.z, xy);
    float wc = 1.0f;
    if (!BRANCH || rr > 0.0f) {   // without the branch rr = 0 makes a NaN of r, beyond no mean
        const float r = IEEE ? sqrtf(rr) : rr * rsqrtf(rr);
        const float2 u = IEEE ? oct_encode((1.0f / r) * pv) : oct_encode_fast(rsqrtf(rr) * pv);
        const float2 mom = dist_taps<FORM, IEEE>(v, p, footprint_issue(u, v.dist_n));
        auto chebyshev = [&]() {
            const float var = fmaxf(mom.y - mom.x * mom.x, 0.0f);
            const float dr = r - mom.x;
            return __fdividef(var, var + dr * dr);
        };
        if constexpr (BRANCH) {
            if (r > mom.x) wc = chebyshev();
        } else {
            const float c = chebyshev();
            wc = rr > 0.0f && r > mom.x ? c : 1.0f;
        }
    }
    return wt * wb * fmaxf(wc, 1e-6f);
}

// Corners that the specialised query takes to a trip of its loop: all eight,
// but two where the power of any gamma is inlined for three channels of each
// (1920 x 1080 points inside the grid, FP32 gamma 2.2: 246 us with eight, 216
// with two, general form 227; in random order 320, 298 and 295; RGB9E5 296, 245
// and 270), and four for an irradiance query of FP32 atlases at gamma 1 (112 us,
// with eight 113; in random order 294, 304, general form 288).  The glossy
// lookup and cascades of that form are no faster so (76 us for points beyond the
// grid, 74 with eight), and with probe offsets fewer cost neighbouring points
// 5 % (119 us, 114; general form 136) and give random order 1 % (327, 331; 320).
// all: a glossy lookup or a cascade.
template <int FORM>
__host__ __device__ constexpr int corners_per_trip(bool all) {
    return QueryForm<FORM>::kAnyGamma ? 2 : FORM == kQueryGamma1 && !all ? 4 : 8;
}

// The specialised query of query_M_look (any FORM but kQueryGeneral): the same
// operations in the same order, except the decode's zero test
// (gamma_decode_g5_pair), with the eight cage corners unrolled, the storage
// format, gamma and offsets fixed at compile time, and the red and green
// channels of the irradiance taps and their decode carried as packed FP32
// pairs (the blue channel scalar).  Bound by instruction issue for
// neighbouring points: 1920 x 1080 of them on 16 x 8 x 16 probes, beyond the
// grid planes on one axis, take 72-84 us by the storage format (general form:
// 142-183 us), with the power of any other gamma 128-142 us (234-278).
// Points in random order are bound by L2 sectors instead (124-165 us).
// EDGES: corners of zero trilinear weight are passed over (no lookup, the
// same sums), which a volume's points on and beyond its grid planes gain
// from: the glossy lookup of 960 x 540 such points 33.6 -> 22.6 us, a
// city frame's hit shading 74 -> 72 us.  Cascades leave it out: a volume of
// weight 0 at its edges is not read there, and their kernels spill more with
// the test (2852 -> 2912 us a frame).
// CORNERS: corners to a trip of the loop (corners_per_trip).
template <int FORM, bool EDGES, int CORNERS>
__device__ __forceinline__ float3 query_M_look_fast(const VolView& v, float3 x, float3 n, float3 wo, float3 look) {
    const LocalPoint q = local_point(v, x, n, wo);
    const Cage k = cage_of(v, q);
    const Footprint fn = footprint_issue(oct_encode(look), v.irr_n);
    const Bilerp wn = bilerp_weights(fn);
    unsigned act = 0;
#pragma unroll
    for (int c = 0; c < 8; ++c) act |= state_active(v.states[k.probe(v, c)]) ? 1u << c : 0u;
    float sumw = 0.0f;
    float3 acc = f3(0.0f, 0.0f, 0.0f);
#pragma unroll CORNERS
    for (int c = 0; c < 8; ++c) {
        if (!(act & (1u << c)) || (EDGES && k.trilinear(c) == 0.0f)) continue;
        const int p = k.probe(v, c);
        const float w = corner_weight<FORM, false, !EDGES>(v, q, k, c, p, n);
        float er, eg, eb;
        f2_unpack(irr_taps<FORM>(v, p, fn, wn, eb), er, eg);
        if constexpr (QueryForm<FORM>::kGamma1) {
            acc.x += w * gamma_decode_half(er, 0.5f);
            acc.y += w * gamma_decode_half(eg, 0.5f);
            acc.z += w * gamma_decode_half(eb, 0.5f);
        } else if constexpr (QueryForm<FORM>::kAnyGamma) {
            acc.x += w * gamma_decode_half(er, v.half_gamma);
            acc.y += w * gamma_decode_half(eg, v.half_gamma);
            acc.z += w * gamma_decode_half(eb, v.half_gamma);
        } else {
            float dr_, dg_;
            f2_unpack(gamma_decode_g5_pair(er, eg), dr_, dg_);
            const float ebc = fmaxf(eb, 1e-30f);
            acc.x += w * dr_;
            acc.y += w * dg_;
            acc.z += w * (ebc * ebc * (ebc * rsqrtf(ebc)));
        }
        sumw += w;
    }
    if (!(sumw > 0.0f)) return f3(0.0f, 0.0f, 0.0f);
    const float inv = 1.0f / sumw;
    const float3 m = inv * acc;
    return f3(m.x * m.x, m.y * m.y, m.z * m.z);
}

// Cosine-weighted mean radiance M at x with normal n, the self-shadow bias
// using w_o (Sec. 4.1 equation), the 8-probe cage (Sec. 2.2): trilinear,
// backface ((1 + n.w_p)/2)^2 + 0.2, Chebyshev visibility, weight floor
// 1e-6 * w_t * w_b, gamma decode (Sec. 4.2) normalised before squaring.
// Per-probe normalisations, the Chebyshev ratio and the square roots of the
// decode use the hardware reciprocal and reciprocal square root.
// `look` is the direction the irradiance tiles are read in: n for the
// irradiance query, the mirror direction for a second-order glossy lookup
// (Sec. 4.4); the bias and the backface weights use n either way.
// FORM: the view's form (query_form); query_M_look_fast serves all but the
// general one.
template <int FORM = kQueryGeneral, bool EDGES = true, int CORNERS = corners_per_trip<FORM>(!EDGES)>
__device__ __forceinline__ float3 query_M_look(const VolView& v, float3 x, float3 n, float3 wo, float3 look) {
    if constexpr (FORM != kQueryGeneral) return query_M_look_fast<FORM, EDGES, CORNERS>(v, x, n, wo, look);
    const LocalPoint q = local_point(v, x, n, wo);
    float g[3] = {(q.hi.x + q.lb.x) / v.spacing.x, (q.hi.y + q.lb.y) / v.spacing.y,
                  (q.hi.z + q.lb.z) / v.spacing.z};
    int cnt[3] = {v.counts.x, v.counts.y, v.counts.z};
    int base[3];
    float fr[3];
    for (int a = 0; a < 3; ++a) {
        float b = floorf(g[a]);
        b = fminf(fmaxf(b, 0.0f), (float)(cnt[a] - 2));
        base[a] = (int)b;
        fr[a] = fminf(fmaxf(g[a] - b, 0.0f), 1.0f);
    }
    float sumw = 0.0f;
    float3 acc = f3(0.0f, 0.0f, 0.0f);
    const Footprint fn = footprint(oct_encode(look), v.irr_n);   // irradiance lookup, the same for every probe
    const Bilerp wn = bilerp_weights(fn);
    // physical indices of the cage's two planes per axis
    const int px0 = wrap_add(base[0], v.shift.x, cnt[0]), px1 = wrap_add(base[0] + 1, v.shift.x, cnt[0]);
    const int py0 = wrap_add(base[1], v.shift.y, cnt[1]), py1 = wrap_add(base[1] + 1, v.shift.y, cnt[1]);
    const int pz0 = wrap_add(base[2], v.shift.z, cnt[2]), pz1 = wrap_add(base[2] + 1, v.shift.z, cnt[2]);
    // the eight states first, as independent loads, so the probe loop below
    // does not wait on one state load per probe
    unsigned act = 0;
#pragma unroll
    for (int c = 0; c < 8; ++c) {
        const int p = (c & 1 ? px1 : px0) + cnt[0] * ((c & 2 ? py1 : py0) + cnt[1] * (c & 4 ? pz1 : pz0));
        act |= state_active(v.states[p]) ? 1u << c : 0u;
    }
#pragma unroll 1
    for (; act != 0; act &= act - 1) {   // active probes in ascending c
        const int c = __ffs(act) - 1;
        int o0 = c & 1, o1 = (c >> 1) & 1, o2 = (c >> 2) & 1;
        int p = (o0 ? px1 : px0) + cnt[0] * ((o1 ? py1 : py0) + cnt[1] * (o2 ? pz1 : pz0));
        float3 a = local_to_probe(v, q, base[0] + o0, base[1] + o1, base[2] + o2);
        if (v.offsets) {   // the probe's own (moved) position; the cage stays on the grid
            const float4 po = __ldg(v.offsets + p);
            a = f3(a.x - po.x, a.y - po.y, a.z - po.z);
        }
        float wt = (o0 ? fr[0] : 1.0f - fr[0]) * (o1 ? fr[1] : 1.0f - fr[1]) * (o2 ? fr[2] : 1.0f - fr[2]);
        float3 dp = f3(-(a.x + q.lo.x), -(a.y + q.lo.y), -(a.z + q.lo.z));   // probe - x
        float dd = dot(dp, dp);
        float cw = dd > 0.0f ? dot(n, dp) * rsqrtf(dd) : 1.0f;
        float hb = (1.0f + cw) * 0.5f;
        float wb = hb * hb + 0.2f;
        float3 pv = a + q.lb;                                                // biased point - probe
        float rr = dot(pv, pv);
        float wc = 1.0f;
        if (rr > 0.0f) {
            float ir = rsqrtf(rr);
            float r = rr * ir;
            const Footprint fd = footprint(oct_encode_fast(ir * pv), v.dist_n);
            float2 mom = sample_dist_at(v, p, fd);
            if (r > mom.x) {
                float var = fmaxf(mom.y - mom.x * mom.x, 0.0f);
                float dr = r - mom.x;
                wc = __fdividef(var, var + dr * dr);
            }
        }
        float w = wt * wb * fmaxf(wc, 1e-6f);
        float3 e = sample_irr_at(v, p, fn, wn);
        acc.x += w * gamma_decode_half(e.x, v.half_gamma);
        acc.y += w * gamma_decode_half(e.y, v.half_gamma);
        acc.z += w * gamma_decode_half(e.z, v.half_gamma);
        sumw += w;
    }
    if (!(sumw > 0.0f)) return f3(0.0f, 0.0f, 0.0f);
    float inv = 1.0f / sumw;
    float3 a = inv * acc;
    return f3(a.x * a.x, a.y * a.y, a.z * a.z);
}

template <int FORM = kQueryGeneral, bool EDGES = true>
__device__ __forceinline__ float3 query_M(const VolView& v, float3 x, float3 n, float3 wo) {
    return query_M_look<FORM, EDGES>(v, x, n, wo, n);
}

// Cascade value M at x (Sec. 7.3): volumes densest first; each volume's
// weight is the product over axes of its linear fall-off over the last cell
// of its blend box; accumulation stops once the weights reach 1; the sum is
// normalised by the weights taken (0 when no volume covers x).
__device__ __forceinline__ float volume_weight(const VolView& v, float3 x) {
    float wx = fminf(fmaxf(fminf(x.x - v.blend_lo.x, v.blend_hi.x - x.x) / v.spacing.x, 0.0f), 1.0f);
    float wy = fminf(fmaxf(fminf(x.y - v.blend_lo.y, v.blend_hi.y - x.y) / v.spacing.y, 0.0f), 1.0f);
    float wz = fminf(fmaxf(fminf(x.z - v.blend_lo.z, v.blend_hi.z - x.z) / v.spacing.z, 0.0f), 1.0f);
    return wx * wy * wz;
}

template <int FORM = kQueryGeneral>
__device__ __forceinline__ float3 cascade_M(const VolView* vols, int n, float3 x, float3 nrm, float3 wo) {
    float sum = 0.0f;
    float3 acc = f3(0.0f, 0.0f, 0.0f);
    for (int k = 0; k < n; ++k) {
        const VolView& v = vols[k];
        float take = fminf(volume_weight(v, x), 1.0f - sum);
        if (!(take > 0.0f)) continue;
        float3 M = query_M<FORM, false>(v, x, nrm, wo);
        acc = acc + take * M;
        sum += take;
        if (sum >= 1.0f) break;
    }
    if (!(sum > 0.0f)) return f3(0.0f, 0.0f, 0.0f);
    return (1.0f / sum) * acc;
}

// Whether points were put in order (order_points).
__device__ __forceinline__ bool points_scattered(const PointOrder& o, int n) {
    return *o.groups > kAdjMaxGroups / 2 * ((n + 31) / 32);
}

}  // namespace ddgi
