// nodes.cuh -- device code shared by the pass kernels and the surrogate kernels:
// descriptors and hashes (Sec. 3.1, Eq. 1, Alg. 1), the FP32 node primitives and one
// interpreter step of a compiled material program (Sec. 2).
#pragma once

#include <cstdint>

#include "pmc_internal.h"

namespace pmc {

// =======================================================================================
// Descriptor and hashes (Sec. 3.1, Eq. 1, Alg. 1)
// =======================================================================================
__device__ __forceinline__ uint32_t d_fmix32(uint32_t h) {
    // MurmurHash3 32-bit finaliser (Appleby)
    h ^= h >> 16;
    h *= 0x85EBCA6Bu;
    h ^= h >> 13;
    h *= 0xC2B2AE35u;
    h ^= h >> 16;
    return h;
}

__device__ __forceinline__ uint64_t d_fmix64(uint64_t k) {
    // MurmurHash3 64-bit finaliser (Appleby)
    k ^= k >> 33;
    k *= 0xFF51AFD7ED558CCDull;
    k ^= k >> 33;
    k *= 0xC4CEB9FE1A85EC53ull;
    k ^= k >> 33;
    return k;
}

__device__ __forceinline__ uint64_t d_splitmix(uint64_t z) {
    // SplitMix64 output function (Steele, Lea & Flood 2014)
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

// Texel index on a virtual texture of 2^level texels per axis.  u * 2^level is exact in
// FP32, so the index is the same as in any wider precision.  fmaxf maps NaN to 0.
__device__ __forceinline__ uint32_t d_texel(float u, uint32_t level) {
    float x = fminf(fmaxf(u, 0.0f), 1.0f);
    uint32_t res = 1u << level;
    uint32_t t = (uint32_t)floorf(x * (float)res);
    return min(t, res - 1u);
}

// Mip level of the virtual texture from the ray-cone footprint (Sec. 3.1, Eq. 1):
// floor(-log2(min(|g1|, |g2|))) + offset, clamped to [0, 13].  The squared norms are formed
// in FP32 with every product and the sum rounded to nearest (no fused multiply-add), and
// the floor is read off the exponent E and fraction f of the smaller one, s = (1 + f) 2^E:
// -log2(sqrt(s)) = -(E + log2(1 + f)) / 2, whose floor is -ceil(E / 2) when f = 0 and
// -floor(E / 2) - 1 otherwise.  A zero or subnormal s (level 63 or more) gives 13 for any
// offset of at least -13; an infinite or NaN one gives 0.
__device__ __forceinline__ uint32_t d_level(float g1u, float g1v, float g2u, float g2v, int32_t offset) {
    const float s1 = __fadd_rn(__fmul_rn(g1u, g1u), __fmul_rn(g1v, g1v));
    const float s2 = __fadd_rn(__fmul_rn(g2u, g2u), __fmul_rn(g2v, g2v));
    if (s1 != s1 || s2 != s2) return 0u;
    const uint32_t b = __float_as_uint(fminf(s1, s2));
    const int be = (int)(b >> 23);   // s >= 0: the sign bit is clear
    if (be == 0) return 13u;
    if (be == 255) return 0u;
    const int E = be - 127;
    const int L = (b & 0x7FFFFFu) ? -((E + 2) >> 1) : -((E + 1) >> 1);
    return (uint32_t)min(13, max(0, L + offset));
}

__device__ __forceinline__ uint64_t d_key(uint32_t mat, uint32_t node, uint32_t level,
                                          uint32_t iu, uint32_t iv) {
    return ((uint64_t)mat << 48) | ((uint64_t)node << 32) | ((uint64_t)level << 26) |
           ((uint64_t)iu << 13) | (uint64_t)iv;
}

// Voxel of one position coordinate on a grid of 2^-level world units: floor(p 2^level)
// clamped to [-512, 511] and offset to [0, 1023]; p 2^level is exact in FP32 (a power-of-two
// scale), so the index is the same in any wider precision; NaN takes the lowest voxel.
__device__ __forceinline__ uint32_t d_voxel(float p, uint32_t level) {
    float x = p * __int_as_float((int)(127u + level) << 23);
    if (!(x >= -512.0f)) x = -512.0f;
    if (x > 511.0f) x = 511.0f;
    return (uint32_t)((int)floorf(x) + 512);
}

// World-position descriptor: (material, node, voxel of the position); bit 31 set.
__device__ __forceinline__ uint64_t d_key_pos(uint32_t mat, uint32_t node, uint32_t level, float px, float py,
                                              float pz) {
    return ((uint64_t)mat << 48) | ((uint64_t)node << 32) | (1ull << 31) | ((uint64_t)d_voxel(px, level) << 20) |
           ((uint64_t)d_voxel(py, level) << 10) | (uint64_t)d_voxel(pz, level);
}

__device__ __forceinline__ void d_address(uint64_t key, uint64_t n_cells, uint32_t pow2_mask,
                                          uint32_t* cell, uint32_t* h2) {
    uint64_t h1 = d_splitmix(key);
    *cell = pow2_mask ? (uint32_t)(h1 & (uint64_t)pow2_mask) : (uint32_t)(h1 % n_cells);
    uint32_t c = (uint32_t)(d_fmix64(key ^ 0x9E3779B97F4A7C15ull) >> 32);
    *h2 = c ? c : 1u;
}

// =======================================================================================
// Node primitives in FP32
// =======================================================================================
__device__ __forceinline__ uint32_t d_lattice(int i, int j, uint32_t seed) {
    // Teschner et al. 2003 primes, xor-combined, then fmix32
    return d_fmix32(((uint32_t)i * 73856093u) ^ ((uint32_t)j * 19349663u) ^ (seed * 83492791u));
}

// The 8 unit gradients at multiples of 45 degrees, indexed by hash & 7; each kernel that
// evaluates noise keeps a copy in shared memory (one 8-byte load per lattice corner).
__device__ __forceinline__ void init_gradients(float2* g) {
    if (threadIdx.x < 8) {
        const float R = 0.70710678118654752f;
        const float gx[8] = {1.0f, R, 0.0f, -R, -1.0f, -R, 0.0f, R};
        const float gy[8] = {0.0f, R, 1.0f, R, 0.0f, -R, -1.0f, -R};
        g[threadIdx.x] = make_float2(gx[threadIdx.x], gy[threadIdx.x]);
    }
}

// Pairs of independent FP32 operations issue as one instruction (Blackwell's packed FP32);
// each lane of a pair rounds exactly as the scalar operation would.
__device__ __forceinline__ float2 f2(float a, float b) { return make_float2(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }

// quintic fade 6t^5 - 15t^4 + 10t^3 of both coordinates at once
__device__ __forceinline__ float2 d_fade2(float2 t) {
    const float2 t3 = mul2(mul2(t, t), t);
    return mul2(t3, fma2(t, fma2(t, f2(6.0f, 6.0f), f2(-15.0f, -15.0f)), f2(10.0f, 10.0f)));
}

__device__ __forceinline__ float d_fade(float t) {
    return t * t * t * fmaf(t, fmaf(t, 6.0f, -15.0f), 10.0f);
}

__device__ __forceinline__ float d_perlin(float x, float y, uint32_t seed, const float2* grad) {
    const float2 p = f2(x, y);
    const float2 f0 = f2(floorf(x), floorf(y));
    const int ix = (int)f0.x, iy = (int)f0.y;
    const float2 fr = fma2(f0, f2(-1.0f, -1.0f), p);          // (fx, fy) = p - floor(p)
    const float2 fr1 = add2(fr, f2(-1.0f, -1.0f));            // (fx - 1, fy - 1)
    // lattice hashes of the four corners: the prime products of x + 1 and y + 1 are those
    // of x and y plus the prime
    const uint32_t ax = (uint32_t)ix * 73856093u, by = (uint32_t)iy * 19349663u, sz = seed * 83492791u;
    const uint32_t ax1 = ax + 73856093u, by1 = by + 19349663u;
    const float2 g00 = grad[d_fmix32(ax ^ by ^ sz) & 7u];
    const float2 g10 = grad[d_fmix32(ax1 ^ by ^ sz) & 7u];
    const float2 g01 = grad[d_fmix32(ax ^ by1 ^ sz) & 7u];
    const float2 g11 = grad[d_fmix32(ax1 ^ by1 ^ sz) & 7u];
    // corner dot products g . (p - corner), each as fmaf(gx, dx, gy dy); scalar, since the
    // corners' gradients arrive in separate registers
    const float2 dA = f2(fmaf(g00.x, fr.x, g00.y * fr.y), fmaf(g01.x, fr.x, g01.y * fr1.y));    // (d00, d01)
    const float2 dB = f2(fmaf(g10.x, fr1.x, g10.y * fr.y), fmaf(g11.x, fr1.x, g11.y * fr1.y));  // (d10, d11)
    const float2 s = d_fade2(fr);
    // (a, b) = dA + s.x (dB - dA); result = a + s.y (b - a)
    const float2 ab = fma2(f2(s.x, s.x), fma2(dA, f2(-1.0f, -1.0f), dB), dA);
    return fmaf(s.y, ab.y - ab.x, ab.x);
}

// ---- the fast form of the noise, for arguments below 2^22 in magnitude ------------------
// floor(x) through one addition of 1.5 x 2^23 rounded down: the sum's bits are FLOOR_BITS +
// floor(x), and subtracting the constant again gives floor(x) as a float.  Both additions are
// packed (two operations per instruction on the FMA pipe), where floorf and the conversion to
// an integer are two instructions per value on the quarter-rate conversion pipe.
constexpr uint32_t FLOOR_BITS = 0x4B400000u;
constexpr uint32_t PRIME_X = 73856093u, PRIME_Y = 19349663u, PRIME_S = 83492791u;

__device__ __forceinline__ float2 floor_sum2(float2 x) { return __fadd2_rd(x, f2(12582912.0f, 12582912.0f)); }
__device__ __forceinline__ float2 floor_of2(float2 t) { return add2(t, f2(-12582912.0f, -12582912.0f)); }
// (integer of a floor sum) x prime, modulo 2^32: the constant's share folds into the addend
__device__ __forceinline__ uint32_t floor_mul(float t, uint32_t prime) {
    return __float_as_uint(t) * prime + (0u - FLOOR_BITS * prime);
}

// The gradient of a lattice corner whose xor-combined prime products are h: fmix32, of which
// the gradient needs the low three bits.  The last multiplier carries a factor of 8, so the
// masked result is the byte offset of the 8-byte table entry.
__device__ __forceinline__ float2 lattice_grad(uint32_t h, const float2* grad) {
    h ^= h >> 16;
    h *= 0x85EBCA6Bu;
    h ^= h >> 13;
    h *= 0xC2B2AE35u << 3;
    return *reinterpret_cast<const float2*>(reinterpret_cast<const char*>(grad) + ((h ^ (h >> 16)) & 0x38u));
}

// Noise at two points A and B (|X|, |Y| < 2^22), every FP32 quantity held as an (A, B) pair so
// that each packed instruction serves both; (noise(A), noise(B)) with the roundings of
// d_perlin.  sz = seed x PRIME_S.
__device__ __forceinline__ float2 d_noise2(float2 X, float2 Y, uint32_t sz, const float2* grad) {
    const float2 tX = floor_sum2(X), tY = floor_sum2(Y);
    const float2 rX = fma2(floor_of2(tX), f2(-1.0f, -1.0f), X), rY = fma2(floor_of2(tY), f2(-1.0f, -1.0f), Y);
    const float2 rX1 = add2(rX, f2(-1.0f, -1.0f)), rY1 = add2(rY, f2(-1.0f, -1.0f));
    const uint32_t axA = floor_mul(tX.x, PRIME_X), byA = floor_mul(tY.x, PRIME_Y);
    const uint32_t axB = floor_mul(tX.y, PRIME_X), byB = floor_mul(tY.y, PRIME_Y);
    const uint32_t axA1 = axA + PRIME_X, byA1 = byA + PRIME_Y;
    const uint32_t axB1 = axB + PRIME_X, byB1 = byB + PRIME_Y;
    const float2 a00 = lattice_grad(axA ^ byA ^ sz, grad), b00 = lattice_grad(axB ^ byB ^ sz, grad);
    const float2 a10 = lattice_grad(axA1 ^ byA ^ sz, grad), b10 = lattice_grad(axB1 ^ byB ^ sz, grad);
    const float2 a01 = lattice_grad(axA ^ byA1 ^ sz, grad), b01 = lattice_grad(axB ^ byB1 ^ sz, grad);
    const float2 a11 = lattice_grad(axA1 ^ byA1 ^ sz, grad), b11 = lattice_grad(axB1 ^ byB1 ^ sz, grad);
    const float2 d00 = f2(fmaf(a00.x, rX.x, a00.y * rY.x), fmaf(b00.x, rX.y, b00.y * rY.y));
    const float2 d10 = f2(fmaf(a10.x, rX1.x, a10.y * rY.x), fmaf(b10.x, rX1.y, b10.y * rY.y));
    const float2 d01 = f2(fmaf(a01.x, rX.x, a01.y * rY1.x), fmaf(b01.x, rX.y, b01.y * rY1.y));
    const float2 d11 = f2(fmaf(a11.x, rX1.x, a11.y * rY1.x), fmaf(b11.x, rX1.y, b11.y * rY1.y));
    const float2 sX = d_fade2(rX), sY = d_fade2(rY);
    const float2 a = fma2(sX, fma2(d00, f2(-1.0f, -1.0f), d10), d00);
    const float2 b = fma2(sX, fma2(d01, f2(-1.0f, -1.0f), d11), d01);
    return fma2(sY, fma2(a, f2(-1.0f, -1.0f), b), a);
}

// The same at one point p = (x, y), the pairs holding its two coordinates.
__device__ __forceinline__ float d_noise(float2 p, uint32_t sz, const float2* grad) {
    const float2 t = floor_sum2(p);
    const float2 fr = fma2(floor_of2(t), f2(-1.0f, -1.0f), p);
    const float2 fr1 = add2(fr, f2(-1.0f, -1.0f));
    const uint32_t ax = floor_mul(t.x, PRIME_X), by = floor_mul(t.y, PRIME_Y);
    const uint32_t ax1 = ax + PRIME_X, by1 = by + PRIME_Y;
    const float2 g00 = lattice_grad(ax ^ by ^ sz, grad), g10 = lattice_grad(ax1 ^ by ^ sz, grad);
    const float2 g01 = lattice_grad(ax ^ by1 ^ sz, grad), g11 = lattice_grad(ax1 ^ by1 ^ sz, grad);
    const float2 dA = f2(fmaf(g00.x, fr.x, g00.y * fr.y), fmaf(g01.x, fr.x, g01.y * fr1.y));
    const float2 dB = f2(fmaf(g10.x, fr1.x, g10.y * fr.y), fmaf(g11.x, fr1.x, g11.y * fr1.y));
    const float2 s = d_fade2(fr);
    const float2 ab = fma2(f2(s.x, s.x), fma2(dA, f2(-1.0f, -1.0f), dB), dA);
    return fmaf(s.y, ab.y - ab.x, ab.x);
}

// clamp to [0, 1] (NaN to 0) as a saturating modifier of the producing instruction
__device__ __forceinline__ float d_clamp01(float x) { return __saturatef(x); }

// q = {scale, lacunarity, gain, 1 / sum of gains}, t = {octaves, seed, limit} (the first two
// integers in floats): below the limit in magnitude, every octave's argument is below 2^22 and
// the fast noise applies; beyond it (and for NaN) d_perlin, with the same results where both do.
__device__ __forceinline__ float d_fbm(float x, float y, const float4 q, const float4 t, const float2* grad) {
    const float scale = q.x, lac = q.y, gain = q.z, inv_norm = q.w;
    const int oct = __float_as_int(t.x);
    const uint32_t seed = (uint32_t)__float_as_int(t.y);
    float sum = 0.0f, amp = 1.0f, freq = scale;
    if (fabsf(x) < t.z && fabsf(y) < t.z) {
        uint32_t sz = seed * PRIME_S;
        for (int k = 0; k < oct; ++k) {
            sum = fmaf(amp, d_noise(mul2(f2(x, y), f2(freq, freq)), sz, grad), sum);
            sz += PRIME_S;
            const float2 af = mul2(f2(amp, freq), f2(gain, lac));
            amp = af.x;
            freq = af.y;
        }
    } else {
#pragma unroll 1
        for (int k = 0; k < oct; ++k) {
            sum = fmaf(amp, d_perlin(x * freq, y * freq, seed + (uint32_t)k, grad), sum);
            const float2 af = mul2(f2(amp, freq), f2(gain, lac));
            amp = af.x;
            freq = af.y;
        }
    }
    return d_clamp01(fmaf(sum, inv_norm, 0.5f));
}

// d_fbm at two points in one octave loop (the amplitude and frequency updates are shared)
__device__ __forceinline__ float2 d_fbm2(float2 X, float2 Y, const float4 q, const float4 t, const float2* grad) {
    const float scale = q.x, lac = q.y, gain = q.z, inv_norm = q.w;
    const int oct = __float_as_int(t.x);
    const uint32_t seed = (uint32_t)__float_as_int(t.y);
    float2 sum = f2(0.0f, 0.0f);
    float amp = 1.0f, freq = scale;
    if (fabsf(X.x) < t.z && fabsf(X.y) < t.z && fabsf(Y.x) < t.z && fabsf(Y.y) < t.z) {
        uint32_t sz = seed * PRIME_S;
        for (int k = 0; k < oct; ++k) {
            const float2 n = d_noise2(mul2(X, f2(freq, freq)), mul2(Y, f2(freq, freq)), sz, grad);
            sum = fma2(f2(amp, amp), n, sum);
            sz += PRIME_S;
            const float2 af = mul2(f2(amp, freq), f2(gain, lac));
            amp = af.x;
            freq = af.y;
        }
    } else {
#pragma unroll 1
        for (int k = 0; k < oct; ++k) {
            float n[2];
#pragma unroll 1
            for (int i = 0; i < 2; ++i)
                n[i] = d_perlin((i ? X.y : X.x) * freq, (i ? Y.y : Y.x) * freq, seed + (uint32_t)k, grad);
            sum = fma2(f2(amp, amp), f2(n[0], n[1]), sum);
            const float2 af = mul2(f2(amp, freq), f2(gain, lac));
            amp = af.x;
            freq = af.y;
        }
    }
    const float2 r = fma2(sum, f2(inv_norm, inv_norm), f2(0.5f, 0.5f));
    return f2(d_clamp01(r.x), d_clamp01(r.y));
}

// x ^ (x >> 16), the first step of fmix32.  It is linear over xor, so applied to the prime
// products of the three columns, the three rows and the seed it serves all nine cells.
__device__ __forceinline__ uint32_t fold16(uint32_t x) { return x ^ (x >> 16); }

// Worley F1.  q = {scale, seed (an integer in a float), limit}: below the limit in magnitude the
// floor goes through floor_sum2, beyond it through floorf, with the same results where both
// apply.
__device__ __forceinline__ float d_voronoi(float x, float y, const float4 q) {
    const float2 sc = mul2(f2(x, y), f2(q.x, q.x));
    float2 f0;
    uint32_t ax, by;
    if (fabsf(x) < q.z && fabsf(y) < q.z) {
        const float2 t = floor_sum2(sc);
        f0 = floor_of2(t);
        ax = floor_mul(t.x, PRIME_X);
        by = floor_mul(t.y, PRIME_Y);
    } else {
        f0 = f2(floorf(sc.x), floorf(sc.y));
        ax = (uint32_t)(int)f0.x * PRIME_X;
        by = (uint32_t)(int)f0.y * PRIME_Y;
    }
    const float2 fr = fma2(f0, f2(-1.0f, -1.0f), sc);
    const uint32_t sz = fold16((uint32_t)__float_as_int(q.y) * PRIME_S);
    const uint32_t col[3] = {fold16(ax - PRIME_X), fold16(ax), fold16(ax + PRIME_X)};
    const uint32_t row[3] = {fold16(by - PRIME_Y) ^ sz, fold16(by) ^ sz, fold16(by + PRIME_Y) ^ sz};
    float best = 3.0e38f;
#pragma unroll
    for (int b = -1; b <= 1; ++b) {
#pragma unroll
        for (int a = -1; a <= 1; ++a) {
            uint32_t h = col[a + 1] ^ row[b + 1];
            h *= 0x85EBCA6Bu;
            h ^= h >> 13;
            h *= 0xC2B2AE35u;
            // the halves of h ^ (h >> 16) as the floats 2^23 + h16: the upper half is the shift
            // itself.  Feature point at cell + 0.25 + 0.5 h16 2^-16 per axis: one fused operation
            // with exact constants, (2^23 + h16) 2^-17 + (a + 0.25 - 64)
            const uint32_t hi = h >> 16;
            const float2 m = f2(__uint_as_float(__byte_perm(h ^ hi, 0x4B000000u, 0x7610)), __uint_as_float(hi | 0x4B000000u));
            const float2 o = fma2(m, f2(0x1p-17f, 0x1p-17f), f2((float)a - 63.75f, (float)b - 63.75f));
            const float2 d = fma2(fr, f2(-1.0f, -1.0f), o);
            best = fminf(best, fmaf(d.x, d.x, d.y * d.y));
        }
    }
    // sqrt(best) as best / sqrt(best) through the reciprocal square root (within a few ulp);
    // best = 0 gives 0 x inf = NaN, which the clamp maps to 0 = sqrt(0)
    return d_clamp01(best * rsqrtf(best));
}

// Parity of an integer-valued FP32 number f as 0 or 1: f - 2 floor(f / 2), exact for every
// finite f (integers beyond 2^24 are even, and the formula gives 0 there).
__device__ __forceinline__ float d_parity(float f) { return fmaf(-2.0f, floorf(f * 0.5f), f); }

struct PointIn {
    float u, v, px, py, pz, nx, ny, nz;
};

// Where a point's inputs come from: registers (the points made by a kernel itself) or the
// grouped arrays.  An interpreter that reads them where its program's input nodes run, instead of
// holding eight floats a point across the whole program, has those registers for the nodes.
struct PointRegs {
    PointIn p;
    __device__ __forceinline__ float u() const { return p.u; }
    __device__ __forceinline__ float v() const { return p.v; }
    __device__ __forceinline__ float px() const { return p.px; }
    __device__ __forceinline__ float py() const { return p.py; }
    __device__ __forceinline__ float pz() const { return p.pz; }
    __device__ __forceinline__ float nx() const { return p.nx; }
    __device__ __forceinline__ float ny() const { return p.ny; }
    __device__ __forceinline__ float nz() const { return p.nz; }
};
struct PointMem {
    const BatchArgs& a;
    uint32_t s;   // grouped index
    __device__ __forceinline__ float u() const { return a.su[s]; }
    __device__ __forceinline__ float v() const { return a.sv[s]; }
    __device__ __forceinline__ float px() const { return a.spx[s]; }
    __device__ __forceinline__ float py() const { return a.spy[s]; }
    __device__ __forceinline__ float pz() const { return a.spz[s]; }
    __device__ __forceinline__ float nx() const { return a.snx[s]; }
    __device__ __forceinline__ float ny() const { return a.sny[s]; }
    __device__ __forceinline__ float nz() const { return a.snz[s]; }
};

// A node's value in the lane's slot file, laid out [row][lane] per warp: one row per channel,
// or a single row for a value whose three channels are equal (noise, Worley, facing and the
// arithmetic on them), so that such a node computes, stores and keeps one channel.  Programs name
// rows by byte offsets from the lane's base (of rows of one point per lane), so an operand is
// one add away from its address.  V = float: one point per lane, float2: two (A = .x, B = .y).
template <class V>
struct Slots {
    static constexpr uint32_t W = sizeof(V) / sizeof(float);
    static constexpr uint32_t CH = ROW_BYTES * W;   // bytes from channel to channel
    static __device__ __forceinline__ const char* at(const char* Vb, uint32_t off) { return Vb + W * off; }
    static __device__ __forceinline__ V get(const char* p, int ch) { return *reinterpret_cast<const V*>(p + ch * CH); }
    static __device__ __forceinline__ void put(char* Vb, uint32_t off, V r0, V r1, V r2) {
        V* o = reinterpret_cast<V*>(Vb + W * off);
        o[0] = r0;
        o[32] = r1;
        o[64] = r2;
    }
    // equal channels: one row, or three for a value that others read by channel
    static __device__ __forceinline__ void put1(char* Vb, uint32_t off, bool one, V r) {
        V* o = reinterpret_cast<V*>(Vb + W * off);
        o[0] = r;
        if (!one) {   // uniform
            o[32] = r;
            o[64] = r;
        }
    }
};
__device__ __forceinline__ float slot_ch(const char* Vb, uint32_t off, int ch) {
    return Slots<float>::get(Slots<float>::at(Vb, off), ch);
}
__device__ __forceinline__ void slot_store(char* Vb, uint32_t off, float r0, float r1, float r2) {
    Slots<float>::put(Vb, off, r0, r1, r2);
}
__device__ __forceinline__ float2 slot2(const char* Vb, uint32_t off, int ch) {
    return Slots<float2>::get(Slots<float2>::at(Vb, off), ch);
}
__device__ __forceinline__ void slot2_store(char* Vb, uint32_t off, float2 r0, float2 r1, float2 r2) {
    Slots<float2>::put(Vb, off, r0, r1, r2);
}
__device__ __forceinline__ float2 sat2(float2 x) { return f2(d_clamp01(x.x), d_clamp01(x.y)); }

// The arithmetic of a node for one point (float) or two (float2); every lane of a pair rounds
// as the scalar form does.
__device__ __forceinline__ float v_sat(float x) { return d_clamp01(x); }
__device__ __forceinline__ float2 v_sat(float2 x) { return sat2(x); }
template <class V>
__device__ __forceinline__ V v_set(float x);
template <>
__device__ __forceinline__ float v_set<float>(float x) { return x; }
template <>
__device__ __forceinline__ float2 v_set<float2>(float x) { return f2(x, x); }
__device__ __forceinline__ float v_fma(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ float2 v_fma(float2 a, float2 b, float2 c) { return fma2(a, b, c); }
__device__ __forceinline__ float v_add(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float2 v_add(float2 a, float2 b) { return add2(a, b); }
__device__ __forceinline__ float v_mul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float2 v_mul(float2 a, float2 b) { return mul2(a, b); }
__device__ __forceinline__ float v_abs(float a) { return fabsf(a); }
__device__ __forceinline__ float2 v_abs(float2 a) { return f2(fabsf(a.x), fabsf(a.y)); }
// x^e for x >= 0 through the hardware base-2 logarithm and exponential (__powf); x = 0 gives 0
// for every e > 0
__device__ __forceinline__ float v_pow(float a, float e) { return __powf(fmaxf(a, 0.0f), e); }
__device__ __forceinline__ float2 v_pow(float2 a, float e) { return f2(v_pow(a.x, e), v_pow(a.y, e)); }
__device__ __forceinline__ float v_fbm(float x, float y, const float4 q, const float4 t, const float2* grad) {
    return d_fbm(x, y, q, t, grad);
}
__device__ __forceinline__ float2 v_fbm(float2 x, float2 y, const float4 q, const float4 t, const float2* grad) {
    return d_fbm2(x, y, q, t, grad);
}
__device__ __forceinline__ float v_voronoi(float x, float y, const float4 q) { return d_voronoi(x, y, q); }
__device__ __forceinline__ float2 v_voronoi(float2 x, float2 y, const float4 q) {
    return f2(d_voronoi(x.x, y.x, q), d_voronoi(x.y, y.y, q));
}
// colour B iff floor(x s) + floor(y s) is odd, i.e. the two parities differ
__device__ __forceinline__ bool checker_odd(float x, float y, float s) {
    const float2 f = mul2(f2(x, y), f2(s, s));
    return d_parity(floorf(f.x)) != d_parity(floorf(f.y));
}

// Piecewise linear ramp at t.  Parameters: {first stop, last stop, second, third (2 if absent)},
// (stop, 1 / segment length) of segments 0..2, padding, colours of stops 0..3 and of the last
// stop, four floats each.
__device__ __forceinline__ void d_ramp(float x, const float* p, const float4 q, float (&o)[3]) {
    const float4* p4 = reinterpret_cast<const float4*>(p);
    const float t = d_clamp01(x);
    const int k = (t >= q.z ? 1 : 0) + (t >= q.w ? 1 : 0);   // interior stops at or below t
    const float2 seg = __ldg(reinterpret_cast<const float2*>(p + 4) + k);
    const float4 ca = __ldg(p4 + 3 + k);
    const float4 cb = __ldg(p4 + 4 + k);
    const float w = (t - seg.x) * seg.y;
    o[0] = fmaf(w, cb.x - ca.x, ca.x);
    o[1] = fmaf(w, cb.y - ca.y, ca.y);
    o[2] = fmaf(w, cb.z - ca.z, ca.z);
    if (t <= q.x) {
        const float4 c0 = __ldg(p4 + 3);
        o[0] = c0.x; o[1] = c0.y; o[2] = c0.z;
    } else if (t >= q.y) {
        const float4 cl = __ldg(p4 + 7);
        o[0] = cl.x; o[1] = cl.y; o[2] = cl.z;
    }
}

// OP per channel of two inputs, with one row (ONE) or three each.
template <class V, bool ONE0, bool ONE1, class OP>
__device__ __forceinline__ void binary_node(char* Vb, const uint4& ins, OP op) {
    using S = Slots<V>;
    const char* a = S::at(Vb, ins.y >> 16);
    const char* b = S::at(Vb, ins.z & 0xFFFFu);
    const uint32_t out = ins.y & 0xFFFFu;
    if (ONE0 && ONE1) {
        S::put1(Vb, out, (ins.x >> 8) & FLAG_ONE_ROW, op(S::get(a, 0), S::get(b, 0)));
    } else {
        const V r0 = op(S::get(a, 0), S::get(b, 0)), r1 = op(S::get(a, ONE0 ? 0 : 1), S::get(b, ONE1 ? 0 : 1)),
                r2 = op(S::get(a, ONE0 ? 0 : 2), S::get(b, ONE1 ? 0 : 2));
        S::put(Vb, out, r0, r1, r2);
    }
}

// One node instruction for one lane, for one point (V = float; A) or two (V = float2: one
// decode, dispatch and parameter load serve both, and their two independent computations
// overlap).  Vb is the lane's base in the slot file.  What kind of rows an operand has is part
// of the operator (DOP_*), so that nothing is tested for it here; every case stores its own
// result, and no values merge after the switch.
template <class V, class PT>
__device__ __forceinline__ void exec_points(const uint4& ins, char* Vb, const PT& A, const PT& B,
                                            const float* __restrict__ params, const float2* grad) {
    using S = Slots<V>;
    constexpr bool TWO = S::W == 2;
    const V zero = v_set<V>(0.0f);
    const uint32_t out = ins.y & 0xFFFFu;
    const bool one = (ins.x >> 8) & FLAG_ONE_ROW;
    const char* i0 = S::at(Vb, ins.y >> 16);
    // a node's parameters start on a 16-byte boundary: vector loads fetch them
    const float* p = params + ins.w;
    const float4* p4 = reinterpret_cast<const float4*>(p);
#define PMC_PICK(f) [&]() -> V { if constexpr (TWO) return f2(A.f(), B.f()); else return A.f(); }()
    auto mix_f = [&](bool node) -> V {
        return v_sat(node ? S::get(S::at(Vb, ins.z >> 16), 0) : v_set<V>(__ldg(p)));
    };
    // a + f (b - a), clamped
    auto mix = [&](V f) {
        return [f](V a, V b) { return v_sat(v_fma(f, v_fma(a, v_set<V>(-1.0f), b), a)); };
    };
    auto add = [](V a, V b) { return v_sat(v_add(a, b)); };
    auto mul = [](V a, V b) { return v_sat(v_mul(a, b)); };
    switch (ins.x & 0xFFu) {
    case DOP_UV: S::put(Vb, out, PMC_PICK(u), PMC_PICK(v), zero); break;
    case DOP_POSITION: S::put(Vb, out, PMC_PICK(px), PMC_PICK(py), PMC_PICK(pz)); break;
    case DOP_NORMAL: S::put(Vb, out, PMC_PICK(nx), PMC_PICK(ny), PMC_PICK(nz)); break;
    case DOP_CONST: {
        const float4 q = __ldg(p4);
        S::put(Vb, out, v_set<V>(q.x), v_set<V>(q.y), v_set<V>(q.z));
        break;
    }
    case DOP_CONST_1: S::put1(Vb, out, true, v_set<V>(__ldg(p))); break;
    case DOP_AFFINE: {
        const float4 q = __ldg(p4);
        const float4 t = __ldg(p4 + 1);
        const V x = S::get(i0, 0), y = S::get(i0, ((ins.x >> 8) & FLAG_ONE_IN) ? 0 : 1);
        S::put(Vb, out, v_fma(v_set<V>(q.x), x, v_fma(v_set<V>(q.y), y, v_set<V>(t.x))),
               v_fma(v_set<V>(q.z), x, v_fma(v_set<V>(q.w), y, v_set<V>(t.y))), zero);
        break;
    }
    case DOP_FBM: {
        const float4 q = __ldg(p4);
        const float4 t = __ldg(p4 + 1);
        S::put1(Vb, out, one, v_fbm(S::get(i0, 0), S::get(i0, ((ins.x >> 8) & FLAG_ONE_IN) ? 0 : 1), q, t, grad));
        break;
    }
    case DOP_VORONOI:
        S::put1(Vb, out, one, v_voronoi(S::get(i0, 0), S::get(i0, ((ins.x >> 8) & FLAG_ONE_IN) ? 0 : 1), __ldg(p4)));
        break;
    case DOP_CHECKER: {
        const float4 q = __ldg(p4);
        const float4 t = __ldg(p4 + 1);
        const V x = S::get(i0, 0), y = S::get(i0, 1);
        if constexpr (TWO) {
            const bool oa = checker_odd(x.x, y.x, q.x), ob = checker_odd(x.y, y.y, q.x);
            S::put(Vb, out, sat2(f2(oa ? t.x : q.y, ob ? t.x : q.y)), sat2(f2(oa ? t.y : q.z, ob ? t.y : q.z)),
                   sat2(f2(oa ? t.z : q.w, ob ? t.z : q.w)));
        } else {
            const bool odd = checker_odd(x, y, q.x);
            S::put(Vb, out, d_clamp01(odd ? t.x : q.y), d_clamp01(odd ? t.y : q.z), d_clamp01(odd ? t.z : q.w));
        }
        break;
    }
    case DOP_RAMP: {
        const float4 q = __ldg(p4);
        const V t = S::get(i0, 0);
        if constexpr (TWO) {
            float x[3], y[3];
            d_ramp(t.x, p, q, x);
            d_ramp(t.y, p, q, y);
            S::put(Vb, out, sat2(f2(x[0], y[0])), sat2(f2(x[1], y[1])), sat2(f2(x[2], y[2])));
        } else {
            float x[3];
            d_ramp(t, p, q, x);
            S::put(Vb, out, d_clamp01(x[0]), d_clamp01(x[1]), d_clamp01(x[2]));
        }
        break;
    }
    case DOP_MIX_33: binary_node<V, false, false>(Vb, ins, mix(mix_f(false))); break;
    case DOP_MIX_31: binary_node<V, false, true>(Vb, ins, mix(mix_f(false))); break;
    case DOP_MIX_13: binary_node<V, true, false>(Vb, ins, mix(mix_f(false))); break;
    case DOP_MIX_11: binary_node<V, true, true>(Vb, ins, mix(mix_f(false))); break;
    case DOP_MIXN_33: binary_node<V, false, false>(Vb, ins, mix(mix_f(true))); break;
    case DOP_MIXN_31: binary_node<V, false, true>(Vb, ins, mix(mix_f(true))); break;
    case DOP_MIXN_13: binary_node<V, true, false>(Vb, ins, mix(mix_f(true))); break;
    case DOP_MIXN_11: binary_node<V, true, true>(Vb, ins, mix(mix_f(true))); break;
    case DOP_ADD_33: binary_node<V, false, false>(Vb, ins, add); break;
    case DOP_ADD_31: binary_node<V, false, true>(Vb, ins, add); break;
    case DOP_ADD_11: binary_node<V, true, true>(Vb, ins, add); break;
    case DOP_MUL_33: binary_node<V, false, false>(Vb, ins, mul); break;
    case DOP_MUL_31: binary_node<V, false, true>(Vb, ins, mul); break;
    case DOP_MUL_11: binary_node<V, true, true>(Vb, ins, mul); break;
    case DOP_POW_3: {
        const float e = __ldg(p);
        const V x0 = S::get(i0, 0), x1 = S::get(i0, 1), x2 = S::get(i0, 2);
        S::put(Vb, out, v_sat(v_pow(x0, e)), v_sat(v_pow(x1, e)), v_sat(v_pow(x2, e)));
        break;
    }
    case DOP_POW_1: S::put1(Vb, out, one, v_sat(v_pow(S::get(i0, 0), __ldg(p)))); break;
    case DOP_FACING: {
        const float4 q = __ldg(p4);
        const bool in1 = (ins.x >> 8) & FLAG_ONE_IN;
        const V d = v_fma(S::get(i0, 0), v_set<V>(q.x),
                          v_fma(S::get(i0, in1 ? 0 : 1), v_set<V>(q.y), v_mul(S::get(i0, in1 ? 0 : 2), v_set<V>(q.z))));
        S::put1(Vb, out, one, v_sat(v_abs(d)));
        break;
    }
    default: __builtin_unreachable();   // the compiler emits no other operator here
    }
#undef PMC_PICK
}

}  // namespace pmc
