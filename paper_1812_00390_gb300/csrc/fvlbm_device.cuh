// Device-side helpers shared by the library's CUDA translation units: the
// D2Q9 lattice of Sec. 2.1 and the storage formats of the state.
#pragma once

#include <cuda_runtime.h>
#include <cuda_fp16.h>
#include <cuda_bf16.h>

#include "fvlbm_internal.h"

namespace fvlbm {

#define EXA(a) ((a) == 1 || (a) == 5 || (a) == 8 ? 1 : ((a) == 3 || (a) == 6 || (a) == 7 ? -1 : 0))
#define EYA(a) ((a) == 2 || (a) == 5 || (a) == 6 ? 1 : ((a) == 4 || (a) == 7 || (a) == 8 ? -1 : 0))

template <typename T>
__device__ __forceinline__ T wgt(int a) {
    return a == 0 ? T(4.0 / 9.0) : (a < 5 ? T(1.0 / 9.0) : T(1.0 / 36.0));
}

// A product that is rounded by itself.  Which of two products in a sum the
// compiler fuses depends on the code around it; where a value is computed in
// several kernels (stage kernels, resident loop, storage formats), the
// operations that could fuse either way are written out, so that all give the
// same bits.
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }

// acc + e v for a velocity component e of -1, 0 or 1 (known when unrolled; a
// product with 0 would be kept, since it is not 0 for an infinite v).
template <typename T> __device__ __forceinline__ T add_e(int e, T acc, T v) {
    return e == 0 ? acc : (e > 0 ? acc + v : acc - v);
}
// e_a . u
template <typename T> __device__ __forceinline__ T dot_e(int a, T ux, T uy) {
    const T x = EXA(a) > 0 ? ux : -ux;
    if (EYA(a) == 0) return EXA(a) == 0 ? T(0) : x;
    if (EXA(a) == 0) return EYA(a) > 0 ? uy : -uy;
    return EYA(a) > 0 ? x + uy : x - uy;
}

// Density and velocity (Sec. 2.1).  FP64 mode: r = rho = sum f.  Deviation
// mode: r = rho - 1 = sum g, kept unrounded by the 1 so that the density
// deviation keeps FP32 relative precision.  FP64 sums by opposite pairs (16
// operations instead of 18, and four lanes that hold a pair each can form the
// same sums: see fvlbm_resident.cuh).
template <typename T, bool DEV>
__device__ __forceinline__ void moments(const T* f, T& r, T& ux, T& uy) {
    T s = 0, mx = 0, my = 0;
    if constexpr (DEV) {
#pragma unroll
        for (int a = 0; a < FVLBM_Q; a++) {
            s += f[a];
            mx = add_e(EXA(a), mx, f[a]);
            my = add_e(EYA(a), my, f[a]);
        }
    } else {
        const T d2 = f[5] - f[7], d3 = f[6] - f[8];
        s = f[0] + (((f[1] + f[3]) + (f[2] + f[4])) + ((f[5] + f[7]) + (f[6] + f[8])));
        mx = (f[1] - f[3]) + (d2 - d3);
        my = (f[2] - f[4]) + (d2 + d3);
    }
    r = s;
    const T inv_rho = T(1) / (DEV ? T(1) + s : s);
    ux = mul_rn(mx, inv_rho);
    uy = mul_rn(my, inv_rho);
}
// u^2
template <typename T> __device__ __forceinline__ T square(T ux, T uy) { return fma(ux, ux, mul_rn(uy, uy)); }

// Eq. (feq).  FP64 mode: r = rho, returns f^eq.  Deviation mode: r = rho - 1,
// returns f^eq - w = w [(rho - 1) + rho (3 e.u + 4.5 (e.u)^2 - 1.5 u^2)].
// The polynomial is evaluated as e.u (3 + 4.5 e.u) - 1.5 u^2 (two fused
// multiply-adds per direction once u^2 is known).
// feq_factor * feq_value: the two factors of the product, for sums that fuse it.
template <typename T, bool DEV> __device__ __forceinline__ T feq_factor(int a, T r) {
    return DEV ? wgt<T>(a) : r * wgt<T>(a);
}
template <typename T, bool DEV>
__device__ __forceinline__ T feq_value(int a, T r, T ux, T uy) {
    const T eu = dot_e(a, ux, uy);
    const T poly = fma(T(4.5), eu, T(3)), uu = square(ux, uy);
    if (DEV) return fma(T(1) + r, fma(eu, poly, -(T(1.5) * uu)), r);
    return fma(eu, poly, fma(T(-1.5), uu, T(1)));
}
template <typename T, bool DEV>
__device__ __forceinline__ T feqs(int a, T r, T ux, T uy) {
    return mul_rn(feq_factor<T, DEV>(a, r), feq_value<T, DEV>(a, r, ux, uy));
}

// Density argument of feqs for a given density.
template <typename T, bool DEV>
__device__ __forceinline__ T rarg(double rho) { return DEV ? T(rho - 1.0) : T(rho); }

// ------------------------------------------------------------------ pairs
// The eight moving directions in four opposite pairs p = (A, B): (1, 3),
// (2, 4), (5, 7), (6, 8).  e_B = -e_A, so that on every face one direction of
// each pair leaves the cell and the other enters it, and the pair shares e.n
// up to its sign.  State, gradients and fluxes are handled a pair at a time:
// in FP32 as packed operations (two FP32 operations per issued instruction;
// GB300 issues FFMA with three distinct registers at 2.4 warp instructions per
// clock and SM, the packed form at 1.9, i.e. 3.8), each half rounded exactly as
// the scalar operation.
__host__ __device__ constexpr int dir_a(int p) { return p == 0 ? 1 : p == 1 ? 2 : p == 2 ? 5 : 6; }
__host__ __device__ constexpr int dir_b(int p) { return p == 0 ? 3 : p == 1 ? 4 : p == 2 ? 7 : 8; }

template <typename T> struct Pair;
template <> struct Pair<float> {
    unsigned long long v;
};
template <> struct Pair<double> {
    double x, y;
};
__device__ __forceinline__ Pair<float> make_pair2(float x, float y) {
    Pair<float> r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(x), "f"(y));
    return r;
}
__device__ __forceinline__ Pair<double> make_pair2(double x, double y) { return {x, y}; }
__device__ __forceinline__ void split2(const Pair<float>& a, float& x, float& y) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(a.v));
}
__device__ __forceinline__ void split2(const Pair<double>& a, double& x, double& y) {
    x = a.x;
    y = a.y;
}
// a * b + c, each half one fused multiply-add
__device__ __forceinline__ Pair<float> fma2(const Pair<float>& a, const Pair<float>& b, const Pair<float>& c) {
    Pair<float> r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
    return r;
}
__device__ __forceinline__ Pair<double> fma2(const Pair<double>& a, const Pair<double>& b, const Pair<double>& c) {
    return {fma(a.x, b.x, c.x), fma(a.y, b.y, c.y)};
}
__device__ __forceinline__ Pair<float> sub2(const Pair<float>& a, const Pair<float>& b) {
    Pair<float> r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ Pair<double> sub2(const Pair<double>& a, const Pair<double>& b) {
    return {a.x - b.x, a.y - b.y};
}

// Four values of type T (the values that leave a cell through one face, one
// per pair; or two pairs) in 16-byte units: one for FP32, two for FP64.
template <typename T> struct Quad {
    T v[4];
};
template <typename T> struct Vec16;   // the 16-byte vector of T
template <> struct Vec16<float> {
    typedef float4 type;
    static constexpr int N = 4;
};
template <> struct Vec16<double> {
    typedef double2 type;
    static constexpr int N = 2;
};
// 16-byte units in a Quad
template <typename T> constexpr int QUAD_UNITS = sizeof(T) / 4;
// A Quad kept in planes: unit u at base[u * stride] (a warp's consecutive rows
// are then 16 bytes apart: no bank conflict, whole lines in global memory).
__device__ __forceinline__ Quad<float> load_quad(const float4* base, int64_t) {
    const float4 a = base[0];
    return {{a.x, a.y, a.z, a.w}};
}
__device__ __forceinline__ Quad<double> load_quad(const double2* base, int64_t stride) {
    const double2 a = base[0], b = base[stride];
    return {{a.x, a.y, b.x, b.y}};
}
__device__ __forceinline__ void store_quad(float4* base, int64_t, const Quad<float>& q) {
    base[0] = make_float4(q.v[0], q.v[1], q.v[2], q.v[3]);
}
__device__ __forceinline__ void store_quad(double2* base, int64_t stride, const Quad<double>& q) {
    base[0] = make_double2(q.v[0], q.v[1]);
    base[stride] = make_double2(q.v[2], q.v[3]);
}

// ------------------------------------------------------------------ storage
// Per-cell arrays are stored in blocks of BLK = 32 consecutive cells (internal
// order).  The state of a block is a row of 16-byte units per cell for the
// pairs of directions, then the remaining values:
//   float    [2][32] float4 (pairs 0, 1 | pairs 2, 3), [32] float f_0
//   double   [4][32] double2 (pairs 0..3), [32] double f_0
//   16-bit   [32] uint4 (rho - 1, rho u_x, rho u_y, n_3 n_4), [32] uint2 (n_5 n_6, n_7 n_8)
// so that a cell moves in two or three vector accesses instead of nine, and a
// halo cell touches 2-3 sectors of 32 bytes instead of nine.
__host__ __device__ __forceinline__ int64_t blk_index(int64_t i, int ncomp) {
    return (i >> BLK_SHIFT) * ((int64_t)ncomp << BLK_SHIFT) + (i & (BLK - 1));
}
// The same in 32-bit arithmetic, for the fused stage kernel, whose solvers
// keep every blocked array below 2^32 elements (checked at set-up).
__host__ __device__ __forceinline__ uint32_t blk_index(uint32_t i, int ncomp) {
    return (i >> BLK_SHIFT) * ((uint32_t)ncomp << BLK_SHIFT) + (i & (BLK - 1));
}

// Whole-cell access to the stored state (T: arithmetic type, DEV: deviation
// mode, the stored quantity is g = f - w).
//  double / float   9 components per cell: g_a (f_a in FP64 mode).
//  __half / bf16    split format: 3 FP32 components rho - 1, rho u_x, rho u_y,
//                   then the six 16-bit non-equilibrium parts
//                   n_a = g_a - g^eq_a(rho, u) of directions a = 3..8, times
//                   a power-of-two scale per (instance, direction), packed in
//                   pairs into three 32-bit components.
//                   n_0, n_1, n_2 follow from sum_a n_a = 0 and
//                   sum_a e_a n_a = 0 (the non-equilibrium part carries no mass
//                   or momentum), so rho and u never round through 16 bits;
//                   only the small non-equilibrium part does.
template <typename S> struct CellIO;

template <typename S> struct PlainIO {
    typedef typename Vec16<S>::type V;
    static constexpr int UNITS = 8 / Vec16<S>::N;    // 16-byte units of the eight moving directions
    static constexpr int64_t BLOCK_BYTES = (int64_t)FVLBM_Q * BLK * sizeof(S);
    // unit u of cell i at pairs(base, i)[u * BLK]; f_0 at rest(base, i)
    template <typename I> __device__ __forceinline__ static const V* pairs(const void* base, I i) {
        return (const V*)((const unsigned char*)base + (size_t)(i >> BLK_SHIFT) * BLOCK_BYTES) + (i & (BLK - 1));
    }
    template <typename I> __device__ __forceinline__ static const S* rest(const void* base, I i) {
        return (const S*)((const unsigned char*)base + (size_t)(i >> BLK_SHIFT) * BLOCK_BYTES + 8 * BLK * sizeof(S)) +
               (i & (BLK - 1));
    }
    template <typename T, bool DEV, typename I>
    __device__ __forceinline__ static void load(const void* base, I i, const InstParam&, T* f) {
        const V* p = pairs(base, i);
        f[0] = (T)*rest(base, i);
#pragma unroll
        for (int h = 0; h < 2; h++) {
            const Quad<S> q = load_quad(p + h * (UNITS / 2) * BLK, BLK);
            f[dir_a(2 * h)] = (T)q.v[0];
            f[dir_b(2 * h)] = (T)q.v[1];
            f[dir_a(2 * h + 1)] = (T)q.v[2];
            f[dir_b(2 * h + 1)] = (T)q.v[3];
        }
    }
    template <typename T, bool DEV, typename I>
    __device__ __forceinline__ static void store(void* base, I i, const InstParam&, const T* f) {
        V* p = (V*)pairs(base, i);
        *(S*)rest(base, i) = (S)f[0];
#pragma unroll
        for (int h = 0; h < 2; h++)
            store_quad(p + h * (UNITS / 2) * BLK, BLK,
                       Quad<S>{{(S)f[dir_a(2 * h)], (S)f[dir_b(2 * h)], (S)f[dir_a(2 * h + 1)], (S)f[dir_b(2 * h + 1)]}});
    }
    // FP64 moments of the stored state: r = sum f (FP64 mode) or sum g (deviation), j = sum e g
    __device__ static void moments64(const void* base, int64_t i, const InstParam& P, double& r, double& jx, double& jy) {
        S f[FVLBM_Q];
        load<S, false>(base, i, P, f);
        r = jx = jy = 0;
#pragma unroll
        for (int a = 0; a < FVLBM_Q; a++) {
            const double x = (double)f[a];
            r += x;
            jx = add_e(EXA(a), jx, x);
            jy = add_e(EYA(a), jy, x);
        }
    }
};
template <> struct CellIO<double> : PlainIO<double> {};
template <> struct CellIO<float> : PlainIO<float> {};

// Unbiased (stochastic) rounding of q to the 16-bit format H: the upper of the
// two neighbouring 16-bit values with probability equal to q's distance from
// the lower one in units of their gap, else the lower one.  Round to nearest
// would lose every update smaller than half a 16-bit step, so that a slowly
// relaxing non-equilibrium part could stay up to about 2^-(p+1) tau / dt of
// itself away from its value (p = 10 bits in FP16, 7 in BF16); unbiased
// rounding leaves only zero-mean noise.  It is done on the bits: a uniform
// random integer below one 16-bit step, in units of q's last FP32 bit, is
// added to q's magnitude and the sum is truncated (rounded toward zero) to the
// 16-bit grid, which rounds up exactly when the random number reaches the
// step minus q's remainder.  BF16 (the same exponent range as FP32) drops 16
// bits of every finite FP32 value.  FP16 adds, with one fused multiply-add, a
// uniform fraction of the grid step at |q| (2^(e - 10) for FP16 normals,
// 2^-24 for its subnormals below 2^-14), whose FP32 sum keeps the same ~13
// random bits, and rounds toward zero: one formula for every magnitude, no
// branch.
// The random word of a cell comes from one integer hash of the bits of its
// six rounded values (the "lowbias32" mixing function of C. Wellons'
// hash-prospector, two multiply-xorshift rounds), spread over the directions
// by odd multipliers: it changes whenever the cell's values do, and equal
// cells round alike, so a cell's result does not depend on where it sits
// (batch, alone, partitioned).
__device__ __forceinline__ uint32_t mix32(uint32_t x) {
    x ^= x >> 16;
    x *= 0x7FEB352Du;
    x ^= x >> 15;
    x *= 0x846CA68Bu;
    x ^= x >> 16;
    return x;
}
// random word of direction a from the cell's hash: the high bits of an odd multiple
__device__ __forceinline__ uint32_t sr_word(uint32_t h, int a) { return h * (0x9E3779B9u + 2u * (uint32_t)a); }
template <typename H> __device__ __forceinline__ uint32_t h_bits_sr(float q, uint32_t rnd);
template <> __device__ __forceinline__ uint32_t h_bits_sr<__half>(float q, uint32_t rnd) {
    const uint32_t b = __float_as_uint(q), mag = b & 0x7FFFFFFFu;
    // FP16 grid step at |q|: 2^(e - 10) for normals, 2^-24 below 2^-14 (subnormals)
    const int e = max((int)(mag >> 23) - 127, -14);
    const float step = __uint_as_float((uint32_t)(e - 10 + 127) << 23);
    const float u = __uint_as_float(0x3F800000u | (rnd >> 9)) - 1.0f;   // uniform in [0, 1)
    const float up = fmaf(u, step, __uint_as_float(mag));
    return __half_as_ushort(__float2half_rz(__uint_as_float(__float_as_uint(up) | (b & 0x80000000u))));
}
template <> __device__ __forceinline__ uint32_t h_bits_sr<__nv_bfloat16>(float q, uint32_t rnd) {
    return (__float_as_uint(q) + (rnd >> 16)) >> 16;
}
template <typename H> __device__ __forceinline__ float h_value(uint32_t bits);
template <> __device__ __forceinline__ float h_value<__half>(uint32_t bits) {
    return __half2float(__ushort_as_half((unsigned short)bits));
}
template <> __device__ __forceinline__ float h_value<__nv_bfloat16>(uint32_t bits) {
    return __bfloat162float(__ushort_as_bfloat16((unsigned short)bits));
}

// Split format: a block of 32 cells holds 32 x (rho - 1, rho u_x, rho u_y, w_0),
// then 32 x (w_1, w_2), word w_q of a cell packing n_{3+2q} (low 16 bits) and
// n_{4+2q} (high 16 bits).
template <typename H> struct SplitIO {
    static_assert(sizeof(H) == 2, "16-bit storage");
    static constexpr int64_t BLOCK_BYTES = BLK * (3 * sizeof(float) + 3 * sizeof(uint32_t));
    template <typename I> __device__ __forceinline__ static const uint4* head(const void* base, I i) {
        return (const uint4*)((const unsigned char*)base + (size_t)(i >> BLK_SHIFT) * BLOCK_BYTES) + (i & (BLK - 1));
    }
    template <typename I> __device__ __forceinline__ static const uint2* tail(const void* base, I i) {
        return (const uint2*)((const unsigned char*)base + (size_t)(i >> BLK_SHIFT) * BLOCK_BYTES + BLK * sizeof(uint4)) +
               (i & (BLK - 1));
    }
    template <typename T>
    __device__ __forceinline__ static void decode(const uint4& h, const uint2& t, const InstParam& P, T* f) {
        const uint32_t w[3] = {h.w, t.x, t.y};
        decode<T>(__uint_as_float(h.x), __uint_as_float(h.y), __uint_as_float(h.z), w, P, f);
    }
    // f of one cell from its stored moments and non-equilibrium words
    template <typename T>
    __device__ static void decode(float dr, float jx, float jy, const uint32_t* w, const InstParam& P, T* f) {
        const float inv_rho = 1.0f / (1.0f + dr), ux = mul_rn(jx, inv_rho), uy = mul_rn(jy, inv_rho);
        float n[FVLBM_Q];
        float s = 0, sx = 0, sy = 0;
#pragma unroll
        for (int a = 3; a < FVLBM_Q; a++) {
            const uint32_t word = w[(a - 3) >> 1];
            n[a] = mul_rn(h_value<H>(((a - 3) & 1) ? word >> 16 : word & 0xFFFFu), P.inv_scale[a]);
            s += n[a];
            sx = add_e(EXA(a), sx, n[a]);
            sy = add_e(EYA(a), sy, n[a]);
        }
        n[1] = -sx;
        n[2] = -sy;
        n[0] = -(s + n[1] + n[2]);
#pragma unroll
        for (int a = 0; a < FVLBM_Q; a++) {
            // one rounding, but for direction 5, whose product is rounded by itself
            // (states decode to the bits that the compiler's own choice gave)
            f[a] = (T)(a == 5 ? feqs<float, true>(a, dr, ux, uy) + n[a]
                              : fma(wgt<float>(a), feq_value<float, true>(a, dr, ux, uy), n[a]));
        }
    }
    template <typename T, bool DEV, typename I>
    __device__ __forceinline__ static void load(const void* base, I i, const InstParam& P, T* f) {
        decode<T>(*head(base, i), *tail(base, i), P, f);
    }
    template <typename T>
    __device__ __forceinline__ static void encode(const InstParam& P, const T* f, uint4& head_out, uint2& tail_out) {
        float dr = 0, jx = 0, jy = 0;
#pragma unroll
        for (int a = 0; a < FVLBM_Q; a++) {
            dr += (float)f[a];
            jx = add_e(EXA(a), jx, (float)f[a]);
            jy = add_e(EYA(a), jy, (float)f[a]);
        }
        const float inv_rho = 1.0f / (1.0f + dr), ux = mul_rn(jx, inv_rho), uy = mul_rn(jy, inv_rho);
        float q[FVLBM_Q];
        uint32_t h = 0x811C9DC5u;
#pragma unroll
        for (int a = 3; a < FVLBM_Q; a++) {
            q[a] = fma(-wgt<float>(a), feq_value<float, true>(a, dr, ux, uy), (float)f[a]) * P.scale[a];
            h = (h ^ __float_as_uint(q[a])) * 0x01000193u;
        }
        h = mix32(h);
        uint32_t bits[FVLBM_Q];
#pragma unroll
        for (int a = 3; a < FVLBM_Q; a++) bits[a] = h_bits_sr<H>(q[a], sr_word(h, a));
        head_out = make_uint4(__float_as_uint(dr), __float_as_uint(jx), __float_as_uint(jy),
                              bits[3] | (bits[4] << 16));
        tail_out = make_uint2(bits[5] | (bits[6] << 16), bits[7] | (bits[8] << 16));
    }
    template <typename T, bool DEV, typename I>
    __device__ __forceinline__ static void store(void* base, I i, const InstParam& P, const T* f) {
        uint4 h;
        uint2 t;
        encode(P, f, h, t);
        *(uint4*)head(base, i) = h;
        *(uint2*)tail(base, i) = t;
    }
    __device__ static void moments64(const void* base, int64_t i, const InstParam&, double& r, double& jx, double& jy) {
        const uint4 h = *head(base, i);
        r = __uint_as_float(h.x);
        jx = __uint_as_float(h.y);
        jy = __uint_as_float(h.z);
    }
};
template <> struct CellIO<__half> : SplitIO<__half> {};
template <> struct CellIO<__nv_bfloat16> : SplitIO<__nv_bfloat16> {};

// Geometry of one cell, blocked by 32 cells: for each face slot k a 2-vector
// of type T each of the least-squares coefficients (GEO_LSQ), face midpoint
// minus centroid (GEO_MID) and face vector over area (GEO_FACE), vector by
// vector, in 16-byte units: two slots per unit in FP32, one in FP64.
template <typename T> struct Vec2;
template <> struct Vec2<float> { typedef float2 type; };
template <> struct Vec2<double> { typedef double2 type; };
enum GeoVec { GEO_LSQ = 0, GEO_MID = 1, GEO_FACE = 2 };

template <typename T, int MAXF> struct GeoRef {
    typedef typename Vec2<T>::type T2;
    typedef typename Vec16<T>::type V;
    static constexpr int PER = 16 / sizeof(T2);          // slots per unit
    static constexpr int UNITS = MAXF / PER;             // units per vector
    const V* g;
    __device__ __forceinline__ GeoRef() {}
    template <typename I>
    __device__ __forceinline__ GeoRef(const void* geo, I i) : g((const V*)geo + blk_index(i, 3 * UNITS)) {}
    // every slot's vector of one kind
    __device__ __forceinline__ void load(int vec, T2* out) const {
#pragma unroll
        for (int u = 0; u < UNITS; u++) {
            const V x = g[(vec * UNITS + u) * BLK];
            if constexpr (PER == 2) {
                out[2 * u] = make_float2(x.x, x.y);
                out[2 * u + 1] = make_float2(x.z, x.w);
            } else {
                out[u] = x;
            }
        }
    }
    __device__ __forceinline__ T2 get(int vec, int k) const {
        return ((const T2*)(g + (vec * UNITS + k / PER) * BLK))[k % PER];
    }
};

// The link words of a cell: uint4 units of four slots, blocked by 32 cells.
template <int MAXF, typename I>
__device__ __forceinline__ void load_links(const uint4* link, I i, uint32_t* d) {
    const uint4* p = link + blk_index(i, MAXF / 4);
#pragma unroll
    for (int u = 0; u < MAXF / 4; u++) {
        const uint4 x = p[u * BLK];
        d[4 * u] = x.x;
        d[4 * u + 1] = x.y;
        d[4 * u + 2] = x.z;
        d[4 * u + 3] = x.w;
    }
}

}  // namespace fvlbm
