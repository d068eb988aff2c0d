// Pieces shared by the two tensor-core encoders of the correctness mode (one CTA per pair of row
// tiles for all atoms; the dictionary split across the CTAs of one launch for fewer rows): the fp16
// operands and the bound of what their rounding does to a correlation, the groups of atoms that hold a row's largest
// correlations, the fp64 arithmetic of the picks.
#pragma once

#include <cuda.h>

#include "common.cuh"
#include "tcgen05_common.cuh"

namespace csr {
namespace exact_tc {

using namespace tc;

constexpr int TILE_M = 128;
constexpr int TILE_N = 256;
constexpr int STAGE_CH = 64;
constexpr uint32_t kKeyMask = 0x7FFFFFE0u;                // |value| without its five lowest mantissa bits
// Adjacent atoms that the sweep takes as one: it keeps their largest |correlation|; which of them that was is found
// when the row is settled (2 KB of the dictionary's fp16 copy gathered per row at d = 128).  Groups of four at d = 128:
// a training step of 65536 rows (N = 8192, s = 8) 1511 us, of eight 1394.
constexpr int G = 8;
constexpr uint32_t FULL = 0xffffffffu;
// What the tensor cores' fp32 accumulation of d exact products of fp16 values (in groups of 16) may add to
// the error of a correlation, relative to ||R|| and the largest norm of an atom.  Measured (checked
// build): below a quarter of it.
constexpr float kAccumRel = 1.0f / 32768.0f;

// The dictionary as the sweeps read it: fp16, times a power of two; largest norm of a (scaled) atom and
// of what the rounding took from one.
struct DictBounds {
    float norm, err, scale;
};
// One block's share of them, as dict_to_f16_kernel leaves it.
constexpr int kMaxDictParts = 296;
struct DictPart {
    float norm2, err2, scale, pad;
};
// All of them put together; every lane of a warp calls and gets the result (at most ten loads a lane).
__device__ __forceinline__ DictBounds dict_bounds(const DictPart* __restrict__ parts, int n_parts, int lane) {
    float norm2 = 0.f, err2 = 0.f;
    for (int i = lane; i < n_parts; i += 32) {
        const float4 v = __ldg(reinterpret_cast<const float4*>(parts) + i);
        norm2 = fmaxf(norm2, v.x);
        err2 = fmaxf(err2, v.y);
    }
    for (int o = 16; o; o >>= 1) {
        norm2 = fmaxf(norm2, __shfl_xor_sync(FULL, norm2, o));
        err2 = fmaxf(err2, __shfl_xor_sync(FULL, err2, o));
    }
    return DictBounds{sqrtf(norm2) * 1.0001f, sqrtf(err2) * 1.0001f, __ldg(&parts[0].scale)};
}

__device__ __forceinline__ uint32_t swz_off(int r, int chunk) {
    const int kblock = chunk >> 3, cc = chunk & 7;
    return kblock * (TILE_M * 128) + (r >> 3) * 1024 + (r & 7) * 128 + ((cc ^ (r & 7)) << 4);
}

// The largest keys of groups seen, in descending order, and the dictionary tiles the first three came from.  A key is a
// group's largest |value| with the group's number inside the thread's part of a dictionary tile in its five lowest bits.
struct Tops {
    uint32_t k0, k1, k2, k3;
    uint32_t i0, i1, i2;
};
__device__ __forceinline__ Tops no_tops() { return Tops{0u, 0u, 0u, 0u, 0u, 0u, 0u}; }

__device__ __forceinline__ void tops_insert(Tops& q, uint32_t k, uint32_t id) {
    const bool p0 = k > q.k0, p1 = k > q.k1, p2 = k > q.k2;
    q.k3 = p2 ? q.k2 : max(q.k3, k);
    q.k2 = p1 ? q.k1 : (p2 ? k : q.k2);
    q.i2 = p1 ? q.i1 : (p2 ? id : q.i2);
    q.k1 = p0 ? q.k0 : (p1 ? k : q.k1);
    q.i1 = p0 ? q.i0 : (p1 ? id : q.i1);
    q.k0 = p0 ? k : q.k0;
    q.i0 = p0 ? id : q.i0;
}
// max(|a|, |b|, |c|)
__device__ __forceinline__ float absmax3(float a, float b, float c) {
    float r;
    asm("max.abs.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}

// The three largest keys of a thread's part of one dictionary tile.
struct Three {
    uint32_t a, b, c;
};
// Two more keys: nine two- and three-input minima and maxima, no branch.
__device__ __forceinline__ void fold2(Three& q, uint32_t g, uint32_t h) {
    const uint32_t x = max(g, h), y = min(g, h);
    const uint32_t s = min(q.a, x), u = max(q.b, y), w = min(q.b, y);
    q.a = max(q.a, x);
    q.c = __vimax3_u32(q.c, w, min(s, u));
    q.b = max(s, u);
}
// Key of the G values from v[J] on (a NaN counts as nothing).
template <int J>
__device__ __forceinline__ uint32_t key_of(const uint32_t (&v)[32], uint32_t tag) {
    auto f = [&](int j) { return __uint_as_float(v[J + j]); };
    const float m = absmax3(absmax3(f(3), f(4), f(5)), absmax3(f(6), f(7), absmax3(f(0), f(1), f(2))), 0.f);
    return (__float_as_uint(m) & kKeyMask) | tag;
}
// 32 columns, whose first group has number T0.
template <int T0, int J = 0>
__device__ __forceinline__ void fold32(const uint32_t (&v)[32], Three& q) {
    if constexpr (J < 32) {
        fold2(q, key_of<J>(v, T0 + J / G), key_of<J + G>(v, T0 + J / G + 1));
        fold32<T0, J + 2 * G>(v, q);
    }
}
// A tile's three largest into the row's: whatever ends up within the band of the final maximum was within the band of
// the running one when it came by, so what stays out can never matter.  A key more than the band above the
// running maximum leaves everything seen so far outside the band and becomes the only one.  The tile's third is not known to be the
// last inside the band: it counts as one too many.  `band`: that of the row, a little widened; negative for a row that is all zero
// (nothing is taken and atom 0 is picked).
__device__ __forceinline__ void merge(Tops& q, const Three& l, uint32_t id, float band) {
    auto val = [](uint32_t k) { return __uint_as_float(k & kKeyMask); };
    if (val(l.a) >= val(q.k0) - band) {
        if (val(l.a) - band > val(q.k0))
            q = Tops{l.a, 0u, 0u, 0u, id, 0u, 0u};
        else
            tops_insert(q, l.a, id);
        const float thr = val(q.k0) - band;
        if (val(l.b) >= thr) {
            tops_insert(q, l.b, id);
            if (val(l.c) >= thr) q.k3 = max(q.k3, l.c);
        }
    }
}

// Folds a thread's 32 * CHUNKS columns of an accumulator into its row's `q` and hands the accumulator back as soon as all of them
// are in registers; HALVES: 64 at a time, for a kernel whose threads have few.
template <int CHUNKS, bool HALVES = false>
__device__ __forceinline__ void drain(uint32_t taddr, Tops& q, uint32_t id, float band, uint64_t* acc_empty, int lane) {
    Three l{0u, 0u, 0u};
    auto back = [&]() {
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(acc_empty);
    };
    if constexpr (HALVES) {
        static_assert(CHUNKS == 4, "two halves of two chunks");
        uint32_t v0[32], v1[32];
        tmem_ld32(taddr + 0, v0);
        tmem_ld32(taddr + 32, v1);
        tmem_wait_ld(v0);
        reg_fence(v1);
        fold32<0>(v0, l);
        fold32<32 / G>(v1, l);
        tmem_ld32(taddr + 64, v0);
        tmem_ld32(taddr + 96, v1);
        tmem_wait_ld(v0);
        reg_fence(v1);
        back();
        fold32<64 / G>(v0, l);
        fold32<96 / G>(v1, l);
    } else {
        uint32_t v0[32], v1[32], v2[32], v3[32];
        tmem_ld32(taddr + 0, v0);
        if constexpr (CHUNKS > 1) tmem_ld32(taddr + 32, v1);
        if constexpr (CHUNKS > 2) tmem_ld32(taddr + 64, v2);
        if constexpr (CHUNKS > 3) tmem_ld32(taddr + 96, v3);
        tmem_wait_ld(v0);
        if constexpr (CHUNKS > 1) reg_fence(v1);
        if constexpr (CHUNKS > 2) reg_fence(v2);
        if constexpr (CHUNKS > 3) reg_fence(v3);
        back();
        fold32<0>(v0, l);
        if constexpr (CHUNKS > 1) fold32<32 / G>(v1, l);
        if constexpr (CHUNKS > 2) fold32<64 / G>(v2, l);
        if constexpr (CHUNKS > 3) fold32<96 / G>(v3, l);
    }
    merge(q, l, id, band);
}

// Barrier of 256 epilogue threads (`bar`: its number) that also tells every one of them whether any of them
// passed `pred`.
__device__ __forceinline__ bool epilogue_barrier_any(bool pred, int bar = 1) {
    uint32_t r;
    asm volatile(
        "{\n"
        ".reg .pred p, q;\n"
        "setp.ne.u32 q, %1, 0;\n"
        "bar.red.or.pred p, %2, 256, q;\n"
        "selp.u32 %0, 1, 0, p;\n"
        "}\n"
        : "=r"(r)
        : "r"(static_cast<uint32_t>(pred)), "r"(bar)
        : "memory");
    return r != 0;
}
__device__ __forceinline__ void epilogue_barrier(int bar = 1) { asm volatile("bar.sync %0, 256;" ::"r"(bar) : "memory"); }

__device__ __forceinline__ double group8_sum(double v) {
    v += __shfl_xor_sync(FULL, v, 1);
    v += __shfl_xor_sync(FULL, v, 2);
    v += __shfl_xor_sync(FULL, v, 4);
    return v;
}
__device__ __forceinline__ double warp_sum(double v) {
    for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(FULL, v, o);
    return v;
}

// The eight lanes that share a row own its channels in pairs: lane l8 has channels 2 (8 k + l8)
// and the next one, k = 0 .. CH / 2 - 1, so that one load or store instruction of the eight lanes
// covers one contiguous run (whole 32-byte sectors of the fp64 row).
// CH channels of one atom (fp32 master copy), as this lane's slice.
template <int CH>
__device__ __forceinline__ void load_atom(const float* __restrict__ atom, int l8, float (&a)[CH]) {
#pragma unroll
    for (int k = 0; k < CH / 2; ++k) {
        const float2 v = __ldg(reinterpret_cast<const float2*>(atom) + 8 * k + l8);
        a[2 * k] = v.x;
        a[2 * k + 1] = v.y;
    }
}
// (four running sums: a single chain of fp64 FMAs would wait out the pipe's latency CH times)
template <int CH>
__device__ __forceinline__ double slice_dot(const double (&R)[CH], const double (&a)[CH]) {
    double c0 = 0.0, c1 = 0.0, c2 = 0.0, c3 = 0.0;
#pragma unroll
    for (int k = 0; k < CH; k += 4) {
        c0 = fma(R[k], a[k], c0);
        c1 = fma(R[k + 1], a[k + 1], c1);
        c2 = fma(R[k + 2], a[k + 2], c2);
        c3 = fma(R[k + 3], a[k + 3], c3);
    }
    return (c0 + c1) + (c2 + c3);
}
template <int CH>
__device__ __forceinline__ void widen(const float (&a)[CH], double (&ad)[CH]) {
#pragma unroll
    for (int k = 0; k < CH; ++k) ad[k] = static_cast<double>(a[k]);
}
template <int CH>
__device__ __forceinline__ double slice_dot(const double (&R)[CH], const float (&a)[CH]) {
    double ad[CH];
    widen<CH>(a, ad);
    return slice_dot<CH>(R, ad);
}

// Two neighbouring channels of a scaled row as fp16, one word, and what the rounding took from them squared, added to
// `err2`.  (A value is brought to fp32 first: what that rounds off, 2^-24 of it, is far inside the allowance
// of row_band.)
__device__ __forceinline__ uint32_t round_pair(float f0, float f1, float& err2) {
    const __half2 h = __floats2half2_rn(f0, f1);
    const float2 w = __half22float2(h);
    const float e0 = f0 - w.x, e1 = f1 - w.y;
    err2 = fmaf(e0, e0, err2);
    err2 = fmaf(e1, e1, err2);
    return *reinterpret_cast<const uint32_t*>(&h);
}
__device__ __forceinline__ float group8_sumf(float v) {
    v += __shfl_xor_sync(FULL, v, 1);
    v += __shfl_xor_sync(FULL, v, 2);
    v += __shfl_xor_sync(FULL, v, 4);
    return v;
}

// This lane's share of ||R||^2.
template <int CH>
__device__ __forceinline__ double norm2_share(const double (&R)[CH]) {
    double n0 = 0.0, n1 = 0.0;
#pragma unroll
    for (int k = 0; k < CH / 2; ++k) {
        n0 = fma(R[2 * k], R[2 * k], n0);
        n1 = fma(R[2 * k + 1], R[2 * k + 1], n1);
    }
    return n0 + n1;
}

// What a row is multiplied by before it is rounded to fp16, from its ||R||^2: the power of two that brings
// ||R|| into [1, 2), so that the operands, the sweep's values and the band keep their precision at any
// norm (the keys of a sweep are only compared with one another and with the band, all in the same
// unit, and a power of two leaves every bit of them as it is).  `norm` gets ||R|| in that unit:
// 0 for a row of zeros; Inf or NaN, and no scaling, for a row that is not finite.
__device__ __forceinline__ double row_scale(double nn, float& norm) {
    const int e = (__double2hiint(nn) >> 20) & 0x7FF;
    const double scale = e == 0 || e == 0x7FF ? 1.0 : __hiloint2double((1023 - ((e - 1023) >> 1)) << 20, 0);
    norm = e == 0 ? 0.f : sqrtf(static_cast<float>(nn * scale * scale));
    return scale;
}
// Half-width of the undecided zone of a row, in the sweep's unit, from its norm and the norm of what rounding it to
// fp16 took from it: twice the error of a correlation, plus the 2^-18 relative truncation of the keys (and half as much again for the fp32 rounding of their differences).  With
// r = r' + e and d = d' + f (r', d' the fp16 values), r.d - r'.d' = e.d + r'.f, which is at most
// ||e|| max ||d|| + ||r'|| max ||f|| (Cauchy-Schwarz): these norms are taken, not assumed, and come to 4e-4 ||R|| for
// unit atoms (a rounding error is 1.9e-4 of its value in the mean square), less than half of what the formats alone
// would promise.
__device__ __forceinline__ float row_band(float norm, float err2, const DictBounds& b) {
    const float err = sqrtf(err2);
    const float half = fmaf(err, b.norm, fmaf(norm + err, b.err, kAccumRel * norm * b.norm));
    return norm > 0.f || norm != norm ? 1.001f * fmaf(2.f, half, norm * b.norm * (1.f / 131072.f)) : 0.f;
}
// From which |correlation| on, relative to ||R||, an atom can be the pick, for a sweep whose largest value was `v0`
// (in the sweep's unit, as band and norm): that value less the band, and half a band for the search's fp32
// rounding.
__device__ __forceinline__ float relative_limit(float v0, float band, float norm, const DictBounds& b) {
    return (v0 - 1.5f * band) / (norm * b.scale);
}

// This lane's CH residual values as the sweep takes them: scaled, fp16, two channels per word; the row's norm and what the rounding
// took from it squared (of all eight lanes of the row).  All lanes of a warp call.  Rows of ordinary norm are scaled and
// measured in fp32: fp64 operations and conversions are what the settling has least of, and nothing here needs more than a few
// bits of the norm.
template <int CH>
struct Operand {
    uint32_t w[CH / 2];
    float norm, err2;
};
template <int CH>
__device__ __forceinline__ Operand<CH> to_operand(const double (&R)[CH]) {
    Operand<CH> o;
    float f[CH], n0 = 0.f, n1 = 0.f, err2 = 0.f;
#pragma unroll
    for (int k = 0; k < CH / 2; ++k) {
        f[2 * k] = static_cast<float>(R[2 * k]);
        f[2 * k + 1] = static_cast<float>(R[2 * k + 1]);
        n0 = fmaf(f[2 * k], f[2 * k], n0);
        n1 = fmaf(f[2 * k + 1], f[2 * k + 1], n1);
    }
    const float nn = group8_sumf(n0 + n1);
    if (__all_sync(FULL, nn >= 0x1p-60f && nn <= 0x1p60f)) {
        const int e = static_cast<int>(__float_as_uint(nn) >> 23) - 127;
        const float scale = __uint_as_float(static_cast<uint32_t>(127 - (e >> 1)) << 23);
        o.norm = sqrtf(nn) * scale;
#pragma unroll
        for (int k = 0; k < CH / 2; ++k) o.w[k] = round_pair(f[2 * k] * scale, f[2 * k + 1] * scale, err2);
    } else {
        const double scale = row_scale(group8_sum(norm2_share<CH>(R)), o.norm);
#pragma unroll
        for (int k = 0; k < CH / 2; ++k)
            o.w[k] = round_pair(static_cast<float>(R[2 * k] * scale), static_cast<float>(R[2 * k + 1] * scale), err2);
    }
    o.err2 = group8_sumf(err2);
    return o;
}

#ifdef CSR_DEBUG_CHECKS
// For a pick taken without re-scoring, with `v` its key's value: what the tensor core's own arithmetic contributed (against the
// fp64 sum of the same fp16 operands, relative to ||R|| and the largest atom) and how much of half the band the
// whole deviation from the fp64 correlation `c` used up.  Both raise words of `diag` (float bits).  Eight lanes of a row call.
template <int CH>
__device__ __forceinline__ void check_value(uint32_t* diag, const double (&R)[CH], const float (&a)[CH], double c, float v, float band, float norm,
                                            const DictBounds& b, int l8, bool count) {
    const double scale = exp2(rint(log2(static_cast<double>(norm) / sqrt(group8_sum(norm2_share<CH>(R))))));   // the power of two that was taken
    double p = 0.0;
#pragma unroll
    for (int k = 0; k < CH; ++k)
        p = fma(static_cast<double>(__half2float(__float2half_rn(static_cast<float>(R[k] * scale)))),
                static_cast<double>(__half2float(__float2half_rn(a[k] * b.scale))), p);
    p = fabs(group8_sum(p));
    if (l8 == 0 && count && band > 0.f) {
        const float own = static_cast<float>(fabs(v - p)) / (norm * b.norm);
        const float use = static_cast<float>(fabs(v - fabs(c) * scale * b.scale)) / (0.5f * band);
        atomicMax(diag, __float_as_uint(own));
        atomicMax(diag + 1, __float_as_uint(use));
    }
}
#endif

// Elements `off` and `off + 1` of X widened to fp64.
__device__ __forceinline__ void load_x2(const void* X, int x_dtype, int64_t off, double& x0, double& x1) {
    if (x_dtype == CSR_DTYPE_F32) {
        const float2 v = __ldg(reinterpret_cast<const float2*>(reinterpret_cast<const float*>(X) + off));
        x0 = v.x;
        x1 = v.y;
    } else {
        const uint32_t w = __ldg(reinterpret_cast<const uint32_t*>(reinterpret_cast<const uint16_t*>(X) + off));
        if (x_dtype == CSR_DTYPE_BF16) {
            x0 = __uint_as_float(w << 16);
            x1 = __uint_as_float(w & 0xFFFF0000u);
        } else {
            const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&w));
            x0 = f.x;
            x1 = f.y;
        }
    }
}

// acc += the products of two pairs of fp16 values, exact, each sum rounded once.
__device__ __forceinline__ void fma2_f16(float& acc0, float& acc1, uint32_t a, uint32_t b) {
    asm("{\n"
        ".reg .b16 al, ah, bl, bh;\n"
        "mov.b32 {al, ah}, %2;\n"
        "mov.b32 {bl, bh}, %3;\n"
        "fma.rn.f32.f16 %0, al, bl, %0;\n"
        "fma.rn.f32.f16 %1, ah, bh, %1;\n"
        "}\n"
        : "+f"(acc0), "+f"(acc1)
        : "r"(a), "r"(b));
}
// The sweep's values of one group again: eight lanes per row, lane l8 holds 16-byte chunks l8 + 8 j of the G atoms and of the row.
template <int D_>
struct GroupAtoms {
    static constexpr int CK = D_ / 64;
    uint4 a[G][CK];
    __device__ __forceinline__ void load(const uint16_t* __restrict__ dict, int n0, int N, int l8) {
#pragma unroll
        for (int i = 0; i < G; ++i) {
            const uint4* src = reinterpret_cast<const uint4*>(dict + static_cast<int64_t>(min(n0 + i, N - 1)) * D_);
#pragma unroll
            for (int j = 0; j < CK; ++j) a[i][j] = __ldg(src + l8 + 8 * j);
        }
    }
    // |r . d| of the group's atom l8, to this lane; negative for one past the dictionary's end.
    __device__ __forceinline__ float value(const uint4 (&r)[CK], int n0, int N, int l8) const {
        float e[G];
#pragma unroll
        for (int i = 0; i < G; ++i) {
            float x = 0.f, y = 0.f;
#pragma unroll
            for (int j = 0; j < CK; ++j) {
                fma2_f16(x, y, r[j].x, a[i][j].x);
                fma2_f16(x, y, r[j].y, a[i][j].y);
                fma2_f16(x, y, r[j].z, a[i][j].z);
                fma2_f16(x, y, r[j].w, a[i][j].w);
            }
            e[i] = x + y;
        }
        // a lane keeps half of its atoms at each step and sends the other half's sums to the lane that keeps those
#pragma unroll
        for (int h = 4; h > 0; h >>= 1) {
            const bool up = l8 & h;
#pragma unroll
            for (int i = 0; i < h; ++i) {
                const float keep = up ? e[i + h] : e[i], send = up ? e[i] : e[i + h];
                e[i] = keep + __shfl_xor_sync(FULL, send, h);
            }
        }
        return n0 + l8 < N ? fabsf(e[0]) : -1.f;
    }
};
// Of the group's values, a bit for each lane of the warp whose atom is within the band of its row's largest.
__device__ __forceinline__ uint32_t inside(float value, float band) {
    float m = value;
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) m = fmaxf(m, __shfl_xor_sync(FULL, m, o));
    return __ballot_sync(FULL, value >= 0.f && !(m - value > band));
}
// One row by the whole warp: the atom of largest fp64 |R . d| in the groups start(0) .. start(groups - 1), the lowest among equals.
template <int D_, typename F>
__device__ __forceinline__ int decide(const float* __restrict__ D, int N, const double* Rrow, int groups, F&& start, int lane) {
    constexpr int CH = D_ / 8;
    const int l8 = lane & 7, grp = lane >> 3;
    double R[CH];
#pragma unroll
    for (int k = 0; k < CH / 2; ++k) {
        const double2 v = __ldcg(reinterpret_cast<const double2*>(Rrow) + 8 * k + l8);
        R[2 * k] = v.x;
        R[2 * k + 1] = v.y;
    }
    double best = -1.0;
    int bn = 0;
#pragma unroll 1
    for (int i = 0; i < groups; ++i) {
        const int n0 = start(i);
        float at[2][CH];                                  // four atoms at a time, eight lanes each
#pragma unroll
        for (int h = 0; h < 2; ++h) load_atom<CH>(D + static_cast<int64_t>(min(n0 + 4 * h + grp, N - 1)) * D_, l8, at[h]);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int n = n0 + 4 * h + grp;
            const double c = fabs(group8_sum(slice_dot<CH>(R, at[h])));
            if (n < N && (c > best || (c == best && n < bn))) {
                best = c;
                bn = n;
            }
        }
    }
#pragma unroll
    for (int o = 8; o < 32; o <<= 1) {
        const double ob = __shfl_xor_sync(FULL, best, o);
        const int on = __shfl_xor_sync(FULL, bn, o);
        if (ob > best || (ob == best && on < bn)) {
            best = ob;
            bn = on;
        }
    }
    return bn;
}

// Arg-max of |R . d_n| over the atoms [n0, n1) for one row, by one warp (all lanes call): its share
// of a row that has more atoms inside the band than the sweep kept track of.  The true arg-max has
// an fp32 value of at least `thresh` times ||R|| (see relative_limit), so an fp32 pass over the row
// divided by its norm collects those atoms, one per lane, and their fp64 correlations decide, the
// lowest atom among equal values.  More than 32 candidates (copies of one atom): every
// atom is scored in fp64.  Returns the value (negative: no candidate) and the atom in `bn`.
// The pass is bound by the latency of the atoms' loads, 16 atoms at a time, eight lanes each.
template <int D_>
static __device__ __noinline__ double rescore_part(const float* __restrict__ D, int n0, int n1, const double* Rrow, float thresh, int lane,
                                                   int* bn) {
    constexpr int QV = D_ / 32;                           // 16-byte loads per lane and atom
    const int l8 = lane & 7, grp = lane >> 3;
    double nn = 0.0;
#pragma unroll
    for (int k = 0; k < 4 * QV; ++k) {
        const double r = __ldcg(Rrow + ((k >> 2) * 8 + l8) * 4 + (k & 3));
        nn = fma(r, r, nn);
    }
    const double inv = 1.0 / sqrt(group8_sum(nn));
    float4 rf[QV];
#pragma unroll
    for (int k = 0; k < QV; ++k) {
        const double* r = Rrow + (8 * k + l8) * 4;
        rf[k] = make_float4(static_cast<float>(__ldcg(r) * inv), static_cast<float>(__ldcg(r + 1) * inv),
                            static_cast<float>(__ldcg(r + 2) * inv), static_cast<float>(__ldcg(r + 3) * inv));
    }
    int mine = 0, count = 0;
#pragma unroll 1
    for (int b = n0; b < n1; b += 16) {
        float4 v[4][QV];
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
            for (int k = 0; k < QV; ++k)
                v[u][k] = __ldg(reinterpret_cast<const float4*>(D + static_cast<int64_t>(min(b + 4 * u + grp, n1 - 1)) * D_) + 8 * k + l8);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            float c = 0.f;
#pragma unroll
            for (int k = 0; k < QV; ++k) {
                c = fmaf(rf[k].x, v[u][k].x, c);
                c = fmaf(rf[k].y, v[u][k].y, c);
                c = fmaf(rf[k].z, v[u][k].z, c);
                c = fmaf(rf[k].w, v[u][k].w, c);
            }
            for (int o = 1; o < 8; o <<= 1) c += __shfl_xor_sync(FULL, c, o);
            const bool in = b + 4 * u + grp < n1 && !(fabsf(c) < thresh);      // (NaN counts as a candidate)
            uint32_t hits = __ballot_sync(FULL, in && l8 == 0);
            while (hits) {
                const int g = __ffs(hits) - 1;
                hits &= hits - 1;
                if (lane == (count & 31)) mine = b + 4 * u + (g >> 3);
                ++count;
            }
        }
    }
    double best = -1.0;
    *bn = 0;
    const bool all = count > 32;
    const int todo = all ? n1 - n0 : count;
    constexpr int PER = D_ / 32;
    for (int j = 0; j < todo; ++j) {
        const int n = all ? n0 + j : __shfl_sync(FULL, mine, j);
        double p = 0.0;
#pragma unroll
        for (int k = 0; k < PER; ++k)
            p = fma(__ldcg(Rrow + lane * PER + k), static_cast<double>(__ldg(D + static_cast<int64_t>(n) * D_ + lane * PER + k)), p);
        const double a = fabs(warp_sum(p));
        if (a > best || (a == best && n < *bn)) {
            best = a;
            *bn = n;
        }
    }
    return best;
}

// What the eight warps found for one row.
struct Rescored {
    double val;
    int n, pad;
};
// One row over the whole dictionary by 256 epilogue threads (all call; `warp`: 0 to 7): the pick, to every thread.
template <int D_>
__device__ __forceinline__ int rescore_row(const float* __restrict__ D, int N, const double* Rrow, float thresh, Rescored* found, int warp,
                                           int lane, int bar = 1) {
    const int per = ((N + 7) / 8 + 15) / 16 * 16;
    const int n0 = min(warp * per, N), n1 = min(n0 + per, N);
    Rescored r{-1.0, 0, 0};
    if (n0 < n1) r.val = rescore_part<D_>(D, n0, n1, Rrow, thresh, lane, &r.n);
    if (lane == 0) found[warp] = r;
    epilogue_barrier(bar);
    Rescored top{-1.0, 0, 0};
    for (int w = 0; w < 8; ++w) {                         // atoms ascend with the warp: the first of equal values is the lowest
        const Rescored o = found[w];
        if (o.val > top.val) top = o;
    }
    epilogue_barrier(bar);
    return top.n;
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
inline EncodeTiledFn tensor_map_encoder() {
    static const EncodeTiledFn fn = [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            return reinterpret_cast<EncodeTiledFn>(p);
        return static_cast<EncodeTiledFn>(nullptr);
    }();
    return fn;
}

// The dictionary's fp16 copy, [N][d]: boxes of box_atoms atoms x 64 channels, 128-byte swizzle;
// atoms past N read as zeros.
inline int dict_map(CUtensorMap* map, void* base, int N, int d, int box_atoms) {
    EncodeTiledFn encode = tensor_map_encoder();
    if (!encode) return fail(CSR_ERR_CUDA, "cuTensorMapEncodeTiled is not available from the driver");
    const cuuint64_t gdim[2] = {(cuuint64_t)d, (cuuint64_t)N};
    const cuuint64_t gstride[1] = {(cuuint64_t)d * 2};
    const cuuint32_t box[2] = {STAGE_CH, (cuuint32_t)box_atoms};
    const cuuint32_t estr[2] = {1, 1};
    const CUresult r = encode(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, base, gdim, gstride, box, estr,
                              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return fail(CSR_ERR_CUDA, "cuTensorMapEncodeTiled failed with code %d", (int)r);
    return CSR_OK;
}

}  // namespace exact_tc
}  // namespace csr
