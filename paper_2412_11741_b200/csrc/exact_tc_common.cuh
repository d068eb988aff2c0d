// Pieces shared by the two tensor-core encoders of the correctness mode (one CTA per pair of row
// tiles for all atoms; the dictionary split across the CTAs of one launch for fewer rows): the fp16
// operands and the bound of what their rounding does to a correlation, the running top five of a row's
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
constexpr int UMMA_K = 16;
constexpr int STAGE_CH = 64;
constexpr uint32_t kKeyMask = 0x7FFFFF80u;                // |value| without its seven lowest mantissa bits
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

// The five largest keys seen, in descending order, and the dictionary tiles the first four came from.
struct Top5 {
    uint32_t k0, k1, k2, k3, k4;
    uint32_t i0, i1, i2, i3;
};
__device__ __forceinline__ Top5 top5_none() { return Top5{0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u}; }

__device__ __forceinline__ void top5_insert(Top5& q, uint32_t k, uint32_t id) {
    const bool p0 = k > q.k0, p1 = k > q.k1, p2 = k > q.k2, p3 = k > q.k3;
    q.k4 = p3 ? q.k3 : max(q.k4, k);
    q.k3 = p2 ? q.k2 : (p3 ? k : q.k3);
    q.i3 = p2 ? q.i2 : (p3 ? id : q.i3);
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

// What the filter lets through and new_best did not settle, one copy for all groups of eight: keys `k0` .. `k7` whose last
// three bits are the place in the group, `rest` the other bits of its tags.  Inserts from the largest down until what is
// left is below the rising threshold.  A value more than the band above the running maximum leaves
// everything seen so far outside the band, so it simply becomes the only entry.  Returns the new
// state and threshold.
struct Top5Thr {
    Top5 q;
    float thr;
};
static __device__ __noinline__ Top5Thr insert_group(Top5 q, float thr, uint32_t k0, uint32_t k1, uint32_t k2, uint32_t k3, uint32_t k4,
                                                    uint32_t k5, uint32_t k6, uint32_t k7, uint32_t rest, uint32_t id, float band) {
    uint32_t k[8] = {k0, k1, k2, k3, k4, k5, k6, k7};
#pragma unroll 1
    for (int trip = 0; trip < 8; ++trip) {
        const uint32_t a = __vimax3_u32(k[0], k[1], k[2]), b = __vimax3_u32(k[3], k[4], k[5]);
        const uint32_t best = max(__vimax3_u32(k[6], k[7], a), b);
        const float val = __uint_as_float(best & kKeyMask);
        if (!(val >= thr)) break;
        const uint32_t key = best | rest;
        if (val > __uint_as_float(q.k0 & kKeyMask) + band)
            q = Top5{key, 0u, 0u, 0u, 0u, id, 0u, 0u, 0u};
        else
            top5_insert(q, key, id);
        thr = __uint_as_float(q.k0 & kKeyMask) - band;
#pragma unroll
        for (int j = 0; j < 8; ++j) k[j] = k[j] == best ? 0u : k[j];
    }
    return Top5Thr{q, thr};
}

// Folds 32 columns of this thread's row into its top five; `tag0` is the tag of v[0] (tags fall
// with the column so that the lowest column wins among equal magnitudes).  Eight values at a
// time are first reduced to their largest magnitude (half an instruction each) and only a group
// that reaches `thr`, the running maximum less the band, is looked at: whatever ends up within the band of the
// final maximum was within the band of the running one when it came by, so what the filter
// drops can never matter.  Nearly always the group's largest is then more than the band above the running
// maximum and above the rest of its group: it becomes the only entry (the second largest of the group is found by
// subtracting the largest from all keys: it turns to zero and the others stay in order).  Everything else
// is a call: the sweep's code has to stay small enough for the instruction cache.  100000 rows, N = 4096, s = 8: 2195 us
// with a call for every group that the filter lets through, 1916 us so.
template <int J = 0>
__device__ __forceinline__ void chunk_top5(const uint32_t (&v)[32], Top5& q, uint32_t id, uint32_t tag0, float& thr, float band) {
    if constexpr (J < 32) {
        const float ga = absmax3(__uint_as_float(v[J]), __uint_as_float(v[J + 1]), __uint_as_float(v[J + 2]));
        const float gb = absmax3(__uint_as_float(v[J + 3]), __uint_as_float(v[J + 4]), __uint_as_float(v[J + 5]));
        const float gc = absmax3(__uint_as_float(v[J + 6]), __uint_as_float(v[J + 7]), ga);
        if (fmaxf(gb, gc) >= thr) {
            uint32_t k[8], u[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) k[j] = (v[J + j] & kKeyMask) | static_cast<uint32_t>(7 - j);
            const uint32_t best = max(__vimax3_u32(k[6], k[7], __vimax3_u32(k[0], k[1], k[2])), __vimax3_u32(k[3], k[4], k[5]));
#pragma unroll
            for (int j = 0; j < 8; ++j) u[j] = k[j] - best;
            const uint32_t next = best + max(__vimax3_u32(u[6], u[7], __vimax3_u32(u[0], u[1], u[2])), __vimax3_u32(u[3], u[4], u[5]));
            const uint32_t rest = tag0 - J - 7u;          // tags of a group are consecutive, the last a multiple of eight
            const float val = __uint_as_float(best & kKeyMask), limit = val - band;
            if (limit > __uint_as_float(q.k0 & kKeyMask) && limit > __uint_as_float(next & kKeyMask)) {
                q = Top5{best | rest, 0u, 0u, 0u, 0u, id, 0u, 0u, 0u};
                thr = limit;
            } else {
                const Top5Thr r = insert_group(q, thr, k[0], k[1], k[2], k[3], k[4], k[5], k[6], k[7], rest, id, band);
                q = r.q;
                thr = r.thr;
            }
        }
        chunk_top5<J + 8>(v, q, id, tag0, thr, band);
    }
}

// Folds `chunks` x 32 columns of an accumulator into `q`, 64 at a time, and hands the accumulator back
// when the last have arrived.  Rolled: with all 128 columns' code in line the sweep outgrows the
// instruction cache.  No load is in flight while a group is inserted (the call may move registers).
// `band`: that of the row, a little widened; negative for a row that is all zero (nothing is
// inserted and atom 0 is taken).
__device__ __forceinline__ void drain(uint32_t taddr, int chunks, Top5& q, uint32_t id, float band, uint64_t* acc_empty, int lane) {
    float thr = __uint_as_float(q.k0 & kKeyMask) - band;
    uint32_t tag0 = 127u;
#pragma unroll 1
    for (int c = 0; c < chunks; c += 2) {
        uint32_t v0[32], v1[32];
        tmem_ld32(taddr + 32 * c, v0);
        if (c + 1 < chunks) {
            tmem_ld32(taddr + 32 * (c + 1), v1);
        } else {
#pragma unroll
            for (int j = 0; j < 32; ++j) v1[j] = 0u;
        }
        tmem_wait_ld(v0);
        reg_fence(v1);
        if (c + 2 >= chunks) {
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(acc_empty);
        }
        chunk_top5(v0, q, id, tag0, thr, band);
        if (c + 1 < chunks) chunk_top5(v1, q, id, tag0 - 32u, thr, band);
        tag0 -= 64u;
    }
}

// The same for 128 columns, handed back as soon as all of them are in registers: for an accumulator that
// the tensor core is waiting for.
__device__ __forceinline__ void drain128(uint32_t taddr, Top5& q, uint32_t id, float band, uint64_t* acc_empty, int lane) {
    uint32_t v0[32], v1[32], v2[32], v3[32];
    tmem_ld32(taddr + 0, v0);
    tmem_ld32(taddr + 32, v1);
    tmem_ld32(taddr + 64, v2);
    tmem_ld32(taddr + 96, v3);
    tmem_wait_ld(v0);
    reg_fence(v1);
    reg_fence(v2);
    reg_fence(v3);
    tc_fence_before();
    __syncwarp();
    if (lane == 0) mbar_arrive(acc_empty);
    float thr = __uint_as_float(q.k0 & kKeyMask) - band;
    chunk_top5(v0, q, id, 127u, thr, band);
    chunk_top5(v1, q, id, 95u, thr, band);
    chunk_top5(v2, q, id, 63u, thr, band);
    chunk_top5(v3, q, id, 31u, thr, band);
}

// Barrier of the 256 epilogue threads that also tells every one of them whether any of them
// passed `pred`.
__device__ __forceinline__ bool epilogue_barrier_any(bool pred) {
    uint32_t r;
    asm volatile(
        "{\n"
        ".reg .pred p, q;\n"
        "setp.ne.u32 q, %1, 0;\n"
        "bar.red.or.pred p, 1, 256, q;\n"
        "selp.u32 %0, 1, 0, p;\n"
        "}\n"
        : "=r"(r)
        : "r"(static_cast<uint32_t>(pred))
        : "memory");
    return r != 0;
}
__device__ __forceinline__ void epilogue_barrier() { asm volatile("bar.sync 1, 256;" ::: "memory"); }

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
__device__ __forceinline__ double slice_dot(const double (&R)[CH], const float (&a)[CH]) {
    double c0 = 0.0, c1 = 0.0, c2 = 0.0, c3 = 0.0;
#pragma unroll
    for (int k = 0; k < CH; k += 4) {
        c0 = fma(R[k], static_cast<double>(a[k]), c0);
        c1 = fma(R[k + 1], static_cast<double>(a[k + 1]), c1);
        c2 = fma(R[k + 2], static_cast<double>(a[k + 2]), c2);
        c3 = fma(R[k + 3], static_cast<double>(a[k + 3]), c3);
    }
    return (c0 + c1) + (c2 + c3);
}

// Two neighbouring channels of a scaled row as fp16, one word, and what the rounding took from them squared, added to
// `err2`.  (A value is brought to fp32 first: what that rounds off, 2^-24 of it, is far inside the allowance
// of row_band.)
__device__ __forceinline__ uint32_t round_pair(double r0, double r1, float& err2) {
    const float f0 = static_cast<float>(r0), f1 = static_cast<float>(r1);
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
// fp16 took from it: twice the error of a correlation, plus the 2^-16 relative truncation of the keys.  With
// r = r' + e and d = d' + f (r', d' the fp16 values), r.d - r'.d' = e.d + r'.f, which is at most
// ||e|| max ||d|| + ||r'|| max ||f|| (Cauchy-Schwarz): these norms are taken, not assumed, and come to 4e-4 ||R|| for
// unit atoms (a rounding error is 1.9e-4 of its value in the mean square), less than half of what the formats alone
// would promise.
__device__ __forceinline__ float row_band(float norm, float err2, const DictBounds& b) {
    const float err = sqrtf(err2);
    const float half = fmaf(err, b.norm, fmaf(norm + err, b.err, kAccumRel * norm * b.norm));
    return norm > 0.f || norm != norm ? 1.001f * fmaf(2.f, half, norm * b.norm * (1.f / 65536.f)) : 0.f;
}
// From which |correlation| on, relative to ||R||, an atom can be the pick, for a sweep whose largest value was `v0`
// (in the sweep's unit, as band and norm): that value less the band, and half a band for the search's fp32
// rounding.
__device__ __forceinline__ float relative_limit(float v0, float band, float norm, const DictBounds& b) {
    return (v0 - 1.5f * band) / (norm * b.scale);
}

// Writes this lane's CH residual values: fp64 to the scratch row (`row`: its first element), `scale` times them as fp16
// to the operand tile.  Returns this lane's share of the rounding's squared norm.
template <int CH>
__device__ __forceinline__ float store_residual(const double (&R)[CH], double scale, double* __restrict__ row, uint8_t* A, int r, int l8,
                                                bool write) {
    float err2 = 0.f;
#pragma unroll
    for (int k = 0; k < CH / 2; ++k) {
        const uint32_t w = round_pair(R[2 * k] * scale, R[2 * k + 1] * scale, err2);
        if (write) {
            reinterpret_cast<double2*>(row)[8 * k + l8] = make_double2(R[2 * k], R[2 * k + 1]);
            // channels 2 (8 k + l8), +1: 16-byte chunk 2 k + l8 / 4 of the row, word l8 % 4 of it
            *reinterpret_cast<uint32_t*>(A + swz_off(r, 2 * k + (l8 >> 2)) + (l8 & 3) * 4) = w;
        }
    }
    return err2;
}

#ifdef CSR_DEBUG_CHECKS
// For a pick taken without re-scoring, with `v` its key's value: what the tensor core's own arithmetic contributed (against the
// fp64 sum of the same fp16 operands, relative to ||R|| and the largest atom) and how much of half the band the
// whole deviation from the fp64 correlation `c` used up.  Both raise words of `diag` (float bits).  Eight lanes of a row call.
template <int CH>
__device__ __forceinline__ void check_value(uint32_t* diag, const double (&R)[CH], const float (&a)[CH], double c, float v, float band, float norm,
                                            const DictBounds& b, int l8, bool count) {
    float unused;
    const double scale = row_scale(group8_sum(norm2_share<CH>(R)), unused);
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
// One row over the whole dictionary by the 256 epilogue threads (all call): the pick, to every thread.
template <int D_>
__device__ __forceinline__ int rescore_row(const float* __restrict__ D, int N, const double* Rrow, float thresh, Rescored* found, int warp,
                                           int lane) {
    const int per = ((N + 7) / 8 + 15) / 16 * 16;
    const int n0 = min(warp * per, N), n1 = min(n0 + per, N);
    Rescored r{-1.0, 0, 0};
    if (n0 < n1) r.val = rescore_part<D_>(D, n0, n1, Rrow, thresh, lane, &r.n);
    if (lane == 0) found[warp] = r;
    epilogue_barrier();
    Rescored top{-1.0, 0, 0};
    for (int w = 0; w < 8; ++w) {                         // atoms ascend with the warp: the first of equal values is the lowest
        const Rescored o = found[w];
        if (o.val > top.val) top = o;
    }
    epilogue_barrier();
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
