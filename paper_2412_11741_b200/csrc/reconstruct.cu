// De-sparse (paper Eq. 12): X_hat[m,:] = sum_g coef[m][g] * D[idx[m][g]][:].
//
// HBM traffic per row is 4*s bytes of codes in and d * sizeof(out) bytes out; the s atom rows a
// row needs are gathered from the dictionary, which is a few MB and stays in L2, so from about
// s = 4 up the kernel is bound by the L2 -> SM gather (s * d * sizeof(atom) bytes per row) or, with
// fp16 atoms up to about s = 8, by instruction issue (0.71 per cycle at s = 8; with the dictionary in the L1, N = 512, nearly
// all of the time is left), not by HBM.  Two things follow:
//   - the atoms can be gathered from the fp16 copy of a prepared dictionary (csr_dict_create)
//     instead of the fp32 master: half the gathered bytes, and with fp16 coefficients (the
//     stored form) the products need no unpacking at all: fma.rn.f32.f16 multiplies two fp16
//     values exactly and accumulates in fp32;
//   - what is left is latency: every warp works on units of 16 (or 8 or 4) consecutive rows whose codes it
//     stages through its own piece of shared memory with cp.async one unit ahead (one coalesced
//     stream instead of a dependent load per row; no block-wide barrier anywhere), and it keeps
//     the gathers of several rows in flight: every lane moves 16 bytes of an atom, so an atom
//     row takes 32, 16 or 8 lanes and a warp instruction serves 1, 2 or 4 rows.
// Accumulation is fp32 in the stored order g = 0 .. s-1 (repeated atoms accumulate).
#include <type_traits>

#include "common.cuh"

namespace csr {
namespace {

constexpr int NT = 256;
constexpr int RW = 16;                                    // most rows per unit of a warp
constexpr int PP = 2;                                     // passes (rows) a lane works on together
constexpr int INFLIGHT = 4;                               // gathers per row issued before their first use

__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(static_cast<uint32_t>(__cvta_generic_to_shared(smem))),
                 "l"(gmem)
                 : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Sums are kept in pairs of neighbouring channels.
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pair(float lo, float hi) {
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void unpair(f32x2 v, float& lo, float& hi) { asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v)); }
__device__ __forceinline__ void fma_pair(f32x2& acc, float c, float a0, float a1) {
    float lo, hi;
    unpair(acc, lo, hi);
    acc = pair(fmaf(c, a0, lo), fmaf(c, a1, hi));
}
// acc += c * the two halves of w: fp16 x fp16 products are exact in fp32, the sum is rounded once (the same value as
// fmaf on the widened operands).  (Widened operands and the packed fma.rn.f32x2: 176 us against 146 for 2^20 rows,
// s = 8, N = 8192.)
__device__ __forceinline__ void fma2_f16(f32x2& acc, uint32_t w, uint16_t c) {
    float a0, a1;
    unpair(acc, a0, a1);
    asm("{\n"
        ".reg .b16 lo, hi;\n"
        "mov.b32 {lo, hi}, %2;\n"
        "fma.rn.f32.f16 %0, lo, %3, %0;\n"
        "fma.rn.f32.f16 %1, hi, %3, %1;\n"
        "}\n"
        : "+f"(a0), "+f"(a1)
        : "r"(w), "h"(c));
    acc = pair(a0, a1);
}

// The 16 bytes of an atom a lane holds: four fp32 channels, or eight fp16 channels.
template <bool F16>
struct Piece;
template <>
struct Piece<false> {
    static constexpr int CH = 4;
    static __device__ __forceinline__ void axpy(f32x2 (&a)[2], float c, const uint4& v) {
        fma_pair(a[0], c, __uint_as_float(v.x), __uint_as_float(v.y));
        fma_pair(a[1], c, __uint_as_float(v.z), __uint_as_float(v.w));
    }
};
template <>
struct Piece<true> {
    static constexpr int CH = 8;
    // fp32 coefficient: the atom's halves are widened first
    static __device__ __forceinline__ void axpy(f32x2 (&a)[4], float c, const uint4& v) {
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&w[q]));
            fma_pair(a[q], c, f.x, f.y);
        }
    }
    // fp16 coefficient, as stored
    static __device__ __forceinline__ void axpy(f32x2 (&a)[4], uint16_t c, const uint4& v) {
        fma2_f16(a[0], v.x, c);
        fma2_f16(a[1], v.y, c);
        fma2_f16(a[2], v.z, c);
        fma2_f16(a[3], v.w, c);
    }
};
// Byte offset of the atom whose index is the low or high half of a word of two.  Where an atom is 256 bytes the
// index's two bytes are put above the lane's (its place in the atom, l * 16): one instruction; elsewhere the lane's
// place is in the base.  With this and two indices clamped at a time, 2^20 rows, s = 8, fp16 atoms, N = 8192 take 139 us
// instead of 144 (an index unpacked, clamped and widened on its own each).
template <int ROW_BYTES>
__device__ __forceinline__ uint32_t piece_lo(uint32_t w, uint32_t lane_off) {
    if constexpr (ROW_BYTES == 256) return __byte_perm(w, lane_off, 0x7104);
    return (w & 0xFFFFu) * ROW_BYTES;
}
template <int ROW_BYTES>
__device__ __forceinline__ uint32_t piece_hi(uint32_t w, uint32_t lane_off) {
    if constexpr (ROW_BYTES == 256) return __byte_perm(w, lane_off, 0x7324);
    return (w >> 16) * ROW_BYTES;
}

__device__ __forceinline__ uint32_t pack2(float lo, float hi, int out_dtype) {
    if (out_dtype == CSR_DTYPE_BF16) {
        __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
        return *reinterpret_cast<uint32_t*>(&v);
    }
    __half2 v = __floats2half2_rn(lo, hi);
    return *reinterpret_cast<uint32_t*>(&v);
}

// CH consecutive channels of one row, starting at element `off` of X_hat.
template <int CH>
__device__ __forceinline__ void store_out(void* out, int out_dtype, int64_t off, const float (&a)[CH]) {
    if (out_dtype == CSR_DTYPE_F32) {
        float4* dst = reinterpret_cast<float4*>(reinterpret_cast<float*>(out) + off);
#pragma unroll
        for (int q = 0; q < CH / 4; ++q) dst[q] = make_float4(a[4 * q], a[4 * q + 1], a[4 * q + 2], a[4 * q + 3]);
    } else if constexpr (CH == 8) {
        uint4 u;
        u.x = pack2(a[0], a[1], out_dtype);
        u.y = pack2(a[2], a[3], out_dtype);
        u.z = pack2(a[4], a[5], out_dtype);
        u.w = pack2(a[6], a[7], out_dtype);
        *reinterpret_cast<uint4*>(reinterpret_cast<uint16_t*>(out) + off) = u;
    } else {
        uint2 u;
        u.x = pack2(a[0], a[1], out_dtype);
        u.y = pack2(a[2], a[3], out_dtype);
        *reinterpret_cast<uint2*>(reinterpret_cast<uint16_t*>(out) + off) = u;
    }
}

// Codes of rows [row0, row0 + rows) into the warp's shared memory as [rows][s].  `fast`: a whole unit inside
// dense, 16-byte aligned code arrays, so it is one contiguous run per array and moves with cp.async;
// otherwise element by element (row strides, the ragged last unit).
__device__ __forceinline__ void stage_codes(uint16_t* s_idx, unsigned char* s_coef, const uint16_t* __restrict__ idx,
                                            const void* __restrict__ coef, int cbytes, int64_t ldc, int64_t row0, int rows,
                                            int s, bool fast, int lane) {
    if (fast) {
        const int n_i = rows * s * 2 / 16, n_c = rows * s * cbytes / 16;
        const char* gi = reinterpret_cast<const char*>(idx + row0 * s);
        const char* gc = static_cast<const char*>(coef) + row0 * s * cbytes;
        for (int q = lane; q < n_i; q += 32) cp_async16(reinterpret_cast<char*>(s_idx) + 16 * q, gi + 16 * q);
        for (int q = lane; q < n_c; q += 32) cp_async16(s_coef + 16 * q, gc + 16 * q);
    } else {
        for (int q = lane; q < rows * s; q += 32) {
            const int r = q / s, g = q - r * s;
            s_idx[q] = idx[(row0 + r) * ldc + g];
            if (cbytes == 2)
                reinterpret_cast<uint16_t*>(s_coef)[q] = reinterpret_cast<const uint16_t*>(coef)[(row0 + r) * ldc + g];
            else
                reinterpret_cast<float*>(s_coef)[q] = reinterpret_cast<const float*>(coef)[(row0 + r) * ldc + g];
        }
    }
}

// Rows r[0..PP) of the staged block, one gather step at a time (any s, rows past M skipped).
template <int CH, int LPR, typename P>
__device__ __forceinline__ void rows_generic(const uint4* __restrict__ Dl, const uint16_t* ci, const unsigned char* cc,
                                             int cbytes, int s, int N, const int (&r)[PP], const bool (&valid)[PP],
                                             f32x2 (&acc)[PP][CH / 2], [[maybe_unused]] uint32_t* status) {
    for (int g0 = 0; g0 < s; g0 += INFLIGHT) {
        uint4 v[PP][INFLIGHT];
        float c[PP][INFLIGHT];
#pragma unroll
        for (int w = 0; w < PP; ++w)
#pragma unroll
            for (int u = 0; u < INFLIGHT; ++u) {
                const int g = g0 + u;
                v[w][u] = make_uint4(0u, 0u, 0u, 0u);
                c[w][u] = 0.f;
                if (g < s && valid[w]) {
                    const int i = min(static_cast<int>(ci[r[w] * s + g]), N - 1);
#ifdef CSR_DEBUG_CHECKS
                    if (static_cast<int>(ci[r[w] * s + g]) >= N) atomicOr(status, kStatusBounds);
#endif
                    c[w][u] = cbytes == 2 ? __half2float(reinterpret_cast<const __half*>(cc)[r[w] * s + g])
                                          : reinterpret_cast<const float*>(cc)[r[w] * s + g];
                    v[w][u] = __ldg(Dl + static_cast<size_t>(i) * LPR);
                }
            }
#pragma unroll
        for (int w = 0; w < PP; ++w)
#pragma unroll
            for (int u = 0; u < INFLIGHT; ++u)
                if (g0 + u < s) P::axpy(acc[w], c[w][u], v[w][u]);
    }
}

// The same for s a multiple of four and rows that all exist: the codes of four steps come out
// of shared memory with one 8-byte load per array (16 bytes for fp32 coefficients), two indices are
// clamped at a time, and nothing is predicated.
template <int CH, int LPR, typename P, bool COEF16>
__device__ __forceinline__ void rows_by_four(const void* __restrict__ Dict, uint32_t lane_off, const uint16_t* ci, const unsigned char* cc,
                                             int s, int N, const int (&r)[PP], f32x2 (&acc)[PP][CH / 2], [[maybe_unused]] uint32_t* status) {
    static_assert(INFLIGHT == 4, "four steps per trip");
    constexpr bool RAW16 = COEF16 && CH == 8;             // fp16 coefficients meet fp16 atoms: no conversion
    using CoefT = typename std::conditional<RAW16, uint16_t, float>::type;
    constexpr int ROW = LPR * 16;
    const uint32_t nmax = static_cast<uint32_t>(N - 1), nmax2 = nmax | (nmax << 16);
    const char* base = static_cast<const char*>(Dict) + (ROW == 256 ? 0u : lane_off);
    const auto piece = [&](uint32_t off) { return __ldg(reinterpret_cast<const uint4*>(base + off)); };
    for (int g0 = 0; g0 < s; g0 += 4) {
        uint4 v[PP][4];
        CoefT c[PP][4];
#pragma unroll
        for (int w = 0; w < PP; ++w) {
            const uint2 iw = *reinterpret_cast<const uint2*>(ci + r[w] * s + g0);
            if constexpr (RAW16) {
                const uint2 cw = *reinterpret_cast<const uint2*>(cc + (r[w] * s + g0) * 2);
                c[w][0] = static_cast<uint16_t>(cw.x & 0xFFFFu);
                c[w][1] = static_cast<uint16_t>(cw.x >> 16);
                c[w][2] = static_cast<uint16_t>(cw.y & 0xFFFFu);
                c[w][3] = static_cast<uint16_t>(cw.y >> 16);
            } else if constexpr (COEF16) {
                const uint2 cw = *reinterpret_cast<const uint2*>(cc + (r[w] * s + g0) * 2);
                const float2 c01 = __half22float2(*reinterpret_cast<const __half2*>(&cw.x));
                const float2 c23 = __half22float2(*reinterpret_cast<const __half2*>(&cw.y));
                c[w][0] = c01.x;
                c[w][1] = c01.y;
                c[w][2] = c23.x;
                c[w][3] = c23.y;
            } else {
                const float4 cw = *reinterpret_cast<const float4*>(cc + (r[w] * s + g0) * 4);
                c[w][0] = cw.x;
                c[w][1] = cw.y;
                c[w][2] = cw.z;
                c[w][3] = cw.w;
            }
#ifdef CSR_DEBUG_CHECKS
            if (max(max(iw.x & 0xFFFFu, iw.x >> 16), max(iw.y & 0xFFFFu, iw.y >> 16)) > nmax) atomicOr(status, kStatusBounds);
#endif
            const uint32_t i01 = __vminu2(iw.x, nmax2), i23 = __vminu2(iw.y, nmax2);
            v[w][0] = piece(piece_lo<ROW>(i01, lane_off));
            v[w][1] = piece(piece_hi<ROW>(i01, lane_off));
            v[w][2] = piece(piece_lo<ROW>(i23, lane_off));
            v[w][3] = piece(piece_hi<ROW>(i23, lane_off));
        }
#pragma unroll
        for (int w = 0; w < PP; ++w)
#pragma unroll
            for (int u = 0; u < 4; ++u) P::axpy(acc[w], c[w][u], v[w][u]);
    }
}

// The same for s a multiple of three (six entries per row is what a 4-byte-per-entry budget of 24 bytes
// gives): three steps per trip, no step of four left half empty.
template <int CH, int LPR, typename P, bool COEF16>
__device__ __forceinline__ void rows_by_three(const uint4* __restrict__ Dl, const uint16_t* ci, const unsigned char* cc, int s,
                                              int N, const int (&r)[PP], f32x2 (&acc)[PP][CH / 2], [[maybe_unused]] uint32_t* status) {
    constexpr bool RAW16 = COEF16 && CH == 8;
    using CoefT = typename std::conditional<RAW16, uint16_t, float>::type;
    const int nmax = N - 1;
    for (int g0 = 0; g0 < s; g0 += 3) {
        uint4 v[PP][3];
        CoefT c[PP][3];
#pragma unroll
        for (int w = 0; w < PP; ++w)
#pragma unroll
            for (int u = 0; u < 3; ++u) {
                const int o = r[w] * s + g0 + u;
                const int i = ci[o];
#ifdef CSR_DEBUG_CHECKS
                if (i > nmax) atomicOr(status, kStatusBounds);
#endif
                if constexpr (RAW16)
                    c[w][u] = reinterpret_cast<const uint16_t*>(cc)[o];
                else if constexpr (COEF16)
                    c[w][u] = __half2float(reinterpret_cast<const __half*>(cc)[o]);
                else
                    c[w][u] = reinterpret_cast<const float*>(cc)[o];
                v[w][u] = __ldg(Dl + static_cast<uint32_t>(min(i, nmax) * LPR));
            }
#pragma unroll
        for (int w = 0; w < PP; ++w)
#pragma unroll
            for (int u = 0; u < 3; ++u) P::axpy(acc[w], c[w][u], v[w][u]);
    }
}

// How the entries of a row are taken: four at a time (s a multiple of four), three at a time, or with
// every step tested.  A kernel of its own for each: together they need more registers than the fp32
// variant's four CTAs per SM leave.
enum class By { Any, Four, Three };

template <int D_, bool F16, By BY>
__global__ void __launch_bounds__(NT, F16 ? 3 : 4)
reconstruct_kernel(const void* __restrict__ Dict, const uint16_t* __restrict__ idx, const void* __restrict__ coef,
                   int coef_dtype, int64_t ldc, int64_t M, int N, int s, void* __restrict__ X_hat, int out_dtype,
                   int64_t ldxh, int dense_codes, int rw, uint32_t* status) {
    using P = Piece<F16>;
    constexpr int CH = P::CH;                             // channels per lane
    constexpr int LPR = D_ / CH;                          // lanes per row: 32, 16 or 8
    constexpr int RPP = 32 / LPR;                         // rows per warp pass
    extern __shared__ __align__(16) unsigned char smem[];
    const int cbytes = coef_dtype == CSR_DTYPE_F16 ? 2 : 4;
    const int stride_i = RW * s * 2, stride_c = RW * s * cbytes;      // multiples of 16 bytes
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned char* mine = smem + warp * 2 * (stride_i + stride_c);   // this warp's two buffers of [idx | coef]
    auto s_idx = [&](int which) { return reinterpret_cast<uint16_t*>(mine + which * (stride_i + stride_c)); };
    auto s_coef = [&](int which) { return mine + which * (stride_i + stride_c) + stride_i; };

    const int sub = lane / LPR, l = lane % LPR;
    [[maybe_unused]] const uint4* Dl = static_cast<const uint4*>(Dict) + l;  // this lane's 16 bytes of atom 0; an atom row is LPR pieces
    const int64_t n_units = (M + rw - 1) / rw;            // units of rw rows
    const int64_t unit_step = (int64_t)gridDim.x * (NT / 32);

    auto unit_fast = [&](int64_t u) { return dense_codes && (u + 1) * rw <= M; };
    int64_t u = (int64_t)blockIdx.x * (NT / 32) + warp;
    int buf = 0;
    if (u < n_units) stage_codes(s_idx(0), s_coef(0), idx, coef, cbytes, ldc, u * rw, (int)min((int64_t)rw, M - u * rw), s, unit_fast(u), lane);
    cp_async_commit();
    for (; u < n_units; u += unit_step, buf ^= 1) {
        const int64_t nu = u + unit_step;
        if (nu < n_units)
            stage_codes(s_idx(buf ^ 1), s_coef(buf ^ 1), idx, coef, cbytes, ldc, nu * rw, (int)min((int64_t)rw, M - nu * rw), s,
                        unit_fast(nu), lane);
        cp_async_commit();
        cp_async_wait<1>();                               // this unit's codes have landed (the next may be in flight)
        __syncwarp();
        const uint16_t* ci = s_idx(buf);
        const unsigned char* cc = s_coef(buf);
        const int rows = (int)min((int64_t)rw, M - u * rw);
#pragma unroll 1
        for (int p = 0; p * RPP < rows; p += PP) {
            int r[PP];
            bool valid[PP];
            f32x2 acc[PP][CH / 2];
#pragma unroll
            for (int w = 0; w < PP; ++w) {
                r[w] = (p + w) * RPP + sub;               // row inside the unit
                valid[w] = r[w] < rows;
                if (BY != By::Any) r[w] = min(r[w], rows - 1);   // (a row past the end repeats the last one and is not stored)
#pragma unroll
                for (int k = 0; k < CH / 2; ++k) acc[w][k] = 0ull;
            }
            if constexpr (BY == By::Four) {
                if (cbytes == 2)
                    rows_by_four<CH, LPR, P, true>(Dict, static_cast<uint32_t>(l) * 16u, ci, cc, s, N, r, acc, status);
                else
                    rows_by_four<CH, LPR, P, false>(Dict, static_cast<uint32_t>(l) * 16u, ci, cc, s, N, r, acc, status);
            } else if constexpr (BY == By::Three) {
                if (cbytes == 2)
                    rows_by_three<CH, LPR, P, true>(Dl, ci, cc, s, N, r, acc, status);
                else
                    rows_by_three<CH, LPR, P, false>(Dl, ci, cc, s, N, r, acc, status);
            } else {
                rows_generic<CH, LPR, P>(Dl, ci, cc, cbytes, s, N, r, valid, acc, status);
            }
#pragma unroll
            for (int w = 0; w < PP; ++w)
                if (valid[w]) {
                    float f[CH];
#pragma unroll
                    for (int k = 0; k < CH / 2; ++k) unpair(acc[w][k], f[2 * k], f[2 * k + 1]);
                    store_out<CH>(X_hat, out_dtype, (u * rw + r[w]) * ldxh + l * CH, f);
                }
        }
        __syncwarp();                                      // the buffer may be refilled
    }
    cp_async_wait<0>();
}

template <int D_, bool F16, By BY>
int launch_by(const ReconstructArgs& a, const void* dict) {
    auto kernel = reconstruct_kernel<D_, F16, BY>;
    const int cbytes = a.coef_dtype == CSR_DTYPE_F16 ? 2 : 4;
    const size_t smem = (size_t)(NT / 32) * 2 * RW * a.s * (2 + cbytes);
    static int ctas_per_sm[64] = {};                       // per device; what the occupancy calculator says for smem = 0
    int dev = 0;
    cudaGetDevice(&dev);
    dev = (dev >= 0 && dev < 64) ? dev : 0;
    int per_sm = ctas_per_sm[dev];
    if (per_sm == 0) {
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, NT, 0) != cudaSuccess || per_sm < 1) per_sm = 4;
        ctas_per_sm[dev] = per_sm;
    }
    // shared memory may hold fewer CTAs than the registers do (227 KB per SM)
    int fit = smem ? (int)((size_t)(227 * 1024) / (smem + 1024)) : per_sm;
    if (fit < 1) fit = 1;
    const int64_t cap = (int64_t)sm_count() * (per_sm < fit ? per_sm : fit);
    // Rows per unit: 16, or 8 or 4 where that leaves a warp at least a tenth fewer rows in all (a last round of
    // units that few warps have): 77777 rows are 1.03 rounds of 16 on 4736 warps, two rounds, or five
    // rounds of 4: 24.6 us in units of 16, 22.6 in units of 4 (s = 6, N = 5001, fp32 atoms, cold caches; both
    // with the steps of three).  Longer units are better otherwise (2^20 rows, s = 8, fp16 atoms, N = 8192: 131 us
    // in units of 16, 166 in units of 4).  Eight rows of codes end on a 16-byte boundary in any case, four if s
    // is even; a trip of a warp takes 32 / lanes per row * PP rows.
    constexpr int trip = 32 / (D_ / Piece<F16>::CH) * PP;
    const int64_t warps = cap * (NT / 32);
    auto rows_of_a_warp = [&](int w) { return ((a.M + w - 1) / w + warps - 1) / warps * w; };
    int rw = RW;
    for (int w : {8, 4})
        if (w >= trip && (w == 8 || a.s % 2 == 0) && 10 * rows_of_a_warp(w) <= 9 * rows_of_a_warp(rw)) rw = w;
    const int64_t n_blocks = ((a.M + rw - 1) / rw + NT / 32 - 1) / (NT / 32);
    const int grid = (int)(n_blocks < cap ? n_blocks : cap);
    if (smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return fail(CSR_ERR_CUDA, "cudaFuncSetAttribute: %s", cudaGetErrorString(e));
    }
    const uintptr_t pi = reinterpret_cast<uintptr_t>(a.idx), pc = reinterpret_cast<uintptr_t>(a.coef);
    const int dense = a.ld_code == a.s && pi % 16 == 0 && pc % 16 == 0;
    kernel<<<grid, NT, smem, a.stream>>>(dict, a.idx, a.coef, a.coef_dtype, a.ld_code, a.M, a.N, a.s, a.X_hat, a.out_dtype, a.ld_xhat,
                                         dense, rw, a.status);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return fail(CSR_ERR_CUDA, "reconstruct launch: %s", cudaGetErrorString(e));
    return CSR_OK;
}

template <int D_, bool F16>
int launch_t(const ReconstructArgs& a, const void* dict) {
    if (a.s % 4 == 0) return launch_by<D_, F16, By::Four>(a, dict);
    if (a.s % 3 == 0) return launch_by<D_, F16, By::Three>(a, dict);
    return launch_by<D_, F16, By::Any>(a, dict);
}

}  // namespace

int launch_reconstruct(const ReconstructArgs& a) {
    if (a.M == 0) return CSR_OK;
    if (a.dict_f16) return a.d == 128 ? launch_t<128, true>(a, a.dict_f16) : launch_t<64, true>(a, a.dict_f16);
    return a.d == 128 ? launch_t<128, false>(a, a.D) : launch_t<64, false>(a, a.D);
}

}  // namespace csr
