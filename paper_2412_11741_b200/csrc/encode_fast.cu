// Fast matching pursuit (paper Eq. 2-4) on the sm_100a tensor cores.
//
// One persistent CTA per SM owns two tiles of 128 input rows at a time and keeps their
// residuals on chip for all s iterations:
//
//   - the residual tiles live in shared memory as bf16, in the K-major 128-byte-swizzled
//     layout tcgen05.mma reads (operand A);
//   - the bf16 copy of the dictionary (a few MB, L2 resident) streams through a ring of
//     shared-memory stages fetched by TMA (operand B).  A stage holds 64 channels of 256
//     atoms (32 KB); every stage feeds both row tiles, so each dictionary byte fetched
//     from L2 serves 256 rows;
//   - tcgen05.mma (M = 128, N = 256, K = 16, bf16 x bf16 -> fp32) writes the 128 x 256
//     correlations of (row tile, atom tile) into that row tile's TMEM accumulator (2 row
//     tiles x 256 columns = all 512 columns).  N = 256 per instruction is what keeps the
//     tensor pipe fed: with N = 128 the operand reads from shared memory (A and B per
//     instruction) need the whole shared-memory bandwidth and the pipe starves;
//   - eight epilogue warps (four per row tile, one thread per row) pull the
//     accumulators out with tcgen05.ld and keep a running arg-max of |correlation| per
//     row.  The plain-ALU work per correlation value is what bounds the kernel next to
//     the tensor pipe, so it is cut in two levels: groups of G adjacent atoms are first
//     reduced to max |value| with 3-input floating-point maxima (absolute value is an
//     operand modifier, half an instruction per value), then the group maximum's low
//     mantissa bits are replaced by a group tag (one logic instruction per group) and a
//     3-input integer max per two groups tracks the largest magnitude and where it was.
//     The first half of an accumulator is processed while its second half is already on
//     its way into registers, so the accumulator is handed back to the tensor core after
//     half of the arithmetic; the two row tiles alternate on the tensor pipe.  The M x N
//     correlations never leave the SM;
//   - at the end of a sweep the four warps of a row tile resolve their rows' picks
//     cooperatively: eight lanes per row gather the G atoms of the row's winning group
//     (bf16, from L2, 128 contiguous bytes or more per request), recompute the G signed
//     correlations as fp32 dot products with the residual row, take the largest in
//     magnitude as (index, coefficient), subtract coefficient * atom and write the bf16
//     residual back into the operand tile; then the MMA warp is released for the next
//     iteration;
//   - codes are collected in shared memory and written as 16-byte vectors (uint16 index,
//     fp16 or fp32 coefficient).
//
// Warp roles: warps 0-3 epilogue of row tile 0, warps 4-7 epilogue of row tile 1 (warp w
// reads TMEM lanes 32*(w%4) .. +31), warp 8 TMA producer, warp 9 TMEM owner and MMA
// issuer.  All hand-offs are mbarriers; every wait is bounded by a wall-clock limit,
// after which the CTA raises a flag in the status word, lets its copies land, frees
// its TMEM and exits.
//
// Few rows (the vectors one decoding step adds, a short prompt, what is left over after whole waves of
// pairs) would leave most SMs idle, each of the others sweeping the whole dictionary s times.  A
// second instantiation (template argument ONE) works on single row tiles: n_splits CTAs (1, 2, 4, 8 or
// 16, a thread-block cluster) hold the same tile and each sweep a slice of the dictionary, both
// accumulators and both epilogue warp groups serving the one tile; after every sweep the rows' maxima
// are exchanged through distributed shared memory in one hop (st.async credited to the peers'
// mbarriers, into the other row tile's memory) and every CTA makes the same pick and update, so all
// s iterations run in one launch.  plan_rows() says which rows run how; the codes are the same bits in
// every case.  The handful of rows that a decoding step adds takes encode_few_kernel instead, which
// holds the dictionary in registers; its correlations are summed in another order, so that it could part
// from the others where two atoms' correlations agree to the width of the key's tag and the last
// bit decides (about one pick in 10^6; none in the tests).  (Where clusters must not be used, n_splits > 1 without ONE sweeps a slice for one
// iteration and leaves the rows' maxima to split_pick_kernel: a launch pair per iteration.)
#include <cuda.h>

#include <atomic>
#include <mutex>

#include "common.cuh"
#include "tcgen05_common.cuh"

namespace csr {
namespace {

using namespace tc;

constexpr int TILE_M = 128;
constexpr int TILE_N = 256;                           // atoms per accumulator / per MMA instruction
constexpr int STAGE_CH = 64;                          // channels per dictionary stage (one 128-byte row)
constexpr int STAGES = 4;
constexpr int NT = 320;
constexpr int PRODUCER_WARP = 8;
constexpr int MMA_WARP = 9;
constexpr uint32_t TMEM_COLS = 512;
constexpr int CODE_BLOCK = 8;                         // codes collected before a flush


// Instruction descriptor: fp32 accumulator, bf16 A and B, both K-major, M = 128, N = 256.
constexpr uint32_t kInstrDesc = instr_desc_bf16(TILE_M, TILE_N);

// ---------------------------------------------------------------------------------------
// shared memory
// ---------------------------------------------------------------------------------------
template <int D_>
struct FastSmem {
    static constexpr int kATileBytes = TILE_M * D_ * 2;          // residual tile: D_/64 blocks of 128 rows x 128 B
    static constexpr int kStageBytes = TILE_N * STAGE_CH * 2;    // 256 atoms x 64 channels
    alignas(1024) uint8_t A[2][kATileBytes];
    alignas(1024) uint8_t B[STAGES][kStageBytes];
    alignas(16) uint16_t code_idx[2 * TILE_M][CODE_BLOCK];
    alignas(16) float code_coef[2 * TILE_M][CODE_BLOCK];
    uint64_t full_b[STAGES];
    uint64_t empty_b[STAGES];
    uint64_t acc_full[2];
    uint64_t acc_empty[2];
    uint64_t res_ready[2];
    uint64_t drained;
    // ONE:
    uint64_t pair_bar;                                 // the second warp group's maxima are in xout
    uint64_t pick_bar;                                 // the rows' winning atoms are in pick_n0 (for the second group)
    uint64_t xbar;                                     // every CTA's maxima have arrived, one phase per iteration
    unsigned long long xout[TILE_M];
    int pick_n0[TILE_M];
    uint32_t tmem_base;
    volatile uint32_t abort;
};


// Byte offset of 16-byte chunk `chunk` (8 channels) of row `r` inside a residual tile.
__device__ __forceinline__ uint32_t swz_off(int r, int chunk) {
    const int khalf = chunk >> 3, cc = chunk & 7;
    return khalf * (TILE_M * 128) + (r >> 3) * 1024 + (r & 7) * 128 + ((cc ^ (r & 7)) << 4);
}

// First atom of the group a (key, tile) pair names.  Whatever the keys say (NaN correlations can
// make a zero-filled column past the dictionary win) the gather that follows stays inside the
// padded bf16 copy; a build with CSR_DEBUG_CHECKS also records that the clamp was needed.
template <int G>
__device__ __forceinline__ int candidate_start(uint32_t best_key, uint32_t best_t, int N, [[maybe_unused]] uint32_t* status) {
    constexpr int NG = TILE_N / G;
    const int n0 = static_cast<int>(best_t) * TILE_N + (NG - 1 - static_cast<int>(best_key & static_cast<uint32_t>(NG - 1))) * G;
    const int last = ((N + 7) / 8) * 8 - G;
#ifdef CSR_DEBUG_CHECKS
    if (n0 > last || n0 < 0) atomicOr(status, kStatusBounds);
#endif
    return min(n0, last);
}

__device__ __forceinline__ float bf_lo(uint32_t u) { return __uint_as_float(u << 16); }
__device__ __forceinline__ float bf_hi(uint32_t u) { return __uint_as_float(u & 0xFFFF0000u); }
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
    __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t*>(&v);
}

// (a & mask) | TAG as one logic instruction: the mask is a kernel argument (so it sits in
// a register) and the tag is the instruction's immediate.
template <uint32_t TAG>
__device__ __forceinline__ uint32_t mask_tag(uint32_t a, uint32_t mask) {
    uint32_t r;
    asm("lop3.b32 %0, %1, %2, %3, 0xEA;" : "=r"(r) : "r"(a), "r"(mask), "n"(TAG));
    return r;
}
// max(|a|, |b|, |c|)
__device__ __forceinline__ float absmax3(float a, float b, float c) {
    float r;
    asm("max.abs.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}

// Key of the group of G values starting at v[J] (column COL0 + J of the accumulator):
// max |value| with its low bits replaced by the tag of the group (higher tag = lower
// column, so that the lowest column wins ties).
template <int G, int COL0, int J>
__device__ __forceinline__ uint32_t group_key(const uint32_t (&v)[32], uint32_t mask) {
    constexpr uint32_t kTag = static_cast<uint32_t>(TILE_N / G - 1 - (COL0 + J) / G);
    if constexpr (G == 1) {
        return mask_tag<kTag>(v[J], mask);                // the mask also clears the sign
    } else {
        float gm;
        if constexpr (G == 2) {
            gm = fmaxf(fabsf(__uint_as_float(v[J])), fabsf(__uint_as_float(v[J + 1])));
        } else if constexpr (G == 4) {
            gm = fmaxf(absmax3(__uint_as_float(v[J]), __uint_as_float(v[J + 1]), __uint_as_float(v[J + 2])),
                       fabsf(__uint_as_float(v[J + 3])));
        } else {
            const float t1 = absmax3(__uint_as_float(v[J]), __uint_as_float(v[J + 1]), __uint_as_float(v[J + 2]));
            const float t2 = absmax3(__uint_as_float(v[J + 3]), __uint_as_float(v[J + 4]), __uint_as_float(v[J + 5]));
            gm = fmaxf(t2, absmax3(__uint_as_float(v[J + 6]), __uint_as_float(v[J + 7]), t1));
        }
        return mask_tag<kTag>(__float_as_uint(gm), mask);
    }
}

// Running key maxima (two independent chains) over the 32 / G groups of a 32-column chunk.
template <int G, int COL0, int J = 0>
__device__ __forceinline__ void chunk_key_max(const uint32_t (&v)[32], uint32_t mask, uint32_t& m0, uint32_t& m1) {
    if constexpr (J < 32) {
        m0 = __vimax3_u32(m0, group_key<G, COL0, J>(v, mask), group_key<G, COL0, J + G>(v, mask));
        m1 = __vimax3_u32(m1, group_key<G, COL0, J + 2 * G>(v, mask), group_key<G, COL0, J + 3 * G>(v, mask));
        chunk_key_max<G, COL0, J + 4 * G>(v, mask, m0, m1);
    }
}

// even += lo(r) * lo(a), odd += hi(r) * hi(a) for one word of two bf16 values each: the product of
// two bf16 values is exact in fp32 and the sum is rounded once (the value fmaf gives on the widened
// operands), and the mixed-precision instruction takes the 16-bit halves as they are.
__device__ __forceinline__ void fma2_bf16(float& even, float& odd, uint32_t r, uint32_t a) {
    asm("{\n"
        ".reg .b16 rl, rh, al, ah;\n"
        "mov.b32 {rl, rh}, %2;\n"
        "mov.b32 {al, ah}, %3;\n"
        "fma.rn.f32.bf16 %0, rl, al, %0;\n"
        "fma.rn.f32.bf16 %1, rh, ah, %1;\n"
        "}\n"
        : "+f"(even), "+f"(odd)
        : "r"(r), "r"(a));
}
// fp32 dot product of eight bf16 pairs (one 16-byte chunk of a residual row and of an atom)
__device__ __forceinline__ void dot8(const uint4& rv, const uint4& av, float& even, float& odd) {
    fma2_bf16(even, odd, rv.x, av.x);
    fma2_bf16(even, odd, rv.y, av.y);
    fma2_bf16(even, odd, rv.z, av.z);
    fma2_bf16(even, odd, rv.w, av.w);
}
// r -= coef * a on one 16-byte chunk, rounded back to bf16
__device__ __forceinline__ uint4 axpy8(const uint4& rv, const uint4& av, float coef) {
    uint4 o;
    o.x = pack_bf16(fmaf(-coef, bf_lo(av.x), bf_lo(rv.x)), fmaf(-coef, bf_hi(av.x), bf_hi(rv.x)));
    o.y = pack_bf16(fmaf(-coef, bf_lo(av.y), bf_lo(rv.y)), fmaf(-coef, bf_hi(av.y), bf_hi(rv.y)));
    o.z = pack_bf16(fmaf(-coef, bf_lo(av.z), bf_lo(rv.z)), fmaf(-coef, bf_hi(av.z), bf_hi(rv.z)));
    o.w = pack_bf16(fmaf(-coef, bf_lo(av.w), bf_lo(rv.w)), fmaf(-coef, bf_hi(av.w), bf_hi(rv.w)));
    return o;
}

// End of a sweep for the 32 rows of one epilogue warp (Eq. 2-4).  Lane i enters with the
// first atom `n0` of the winning group of row q*32 + i.  Eight lanes work on one row (four
// rows per pass, eight passes): each lane gathers its 1/8 of the G candidate atoms (one
// contiguous run of G * 2 * D_ bytes per row), the G signed correlations with the row's
// residual are rebuilt as fp32 dot products and summed over the eight lanes, the largest
// in magnitude (lowest atom on ties) gives the index and the coefficient, and, unless
// this was the last iteration, the residual row in the operand tile becomes
// R - coef * atom.  The code goes to the row's slot in the shared-memory staging arrays.
// With SKIP, groups of (at most four) passes none of whose rows is set in `row_mask` (bit i =
// row i of the warp's 32 is a row of X) are left out: with few rows the pick is on the
// critical path of every iteration.
template <int D_, int G, bool SKIP = false>
__device__ __forceinline__ void pick_and_update(uint8_t* Atile, int q, int lane, const uint16_t* __restrict__ Db,
                                                int n0, bool update, uint16_t (*code_idx)[CODE_BLOCK],
                                                float (*code_coef)[CODE_BLOCK], int gi, uint32_t row_mask = 0xffffffffu) {
    constexpr int CH = D_ / 64;                           // 16-byte chunks per lane per atom
    constexpr int APR = D_ / 8;                           // 16-byte chunks per atom row
    constexpr int LPP = G * CH;                           // gathered chunks per lane per pass
    constexpr int WAVE0 = (32 / LPP) < 8 ? (32 / LPP) : 8;
    constexpr int WAVE = SKIP && WAVE0 > 4 ? 4 : WAVE0;   // passes whose gathers are in flight together
    const int sub = lane >> 3, l8 = lane & 7;
#pragma unroll
    for (int w0 = 0; w0 < 8; w0 += WAVE) {
        if (SKIP && ((row_mask >> (w0 * 4)) & ((1ull << (4 * WAVE)) - 1)) == 0) continue;
        uint4 atom[WAVE][G][CH];
        int base[WAVE];
#pragma unroll
        for (int it = 0; it < WAVE; ++it) {
            base[it] = __shfl_sync(0xffffffffu, n0, (w0 + it) * 4 + sub);
            const uint4* src = reinterpret_cast<const uint4*>(Db + static_cast<size_t>(base[it]) * D_) + l8 * CH;
#pragma unroll
            for (int j = 0; j < G; ++j)
#pragma unroll
                for (int c = 0; c < CH; ++c) atom[it][j][c] = __ldg(src + j * APR + c);
        }
#pragma unroll
        for (int it = 0; it < WAVE; ++it) {
            const int i = (w0 + it) * 4 + sub;            // row inside the warp's 32
            const int r = q * 32 + i;                     // row inside the tile
            uint4 rv[CH];
#pragma unroll
            for (int c = 0; c < CH; ++c) rv[c] = *reinterpret_cast<const uint4*>(Atile + swz_off(r, l8 * CH + c));
            float dot[G];
#pragma unroll
            for (int j = 0; j < G; ++j) {
                float ev = 0.f, od = 0.f;
#pragma unroll
                for (int c = 0; c < CH; ++c) dot8(rv[c], atom[it][j][c], ev, od);
                dot[j] = ev + od;
            }
#pragma unroll
            for (int m = 1; m < 8; m <<= 1)
#pragma unroll
                for (int j = 0; j < G; ++j) dot[j] += __shfl_xor_sync(0xffffffffu, dot[j], m);
            float coef = dot[0];
            int jb = 0;
#pragma unroll
            for (int j = 1; j < G; ++j)
                if (fabsf(dot[j]) > fabsf(coef)) {
                    coef = dot[j];
                    jb = j;
                }
            if (update) {
#pragma unroll
                for (int c = 0; c < CH; ++c) {
                    uint4 av = atom[it][0][c];
#pragma unroll
                    for (int j = 1; j < G; ++j)
                        if (jb == j) av = atom[it][j][c];
                    *reinterpret_cast<uint4*>(Atile + swz_off(r, l8 * CH + c)) = axpy8(rv[c], av, coef);
                }
            }
            if (l8 == 0) {
                code_idx[r][gi] = static_cast<uint16_t>(base[it] + jb);
                code_coef[r][gi] = coef;
            }
        }
    }
}

// ---------------------------------------------------------------------------------------
// dictionary preparation: fp32 -> bf16 copy, same [N][d] layout, zeros up to a multiple of eight atoms
// ---------------------------------------------------------------------------------------
// The encoder that follows may be launched with programmatic stream serialization (EncodeArgs::after_copy): its CTAs come
// up beside this kernel's, load their rows and wait for its end before they touch the copy.  4160 fp32 rows, N = 1024,
// s = 8: 45.1 us one after the other, 42.0 so; 100003 rows, N = 5001, d = 64, whose padding was a launch of its own: 432 -> 428.
__device__ __forceinline__ void next_may_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void wait_for_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

__global__ void dict_to_bf16_kernel(const float4* __restrict__ src, uint2* __restrict__ dst, int64_t n_vec4, int64_t n_padded) {
    next_may_start();
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n_padded; i += (int64_t)gridDim.x * blockDim.x) {
        uint2 o = make_uint2(0u, 0u);
        if (i < n_vec4) {
            const float4 v = src[i];
            o.x = pack_bf16(v.x, v.y);
            o.y = pack_bf16(v.z, v.w);
        }
        dst[i] = o;
    }
}

// ---------------------------------------------------------------------------------------
// few rows: the dictionary is split across CTAs, one iteration per launch
// ---------------------------------------------------------------------------------------
// R_0 = x rounded to bf16, dense [M][d]; one thread per 16-byte chunk of eight channels.
template <int D_>
__global__ void rows_to_bf16_kernel(const void* __restrict__ X, int x_dtype, int64_t ldx, int64_t M, uint4* __restrict__ Rb) {
    constexpr int CHUNKS = D_ / 8;
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= M * CHUNKS) return;
    const int64_t m = i / CHUNKS;
    const int c = (int)(i % CHUNKS);
    uint4 v;
    if (x_dtype == CSR_DTYPE_BF16) {
        v = *reinterpret_cast<const uint4*>(reinterpret_cast<const uint16_t*>(X) + m * ldx + 8 * c);
    } else {
        float f[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) f[k] = load_elem(X, x_dtype, m * ldx + 8 * c + k);
        v.x = pack_bf16(f[0], f[1]);
        v.y = pack_bf16(f[2], f[3]);
        v.z = pack_bf16(f[4], f[5]);
        v.w = pack_bf16(f[6], f[7]);
    }
    Rb[i] = v;
}

// Pick of one iteration for the split sweep: merges a row's per-CTA (key, tile) pairs (largest
// key, lowest tile among equal keys: the order in which one CTA would have met them), then
// does exactly what pick_and_update does, on the residual rows kept in global memory.
// Eight lanes per row, four rows per warp.
template <int D_, int G>
__global__ void __launch_bounds__(128)
split_pick_kernel(const uint16_t* __restrict__ Db, int N, uint4* __restrict__ Rb, const uint2* __restrict__ partial,
                  int n_splits, int64_t M, int g, int update, uint16_t* __restrict__ out_idx, void* __restrict__ out_coef, int coef_dtype,
                  int64_t ldc) {
    constexpr int CH = D_ / 64;
    constexpr int APR = D_ / 8;
    constexpr int NG = TILE_N / G;
    const int lane = threadIdx.x & 31, sub = lane >> 3, l8 = lane & 7;
    const int64_t m = ((int64_t)blockIdx.x * 4 + (threadIdx.x >> 5)) * 4 + sub;
    const bool valid = m < M;
    uint32_t key = 0, t = 0;
    if (valid) {
        for (int j = l8; j < n_splits; j += 8) {
            const uint2 pr = partial[m * n_splits + j];
            if (pr.x > key || (pr.x == key && pr.y < t)) {
                key = pr.x;
                t = pr.y;
            }
        }
    }
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) {
        const uint32_t ok = __shfl_xor_sync(0xffffffffu, key, o), ot = __shfl_xor_sync(0xffffffffu, t, o);
        if (ok > key || (ok == key && ot < t)) {
            key = ok;
            t = ot;
        }
    }
    const int n0 = min(static_cast<int>(t) * TILE_N + (NG - 1 - static_cast<int>(key & static_cast<uint32_t>(NG - 1))) * G,
                       ((N + 7) / 8) * 8 - G);     // as in the one-launch kernel: never past the padded copy
    const int64_t mr = valid ? m : 0;
    uint4 atom[G][CH], rv[CH];
#pragma unroll
    for (int c = 0; c < CH; ++c) {
        rv[c] = Rb[mr * APR + l8 * CH + c];
#pragma unroll
        for (int j = 0; j < G; ++j)
            atom[j][c] = __ldg(reinterpret_cast<const uint4*>(Db + static_cast<size_t>(n0) * D_) + j * APR + l8 * CH + c);
    }
    float dot[G];
#pragma unroll
    for (int j = 0; j < G; ++j) {
        float ev = 0.f, od = 0.f;
#pragma unroll
        for (int c = 0; c < CH; ++c) dot8(rv[c], atom[j][c], ev, od);
        dot[j] = ev + od;
    }
#pragma unroll
    for (int o = 1; o < 8; o <<= 1)
#pragma unroll
        for (int j = 0; j < G; ++j) dot[j] += __shfl_xor_sync(0xffffffffu, dot[j], o);
    if (!valid) return;
    float coef = dot[0];
    int jb = 0;
#pragma unroll
    for (int j = 1; j < G; ++j)
        if (fabsf(dot[j]) > fabsf(coef)) {
            coef = dot[j];
            jb = j;
        }
    if (update) {
#pragma unroll
        for (int c = 0; c < CH; ++c) {
            uint4 av = atom[0][c];
#pragma unroll
            for (int j = 1; j < G; ++j)
                if (jb == j) av = atom[j][c];
            Rb[m * APR + l8 * CH + c] = axpy8(rv[c], av, coef);
        }
    }
    if (l8 == 0) {
        out_idx[m * ldc + g] = static_cast<uint16_t>(n0 + jb);
        if (coef_dtype == CSR_DTYPE_F16)
            reinterpret_cast<__half*>(out_coef)[m * ldc + g] = __float2half_rn(coef);
        else
            reinterpret_cast<float*>(out_coef)[m * ldc + g] = coef;
    }
}

// ---------------------------------------------------------------------------------------
// the encoder
// ---------------------------------------------------------------------------------------
template <int D_, int G, bool ONE>
__global__ void __launch_bounds__(NT, 1)
encode_fast_kernel(const __grid_constant__ CUtensorMap tmap_d, const uint16_t* __restrict__ Db,
                   const void* __restrict__ X, int x_dtype, int64_t ldx, int64_t M, int N, int s,
                   uint16_t* __restrict__ out_idx, void* __restrict__ out_coef, int coef_dtype, int64_t ldc, int vec_codes,
                   uint32_t key_mask, uint32_t* status, int n_splits, uint2* __restrict__ partial,
                   unsigned long long wait_limit_ns) {
    using S = FastSmem<D_>;
    extern __shared__ uint8_t smem_raw[];
    S& sm = *reinterpret_cast<S*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));

    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    const int T = (N + TILE_N - 1) / TILE_N;                // dictionary tiles per sweep (the last may be half)
    const int64_t n_pairs = ONE ? (M + TILE_M - 1) / TILE_M : (M + 2 * TILE_M - 1) / (2 * TILE_M);   // (ONE: single tiles)
    // n_splits > 1: n_splits CTAs share the rows, CTA j sweeping the dictionary tiles j, j + n_splits, ...
    //  - ONE: they are one thread-block cluster, hold the same single row tile and run all s
    //    iterations.  Only the first row tile exists; the two accumulators take the CTA's
    //    dictionary tiles in turn and the second group of epilogue warps drains the second
    //    accumulator for the same rows; the unused second row tile holds the exchange buffers, large
    //    enough for every CTA to hear from every CTA directly.  CTA 0 of the cluster writes the codes.
    //  - otherwise ONE iteration per launch (s == 1 is passed) on pairs of row tiles: each row's
    //    best (key, tile) goes to `partial` and the pick kernel takes over.
    const int t_begin = n_splits > 1 ? (int)(blockIdx.x % n_splits) : 0;
    const int t_step = n_splits > 1 ? n_splits : 1;
    const int64_t pair_first = n_splits > 1 ? blockIdx.x / n_splits : blockIdx.x;
    const int64_t pair_step = n_splits > 1 ? gridDim.x / n_splits : gridDim.x;
    constexpr int KH = D_ / STAGE_CH;                       // stages per dictionary tile
    constexpr int CHUNKS = D_ / 8;                          // 16-byte chunks per row
    constexpr int NG = TILE_N / G;                          // arg-max groups per accumulator
    const WaitCtx wc{&sm.abort, status, wait_limit_ns};

    if (threadIdx.x == 0) {
        for (int i = 0; i < STAGES; ++i) {
            mbar_init(&sm.full_b[i], 1);
            mbar_init(&sm.empty_b[i], 1);
        }
        for (int t = 0; t < 2; ++t) {
            mbar_init(&sm.acc_full[t], 1);
            mbar_init(&sm.acc_empty[t], 4);
            // (with one tile of rows both warp groups update rows of it)
            mbar_init(&sm.res_ready[t], ONE ? 2 * TILE_M : TILE_M);
        }
        mbar_init(&sm.drained, 1);
        if constexpr (ONE) {
            mbar_init(&sm.xbar, 1);
            mbar_expect_tx(&sm.xbar, static_cast<uint32_t>(n_splits) * TILE_M * 8);
            mbar_init(&sm.pair_bar, TILE_M);
            mbar_init(&sm.pick_bar, TILE_M);
        }
        sm.abort = 0;
        fence_barrier_init();
    }
    if (warp == MMA_WARP) {
        tmem_alloc(&sm.tmem_base, TMEM_COLS);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = sm.tmem_base;
    // no CTA touches a peer's barrier or words before every peer has set them up
    if constexpr (ONE) cluster_sync_all();
    [[maybe_unused]] uint32_t x_phases = 0;                 // phases of xbar that thread 0 has waited out

    if (warp == PRODUCER_WARP) {
        // ------------------------------ TMA producer ------------------------------
        if (lane == 0) {
            asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmap_d)) : "memory");
            wait_for_previous();                              // the bf16 copy
            uint32_t p = 0;
            bool ok = true;
            for (int64_t pair = pair_first; pair < n_pairs && ok; pair += pair_step) {
                for (int g = 0; g < s && ok; ++g) {
                    for (int t = t_begin; t < T && ok; t += t_step) {
                        for (int h = 0; h < KH; ++h, ++p) {
                            const int stage = p % STAGES;
                            if (!wait_bounded(&sm.empty_b[stage], ((p / STAGES) & 1) ^ 1, wc)) {
                                ok = false;
                                break;
                            }
                            // rows past N (a half tile at the end) arrive as zeros and count as bytes
                            mbar_expect_tx(&sm.full_b[stage], S::kStageBytes);
                            tma_load_2d(&sm.B[stage][0], &tmap_d, h * STAGE_CH, t * TILE_N, &sm.full_b[stage]);
                        }
                    }
                }
            }
            if (!ok) {
                // let the copies already issued land before the CTA goes away
                const uint32_t first = p > STAGES ? p - STAGES : 0;
                for (uint32_t qq = first; qq < p; ++qq) {
                    const unsigned long long t0 = globaltimer_ns();
                    while (!mbar_try_wait(&sm.full_b[qq % STAGES], (qq / STAGES) & 1))
                        if (globaltimer_ns() - t0 > 20000000ull) break;
                }
            }
        }
    } else if (warp == MMA_WARP) {
        // ------------------------------ MMA issuer ------------------------------
        // (the whole warp runs this, one elected lane issues: see umma_f16_block)
        const uint32_t tmem_d = warp_uniform(tmem_base);
        if constexpr (ONE) {
            // one row tile; the CTA's dictionary tiles go to the two accumulators in turn
            uint32_t p = 0, accn[2] = {0u, 0u};
            bool ok = true;
            for (int g = 0; g < s && ok; ++g) {
                if (!warp_wait_bounded(&sm.res_ready[0], g & 1, wc)) {
                    ok = false;
                    break;
                }
                int j = 0;
                for (int t = t_begin; t < T && ok; t += t_step, p += KH, ++j) {
                    const int acc = j & 1;
                    if (!warp_wait_bounded(&sm.acc_empty[acc], (accn[acc] & 1) ^ 1, wc)) {
                        ok = false;
                        break;
                    }
                    const uint32_t d_tmem = tmem_d + acc * TILE_N;
#pragma unroll
                    for (int h = 0; h < KH; ++h) {
                        const uint32_t ps = p + h;
                        const int stage = ps % STAGES;
                        if (!warp_wait_bounded(&sm.full_b[stage], (ps / STAGES) & 1, wc)) {
                            ok = false;
                            break;
                        }
                        tc_fence_after();
                        const uint64_t a0 = make_smem_desc(smem_u32(&sm.A[0][h * (TILE_M * 128)]));
                        const uint64_t b0 = make_smem_desc(smem_u32(&sm.B[stage][0]));
                        if (h < KH - 1)
                            umma_f16_block(d_tmem, a0, b0, kInstrDesc, h, &sm.empty_b[stage]);
                        else
                            umma_f16_block(d_tmem, a0, b0, kInstrDesc, h, &sm.empty_b[stage], &sm.acc_full[acc]);
                    }
                    if (ok) ++accn[acc];
                }
            }
            if (!ok) {
                umma_commit(&sm.drained);
                const unsigned long long t0 = globaltimer_ns();
                while (!mbar_try_wait(&sm.drained, 0))
                    if (globaltimer_ns() - t0 > 20000000ull) break;
            }
        } else {
            uint32_t p = 0, accn = 0, steps = 0;
            bool ok = true;
            for (int64_t pair = pair_first; pair < n_pairs && ok; pair += pair_step) {
                for (int g = 0; g < s && ok; ++g, ++steps) {
                    for (int t = t_begin; t < T && ok; t += t_step, p += KH, ++accn) {
#pragma unroll
                        for (int tile = 0; tile < 2; ++tile) {
                            if (t == t_begin) ok = warp_wait_bounded(&sm.res_ready[tile], steps & 1, wc);
                            if (ok) ok = warp_wait_bounded(&sm.acc_empty[tile], (accn & 1) ^ 1, wc);
                            const uint32_t d_tmem = tmem_d + tile * TILE_N;
#pragma unroll
                            for (int h = 0; h < KH; ++h) {
                                const uint32_t ps = p + h;
                                const int stage = ps % STAGES;
                                if (tile == 0 && ok) ok = warp_wait_bounded(&sm.full_b[stage], (ps / STAGES) & 1, wc);
                                if (!ok) break;
                                tc_fence_after();
                                const uint64_t a0 = make_smem_desc(smem_u32(&sm.A[tile][h * (TILE_M * 128)]));
                                const uint64_t b0 = make_smem_desc(smem_u32(&sm.B[stage][0]));
                                // (the second row tile is the last reader of a stage)
                                if (h < KH - 1 && tile == 0)
                                    umma_f16_block(d_tmem, a0, b0, kInstrDesc, h);
                                else if (h < KH - 1)
                                    umma_f16_block(d_tmem, a0, b0, kInstrDesc, h, &sm.empty_b[stage]);
                                else if (tile == 0)
                                    umma_f16_block(d_tmem, a0, b0, kInstrDesc, h, &sm.acc_full[tile]);
                                else
                                    umma_f16_block(d_tmem, a0, b0, kInstrDesc, h, &sm.empty_b[stage], &sm.acc_full[tile]);
                            }
                            if (!ok) break;
                        }
                    }
                }
            }
            if (!ok) {
                // wait (bounded) until the tensor core has stopped writing TMEM
                umma_commit(&sm.drained);
                const unsigned long long t0 = globaltimer_ns();
                while (!mbar_try_wait(&sm.drained, 0))
                    if (globaltimer_ns() - t0 > 20000000ull) break;
            }
        }
    } else {
        // ------------------------------ epilogue ------------------------------
        const int acc = warp >> 2;                        // the accumulator this warp drains
        const int tile = ONE ? 0 : acc;               // the row tile its rows belong to
        const int q = warp & 3;
        const int r = q * 32 + lane;                      // row inside the tile == TMEM lane
        const int slot = tile * TILE_M + r;               // row inside the CTA's pair
        uint8_t* Atile = &sm.A[tile][0];
        uint16_t (*code_idx)[CODE_BLOCK] = &sm.code_idx[tile * TILE_M];
        float (*code_coef)[CODE_BLOCK] = &sm.code_coef[tile * TILE_M];
        const uint32_t taddr = tmem_base + (static_cast<uint32_t>(q * 32) << 16) + acc * TILE_N;
        uint32_t accn = 0;
        [[maybe_unused]] uint32_t xn = 0;
        bool ok = true;
        const bool writes_codes = !ONE || t_begin == 0;
        for (int64_t pair = pair_first; pair < n_pairs && ok; pair += pair_step) {
            const int64_t m = pair * (ONE ? TILE_M : 2 * TILE_M) + slot;
            const bool valid = m < M;
            uint32_t row_mask = 0xffffffffu;
            if constexpr (ONE) row_mask = __ballot_sync(0xffffffffu, valid);
            // ---- R_0 = x, rounded to bf16, into the operand tile ----
            if (ONE && acc == 1) {
                // the second warp group has no rows of its own
            } else if (x_dtype == CSR_DTYPE_BF16) {
                const uint4* src = reinterpret_cast<const uint4*>(reinterpret_cast<const uint16_t*>(X) + m * ldx);
#pragma unroll
                for (int c = 0; c < CHUNKS; ++c) {
                    uint4 v = make_uint4(0u, 0u, 0u, 0u);
                    if (valid) v = __ldg(src + c);
                    *reinterpret_cast<uint4*>(Atile + swz_off(r, c)) = v;
                }
            } else if (x_dtype == CSR_DTYPE_F16) {
                const uint4* src = reinterpret_cast<const uint4*>(reinterpret_cast<const uint16_t*>(X) + m * ldx);
#pragma unroll
                for (int c = 0; c < CHUNKS; ++c) {
                    uint4 h = make_uint4(0u, 0u, 0u, 0u);
                    if (valid) h = __ldg(src + c);
                    const __half2* hp = reinterpret_cast<const __half2*>(&h);
                    const float2 f0 = __half22float2(hp[0]), f1 = __half22float2(hp[1]);
                    const float2 f2 = __half22float2(hp[2]), f3 = __half22float2(hp[3]);
                    uint4 v;
                    v.x = pack_bf16(f0.x, f0.y);
                    v.y = pack_bf16(f1.x, f1.y);
                    v.z = pack_bf16(f2.x, f2.y);
                    v.w = pack_bf16(f3.x, f3.y);
                    *reinterpret_cast<uint4*>(Atile + swz_off(r, c)) = v;
                }
            } else {
                const float4* src = reinterpret_cast<const float4*>(reinterpret_cast<const float*>(X) + m * ldx);
#pragma unroll
                for (int c = 0; c < CHUNKS; ++c) {
                    float4 a = make_float4(0.f, 0.f, 0.f, 0.f), b = a;
                    if (valid) {
                        a = __ldg(src + 2 * c);
                        b = __ldg(src + 2 * c + 1);
                    }
                    uint4 v;
                    v.x = pack_bf16(a.x, a.y);
                    v.y = pack_bf16(a.z, a.w);
                    v.z = pack_bf16(b.x, b.y);
                    v.w = pack_bf16(b.z, b.w);
                    *reinterpret_cast<uint4*>(Atile + swz_off(r, c)) = v;
                }
            }
            fence_proxy_async_smem();
            mbar_arrive(&sm.res_ready[tile]);
            wait_for_previous();                              // (the picks read the copy too)

            for (int g = 0; g < s && ok; ++g) {
                // ---- sweep: running arg-max of |correlation| over all atom tiles ----
                uint32_t best_key = 0, best_t = 0;
                [[maybe_unused]] int n0_other = 0;
                for (int t = t_begin + (ONE ? acc * t_step : 0); t < T; t += (ONE ? 2 : 1) * t_step, ++accn) {
                    bool got = wait_bounded(&sm.acc_full[acc], accn & 1, wc);
                    got = __all_sync(0xffffffffu, got);
                    if (!got) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    uint32_t v0[32], v1[32], v2[32], v3[32];
                    uint32_t k0 = 0, k1 = 0;
                    tmem_ld32(taddr + 0, v0);
                    tmem_ld32(taddr + 32, v1);
                    tmem_ld32(taddr + 64, v2);
                    tmem_ld32(taddr + 96, v3);
                    tmem_wait_ld(v0);
                    reg_fence(v1);
                    reg_fence(v2);
                    reg_fence(v3);
                    chunk_key_max<G, 0>(v0, key_mask, k0, k1);
                    tmem_ld32(taddr + 128, v0);
                    chunk_key_max<G, 32>(v1, key_mask, k0, k1);
                    tmem_ld32(taddr + 160, v1);
                    chunk_key_max<G, 64>(v2, key_mask, k0, k1);
                    tmem_ld32(taddr + 192, v2);
                    chunk_key_max<G, 96>(v3, key_mask, k0, k1);
                    tmem_ld32(taddr + 224, v3);
                    tmem_wait_ld(v0);
                    reg_fence(v1);
                    reg_fence(v2);
                    reg_fence(v3);
                    // every column of this accumulator is in registers: hand it back
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&sm.acc_empty[acc]);
                    chunk_key_max<G, 128>(v0, key_mask, k0, k1);
                    chunk_key_max<G, 160>(v1, key_mask, k0, k1);
                    chunk_key_max<G, 192>(v2, key_mask, k0, k1);
                    chunk_key_max<G, 224>(v3, key_mask, k0, k1);
                    const uint32_t key = k0 > k1 ? k0 : k1;
                    if (key > best_key) {
                        best_key = key;
                        best_t = t;
                    }
                }
                if (!ok) break;
                if (!ONE && partial) {                       // split sweep: the pick kernel takes over
                    if (valid) partial[m * n_splits + t_begin] = make_uint2(best_key, best_t);
                    continue;
                }
                if constexpr (ONE) {
                    // ---- the row's best over this CTA's tiles (both accumulators), then over the
                    // whole dictionary: every CTA sends its (key, ~tile) of the row to every CTA.
                    // The entries are double-buffered by iteration: a peer writes iteration g + 2's
                    // only after it has heard this CTA's iteration g + 1, which the thread that
                    // reads the entries sends after it has read iteration g's. ----
                    unsigned long long mine = (static_cast<unsigned long long>(best_key) << 32) | (0xFFFFFFFFu - best_t);
                    // (a CTA with a single dictionary tile has no use for the second group, which
                    // would otherwise run ahead of the first: nothing paces it but its sweep)
                    const bool two_groups = t_begin + t_step < T;
                    bool got = true;
                    if (acc == 1) {
                        if (two_groups) {
                            sm.xout[r] = mine;
                            mbar_arrive(&sm.pair_bar);
                        }
                        // the second half of every warp's rows is picked and updated by this group
                        got = wait_bounded(&sm.pick_bar, xn & 1, wc);
                    } else if (two_groups) {
                        got = wait_bounded(&sm.pair_bar, xn & 1, wc);
                    }
                    if (got && acc == 0 && two_groups) {
                        const unsigned long long other = *reinterpret_cast<volatile unsigned long long*>(&sm.xout[r]);
                        mine = other > mine ? other : mine;
                    }
                    if (got && acc == 0 && n_splits > 1) {
                        constexpr int XMAX = FastSmem<D_>::kATileBytes / (2 * TILE_M * 8);   // CTAs the buffers hold
                        unsigned long long* xg = reinterpret_cast<unsigned long long*>(&sm.A[1][0]) + (xn & 1) * XMAX * TILE_M;
                        const uint32_t dst = smem_u32(&xg[t_begin * TILE_M + r]), bar = smem_u32(&sm.xbar);
                        for (int c = 0; c < n_splits; ++c) st_async_u64(map_to_cta(dst, c), mine, map_to_cta(bar, c));
                        got = wait_bounded_cluster(&sm.xbar, xn & 1, wc);
                        if (got) {
                            if (r == 0) {
                                mbar_expect_tx(&sm.xbar, static_cast<uint32_t>(n_splits) * TILE_M * 8);
                                ++x_phases;
                            }
                            unsigned long long top = 0ull;
                            for (int c = 0; c < n_splits; ++c) {
                                const unsigned long long v = *reinterpret_cast<volatile unsigned long long*>(&xg[c * TILE_M + r]);
                                top = v > top ? v : top;
                            }
                            mine = top;
                        }
                    }
                    got = __all_sync(0xffffffffu, got);
                    if (!got) {
                        ok = false;
                        break;
                    }
                    ++xn;
                    best_key = static_cast<uint32_t>(mine >> 32);
                    best_t = 0xFFFFFFFFu - static_cast<uint32_t>(mine);
                    if (acc == 0) {
                        sm.pick_n0[r] = candidate_start<G>(best_key, best_t, N, status);
                        mbar_arrive(&sm.pick_bar);
                        row_mask &= 0x0000FFFFu;
                    } else {
                        n0_other = *reinterpret_cast<volatile int*>(&sm.pick_n0[r]);
                        row_mask &= 0xFFFF0000u;
                    }
                }
                // ---- pick, signed coefficient, residual update ----
                const int gi = g & (CODE_BLOCK - 1);
                int n0 = candidate_start<G>(best_key, best_t, N, status);
                if (ONE && acc == 1) n0 = n0_other;
                if constexpr (ONE)
                    pick_and_update<D_, G, true>(Atile, q, lane, Db, n0, g + 1 < s, code_idx, code_coef, gi, row_mask);
                else
                    pick_and_update<D_, G>(Atile, q, lane, Db, n0, g + 1 < s, code_idx, code_coef, gi);
                if (g + 1 < s) {
                    fence_proxy_async_smem();
                    mbar_arrive(&sm.res_ready[tile]);
                }
                __syncwarp();
                // ---- flush the collected codes eight at a time ----
                if ((gi == CODE_BLOCK - 1 || g == s - 1) && valid && writes_codes && (!ONE || (lane < 16) == (acc == 0))) {
                    const int g0 = g - gi;
                    const int64_t o = m * ldc + g0;
                    if (gi == CODE_BLOCK - 1 && vec_codes) {
                        *reinterpret_cast<uint4*>(out_idx + o) = *reinterpret_cast<const uint4*>(&sm.code_idx[slot][0]);
                        const float4 f0 = *reinterpret_cast<const float4*>(&sm.code_coef[slot][0]);
                        const float4 f1 = *reinterpret_cast<const float4*>(&sm.code_coef[slot][4]);
                        if (coef_dtype == CSR_DTYPE_F16) {
                            __half2 h0 = __floats2half2_rn(f0.x, f0.y), h1 = __floats2half2_rn(f0.z, f0.w);
                            __half2 h2 = __floats2half2_rn(f1.x, f1.y), h3 = __floats2half2_rn(f1.z, f1.w);
                            uint4 u;
                            u.x = *reinterpret_cast<uint32_t*>(&h0);
                            u.y = *reinterpret_cast<uint32_t*>(&h1);
                            u.z = *reinterpret_cast<uint32_t*>(&h2);
                            u.w = *reinterpret_cast<uint32_t*>(&h3);
                            *reinterpret_cast<uint4*>(reinterpret_cast<__half*>(out_coef) + o) = u;
                        } else {
                            float4* dst = reinterpret_cast<float4*>(reinterpret_cast<float*>(out_coef) + o);
                            dst[0] = f0;
                            dst[1] = f1;
                        }
                    } else {
                        for (int j = 0; j <= gi; ++j) {
                            out_idx[o + j] = sm.code_idx[slot][j];
                            if (coef_dtype == CSR_DTYPE_F16)
                                reinterpret_cast<__half*>(out_coef)[o + j] = __float2half_rn(sm.code_coef[slot][j]);
                            else
                                reinterpret_cast<float*>(out_coef)[o + j] = sm.code_coef[slot][j];
                        }
                    }
                }
                __syncwarp();
            }
        }
    }

    // ------------------------------ teardown ------------------------------
    tc_fence_before();
    __syncthreads();
    if (warp == MMA_WARP) {
        tc_fence_after();
        tmem_dealloc(tmem_base, TMEM_COLS);
    }
    // A CTA's shared memory must outlive its peers' last writes to it: a CTA that has done all iterations
    // has waited for every one of them, one that has given up has not.
    if constexpr (ONE) {
        cluster_sync_all();
        if (sm.abort != 0 && threadIdx.x == 0 && n_splits > 1)
            let_words_land(&sm.xbar, x_phases, static_cast<uint32_t>(n_splits) * TILE_M * 8);
    }
}

// ---------------------------------------------------------------------------------------
// a handful of rows: the dictionary in registers
// ---------------------------------------------------------------------------------------
// What one decoding step adds is 8 to 128 rows.  A 128-row MMA spends 2100 cycles on 512 atoms whatever
// the rows, and with its hand-offs a sweep of two dictionary tiles takes 4000.  Here a cluster of up to 16
// CTAs keeps the dictionary in registers for all s iterations, 16 warps with MT * 16 atoms each as the A
// fragments of mma.sync m16n8k16 (64 registers), and 8 * NTL residual rows (B, bf16, in shared
// memory) are all that moves: a sweep is 16 * NTL instructions per warp.  The maxima go through one
// shared-memory table and one hop through distributed shared memory, a warp per row; every CTA makes
// the same pick and the same residual update on its own copy of the rows.
// A lane of quarter q holds channels q * D_/4 ..: the k positions of the fragments are dealt out so that
// its share of an atom or of a row is contiguous (a dot product does not mind the order; the
// correlations may differ from tcgen05's in the last bit).
constexpr int RT_THREADS = 512, RT_WARPS = RT_THREADS / 32;
template <int D_, int NTL>
struct FewSmem {
    static constexpr int ROWS = 8 * NTL;
    static constexpr int LD = D_ / 2 + 4;                 // words per residual row: rows 4 banks apart, 16-byte aligned
    alignas(16) uint32_t R[ROWS][LD];                     // residual rows, bf16
    unsigned long long best[ROWS][RT_WARPS];              // (key, ~tile) of each warp's atoms
    unsigned long long from[2][ROWS][16];                 // ... of each CTA's, double-buffered by iteration
    uint64_t bar[ROWS];                                   // one per row: every CTA's word has arrived
    volatile uint32_t abort;
};

__device__ __forceinline__ void mma_bf16_16816(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ unsigned long long max_u64(unsigned long long a, unsigned long long b) { return a > b ? a : b; }

template <int D_, int G, int NTL>
__global__ void __launch_bounds__(RT_THREADS, 1)
encode_few_kernel(const uint16_t* __restrict__ Db, const void* __restrict__ X, int x_dtype, int64_t ldx, int64_t M, int N, int s,
                  uint16_t* __restrict__ out_idx, void* __restrict__ out_coef, int coef_dtype, int64_t ldc, uint32_t key_mask,
                  uint32_t* status, int n_ctas, unsigned long long wait_limit_ns) {
    using S = FewSmem<D_, NTL>;
    constexpr int ROWS = S::ROWS, MT = D_ == 128 ? 2 : 4, KT = D_ / 16;
    constexpr int NG = TILE_N / G;
    __shared__ S sm;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int cta = static_cast<int>(blockIdx.x) % n_ctas;
    const int64_t m0 = static_cast<int64_t>(blockIdx.x / n_ctas) * ROWS;
    const int q4 = lane & 3, l4 = lane >> 2;
    const int n_pad = (N + 7) / 8 * 8;
    const WaitCtx wc{&sm.abort, status, wait_limit_ns};
    if (threadIdx.x < ROWS) {
        mbar_init(&sm.bar[threadIdx.x], 1);
        mbar_expect_tx(&sm.bar[threadIdx.x], static_cast<uint32_t>(n_ctas) * 8);
    }
    if (threadIdx.x == 0) {
        sm.abort = 0;
        fence_barrier_init();
    }
    wait_for_previous();
    // ---- this warp's atoms ----
    const int a0 = (cta * RT_WARPS + warp) * (MT * 16);   // atoms a0 + 16 mt + l4 (+ 8)
    uint32_t A[MT][KT][4];
#pragma unroll
    for (int mt = 0; mt < MT; ++mt)
#pragma unroll
        for (int hi = 0; hi < 2; ++hi) {
            const int n = a0 + 16 * mt + 8 * hi + l4;
            const uint4* src = reinterpret_cast<const uint4*>(Db + static_cast<size_t>(n < n_pad ? n : 0) * D_ + q4 * (D_ / 4));
#pragma unroll
            for (int c = 0; c < D_ / 32; ++c) {           // eight channels: two k tiles of four
                uint4 v = __ldg(src + c);
                if (n >= n_pad) v = make_uint4(0u, 0u, 0u, 0u);
                A[mt][2 * c][hi] = v.x;
                A[mt][2 * c][2 + hi] = v.y;
                A[mt][2 * c + 1][hi] = v.z;
                A[mt][2 * c + 1][2 + hi] = v.w;
            }
        }
    // ---- R_0 = x, rounded to bf16 (rows past M: zeros) ----
    for (int f = threadIdx.x; f < ROWS * (D_ / 8); f += RT_THREADS) {
        const int r = f / (D_ / 8), c = f % (D_ / 8);
        uint4 v = make_uint4(0u, 0u, 0u, 0u);
        if (m0 + r < M) {
            const int64_t o = (m0 + r) * ldx + 8 * c;
            if (x_dtype == CSR_DTYPE_BF16) {
                v = *reinterpret_cast<const uint4*>(reinterpret_cast<const uint16_t*>(X) + o);
            } else {
                float x[8];
#pragma unroll
                for (int k = 0; k < 8; ++k) x[k] = load_elem(X, x_dtype, o + k);
                v = make_uint4(pack_bf16(x[0], x[1]), pack_bf16(x[2], x[3]), pack_bf16(x[4], x[5]), pack_bf16(x[6], x[7]));
            }
        }
        *reinterpret_cast<uint4*>(&sm.R[r][4 * c]) = v;
    }
    __syncthreads();
    if (n_ctas > 1) cluster_sync_all();                   // no CTA touches a peer's barriers before they are set up

    uint32_t phases = 0;                                  // set on giving up: of this warp's row's barrier, waited out
    static_assert(ROWS <= RT_WARPS, "a warp has at most one row");
    for (int g = 0; g < s; ++g) {
        // ---- sweep ----
#pragma unroll
        for (int nt = 0; nt < NTL; ++nt) {
            float c[MT][4];
#pragma unroll
            for (int mt = 0; mt < MT; ++mt)
#pragma unroll
                for (int i = 0; i < 4; ++i) c[mt][i] = 0.f;
            const uint4* row = reinterpret_cast<const uint4*>(&sm.R[8 * nt + l4][q4 * (D_ / 8)]);
#pragma unroll
            for (int ch = 0; ch < D_ / 32; ++ch) {
                const uint4 b = row[ch];
#pragma unroll
                for (int mt = 0; mt < MT; ++mt) {
                    mma_bf16_16816(c[mt], A[mt][2 * ch], b.x, b.y);
                    mma_bf16_16816(c[mt], A[mt][2 * ch + 1], b.z, b.w);
                }
            }
            // this lane: atoms a0 + 16 mt + l4 (c0, c1) and + 8 (c2, c3) of rows 8 nt + 2 q4 (c0, c2) and + 1 (c1, c3)
            unsigned long long k0, k1;
            auto largest = [&]() {
                k0 = k1 = 0ull;
#pragma unroll
                for (int mt = 0; mt < MT; ++mt)
#pragma unroll
                    for (int hi = 0; hi < 2; ++hi) {
                        const int n = a0 + 16 * mt + 8 * hi + l4;
                        const uint32_t tag = static_cast<uint32_t>(NG - 1 - (n & (TILE_N - 1)) / G), low = 0xFFFFFFFFu - static_cast<uint32_t>(n / TILE_N);
                        const uint32_t v0 = (__float_as_uint(c[mt][2 * hi]) & 0x7FFFFFFFu & key_mask) | tag;
                        const uint32_t v1 = (__float_as_uint(c[mt][2 * hi + 1]) & 0x7FFFFFFFu & key_mask) | tag;
                        if (n < n_pad) {
                            k0 = max_u64(k0, (static_cast<unsigned long long>(v0) << 32) | low);
                            k1 = max_u64(k1, (static_cast<unsigned long long>(v1) << 32) | low);
                        }
                    }
            };
            largest();
            if constexpr (G > 1) {
                // A key above those of Inf is a NaN's, which only rows that are not finite have.  As in group_key, the NaNs
                // of a group count only where all of it is NaN.
                constexpr uint32_t kInfKey = 0x7F800000u | (NG - 1);
                if (__any_sync(0xffffffffu, max(static_cast<uint32_t>(k0 >> 32), static_cast<uint32_t>(k1 >> 32)) > kInfKey)) {
#pragma unroll
                    for (int mt = 0; mt < MT; ++mt)
#pragma unroll
                        for (int i = 0; i < 4; ++i)
#pragma unroll
                            for (int o = 4; o < 4 * G; o <<= 1)
                                c[mt][i] = fmaxf(fabsf(c[mt][i]), fabsf(__shfl_xor_sync(0xffffffffu, c[mt][i], o)));
                    largest();
                }
            }
#pragma unroll
            for (int o = 4; o < 32; o <<= 1) {
                k0 = max_u64(k0, __shfl_xor_sync(0xffffffffu, k0, o));
                k1 = max_u64(k1, __shfl_xor_sync(0xffffffffu, k1, o));
            }
            if (l4 == 0) {
                sm.best[8 * nt + 2 * q4][warp] = k0;
                sm.best[8 * nt + 2 * q4 + 1][warp] = k1;
            }
        }
        __syncthreads();
        // ---- a warp per row: merge, exchange, pick, update ----
        bool got = true;
#pragma unroll
        for (int rr = 0; rr < ROWS; rr += RT_WARPS) {     // everyone's words are on their way before any is waited for
            const int r = rr + warp;
            if (ROWS < RT_WARPS && r >= ROWS) continue;
            unsigned long long k = sm.best[r][lane & 15];
#pragma unroll
            for (int o = 1; o < 16; o <<= 1) k = max_u64(k, __shfl_xor_sync(0xffffffffu, k, o));
            if (n_ctas == 1) {
                if (lane == 0) sm.from[g & 1][r][0] = k;
            } else if (lane < n_ctas) {
                st_async_u64(map_to_cta(smem_u32(&sm.from[g & 1][r][cta]), lane), k, map_to_cta(smem_u32(&sm.bar[r]), lane));
            }
        }
        __syncwarp();
#pragma unroll
        for (int rr = 0; rr < ROWS; rr += RT_WARPS) {
            const int r = rr + warp;
            if (ROWS < RT_WARPS && r >= ROWS) continue;
            if (n_ctas > 1 && got) {
                got = wait_bounded_cluster(&sm.bar[r], g & 1, wc);
                got = __all_sync(0xffffffffu, got);
                if (got && lane == 0) mbar_expect_tx(&sm.bar[r], static_cast<uint32_t>(n_ctas) * 8);      // the next iteration's
            }
            if (!got) continue;
            unsigned long long k = lane < n_ctas ? *reinterpret_cast<volatile unsigned long long*>(&sm.from[g & 1][r][lane]) : 0ull;
#pragma unroll
            for (int o = 1; o < 16; o <<= 1) k = max_u64(k, __shfl_xor_sync(0xffffffffu, k, o));
            k = __shfl_sync(0xffffffffu, k, 0);
            const int n0 = candidate_start<G>(static_cast<uint32_t>(k >> 32), 0xFFFFFFFFu - static_cast<uint32_t>(k), N, status);
            // the arithmetic of pick_and_update: eight lanes (four times the same here) with CH chunks each
            constexpr int CH = D_ / 64, APR = D_ / 8;
            const int l8 = lane & 7;
            uint4 atom[G][CH], rv[CH];
            const uint4* src = reinterpret_cast<const uint4*>(Db + static_cast<size_t>(n0) * D_) + l8 * CH;
#pragma unroll
            for (int j = 0; j < G; ++j)
#pragma unroll
                for (int c = 0; c < CH; ++c) atom[j][c] = __ldg(src + j * APR + c);
#pragma unroll
            for (int c = 0; c < CH; ++c) rv[c] = *reinterpret_cast<const uint4*>(&sm.R[r][4 * (l8 * CH + c)]);
            float dot[G];
#pragma unroll
            for (int j = 0; j < G; ++j) {
                float ev = 0.f, od = 0.f;
#pragma unroll
                for (int c = 0; c < CH; ++c) dot8(rv[c], atom[j][c], ev, od);
                dot[j] = ev + od;
            }
#pragma unroll
            for (int o = 1; o < 8; o <<= 1)
#pragma unroll
                for (int j = 0; j < G; ++j) dot[j] += __shfl_xor_sync(0xffffffffu, dot[j], o);
            float coef = dot[0];
            int jb = 0;
#pragma unroll
            for (int j = 1; j < G; ++j)
                if (fabsf(dot[j]) > fabsf(coef)) {
                    coef = dot[j];
                    jb = j;
                }
            __syncwarp();                                  // every lane has read its part of the row
            if (lane < 8) {
#pragma unroll
                for (int c = 0; c < CH; ++c) {
                    uint4 av = atom[0][c];
#pragma unroll
                    for (int j = 1; j < G; ++j)
                        if (jb == j) av = atom[j][c];
                    *reinterpret_cast<uint4*>(&sm.R[r][4 * (l8 * CH + c)]) = axpy8(rv[c], av, coef);
                }
            }
            const int64_t m = m0 + r;
            if (cta == 0 && lane == 0 && m < M) {
                out_idx[m * ldc + g] = static_cast<uint16_t>(n0 + jb);
                if (coef_dtype == CSR_DTYPE_F16)
                    reinterpret_cast<__half*>(out_coef)[m * ldc + g] = __float2half_rn(coef);
                else
                    reinterpret_cast<float*>(out_coef)[m * ldc + g] = coef;
            }
        }
        if (__syncthreads_or(!got || sm.abort != 0)) {
            phases = g + (got ? 1 : 0);
            break;
        }
    }
    // a CTA's shared memory must outlive its peers' last writes to it, also when it has given up
    if (n_ctas > 1) {
        cluster_sync_all();
        if (sm.abort != 0 && lane == 0 && warp < ROWS) let_words_land(&sm.bar[warp], phases, static_cast<uint32_t>(n_ctas) * 8);
    }
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn get_encode_tiled() {
    static const EncodeTiledFn fn = [] {               // initialised once, also with concurrent callers
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            return reinterpret_cast<EncodeTiledFn>(p);
        return static_cast<EncodeTiledFn>(nullptr);
    }();
    return fn;
}

constexpr int kClusterLaunchRefused = 1;                  // internal: not a CSR_ERR_* code

template <int D_, int G>
void cluster_config(cudaLaunchConfig_t& cfg, cudaLaunchAttribute* attr, int cluster_ctas, int grid, size_t smem,
                    cudaStream_t stream) {
    cfg.gridDim = dim3((unsigned)grid, 1, 1);
    cfg.blockDim = dim3(NT, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)cluster_ctas;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
}

// Adds to cfg that its CTAs may come up before the kernel in front of them has ended.
void beside_previous(cudaLaunchConfig_t& cfg, cudaLaunchAttribute* attr) {
    attr[cfg.numAttrs].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[cfg.numAttrs].val.programmaticStreamSerializationAllowed = 1;
    ++cfg.numAttrs;
}

// How many clusters of `cluster_ctas` CTAs of the encoder the device holds at once (0: none,
// or clusters of that size cannot be launched here).  Asked once per size.
template <int D_, int G>
int max_clusters(int cluster_ctas) {
    static int cached_dev[64][17] = {};                // per device: 0 = not asked yet, -1 = none
    static std::mutex mu;
    int dev = 0;
    if (cluster_ctas < 2 || cluster_ctas > 16 || cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
    std::lock_guard<std::mutex> lk(mu);
    int* cached = cached_dev[dev];                     // (function attributes are per device as well)
    if (cached[cluster_ctas] == 0) {
        const size_t smem = sizeof(FastSmem<D_>) + 1024;
        int n = 0;
        bool good = cudaFuncSetAttribute(encode_fast_kernel<D_, G, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)smem) == cudaSuccess;
        if (good && cluster_ctas > 8)
            good = cudaFuncSetAttribute(encode_fast_kernel<D_, G, true>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) ==
                   cudaSuccess;
        if (good) {
            cudaLaunchConfig_t cfg = {};
            cudaLaunchAttribute attr[1];
            cluster_config<D_, G>(cfg, attr, cluster_ctas, cluster_ctas, smem, 0);
            good = cudaOccupancyMaxActiveClusters(&n, encode_fast_kernel<D_, G, true>, &cfg) == cudaSuccess;
        }
        if (!good) {
            cudaGetLastError();                        // a refusal is an answer, not a failure of the call
            n = 0;
        }
        cached[cluster_ctas] = n > 0 ? n : -1;
    }
    return cached[cluster_ctas] > 0 ? cached[cluster_ctas] : 0;
}

// Pairs of row tiles, one CTA each over the whole dictionary (n_splits = 0), or one iteration of the
// split without clusters; or, with `tile_splits` > 0, single row tiles, tile_splits CTAs each.
template <int D_, int G>
int launch(const EncodeArgs& a, const CUtensorMap& tmap, const uint16_t* Db, uint32_t* status, int n_splits, uint2* partial,
           int tile_splits = 0) {
    const size_t smem = sizeof(FastSmem<D_>) + 1024;
    auto kernel = tile_splits > 0 ? encode_fast_kernel<D_, G, true> : encode_fast_kernel<D_, G, false>;
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return fail(CSR_ERR_CUDA, "cudaFuncSetAttribute: %s", cudaGetErrorString(e));
    // keys keep the magnitude bits above the group tag; with G == 1 the key is built from the
    // raw value, so the mask clears the sign bit as well
    const uint32_t key_mask = (G == 1 ? 0x7FFFFFFFu : 0xFFFFFFFFu) & ~static_cast<uint32_t>(TILE_N / G - 1);
    // 16-byte code stores need eight codes per flush and 16-byte aligned rows in both arrays
    const uintptr_t ci = reinterpret_cast<uintptr_t>(a.out_idx), cc = reinterpret_cast<uintptr_t>(a.out_coef);
    const int vec_codes = (a.s % 8 == 0) && (a.ld_code % 8 == 0) && (ci % 16 == 0) && (cc % 16 == 0);
    const int64_t n_pairs = (a.M + 2 * TILE_M - 1) / (2 * TILE_M), n_tiles = (a.M + TILE_M - 1) / TILE_M;
    const int grid = tile_splits > 0 ? (int)(n_tiles * tile_splits)
                     : n_splits > 1  ? (int)(n_pairs * n_splits)
                                     : (int)(n_pairs < (int64_t)sm_count() ? n_pairs : (int64_t)sm_count());
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[2];
    cluster_config<D_, G>(cfg, attr, tile_splits > 1 ? tile_splits : 1, grid, smem, a.stream);
    if (tile_splits <= 1) cfg.numAttrs = 0;
    if (a.after_copy) beside_previous(cfg, attr);
    e = cudaLaunchKernelEx(&cfg, kernel, tmap, Db, a.X, a.x_dtype, a.ldx, a.M, a.N, a.s, a.out_idx, a.out_coef, a.coef_dtype,
                           a.ld_code, vec_codes, key_mask, status, tile_splits > 0 ? tile_splits : n_splits, partial,
                           options().wait_limit_ns);
    if (e != cudaSuccess && tile_splits > 1) {             // refused at launch (nothing ran): the caller takes another path
        cudaGetLastError();
        return kClusterLaunchRefused;
    }
    if (e != cudaSuccess) return fail(CSR_ERR_CUDA, "encode_fast launch: %s", cudaGetErrorString(e));
    return CSR_OK;
}

// Atoms per arg-max group.  Larger groups save arg-max arithmetic during the sweep (which
// grows with N) and cost a wider gather at the end of every sweep (which does not); the
// defaults are where the measured crossovers lie.  The option "fast_group" (1, 2, 4 or 8)
// overrides them; it is a tuning knob only: every setting picks, per row, an atom whose bf16
// correlation is the largest to within the width of the group tag.
int group_size(int d, int N) {
    const int v = options().fast_group;
    if (v == 1 || v == 2 || v == 4 || v == 8) return v;
    if (d == 64) return N <= 2048 ? 2 : 4;
    return 1;
}

// How M rows are run: `pair_rows` of them as whole waves of pairs of row tiles, one CTA per pair, then up
// to two launches of single row tiles with splits[k] CTAs per tile.  A pair shares each dictionary
// stage between its two tiles and is the cheapest way to fill the chip; single tiles spread what
// does not.  The estimates are fits of this kernel's measured time per iteration in us (M from 64 to
// 28000, N from 512 to 16384, s = 8): pairs 3.3 + 1.55 per 256-atom tile of the dictionary (d = 64: 3.0
// + 1.05), single tiles 4.1 + 0.75 per tile of the CTA's slice (d = 64: 3.2 + 0.48).  Some of it, in us
// a call of 8 iterations at N = 1024 / 8192, d = 128, this plan against clusters of up to 16 CTAs
// on pairs of row tiles: 64 rows 35 / 45 against 47 / 45; 1100 rows 37 / 58 against 54 / 74; 4160 rows
// 40 / 83 against 56 / 140; 9400 rows 45 / 131 against 68 / 233; 18900 rows 54 / 227 against 70 / 237.
// Problems side by side (a grouped call) share the chip: a plan that gives each all of it has their
// clusters wait for one another.  Measured in us, two / four problems, d = 128, s = 16, planned for the whole
// chip against for their share of it: 128 rows N = 4096 96 / 143 against 83 / 86; 1024 rows N = 1024 95 / 187
// against 74 / 85, N = 8192 214 / 321 against 155 / 161; 9472 rows N = 1024 167 / 327 against 102 / 156.
struct RowPlan {
    int64_t pair_rows;
    int64_t tile_rows[2];
    int splits[2];
    float us;                // an iteration of what follows the whole waves
};
// Rounds in which the GPU gets through n units of a call, `cap` at a time, with `load` times as many rows in flight.
int64_t rounds_of(int64_t n, int64_t cap, float load) {
    return (static_cast<int64_t>(ceilf(static_cast<float>(n) * load - 1e-3f)) + cap - 1) / cap;
}
template <int D_, int G>
RowPlan plan_rows(int64_t M, int N, float load) {
    const int T = (N + TILE_N - 1) / TILE_N;
    const int64_t sms = sm_count(), wave = sms * 2 * TILE_M;
    const int64_t rest = M % wave, tiles = (rest + TILE_M - 1) / TILE_M;
    constexpr float kPair0 = D_ == 128 ? 3.3f : 3.0f, kPair1 = D_ == 128 ? 1.55f : 1.05f;
    constexpr float kTile0 = D_ == 128 ? 4.1f : 3.2f, kTile1 = D_ == 128 ? 0.75f : 0.48f;
    constexpr int kMost = FastSmem<D_>::kATileBytes / (2 * TILE_M * 8);       // the exchange buffers bound the cluster
    // n row tiles in one launch: the best number of CTAs per tile
    auto best_split = [&](int64_t n, float* cost) {
        int best = 1;
        *cost = (float)rounds_of(n, sms, load) * (kTile0 + kTile1 * T);
        for (int ns = 2; ns <= kMost && ns <= T; ns *= 2) {
            const int nc = max_clusters<D_, G>(ns);
            if (nc < 1) continue;
            const float c = (float)rounds_of(n, nc, load) * (kTile0 + kTile1 * ((T + ns - 1) / ns));
            if (c < *cost) {
                *cost = c;
                best = ns;
            }
        }
        return best;
    };
    RowPlan p{M, {0, 0}, {0, 0}, 0.f};
    if (tiles == 0) return p;
    float least = (float)rounds_of((tiles + 1) / 2, sms, load) * (kPair0 + kPair1 * T), cost;
    p.us = least;
    const int one = best_split(tiles, &cost);
    if (cost < least) {
        least = cost;
        p = RowPlan{M - rest, {rest, 0}, {one, 0}, cost};
    }
    if (tiles > sms) {                                     // a whole wave of single tiles, then the others over the whole chip
        const int two = best_split(tiles - sms, &cost);
        cost += (float)rounds_of(sms, sms, load) * (kTile0 + kTile1 * T);
        if (cost < least) p = RowPlan{M - rest, {sms * TILE_M, rest - sms * TILE_M}, {1, two}, cost};
    }
    return p;
}

// A handful of rows (see encode_few_kernel): atoms a CTA holds, and how many CTAs the dictionary takes
// (0: it does not fit).
template <int D_>
int few_ctas(int N) {
    constexpr int kAtoms = RT_WARPS * 16 * (D_ == 128 ? 2 : 4);
    int n = 1;
    while (n <= 16 && n * kAtoms < (N + 7) / 8 * 8) n *= 2;
    return n <= 16 ? n : 0;
}
// Rows per cluster of encode_few_kernel, 8 or 16 (0: row tiles are faster).  Measured, s = 16, in us, this
// kernel with 8 rows / 16 rows per cluster against row tiles: 8 rows N = 1000 33 / 33 / 57, N = 8192 35 / 49 /
// 78; 64 rows N = 8192 (8 clusters of 16, more than the chip holds at once) 68 / 49 / 84; 128 rows
// N = 1000 33 / 47 / 68.  Per iteration 2.2 us (8 rows) and 3.05 (16 rows) a round of clusters, at d = 64 (a
// warp holds twice the atoms, half the channels) as at d = 128: 8 rows N = 1000 35 / 51 / 51, 512 rows
// N = 1000 35 / 51 / 57, 128 rows N = 4096 43 / 59 / 76, 512 rows N = 4096 80 / 61 / 76, 128 rows N = 8192
// 80 / 60 / 90, 256 rows N = 8192 117 / 115 / 92 (d = 64, cold caches).
template <int D_, int G>
int few_rows_per_cluster(int64_t M, int N, float load) {
    const int n_ctas = few_ctas<D_>(N);
    if (n_ctas == 0 || M > 4096) return 0;
    const int fit = n_ctas == 1 ? sm_count() : max_clusters<D_, G>(n_ctas);
    if (fit < 1) return 0;
    auto rounds = [&](int rows) { return (float)rounds_of((M + rows - 1) / rows, fit, load); };
    const float c8 = 2.2f * rounds(8), c16 = 3.05f * rounds(16), few = c8 <= c16 ? c8 : c16;
    if (few >= plan_rows<D_, G>(M, N, load).us) return 0;
    return c8 <= c16 ? 8 : 16;
}

template <int D_, int G, int NTL>
int launch_few(const EncodeArgs& a, const uint16_t* Db, uint32_t* status) {
    auto kernel = encode_few_kernel<D_, G, NTL>;
    const int n_ctas = few_ctas<D_>(a.N);
    cudaError_t e = n_ctas > 8 ? cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) : cudaSuccess;
    if (e == cudaSuccess) {
        const uint32_t key_mask = ~static_cast<uint32_t>(TILE_N / G - 1);
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute attr[2];
        cluster_config<D_, G>(cfg, attr, n_ctas, (int)((a.M + 8 * NTL - 1) / (8 * NTL)) * n_ctas, 0, a.stream);
        cfg.blockDim = dim3(RT_THREADS, 1, 1);
        if (n_ctas == 1) cfg.numAttrs = 0;
        if (a.after_copy) beside_previous(cfg, attr);
        e = cudaLaunchKernelEx(&cfg, kernel, Db, a.X, a.x_dtype, a.ldx, a.M, a.N, a.s, a.out_idx, a.out_coef, a.coef_dtype, a.ld_code,
                               key_mask, status, n_ctas, options().wait_limit_ns);
    }
    if (e != cudaSuccess) {                                // refused at launch (nothing ran): the caller takes another path
        cudaGetLastError();
        return kClusterLaunchRefused;
    }
    return CSR_OK;
}

template <int D_, int G>
int launch_planned(const EncodeArgs& a, const CUtensorMap& tmap, const uint16_t* Db, uint32_t* status) {
    if (options().fast_split == 0) {
        const int rows = few_rows_per_cluster<D_, G>(a.M, a.N, a.load);
        if (rows > 0) {
            const int rc = rows == 8 ? launch_few<D_, G, 1>(a, Db, status) : launch_few<D_, G, 2>(a, Db, status);
            if (rc != kClusterLaunchRefused) return rc;
        }
    }
    // (the option forces pairs only)
    const RowPlan p = options().fast_split == 0 ? plan_rows<D_, G>(a.M, a.N, a.load) : RowPlan{a.M, {0, 0}, {0, 0}, 0.f};
    auto rows_from = [&](int64_t r0, int64_t m) {
        EncodeArgs b = a;
        b.after_copy = a.after_copy && r0 == 0;            // (the launches after the first follow an encoder)
        b.X = static_cast<const char*>(a.X) + (size_t)r0 * a.ldx * dtype_size(a.x_dtype);
        b.out_idx = a.out_idx + r0 * a.ld_code;
        b.out_coef = static_cast<char*>(a.out_coef) + (size_t)r0 * a.ld_code * (a.coef_dtype == CSR_DTYPE_F16 ? 2 : 4);
        b.M = m;
        return b;
    };
    if (p.pair_rows)
        if (int rc = launch<D_, G>(rows_from(0, p.pair_rows), tmap, Db, status, 0, nullptr)) return rc;
    int64_t r0 = p.pair_rows;
    for (int k = 0; k < 2; ++k) {
        if (p.tile_rows[k] == 0) continue;
        const EncodeArgs b = rows_from(r0, p.tile_rows[k]);
        int rc = launch<D_, G>(b, tmap, Db, status, 0, nullptr, p.splits[k]);
        if (rc == kClusterLaunchRefused) rc = launch<D_, G>(b, tmap, Db, status, 0, nullptr, 1);
        if (rc != CSR_OK) return rc;
        r0 += p.tile_rows[k];
    }
    return CSR_OK;
}

template <int D_>
int launch_d(const EncodeArgs& a, const CUtensorMap& tmap, const uint16_t* Db, uint32_t* status) {
    switch (group_size(D_, a.N)) {
        case 1: return launch_planned<D_, 1>(a, tmap, Db, status);
        case 2: return launch_planned<D_, 2>(a, tmap, Db, status);
        case 8: return launch_planned<D_, 8>(a, tmap, Db, status);
        default: return launch_planned<D_, 4>(a, tmap, Db, status);
    }
}

// Without clusters: how many CTAs share a pair of row tiles (1 = the whole dictionary per CTA).
int split_count(int64_t M, int N) {
    const int64_t n_pairs = (M + 2 * TILE_M - 1) / (2 * TILE_M);
    const int T = (N + TILE_N - 1) / TILE_N;
    if (n_pairs < 1 || n_pairs * 2 > sm_count() || T < 2) return 1;
    int ns = (int)(sm_count() / n_pairs);
    if (ns > T) ns = T;
    if (ns > 32) ns = 32;
    // Worth it only if an iteration's sweep over all T tiles by one CTA (about 1.55 us per
    // tile, measured) outlasts two launches (about 12 us) plus the sweep of a slice.
    const float whole = 1.55f * T, sliced = 12.f + 1.6f * ((T + ns - 1) / ns);
    return whole > 1.2f * sliced ? ns : 1;
}
size_t align256(size_t x) { return (x + 255) / 256 * 256; }

// One launch of the sweep (every CTA a slice of the dictionary, s = 1) and one of the pick
// per iteration; the residual rows live in global memory as bf16 in between.
template <int D_, int G>
int run_split_g(const EncodeArgs& a, const CUtensorMap& tmap, const uint16_t* Db, uint32_t* status, void* scratch) {
    const int ns = split_count(a.M, a.N);
    uint4* Rb = static_cast<uint4*>(scratch);
    uint2* partial = reinterpret_cast<uint2*>(static_cast<char*>(scratch) + align256((size_t)a.M * D_ * 2));
    const int64_t chunks = a.M * (D_ / 8);
    rows_to_bf16_kernel<D_><<<(unsigned)((chunks + 255) / 256), 256, 0, a.stream>>>(a.X, a.x_dtype, a.ldx, a.M, Rb);
    EncodeArgs b = a;
    b.after_copy = false;
    b.X = Rb;
    b.x_dtype = CSR_DTYPE_BF16;
    b.ldx = D_;
    b.s = 1;
    const unsigned pick_blocks = (unsigned)((a.M + 15) / 16);
    for (int g = 0; g < a.s; ++g) {
        if (int rc = launch<D_, G>(b, tmap, Db, status, ns, partial)) return rc;
        split_pick_kernel<D_, G><<<pick_blocks, 128, 0, a.stream>>>(Db, a.N, Rb, partial, ns, a.M, g, g + 1 < a.s, a.out_idx, a.out_coef,
                                                                a.coef_dtype, a.ld_code);
    }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return fail(CSR_ERR_CUDA, "encode_fast split launch: %s", cudaGetErrorString(e));
    return CSR_OK;
}

template <int D_>
int run_split(const EncodeArgs& a, const CUtensorMap& tmap, const uint16_t* Db, uint32_t* status, void* scratch) {
    switch (group_size(D_, a.N)) {
        case 1: return run_split_g<D_, 1>(a, tmap, Db, status, scratch);
        case 2: return run_split_g<D_, 2>(a, tmap, Db, status, scratch);
        case 8: return run_split_g<D_, 8>(a, tmap, Db, status, scratch);
        default: return run_split_g<D_, 4>(a, tmap, Db, status, scratch);
    }
}

}  // namespace

bool encode_fast_split_applies(int64_t M, int N) { return M > 0 && split_count(M, N) > 1; }
size_t encode_fast_split_scratch_bytes(int64_t M, int d, int N) {
    return align256((size_t)M * d * 2) + align256((size_t)M * split_count(M, N) * sizeof(uint2));
}

// The bf16 copy holds N rounded up to a multiple of 8 atoms; the extra rows are zero, so a
// group of up to 8 candidate atoms never reaches past the copy.
static int padded_atoms(int N) { return (N + 7) / 8 * 8; }
size_t encode_fast_workspace_bytes(int d, int N) { return (size_t)padded_atoms(N) * (size_t)d * 2; }

int prepare_fast_dictionary(const float* D, int N, int d, void* workspace, cudaStream_t stream) {
    if ((reinterpret_cast<uintptr_t>(workspace) & 1023u) != 0)
        return fail(CSR_ERR_ALIGNMENT, "internal: dictionary scratch not 1024-byte aligned");
    const int64_t n_vec4 = (int64_t)N * d / 4, n_padded = (int64_t)padded_atoms(N) * d / 4;
    int blocks = (int)((n_padded + 255) / 256);
    if (blocks > 4 * sm_count()) blocks = 4 * sm_count();
    dict_to_bf16_kernel<<<blocks, 256, 0, stream>>>(reinterpret_cast<const float4*>(D), reinterpret_cast<uint2*>(workspace), n_vec4,
                                                    n_padded);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return fail(CSR_ERR_CUDA, "dict_to_bf16 launch: %s", cudaGetErrorString(e));
    return CSR_OK;
}

// Has the runtime load the code of every kernel that a call of any number of rows may launch for this d and
// N (it loads a kernel when that is first asked for, and its code takes device memory).
template <int D_>
static int load_kernels(int G) {
    auto load = [](auto... kernels) {
        cudaFuncAttributes at;
        cudaError_t e = cudaFuncGetAttributes(&at, dict_to_bf16_kernel);
        for (const void* k : {reinterpret_cast<const void*>(kernels)...})
            if (e == cudaSuccess) e = cudaFuncGetAttributes(&at, k);
        return e;
    };
    auto of = [&](auto g) {
        constexpr int g_ = decltype(g)::value;
        return load(encode_fast_kernel<D_, g_, false>, encode_fast_kernel<D_, g_, true>, encode_few_kernel<D_, g_, 1>,
                    encode_few_kernel<D_, g_, 2>);
    };
    using std::integral_constant;
    const cudaError_t e = G == 1   ? of(integral_constant<int, 1>{})
                          : G == 2 ? of(integral_constant<int, 2>{})
                          : G == 8 ? of(integral_constant<int, 8>{})
                                   : of(integral_constant<int, 4>{});
    return e == cudaSuccess ? CSR_OK : fail(CSR_ERR_CUDA, "loading the encoder's kernels: %s", cudaGetErrorString(e));
}
int load_fast_kernels(int d, int N) {
    static std::atomic<uint32_t> loaded[64];              // per device, a bit for each d and group size
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess || dev < 0 || dev >= 64) return fail(CSR_ERR_CUDA, "cudaGetDevice: %s", cudaGetErrorString(e));
    const int G = group_size(d, N);
    const uint32_t bit = static_cast<uint32_t>(G) << (d == 128 ? 8 : 0);
    if (loaded[dev].load() & bit) return CSR_OK;
    if (int rc = d == 128 ? load_kernels<128>(G) : load_kernels<64>(G)) return rc;
    loaded[dev].fetch_or(bit);
    return CSR_OK;
}

int launch_encode_fast(const EncodeArgs& a, void* workspace, uint32_t* status) {
    if (a.M == 0) return CSR_OK;
    if (int rc = prepare_fast_dictionary(a.D, a.N, a.d, workspace, a.stream)) return rc;
    EncodeArgs b = a;
    b.after_copy = true;
    return launch_encode_fast_prepared(b, workspace, status, nullptr);
}

int launch_encode_fast_prepared(const EncodeArgs& a, const void* dict_bf16, uint32_t* status, void* split_scratch) {
    if (a.M == 0) return CSR_OK;
    void* workspace = const_cast<void*>(dict_bf16);
    if ((reinterpret_cast<uintptr_t>(workspace) & 1023u) != 0)
        return fail(CSR_ERR_ALIGNMENT, "internal: dictionary scratch not 1024-byte aligned");
    EncodeTiledFn encode = get_encode_tiled();
    if (!encode) return fail(CSR_ERR_CUDA, "cuTensorMapEncodeTiled is not available from the driver");
    const int n_pad = padded_atoms(a.N);

    // rows past the padded copy (the rest of the last 256-atom tile) are filled with zeros by TMA
    CUtensorMap tmap;
    const cuuint64_t gdim[2] = {(cuuint64_t)a.d, (cuuint64_t)n_pad};
    const cuuint64_t gstride[1] = {(cuuint64_t)a.d * 2};
    const cuuint32_t box[2] = {64, (cuuint32_t)TILE_N};
    const cuuint32_t estr[2] = {1, 1};
    CUresult r = encode(&tmap, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, workspace, gdim, gstride, box, estr,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return fail(CSR_ERR_CUDA, "cuTensorMapEncodeTiled failed with code %d", (int)r);

    const uint16_t* Db = static_cast<const uint16_t*>(workspace);
    // no clusters wanted: with scratch, a sweep launch and a pick launch per iteration
    if (split_scratch) {
        if (a.d == 128) return run_split<128>(a, tmap, Db, status, split_scratch);
        return run_split<64>(a, tmap, Db, status, split_scratch);
    }
    if (a.d == 128) return launch_d<128>(a, tmap, Db, status);
    return launch_d<64>(a, tmap, Db, status);
}

}  // namespace csr
