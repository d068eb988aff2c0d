// Attention straight from the codes ("De-Sparse to restore": the restored tensor
// X~ = D r of Eq. 12 "will be used in the attention score calculation").  Because X~ is
// linear in the atoms, neither product needs X~ in memory:
//
//   scores[t] = scale * q . x~_t   = sum_g coef[t][g] * p[idx[t][g]],    p = scale * D q
//   out       = sum_t w[t] * x~_t  = sum_n a[n] * D[n][:],               a[n] = sum_{(t,g): idx[t][g] = n} w[t] coef[t][g]
//
// HBM traffic per token is the 4*s bytes of its code (plus 4 bytes per query head of score
// or weight) instead of the 2*d bytes of a restored bf16 row written and read again.
//
// Four launches and a small sum:
//   qd_kernel          p for all B*H query heads, fp32, channels summed in ascending order, written as
//                      [b][group of HG heads][atom][HG];
//   key_scores_kernel  CTAs take contiguous ranges of (stream, head group, chunk of tokens), keep the
//                      group's p in shared memory and stream the codes, one thread per token, the s
//                      terms summed in stored order.  Inside csr_decode_attention it also leaves the
//                      softmax statistics (running maximum and sum of exponentials) of its part of
//                      each row, and the largest l1-norm of a token's value coefficients per chunk;
//   value_scatter_kernel  units of (stream, head group, piece of the tokens): scatters w * coef into
//                      a[head][N] in shared memory with integer atomics and stores the table.  Inside
//                      csr_decode_attention it turns the scores into weights on the way (in place);
//   ad_kernel          out = a D in fp32, the pieces summed in order on the way in, the atoms cut into
//                      slices; add_slices_kernel adds the slices' results in a fixed order.
// Measured (64 streams x 16384 tokens, 4 heads each, s = 16, N = 8192, d = 128; each kernel alone with
// cold caches): 21 / 40 / 53 / 21 / 5 us, together 134 us with the launches overlapped; as six launches
// with the softmax a kernel of its own, the bounds of the scatter a pass over the codes and four
// times the slices, 24 / 35 + 12 / 64 / 29 / 13 us, 166 us.  8 streams x 4099 tokens: 36 us, was 70.
// What bounds them: fp32 FMAs and operand loads (qd, ad), shared-memory gathers at about 16 cycles per
// 16-byte warp access (scores), shared-memory atomics at 17.5 per ns and SM (scatter).
// Every floating-point sum is taken in a fixed order and the tables are accumulated in fixed point,
// so the result is the same bits on every run.
#include <type_traits>

#include "common.cuh"

namespace csr {
namespace {

constexpr int NT = 256;
// Threads of the code-streaming kernels = tokens of a chunk.  (1024 leave 64 registers a thread: the codes
// fetched ahead went to local memory and, the table having most of the L1, to the L2: 77 instead of
// 40 us for the scores of 64 streams x 16384 tokens x 4 heads.)
constexpr int NTHR = 512;
// CTAs per SM that their registers allow
template <int HGP>
__host__ __device__ constexpr int ctas_per_sm() {
    return HGP <= 2 ? 2 : 1;
}
// Where a row's running maximum starts: finite, so that exp(score - maximum) adds nothing for a score of -Inf and
// NaN for one of NaN (from -Inf on, fmaxf and the difference would lose a NaN that came first).
constexpr float kLowest = -3.402823466e38f;

__device__ __forceinline__ float load_coef(const void* coef, int coef_dtype, int64_t off) {
    return coef_dtype == CSR_DTYPE_F16 ? __half2float(reinterpret_cast<const __half*>(coef)[off])
                                       : reinterpret_cast<const float*>(coef)[off];
}
__device__ __forceinline__ void cp_async16(void* smem, const void* gmem, bool in) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(static_cast<uint32_t>(__cvta_generic_to_shared(smem))), "l"(gmem),
                 "r"(in ? 16 : 0)
                 : "memory");
}
// The kernels of one call are launched with programmatic stream serialization: the next one's CTAs come up
// as soon as every CTA of this one has said so, do what does not depend on it (codes, atoms and
// queries were there before the first of them started) and wait for its end here.
__device__ __forceinline__ void next_may_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void wait_for_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// ---- P[b][h / HG][n][h % HG] = scale * Q[r][:] . D[n][:]  (r = b*H + h) ---------------------
// CTA = RT rows x AT atoms, all channels staged at once: the loads of a CTA are one memory latency
// (a tile staged eight channels at a time took sixteen).  Thread = RT / 16 rows x AT / 16 atoms;
// both operands lie row by row, 4 words apart beyond a multiple of 32 banks, and are read four
// channels per load.  Bound by fp32 FMA issue from about 256 rows on, by latency below.
template <int D_, int RT, int AT>
__global__ void __launch_bounds__(NT)
qd_kernel(const float* __restrict__ D, int N, const void* __restrict__ Q, int q_dtype, int R, int H, int HG, float scale,
          float* __restrict__ P, uint32_t* __restrict__ zero, int n_zero) {
    constexpr int LD = D_ + 4, RPT = RT / 16, APT = AT / 16;
    extern __shared__ __align__(16) float qd_smem[];
    float* As = qd_smem;                                  // [RT][LD]
    float* Bs = qd_smem + RT * LD;                        // [AT][LD]
    const int r0 = blockIdx.y * RT, n0 = blockIdx.x * AT;
    for (int i = (blockIdx.y * gridDim.x + blockIdx.x) * NT + threadIdx.x; i < n_zero; i += gridDim.x * gridDim.y * NT) zero[i] = 0u;
    next_may_start();
    // two halves of the channels, the second on its way while the first is multiplied
    constexpr int HC = D_ / 8;                            // float4 per row and half
#pragma unroll
    for (int half = 0; half < 2; ++half) {
#pragma unroll
        for (int f = threadIdx.x; f < AT * HC; f += NT) {
            const int n = f / HC, c = half * HC + f % HC;
            const bool in = n0 + n < N;
            cp_async16(Bs + n * LD + 4 * c, D + (int64_t)(in ? n0 + n : 0) * D_ + 4 * c, in);
        }
        cp_async_commit();
    }
#pragma unroll
    for (int f = threadIdx.x; f < RT * (D_ / 4); f += NT) {
        const int r = f / (D_ / 4), c = f % (D_ / 4);
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (r0 + r < R) {
            const int64_t off = (int64_t)(r0 + r) * D_ + 4 * c;
            if (q_dtype == CSR_DTYPE_F32) {
                v = *reinterpret_cast<const float4*>(static_cast<const float*>(Q) + off);
            } else {
                const uint2 w = *reinterpret_cast<const uint2*>(static_cast<const uint16_t*>(Q) + off);
                if (q_dtype == CSR_DTYPE_BF16) {
                    v = make_float4(__uint_as_float(w.x << 16), __uint_as_float(w.x & 0xFFFF0000u), __uint_as_float(w.y << 16),
                                    __uint_as_float(w.y & 0xFFFF0000u));
                } else {
                    const float2 a = __half22float2(*reinterpret_cast<const __half2*>(&w.x));
                    const float2 b = __half22float2(*reinterpret_cast<const __half2*>(&w.y));
                    v = make_float4(a.x, a.y, b.x, b.y);
                }
            }
        }
        *reinterpret_cast<float4*>(As + r * LD + 4 * c) = v;
    }
    cp_async_wait<1>();
    __syncthreads();
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    float acc[RPT][APT];
#pragma unroll
    for (int i = 0; i < RPT; ++i)
#pragma unroll
        for (int j = 0; j < APT; ++j) acc[i][j] = 0.f;
#pragma unroll 4
    for (int k = 0; k < D_; k += 4) {
        if (k == D_ / 2) {
            cp_async_wait<0>();
            __syncthreads();
        }
        float4 a[RPT], b[APT];
#pragma unroll
        for (int i = 0; i < RPT; ++i) a[i] = *reinterpret_cast<const float4*>(As + (ty * RPT + i) * LD + k);
#pragma unroll
        for (int j = 0; j < APT; ++j) b[j] = *reinterpret_cast<const float4*>(Bs + (tx + 16 * j) * LD + k);
#pragma unroll
        for (int i = 0; i < RPT; ++i)
#pragma unroll
            for (int j = 0; j < APT; ++j) {
                acc[i][j] = fmaf(a[i].x, b[j].x, acc[i][j]);
                acc[i][j] = fmaf(a[i].y, b[j].y, acc[i][j]);
                acc[i][j] = fmaf(a[i].z, b[j].z, acc[i][j]);
                acc[i][j] = fmaf(a[i].w, b[j].w, acc[i][j]);
            }
    }
    const int groups = (H + HG - 1) / HG;
    const int rr = r0 + ty * RPT;
    const bool whole = HG % RPT == 0 && H % HG == 0 && rr + RPT <= R;   // this thread's rows lie side by side in one group
#pragma unroll
    for (int j = 0; j < APT; ++j) {
        const int n = n0 + tx + 16 * j;
        if (n >= N) continue;
        if (whole) {
            const int b = rr / H, h = rr % H;
            float* dst = P + (((int64_t)b * groups + h / HG) * N + n) * HG + h % HG;
            if constexpr (RPT == 4)
                *reinterpret_cast<float4*>(dst) = make_float4(scale * acc[0][j], scale * acc[1][j], scale * acc[2][j], scale * acc[3][j]);
            else
                *reinterpret_cast<float2*>(dst) = make_float2(scale * acc[0][j], scale * acc[1][j]);
        } else {
#pragma unroll
            for (int i = 0; i < RPT; ++i) {
                const int r = rr + i;
                if (r < R) P[(((int64_t)(r / H) * groups + r % H / HG) * N + n) * HG + r % H % HG] = scale * acc[i][j];
            }
        }
    }
}

// ---- part[slice][r][:] = sum_{n in slice} (sum_pieces A[b][group][piece][h][n]) * D[n][:] ------
// CTA = RT rows x all channels x one slice of the atoms, 64 atoms at a time; thread = RT / 16 rows x
// D_ / 16 channels.  A tile's loads (D by cp.async, the first two pieces of A into registers) are issued
// before the tile before it is multiplied.  Both operands are read as float4 (four atoms of a row of
// A, four channels of an atom).
constexpr int OA = 64;    // atoms per tile
template <int D_, int RT>
constexpr size_t ad_smem_bytes() {
    return 2 * (RT * (OA + 4) + OA * (D_ + 4)) * sizeof(float);
}
template <int D_, int RT>
__global__ void __launch_bounds__(NT)
ad_kernel(const float* __restrict__ D, int N, const float* A, int R, int H, int HG, int pieces, int atoms_per_slice,
          float* __restrict__ part) {
    extern __shared__ __align__(16) float ad_smem[];
    constexpr int LDA = OA + 4, LDB = D_ + 4;
    float* As = ad_smem;                                  // [2][RT][LDA]
    float* Bs = ad_smem + 2 * RT * LDA;                   // [2][OA][LDB]
    constexpr int RPT = RT / 16, CPT = D_ / 16;           // rows, channels per thread
    constexpr int AV = RT * OA / 4 / NT;                  // float4 of A per thread per tile
    const int tid = threadIdx.x;
    const int tx = tid & 15, ty = tid >> 4;
    const int r0 = blockIdx.y * RT;
    const int nb = blockIdx.x * atoms_per_slice;
    const int ne = min(nb + atoms_per_slice, N);
    const int groups = (H + HG - 1) / HG;
    const int64_t piece_stride = (int64_t)HG * N;
    const bool vec_a = (N % 4) == 0;                       // rows of A start on 16-byte boundaries
    // this thread's rows of A: rows tid / 16 + 16 u of the block, atoms 4 (tid % 16) .. of a tile
    const int a_col = 4 * (tid % (OA / 4));
    const float* src[AV];
#pragma unroll
    for (int u = 0; u < AV; ++u) {
        const int r = r0 + tid / (OA / 4) + u * (NT / (OA / 4));
        src[u] = r < R ? A + (((int64_t)(r / H) * groups + r % H / HG) * pieces * HG + r % H % HG) * N + a_col : nullptr;
    }
    const auto load_a = [&](int u, int pc, int n0) {
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        const int n = n0 + a_col;
        if (!src[u] || n >= ne) return v;
        const float* p = src[u] + pc * piece_stride + n0;
        if (vec_a && n + 3 < ne) return *reinterpret_cast<const float4*>(p);
        v.x = p[0];
        if (n + 1 < ne) v.y = p[1];
        if (n + 2 < ne) v.z = p[2];
        if (n + 3 < ne) v.w = p[3];
        return v;
    };
    const auto load_d = [&](int n0, int buf) {
#pragma unroll
        for (int f = tid; f < OA * D_ / 4; f += NT) {
            const int n = f / (D_ / 4), c = f % (D_ / 4);
            const bool in = n0 + n < ne;
            cp_async16(Bs + (buf * OA + n) * LDB + 4 * c, D + (int64_t)(in ? n0 + n : 0) * D_ + 4 * c, in);
        }
        cp_async_commit();
    };
    float4 p0[AV], p1[AV];
    const auto load_pieces = [&](int n0) {
#pragma unroll
        for (int u = 0; u < AV; ++u) {
            p0[u] = load_a(u, 0, n0);
            p1[u] = pieces > 1 ? load_a(u, 1, n0) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
    };
    float acc[RPT][CPT];
#pragma unroll
    for (int i = 0; i < RPT; ++i)
#pragma unroll
        for (int j = 0; j < CPT; ++j) acc[i][j] = 0.f;
    next_may_start();
    load_d(nb, 0);
    wait_for_previous();                                  // the tables
    load_pieces(nb);
    int buf = 0;
    for (int n0 = nb; n0 < ne; n0 += OA, buf ^= 1) {
        const auto add = [](float4& a, const float4& v) {
            a.x += v.x;
            a.y += v.y;
            a.z += v.z;
            a.w += v.w;
        };
#pragma unroll
        for (int u = 0; u < AV; ++u) add(p0[u], p1[u]);
#pragma unroll 4
        for (int pc = 2; pc < pieces; ++pc)
#pragma unroll
            for (int u = 0; u < AV; ++u) add(p0[u], load_a(u, pc, n0));
#pragma unroll
        for (int u = 0; u < AV; ++u)
            *reinterpret_cast<float4*>(As + (buf * RT + tid / (OA / 4) + u * (NT / (OA / 4))) * LDA + a_col) = p0[u];
        cp_async_wait<0>();
        __syncthreads();                                   // (also: the buffers of the tile before the last are free)
        if (n0 + OA < ne) {
            load_d(n0 + OA, buf ^ 1);
            load_pieces(n0 + OA);
        }
        const float* At = As + buf * RT * LDA;
        const float* Bt = Bs + buf * OA * LDB;
#pragma unroll 4
        for (int k = 0; k < OA; k += 4) {
            float4 a[RPT];
#pragma unroll
            for (int i = 0; i < RPT; ++i) a[i] = *reinterpret_cast<const float4*>(At + (ty * RPT + i) * LDA + k);
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) {
                float b[CPT];
#pragma unroll
                for (int q = 0; q < CPT / 4; ++q) {
                    const float4 b4 = *reinterpret_cast<const float4*>(Bt + (k + kk) * LDB + q * 64 + tx * 4);
                    b[4 * q + 0] = b4.x;
                    b[4 * q + 1] = b4.y;
                    b[4 * q + 2] = b4.z;
                    b[4 * q + 3] = b4.w;
                }
#pragma unroll
                for (int i = 0; i < RPT; ++i) {
                    const float x = kk == 0 ? a[i].x : kk == 1 ? a[i].y : kk == 2 ? a[i].z : a[i].w;
#pragma unroll
                    for (int j = 0; j < CPT; ++j) acc[i][j] = fmaf(x, b[j], acc[i][j]);
                }
            }
        }
    }
#pragma unroll
    for (int i = 0; i < RPT; ++i) {
        const int r = r0 + ty * RPT + i;
        if (r >= R) continue;
        float* dst = part + ((int64_t)blockIdx.x * R + r) * D_;
#pragma unroll
        for (int q = 0; q < CPT / 4; ++q)
            *reinterpret_cast<float4*>(dst + q * 64 + tx * 4) =
                make_float4(acc[i][4 * q + 0], acc[i][4 * q + 1], acc[i][4 * q + 2], acc[i][4 * q + 3]);
    }
}

// out = part[0] + part[1] + ...: eight threads per four outputs take every eighth slice each, ascending,
// and their sums are added in order.  (One thread per output and all slices after one another
// was a chain of L2 latencies: 12 us for 128 slices.)
constexpr int SUM_X = 32, SUM_Y = 8;
__global__ void __launch_bounds__(SUM_X * SUM_Y)
add_slices_kernel(const float4* part, int slices, int64_t n4, float4* __restrict__ out) {
    __shared__ float4 sum[SUM_Y][SUM_X];
    const int x = threadIdx.x % SUM_X, y = threadIdx.x / SUM_X;
    const int64_t j = (int64_t)blockIdx.x * SUM_X + x;
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    wait_for_previous();
    if (j < n4) {
#pragma unroll 8
        for (int sl = y; sl < slices; sl += SUM_Y) {
            const float4 p = part[(int64_t)sl * n4 + j];
            v.x += p.x;
            v.y += p.y;
            v.z += p.z;
            v.w += p.w;
        }
    }
    sum[y][x] = v;
    __syncthreads();
    if (y == 0 && j < n4) {
#pragma unroll
        for (int q = 1; q < SUM_Y; ++q) {
            const float4 p = sum[q][x];
            v.x += p.x;
            v.y += p.y;
            v.z += p.z;
            v.w += p.w;
        }
        out[j] = v;
    }
}

// Eight consecutive codes of one token (16-byte loads; the caller guarantees s % 8 == 0 and
// 16-byte aligned arrays, so every block of eight starts on a 16-byte boundary).
__device__ __forceinline__ void load_coefs8(const void* coef, int coef_dtype, int64_t off, float (&c)[8]) {
    if (coef_dtype == CSR_DTYPE_F16) {
        const uint4 cv = *reinterpret_cast<const uint4*>(reinterpret_cast<const __half*>(coef) + off);
        const __half2* h = reinterpret_cast<const __half2*>(&cv);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float2 f = __half22float2(h[j]);
            c[2 * j] = f.x;
            c[2 * j + 1] = f.y;
        }
    } else {
        const float4 a = *reinterpret_cast<const float4*>(reinterpret_cast<const float*>(coef) + off);
        const float4 b = *reinterpret_cast<const float4*>(reinterpret_cast<const float*>(coef) + off + 4);
        c[0] = a.x; c[1] = a.y; c[2] = a.z; c[3] = a.w; c[4] = b.x; c[5] = b.y; c[6] = b.z; c[7] = b.w;
    }
}
__device__ __forceinline__ void load_codes8(const uint16_t* idx, const void* coef, int coef_dtype, int64_t off, int (&i)[8],
                                            float (&c)[8]) {
    const uint4 iv = *reinterpret_cast<const uint4*>(idx + off);
    i[0] = iv.x & 0xFFFF; i[1] = iv.x >> 16; i[2] = iv.y & 0xFFFF; i[3] = iv.y >> 16;
    i[4] = iv.z & 0xFFFF; i[5] = iv.z >> 16; i[6] = iv.w & 0xFFFF; i[7] = iv.w >> 16;
    load_coefs8(coef, coef_dtype, off, c);
}

// The codes of one token in registers, for fp16 coefficients and s = 8 * SV in 16-byte aligned arrays: a
// thread asks for its next token's codes as it uses up those of the current one, so a chunk's memory
// latency passes while the chunk before it is worked on.  (All warps of a CTA start together at the
// table load and stay in step: without this each chunk cost its latency in full.)
template <int SV>
struct TokenCodes {
    uint4 i[SV], c[SV];
    __device__ __forceinline__ void fetch(int j, const uint16_t* idx, const void* coef, int64_t o) {
        i[j] = __ldg(reinterpret_cast<const uint4*>(idx + o) + j);
        c[j] = __ldg(reinterpret_cast<const uint4*>(static_cast<const uint16_t*>(coef) + o) + j);
    }
};
// Calls f(atom, coef) for the eight entries of one block.
template <typename F>
__device__ __forceinline__ void for_block(const uint4& iv, const uint4& cv, int N, F&& f) {
    const uint32_t iw[4] = {iv.x, iv.y, iv.z, iv.w}, cw[4] = {cv.x, cv.y, cv.z, cv.w};
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const float2 c = __half22float2(*reinterpret_cast<const __half2*>(&cw[q]));
        const int i0 = iw[q] & 0xFFFF, i1 = iw[q] >> 16;
        f(i0 < N ? i0 : N - 1, c.x);
        f(i1 < N ? i1 : N - 1, c.y);
    }
}
__device__ __forceinline__ float block_l1(const uint4& cv) {
    const uint32_t cw[4] = {cv.x, cv.y, cv.z, cv.w};
    float l1 = 0.f;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const float2 c = __half22float2(*reinterpret_cast<const __half2*>(&cw[q]));
        l1 += fabsf(c.x) + fabsf(c.y);
    }
    return l1;
}

// ---- code streams --------------------------------------------------------------------------
// The table is interleaved, tab[atom][HGP] with HGP = 1, 2, 4 or 8 query heads side by side, so
// that one vector access per stored entry serves all heads of the group.
template <int HGP>
struct HeadVec {
    float v[HGP];
};
template <int HGP>
__device__ __forceinline__ HeadVec<HGP> load_heads(const float* p) {
    HeadVec<HGP> r;
    if constexpr (HGP == 1) {
        r.v[0] = p[0];
    } else if constexpr (HGP == 2) {
        const float2 t = *reinterpret_cast<const float2*>(p);
        r.v[0] = t.x;
        r.v[1] = t.y;
    } else {
#pragma unroll
        for (int q = 0; q < HGP / 4; ++q) {
            const float4 t = *reinterpret_cast<const float4*>(p + 4 * q);
            r.v[4 * q + 0] = t.x;
            r.v[4 * q + 1] = t.y;
            r.v[4 * q + 2] = t.z;
            r.v[4 * q + 3] = t.w;
        }
    }
    return r;
}

// Calls f(g, atom, coef) for the s stored entries of the token whose codes start at `o`.
template <typename F>
__device__ __forceinline__ void for_each_code(const uint16_t* idx, const void* coef, int coef_dtype, int64_t o, int s, int N,
                                              int vec, F&& f) {
    if (vec) {
        for (int g0 = 0; g0 < s; g0 += 8) {
            int i8[8];
            float c8[8];
            load_codes8(idx, coef, coef_dtype, o + g0, i8, c8);
#pragma unroll
            for (int g = 0; g < 8; ++g) f(i8[g] < N ? i8[g] : N - 1, c8[g]);
        }
    } else {
        for (int g = 0; g < s; ++g) {
            const int i = idx[o + g];
            f(i < N ? i : N - 1, load_coef(coef, coef_dtype, o + g));
        }
    }
}

// The coefficients alone.
template <typename F>
__device__ __forceinline__ void for_each_coef(const void* coef, int coef_dtype, int64_t o, int s, int vec, F&& f) {
    if (vec) {
        for (int g0 = 0; g0 < s; g0 += 8) {
            float c8[8];
            load_coefs8(coef, coef_dtype, o + g0, c8);
#pragma unroll
            for (int g = 0; g < 8; ++g) f(c8[g]);
        }
    } else {
        for (int g = 0; g < s; ++g) f(load_coef(coef, coef_dtype, o + g));
    }
}

// Contiguous, balanced ranges of the work items (stream and head group, chunk) over the CTAs: CTA c has the
// items [total * c / grid, total * (c + 1) / grid).
struct Ranges {
    int64_t total, chunks;                                 // items, items per stream and head group
    int grid;
    __host__ __device__ int64_t first(int c) const { return total * c / grid; }
    __host__ __device__ int owner(int64_t w) const { return static_cast<int>(((w + 1) * grid + total - 1) / total - 1); }
};

// What csr_decode_attention's scatter needs to turn scores into weights and to scale its tables.
struct KeyStats {
    float2* ml;             // [b][group][slot][HGP]: (maximum, sum of exponentials) of a CTA's part of a row
    int slots;              // slots reserved per (b, group)
    uint32_t* u;            // [b][chunk]: largest l1-norm of a token's value coefficients, float bits (NaN counts as Inf)
    const void* v_coef;     // [b][t][v_s]
    int v_s, v_vec;
};

// SV: the codes' blocks of eight per token, fetched a token ahead (0: any s, any coefficient type).
template <int HGP, bool STATS, int SV>
__global__ void __launch_bounds__(NTHR, ctas_per_sm<HGP>())
key_scores_kernel(const float* P, int N, int H, const uint16_t* __restrict__ idx, const void* __restrict__ coef,
                  int coef_dtype, int64_t T, int s, int vec, float* __restrict__ scores, Ranges rg, KeyStats st) {
    extern __shared__ __align__(16) float tab[];           // [N][HGP]
    __shared__ float2 red[NTHR / 32][HGP];
    const int groups = (H + HGP - 1) / HGP;
    const int chunks = static_cast<int>(rg.chunks);
    const int64_t w0 = rg.first(blockIdx.x);
    int left = static_cast<int>(rg.first(blockIdx.x + 1) - w0);            // items of this CTA
    // the current item (no divisions in the loop: they would cost as much as the work)
    int chunk = static_cast<int>(w0 % chunks), group = static_cast<int>(w0 / chunks % groups), b = static_cast<int>(w0 / chunks / groups);
    bool fresh = true;                                     // another table is needed
    float m[HGP], l[HGP];
    TokenCodes<SV ? SV : 1> tc;
    uint4 vc[2];                                           // the token's value coefficients (v_s = 8 or 16)
    const bool v_regs = STATS && SV > 0 && st.v_vec && st.v_s <= 16;
    // this thread's token of a chunk, as an offset into [b][t] (what is fetched past a row's end is not used)
    const auto token = [&](int bb, int cc) {
        const int64_t t = static_cast<int64_t>(cc) * NTHR + threadIdx.x;
        return bb * T + (t < T ? t : T - 1);
    };
    if constexpr (SV > 0) {
        if (left > 0) {
            const int64_t o = token(b, chunk);
#pragma unroll
            for (int j = 0; j < SV; ++j) tc.fetch(j, idx, coef, o * s);
            if (v_regs) {
                vc[0] = __ldg(reinterpret_cast<const uint4*>(static_cast<const uint16_t*>(st.v_coef) + o * st.v_s));
                if (st.v_s > 8) vc[1] = __ldg(reinterpret_cast<const uint4*>(static_cast<const uint16_t*>(st.v_coef) + o * st.v_s) + 1);
            }
        }
    }
    next_may_start();
    wait_for_previous();                                  // P
    for (; left > 0; --left) {
        const int h0 = group * HGP;
        const int hg = H - h0 < HGP ? H - h0 : HGP;
        const int64_t bg = static_cast<int64_t>(b) * groups + group;
        // the item after this one
        int chunk_n = chunk + 1, group_n = group, b_n = b;
        if (chunk_n == chunks) {
            chunk_n = 0;
            if (++group_n == groups) {
                group_n = 0;
                ++b_n;
            }
        }
        if (fresh) {
            __syncthreads();
            const float* src = P + bg * N * HGP;
            if (HGP >= 4 || (N * HGP) % 4 == 0) {          // the group's table, as it lies (16-byte aligned in either case)
                const float4* s4 = reinterpret_cast<const float4*>(src);
                float4* t4 = reinterpret_cast<float4*>(tab);
                const int n4 = N * HGP / 4;
#pragma unroll 8
                for (int j = threadIdx.x; j < n4; j += NTHR) t4[j] = s4[j];
            } else {
                for (int j = threadIdx.x; j < N * HGP; j += NTHR) tab[j] = src[j];
            }
            if constexpr (STATS) {
#pragma unroll
                for (int h = 0; h < HGP; ++h) {
                    m[h] = kLowest;
                    l[h] = 0.f;
                }
            }
            __syncthreads();
        }
        const int64_t t = static_cast<int64_t>(chunk) * NTHR + threadIdx.x;
        float acc[HGP];
#pragma unroll
        for (int h = 0; h < HGP; ++h) acc[h] = 0.f;
        const auto add = [&](int i, float c) {
            const HeadVec<HGP> pv = load_heads<HGP>(tab + i * HGP);
#pragma unroll
            for (int h = 0; h < HGP; ++h) acc[h] = fmaf(c, pv.v[h], acc[h]);
        };
        [[maybe_unused]] float l1 = 0.f;                   // all of a token's entries may name the same atom
        if constexpr (SV > 0) {
            const int64_t next = left > 1 ? token(b_n, chunk_n) : 0;
#pragma unroll
            for (int j = 0; j < SV; ++j) {
                for_block(tc.i[j], tc.c[j], N, add);
                tc.fetch(j, idx, coef, next * s);
            }
            if (v_regs) {
                const uint4* nv = reinterpret_cast<const uint4*>(static_cast<const uint16_t*>(st.v_coef) + next * st.v_s);
                l1 = block_l1(vc[0]);
                vc[0] = __ldg(nv);
                if (st.v_s > 8) {
                    l1 += block_l1(vc[1]);
                    vc[1] = __ldg(nv + 1);
                }
                if (t >= T) l1 = 0.f;
            }
        } else if (t < T) {
            for_each_code(idx, coef, coef_dtype, ((int64_t)b * T + t) * s, s, N, vec, add);
        }
        if (t < T) {
#pragma unroll
            for (int h = 0; h < HGP; ++h)
                if (h < hg) scores[((int64_t)b * H + h0 + h) * T + t] = acc[h];
            if constexpr (STATS) {
#pragma unroll
                for (int h = 0; h < HGP; ++h) {
                    const float mn = fmaxf(m[h], acc[h]);
                    l[h] = l[h] * __expf(m[h] - mn) + __expf(acc[h] - mn);
                    m[h] = mn;
                }
            }
        }
        if constexpr (STATS) {
            if (h0 == 0) {                                 // once per token, whatever the number of groups
                if (!v_regs && t < T)
                    for_each_coef(st.v_coef, coef_dtype, ((int64_t)b * T + t) * st.v_s, st.v_s, st.v_vec, [&](float c) { l1 += fabsf(c); });
                const uint32_t top = __reduce_max_sync(0xffffffffu, __float_as_uint(l1 == l1 ? l1 : INFINITY));
                if ((threadIdx.x & 31) == 0) atomicMax(st.u + (int64_t)b * chunks + chunk, top);
            }
            if (left == 1 || chunk_n == 0) {               // this CTA's last item of the row
                const int warp = threadIdx.x >> 5;
#pragma unroll
                for (int h = 0; h < HGP; ++h) {
                    float mw = m[h];
                    for (int o = 16; o; o >>= 1) mw = fmaxf(mw, __shfl_xor_sync(0xffffffffu, mw, o));
                    float lw = l[h] * expf(m[h] - mw);
                    for (int o = 16; o; o >>= 1) lw += __shfl_xor_sync(0xffffffffu, lw, o);
                    if ((threadIdx.x & 31) == 0) red[warp][h] = make_float2(mw, lw);
                }
                __syncthreads();
                if (threadIdx.x < HGP) {
                    const int h = threadIdx.x;
                    float mx = kLowest, sum = 0.f;
                    for (int q = 0; q < NTHR / 32; ++q) mx = fmaxf(mx, red[q][h].x);
                    for (int q = 0; q < NTHR / 32; ++q) sum += red[q][h].y * expf(red[q][h].x - mx);
                    const int slot = blockIdx.x - rg.owner(bg * rg.chunks);
                    st.ml[(bg * st.slots + slot) * HGP + h] = make_float2(mx, sum);
                }
                // (the next row's table load begins with a barrier)
            }
        }
        fresh = chunk_n == 0;
        chunk = chunk_n;
        group = group_n;
        b = b_n;
    }
}

// Block-wide maximum / sum of one value per thread, returned to every thread; the order of the
// additions is fixed.
__device__ __forceinline__ float block_max(float v, float* red) {
    for (int o = 16; o; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    __syncthreads();
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    float r = red[0];
    for (int j = 1; j < NTHR / 32; ++j) r = fmaxf(r, red[j]);
    return r;
}
__device__ __forceinline__ float block_sum(float v, float* red) {
    for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    float r = 0.f;
    for (int j = 0; j < NTHR / 32; ++j) r += red[j];
    return r;
}

// Unit of work = (code stream, head group, piece): a contiguous range of the stream's token chunks.  The
// CTA owns the unit's table, so its result is stored, not added.
//
// The table is accumulated in 32-bit fixed point: integer shared-memory atomics run at more
// than twice the rate of fp32 ones (measured 17.5 against 7.7 per ns per SM), and integer
// addition does not depend on the order, so the table is the same on every run.  A first
// pass over the unit's weights and coefficients gives, per head, S = sum |w_t| and
// U = max over tokens of sum_g |coef[t][g]| (a token's entries may all name one atom); no
// table entry can exceed S * U in magnitude, and the scale is the power
// of two that maps S * U to at most 2^30; the roundings of the individual terms, half a unit
// each, add at most 2^29 (a unit has no more than 2^30 terms) and stay inside the 32-bit
// range.  Each term w * coef is rounded once to fp32, as a floating-point accumulation would,
// and once to the grid, whose step is between 2^-30 and 2^-29 of S * U: it grows with the tokens of a
// unit (see plan_split).  A unit whose S or U is not finite falls back to fp32 atomics, so
// that NaN and Inf still reach the output.
// STATS: W holds scores; the first pass makes them weights (softmax over the row, from the statistics the
// scores kernel left) and reads no codes: U is there already.
template <int HGP, bool STATS, int SV>
__global__ void __launch_bounds__(NTHR, ctas_per_sm<HGP>())
value_scatter_kernel(int N, float* W, int B, int H, const uint16_t* __restrict__ idx, const void* __restrict__ coef, int coef_dtype,
                     int64_t T, int s, int vec, int pieces, float* __restrict__ A, Ranges rg, KeyStats st) {
    extern __shared__ __align__(16) float tab[];           // [HGP][N]: scalar atomics want the heads apart
    __shared__ float red[NTHR / 32];
    __shared__ float row_max[HGP], row_inv[HGP];
    int* itab = reinterpret_cast<int*>(tab);
    const int groups = (H + HGP - 1) / HGP;
    const int64_t chunks_per_b = (T + NTHR - 1) / NTHR;
    const int64_t units = (int64_t)B * groups * pieces;
    next_may_start();
    bool waited = false;
    for (int64_t unit = blockIdx.x; unit < units; unit += gridDim.x) {
        const int64_t bg = unit / pieces;
        const int b = static_cast<int>(bg / groups), piece = static_cast<int>(unit % pieces);
        const int h0 = static_cast<int>(bg % groups) * HGP;
        const int hg = H - h0 < HGP ? H - h0 : HGP;
        const int64_t c0 = chunks_per_b * piece / pieces, c1 = chunks_per_b * (piece + 1) / pieces;
        float* Wb = W + ((int64_t)b * H + h0) * T;
        __syncthreads();
        if ((N * HGP) % 4 == 0) {
            for (int j = threadIdx.x; j < N * HGP / 4; j += NTHR) reinterpret_cast<float4*>(tab)[j] = make_float4(0.f, 0.f, 0.f, 0.f);
        } else {
            for (int j = threadIdx.x; j < N * HGP; j += NTHR) tab[j] = 0.f;   // +0.0f and integer 0 share their bits
        }
        if (!waited) {                                     // the scores and their statistics (the first table is cleared meanwhile)
            wait_for_previous();
            waited = true;
        }
        // ---- pass 1: bounds ----
        float umax = 0.f, sw[HGP];
#pragma unroll
        for (int h = 0; h < HGP; ++h) sw[h] = 0.f;
        if constexpr (STATS) {
            if (threadIdx.x < HGP) {                       // (a handful of slots: one thread per head)
                const int slots = rg.owner((bg + 1) * rg.chunks - 1) - rg.owner(bg * rg.chunks) + 1;
                const float2* ml = st.ml + bg * st.slots * HGP + threadIdx.x;
                float mx = kLowest, sum = 0.f;
                for (int q = 0; q < slots; ++q) mx = fmaxf(mx, ml[q * HGP].x);
                for (int q = 0; q < slots; ++q) sum += ml[q * HGP].y * expf(ml[q * HGP].x - mx);
                row_max[threadIdx.x] = mx;
                row_inv[threadIdx.x] = 1.0f / sum;
            }
            for (int64_t c = c0 + threadIdx.x; c < c1; c += NTHR) umax = fmaxf(umax, __uint_as_float(st.u[(int64_t)b * rg.chunks + c]));
            __syncthreads();
            // (four chunks' scores are read before the first weight is written: one latency for the four)
            for (int64_t c = c0; c < c1; c += 4) {
                float sc[4][HGP];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int64_t t = (c + u) * NTHR + threadIdx.x;
#pragma unroll
                    for (int h = 0; h < HGP; ++h) sc[u][h] = c + u < c1 && t < T && h < hg ? Wb[h * T + t] : 0.f;
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int64_t t = (c + u) * NTHR + threadIdx.x;
                    if (c + u >= c1 || t >= T) continue;
#pragma unroll
                    for (int h = 0; h < HGP; ++h)
                        if (h < hg) {
                            const float w = __expf(sc[u][h] - row_max[h]) * row_inv[h];
                            Wb[h * T + t] = w;
                            sw[h] += fabsf(w);
                        }
                }
            }
        } else {
            for (int64_t c = c0; c < c1; ++c) {
                const int64_t t = c * NTHR + threadIdx.x;
                if (t >= T) continue;
#pragma unroll
                for (int h = 0; h < HGP; ++h)
                    if (h < hg) sw[h] += fabsf(Wb[h * T + t]);
                float l1 = 0.f;                            // all of a token's entries may name the same atom
                for_each_coef(coef, coef_dtype, ((int64_t)b * T + t) * s, s, vec, [&](float cf) { l1 += fabsf(cf); });
                umax = l1 == l1 ? fmaxf(umax, l1) : INFINITY;
            }
        }
        umax = block_max(umax, red);
        float scale[HGP], inv_scale[HGP];
        // (the half-unit roundings of the terms must stay inside the range too)
        bool fixed_point = umax < INFINITY && (c1 - c0) * NTHR * static_cast<int64_t>(s) <= (1ll << 30);
#pragma unroll
        for (int h = 0; h < HGP; ++h) {
            const float S = block_sum(sw[h], red);
            const float bound = S * umax;
            if (!(bound < INFINITY)) fixed_point = false;                 // Inf or NaN
            int e = 0;
            if (bound > 0.f) e = 30 - (ilogbf(bound) + 1);                // 2^e * bound <= 2^30
            e = e > 96 ? 96 : e < -96 ? -96 : e;
            scale[h] = ldexpf(1.f, e);
            inv_scale[h] = ldexpf(1.f, -e);
        }
        __syncthreads();
        // ---- pass 2: scatter ----
        // (the heads past the last one have weight zero and table rows of their own: a test per atomic was a
        // branch per atomic, 20 instructions for each: 73 instead of 52 us)
        const auto add_fixed = [&](const float (&wv)[HGP], int i, float cf) {
            int* at = itab + i;
#pragma unroll
            for (int h = 0; h < HGP; ++h) atomicAdd(at + h * N, __float2int_rn(wv[h] * cf));
        };
        const auto weights = [&](int64_t t, float (&wv)[HGP]) {
#pragma unroll
            for (int h = 0; h < HGP; ++h) wv[h] = h < hg ? Wb[h * T + t] * scale[h] : 0.f;   // exact: a power of two
        };
        if (SV > 0 && fixed_point) {
            TokenCodes<SV ? SV : 1> tc;
            float wn[HGP];
            int64_t t = c0 * NTHR + threadIdx.x;
            const int64_t tn = c1 * NTHR < T ? c1 * NTHR : T;                  // end of this unit's tokens
            if (t < tn) {
#pragma unroll
                for (int j = 0; j < SV; ++j) tc.fetch(j, idx, coef, ((int64_t)b * T + t) * s);
                weights(t, wn);
            }
            for (; t < tn; t += NTHR) {
                float wv[HGP];
#pragma unroll
                for (int h = 0; h < HGP; ++h) wv[h] = wn[h];
                const int64_t next = t + NTHR < tn ? t + NTHR : t;
                weights(next, wn);
#pragma unroll
                for (int j = 0; j < SV; ++j) {
                    const uint4 iv = tc.i[j], cv = tc.c[j];
                    tc.fetch(j, idx, coef, ((int64_t)b * T + next) * s);
                    for_block(iv, cv, N, [&](int i, float cf) { add_fixed(wv, i, cf); });
                }
            }
        } else {
            for (int64_t c = c0; c < c1; ++c) {
                const int64_t t = c * NTHR + threadIdx.x;
                if (t >= T) continue;
                float wv[HGP];
                if (fixed_point) {
                    weights(t, wv);
                    for_each_code(idx, coef, coef_dtype, ((int64_t)b * T + t) * s, s, N, vec, [&](int i, float cf) { add_fixed(wv, i, cf); });
                } else {
#pragma unroll
                    for (int h = 0; h < HGP; ++h) wv[h] = h < hg ? Wb[h * T + t] : 0.f;
                    for_each_code(idx, coef, coef_dtype, ((int64_t)b * T + t) * s, s, N, vec, [&](int i, float cf) {
#pragma unroll
                        for (int h = 0; h < HGP; ++h) atomicAdd(&tab[h * N + i], wv[h] * cf);
                    });
                }
            }
        }
        __syncthreads();
        float* dst = A + unit * HGP * N;                   // [HGP][N] of this unit
        if (fixed_point) {
#pragma unroll
            for (int h = 0; h < HGP; ++h)
                if (h < hg)
                    for (int j = threadIdx.x; j < N; j += NTHR) dst[h * N + j] = static_cast<float>(itab[h * N + j]) * inv_scale[h];
        } else {
            for (int j = threadIdx.x; j < hg * N; j += NTHR) dst[j] = tab[j];
        }
    }
}

// ---- launch plans ------------------------------------------------------------------------------
// Query heads per group (8, 4, 2 or 1; 0 = not even one head's N values fit in shared memory).  As many
// heads as fit share a pass over the codes, but not so many that there are fewer (stream, group,
// chunk) items than SMs: at 8 streams x 4099 tokens x 4 heads, N = 8192, one head per group (288
// items) takes 10 + 10 us of scores and scatter, the four heads together (40 chunks of 1024) took
// 9 + 5 (softmax) + 16.
struct Split {
    int hg, groups, pieces;
    int64_t chunks;
    Ranges ranges;          // of the scores kernel
};
Split plan_split(int B, int H, int N, int64_t T) {
    Split p{};
    const int sms = sm_count();
    int hg = 8;
    while (hg > 1 && (hg / 2 >= H || (size_t)hg * N * 4 > 200 * 1024)) hg /= 2;
    if ((size_t)hg * N * 4 > 200 * 1024) return p;
    p.chunks = (T + NTHR - 1) / NTHR;
    auto items = [&](int g) { return (int64_t)B * ((H + g - 1) / g) * p.chunks; };
    while (hg > 1 && items(hg) < sms) hg /= 2;
    p.hg = hg;
    p.groups = (H + hg - 1) / hg;
    const int64_t total = items(hg), cap = (int64_t)sms * (hg <= 2 && (size_t)hg * N * 4 <= 100 * 1024 ? 2 : 1);
    p.ranges = Ranges{total, p.chunks, (int)(total < cap ? total : cap)};
    // pieces of a stream's tokens for the value scatter: a unit per SM, no more than there are chunks (each
    // unit's table is cleared, stored and read back by ad_kernel)
    int64_t k = sms / ((int64_t)B * p.groups);
    // ... but at least half as many as a stream has SMs, down to units of 2048 tokens: a unit's grid step grows
    // with its share of the weights, and however many groups the heads are cut into, the step stays at
    // what one group per stream has with 2^29 for the grid's range
    const int64_t fine = (p.chunks + 1) / 2, share = sms / B, least = ((share < fine ? share : fine) + 1) / 2;
    if (k < least) k = least;
    if (k > p.chunks) k = p.chunks;
    p.pieces = k < 1 ? 1 : (int)k;
    return p;
}
int slots_of(const Split& p) { return (int)((p.chunks * p.ranges.grid + p.ranges.total - 1) / p.ranges.total) + 2; }

size_t align16(size_t x) { return (x + 15) / 16 * 16; }
size_t p_floats(const Split& p, int B, int N) { return align16((size_t)B * p.groups * N * p.hg); }
size_t a_floats(const Split& p, int B, int N) { return align16((size_t)B * p.groups * p.pieces * p.hg * N); }
// slices of the atoms for out = A D: about two CTAs per SM
int ad_slices(int R, int rt, int N, int* per_slice) {
    const int row_blocks = (R + rt - 1) / rt;
    int slices = 2 * sm_count() / row_blocks;
    const int most = (N + OA - 1) / OA;
    if (slices > most) slices = most;
    if (slices < 1) slices = 1;
    *per_slice = ((N + slices - 1) / slices + OA - 1) / OA * OA;
    return (N + *per_slice - 1) / *per_slice;
}
int row_tile(int R) { return R <= 32 ? 32 : 64; }

// One launch; `overlap`: its CTAs may come up before the previous kernel of this call has ended.
template <typename... P, typename... A>
cudaError_t launch(void (*kernel)(P...), dim3 grid, int threads, size_t smem, cudaStream_t stream, bool overlap, A... args) {
    if (smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    cfg.gridDim = grid;
    cfg.blockDim = dim3((unsigned)threads, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = overlap ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

template <int D_, int RT, int AT>
cudaError_t run_qd(const AttnArgs& a, const Split& p, float* P, uint32_t* zero, int n_zero) {
    constexpr size_t smem = (size_t)(RT + AT) * (D_ + 4) * sizeof(float);
    const int R = a.B * a.H;
    const dim3 grid((a.N + AT - 1) / AT, (R + RT - 1) / RT);
    return launch(qd_kernel<D_, RT, AT>, grid, NT, smem, a.stream, false, a.D, a.N, a.Q, a.q_dtype, R, a.H, p.hg, a.scale, P, zero, n_zero);
}

template <int HGP, bool STATS, int SV>
cudaError_t run_keys(const AttnArgs& a, const Split& p, const float* P, const KeyStats& st) {
    return launch(key_scores_kernel<HGP, STATS, SV>, dim3(p.ranges.grid), NTHR, (size_t)HGP * a.N * 4, a.stream, true, P, a.N, a.H, a.idx,
                  a.coef, a.coef_dtype, a.T, a.s, a.s % 8 == 0, a.out, p.ranges, st);
}
template <int HGP, bool STATS, int SV>
cudaError_t run_scatter(const AttnArgs& a, const Split& p, float* W, float* A, const KeyStats& st, const Ranges& rg) {
    const int64_t units = (int64_t)a.B * p.groups * p.pieces, cap = (int64_t)sm_count() * ctas_per_sm<HGP>();
    // (alone, its weights are the caller's: nothing of this call precedes it)
    return launch(value_scatter_kernel<HGP, STATS, SV>, dim3((unsigned)(units < cap ? units : cap)), NTHR, (size_t)HGP * a.N * 4, a.stream,
                  STATS, a.N, W, a.B, a.H, a.idx, a.coef, a.coef_dtype, a.T, a.s, a.s % 8 == 0, p.pieces, A, rg, st);
}
// f(integral_constant HGP, integral_constant SV) of the plan and the codes
template <typename F>
cudaError_t dispatch(const Split& p, const AttnArgs& a, F&& f) {
    using std::integral_constant;
    const int sv = a.coef_dtype == CSR_DTYPE_F16 && (a.s == 8 || a.s == 16) ? a.s / 8 : 0;
    auto with_codes = [&](auto hg) {
        return sv == 1   ? f(hg, integral_constant<int, 1>{})
               : sv == 2 ? f(hg, integral_constant<int, 2>{})
                         : f(hg, integral_constant<int, 0>{});
    };
    switch (p.hg) {
        case 8: return with_codes(integral_constant<int, 8>{});
        case 4: return with_codes(integral_constant<int, 4>{});
        case 2: return with_codes(integral_constant<int, 2>{});
        default: return with_codes(integral_constant<int, 1>{});
    }
}

int run_scores(const AttnArgs& a, const Split& p, float* P, const KeyStats* st, int n_zero) {
    const int R = a.B * a.H;
    uint32_t* zero = st ? st->u : nullptr;
    cudaError_t e;
    if (row_tile(R) == 32)
        e = a.d == 128 ? run_qd<128, 32, 64>(a, p, P, zero, n_zero) : run_qd<64, 32, 64>(a, p, P, zero, n_zero);
    else
        e = a.d == 128 ? run_qd<128, 64, 128>(a, p, P, zero, n_zero) : run_qd<64, 64, 128>(a, p, P, zero, n_zero);
    if (e == cudaSuccess)
        e = dispatch(p, a, [&](auto hg, auto sv) {
            return st ? run_keys<hg.value, true, sv.value>(a, p, P, *st)
                      : run_keys<hg.value, false, sv.value>(a, p, P, KeyStats{});
        });
    return e == cudaSuccess ? CSR_OK : fail(CSR_ERR_CUDA, "key_scores launch: %s", cudaGetErrorString(e));
}

// scratch: [tables][the slices' results]
int run_mix(const AttnArgs& a, const Split& p, float* W, float* A, const KeyStats* st, const Ranges& rg) {
    cudaError_t e = dispatch(p, a, [&](auto hg, auto sv) {
        return st ? run_scatter<hg.value, true, sv.value>(a, p, W, A, *st, rg)
                  : run_scatter<hg.value, false, sv.value>(a, p, W, A, KeyStats{}, Ranges{});
    });
    if (e != cudaSuccess) return fail(CSR_ERR_CUDA, "value_scatter launch: %s", cudaGetErrorString(e));
    const int R = a.B * a.H, rt = row_tile(R);
    int per_slice = 0;
    const int slices = ad_slices(R, rt, a.N, &per_slice);
    float* part = slices > 1 ? A + a_floats(p, a.B, a.N) : a.out;
    const dim3 grid(slices, (R + rt - 1) / rt);
    auto run_ad = [&](auto d, auto rows) {
        constexpr size_t smem = ad_smem_bytes<d.value, rows.value>();
        return launch(ad_kernel<d.value, rows.value>, grid, NT, smem, a.stream, true, a.D, a.N, A, R, a.H, p.hg, p.pieces, per_slice, part);
    };
    using std::integral_constant;
    if (a.d == 128)
        e = rt == 32 ? run_ad(integral_constant<int, 128>{}, integral_constant<int, 32>{})
                     : run_ad(integral_constant<int, 128>{}, integral_constant<int, 64>{});
    else
        e = rt == 32 ? run_ad(integral_constant<int, 64>{}, integral_constant<int, 32>{})
                     : run_ad(integral_constant<int, 64>{}, integral_constant<int, 64>{});
    if (e == cudaSuccess && slices > 1) {
        const int64_t n4 = (int64_t)R * a.d / 4;
        e = launch(add_slices_kernel, dim3((unsigned)((n4 + SUM_X - 1) / SUM_X)), SUM_X * SUM_Y, 0, a.stream, true,
                   reinterpret_cast<const float4*>(part), slices, n4, reinterpret_cast<float4*>(a.out));
    }
    return e == cudaSuccess ? CSR_OK : fail(CSR_ERR_CUDA, "value_mix launch: %s", cudaGetErrorString(e));
}

int too_large(int N) { return fail(CSR_ERR_UNSUPPORTED, "N = %d: one head's N fp32 values do not fit in shared memory", N); }

size_t mix_bytes(const Split& p, int B, int H, int N) {
    int per_slice = 0;
    const int R = B * H, slices = ad_slices(R, row_tile(R), N, &per_slice);
    return (a_floats(p, B, N) + (size_t)slices * R * 128) * sizeof(float);
}

}  // namespace

size_t key_scores_scratch_bytes(int B, int H, int N, int64_t T) {
    const Split p = plan_split(B, H, N, T);
    return p.hg ? p_floats(p, B, N) * sizeof(float) : 0;
}
size_t value_mix_scratch_bytes(int B, int H, int N, int64_t T) {
    const Split p = plan_split(B, H, N, T);
    return p.hg ? mix_bytes(p, B, H, N) : 0;
}
// [statistics][largest norms per chunk][the scores' table or the mix's tables: one after the other]
static size_t stats_bytes(const Split& k, int B) {
    return align16((size_t)B * k.groups * slots_of(k) * k.hg * sizeof(float2)) + align16((size_t)B * k.chunks * 4);
}
size_t decode_attention_scratch_bytes(int B, int H, int Nk, int Nv, int64_t T) {
    // one plan for both sides (the statistics and norms are per group and chunk): the larger dictionary's
    const Split p = plan_split(B, H, Nk > Nv ? Nk : Nv, T);
    if (!p.hg) return 0;
    const size_t kb = p_floats(p, B, Nk) * sizeof(float), vb = mix_bytes(p, B, H, Nv);
    return stats_bytes(p, B) + (kb > vb ? kb : vb);
}

int launch_key_scores(const AttnArgs& a, float* scratch) {
    if (a.B == 0 || a.T == 0 || a.H == 0) return CSR_OK;
    const Split p = plan_split(a.B, a.H, a.N, a.T);
    if (!p.hg) return too_large(a.N);
    return run_scores(a, p, scratch, nullptr, 0);
}

int launch_value_mix(const AttnArgs& a, float* scratch) {
    if (a.B == 0 || a.H == 0) return CSR_OK;
    if (a.T == 0) {
        cudaError_t e0 = cudaMemsetAsync(a.out, 0, (size_t)a.B * a.H * a.d * sizeof(float), a.stream);
        if (e0 != cudaSuccess) return fail(CSR_ERR_CUDA, "cudaMemsetAsync: %s", cudaGetErrorString(e0));
        return CSR_OK;
    }
    const Split p = plan_split(a.B, a.H, a.N, a.T);
    if (!p.hg) return too_large(a.N);
    return run_mix(a, p, const_cast<float*>(static_cast<const float*>(a.Q)), scratch, nullptr, Ranges{});
}

int launch_decode_attention(const AttnArgs& k, const AttnArgs& v, void* scratch) {
    if (k.B == 0 || k.H == 0) return CSR_OK;
    const Split p = plan_split(k.B, k.H, k.N > v.N ? k.N : v.N, k.T);
    if (!p.hg) return too_large(k.N > v.N ? k.N : v.N);
    char* q = static_cast<char*>(scratch);
    KeyStats st;
    st.ml = reinterpret_cast<float2*>(q);
    st.slots = slots_of(p);
    st.u = reinterpret_cast<uint32_t*>(q + align16((size_t)k.B * p.groups * st.slots * p.hg * sizeof(float2)));
    st.v_coef = v.coef;
    st.v_s = v.s;
    st.v_vec = v.s % 8 == 0;
    float* rest = reinterpret_cast<float*>(q + stats_bytes(p, k.B));
    if (int rc = run_scores(k, p, rest, &st, (int)(k.B * p.chunks))) return rc;
    return run_mix(v, p, k.out, rest, &st, p.ranges);
}

}  // namespace csr
