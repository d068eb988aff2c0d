// Correctness-mode matching pursuit (paper Eq. 2-4) with the sweep on the sm_100a tensor cores.
//
// The picks must be those of an fp64 evaluation of the pursuit.  An fp16 product cannot decide
// them, but it can bound them: with r = r' + e and d = d' + f (r', d' the fp16 values the tensor cores
// read), a correlation r.d differs from r'.d' by at most ||e|| max ||d|| + ||r'|| max ||f||, and all of these
// norms are known (row_band in exact_tc_common.cuh): about 4e-4 ||R||, plus what the fp32 accumulation adds.
// So every correlation of a sweep is known to within a band of about 8e-4 ||R||, which decides 95 % of
// the rows; for the others the candidates inside the band are re-scored in fp64.
//
// One persistent CTA per SM owns two tiles of 128 rows for all s iterations:
//   - the fp64 residuals live in a per-CTA scratch area in global memory (256 KB, L2 resident);
//     the rows as fp16, scaled by a power of two to a norm in [1, 2), are the
//     tcgen05.mma A operands in shared memory (K-major, 128-byte swizzle, 2 row tiles);
//   - the dictionary's fp16 copy (made once per call) streams through a ring of 32 KB stages fetched
//     by TMA: 64 channels of 256 atoms per stage, used by both row tiles;
//   - each row tile has one 256-column fp32 accumulator in TMEM.  All eight epilogue warps drain
//     every accumulator: warp w reads the 32 TMEM lanes of w % 4 and the 128 columns of w / 4, i.e.
//     all of them sit in registers after one round of loads and the accumulator goes straight back
//     to the tensor core.  Groups of eight adjacent atoms are reduced to their largest magnitude, a key being
//     that with its five lowest mantissa bits replaced by the group's number, and each thread keeps the tile's three
//     largest keys, all without a branch; those within the band of the row's running maximum then join
//     the four largest keys of its half row (three of them with the tile they came from);
//   - at the end of a sweep the halves meet in shared memory, and each warp settles its 32 rows,
//     eight lanes per row: the values of the group with the largest key are computed again from the fp16 operands.  Rows
//     whose best atom is further than the band above the rest of its group and above every other group
//     take it; otherwise all atoms of the groups inside the band (the first three of either half) are compared in
//     fp64, a row at a time by the warp; rows where the fourth of a half is inside too are searched for in the
//     whole dictionary (fp32 filter, then fp64) by the eight warps together.  Coefficient (Eq. 2,
//     signed) and residual update (Eq. 4) are fp64, as in the plain-ALU encoder.
// What bounds it: the epilogue and the settling, no longer the MMAs (2048 cycles per 256 atoms and pair of row tiles).
// Three bf16 products per correlation, whose band was 2^-12 ||R||, took 6144: 100000 rows, N = 4096, s = 8,
// 2441 us so and 2195 us with one fp16 product; a training step of 65536 rows (N = 8192, s = 8) 2992 and 2332 us.
// Warp roles: 0-7 epilogue, 8 TMA producer, 9 TMEM owner and MMA issuer.  All waits are bounded.
#include "exact_tc_common.cuh"

namespace csr {
namespace {

using namespace exact_tc;

constexpr int NT = 320;
constexpr int PRODUCER_WARP = 8;
constexpr int MMA_WARP = 9;
constexpr int ROWS = 2 * TILE_M;                          // rows a CTA holds at a time
constexpr uint32_t TMEM_COLS = 512;
constexpr uint32_t kInstrDesc = instr_desc_f16(TILE_M, TILE_N);

template <int D_>
struct TcSmem {
    static constexpr int kStages = D_ == 128 ? 4 : 5;
    static constexpr int kATileBytes = TILE_M * D_ * 2;
    static constexpr int kStageBytes = TILE_N * STAGE_CH * 2;
    alignas(1024) uint8_t A[2][kATileBytes];
    alignas(1024) uint8_t B[kStages][kStageBytes];
    uint32_t xchg[5][TILE_M];                                    // one half's largest keys of a row tile (and the rows' bands)
    uint64_t full_b[kStages];
    uint64_t empty_b[kStages];
    uint64_t acc_full[2];
    uint64_t acc_empty[2];
    uint64_t res_ready;
    uint64_t drained;
    uint32_t tmem_base;
    volatile uint32_t abort;
};

template <int D_>
__global__ void __launch_bounds__(NT, 1)
encode_exact_tc_kernel(const __grid_constant__ CUtensorMap tmap_d, const uint16_t* __restrict__ dict, const DictPart* __restrict__ parts, int n_parts, const float* __restrict__ D, const void* __restrict__ X, int x_dtype, int64_t ldx, int64_t M, int N, int s,
                       uint16_t* __restrict__ out_idx, void* __restrict__ out_coef, int coef_dtype, int64_t ldc,
                       double* __restrict__ Rd_all, uint32_t* status, [[maybe_unused]] uint32_t* diag,
                       unsigned long long wait_limit_ns) {
    using S = TcSmem<D_>;
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    if ((smem_u32(smem_raw) & 1023u) != 0) {              // the swizzled tiles need this; never seen otherwise
        if (threadIdx.x == 0) atomicOr(status, kStatusLayout);
        return;
    }
    S& sm = *reinterpret_cast<S*>(smem_raw);

    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    const int T = (N + TILE_N - 1) / TILE_N;
    const int64_t n_pairs = (M + ROWS - 1) / ROWS;
    constexpr int KH = D_ / STAGE_CH;                       // 64-channel blocks per row
    constexpr int STAGES = S::kStages;
    const WaitCtx wc{&sm.abort, status, wait_limit_ns};

    if (threadIdx.x == 0) {
        for (int i = 0; i < STAGES; ++i) {
            mbar_init(&sm.full_b[i], 1);
            mbar_init(&sm.empty_b[i], 1);
        }
        for (int t = 0; t < 2; ++t) {
            mbar_init(&sm.acc_full[t], 1);
            mbar_init(&sm.acc_empty[t], 8);
        }
        mbar_init(&sm.res_ready, ROWS);
        mbar_init(&sm.drained, 1);
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

    if (warp == PRODUCER_WARP) {
        // ------------------------------ TMA producer ------------------------------
        if (lane == 0) {
            asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmap_d)) : "memory");
            uint32_t p = 0;
            bool ok = true;
            for (int64_t pair = blockIdx.x; pair < n_pairs && ok; pair += gridDim.x) {
                for (int g = 0; g < s && ok; ++g) {
                    for (int t = 0; t < T && ok; ++t) {
                        for (int h = 0; h < KH; ++h, ++p) {
                            const int stage = p % STAGES;
                            if (!wait_bounded_suspended(&sm.empty_b[stage], ((p / STAGES) & 1) ^ 1, wc, 2000)) {
                                ok = false;
                                break;
                            }
                            // atoms past N arrive as zeros and count as bytes
                            mbar_expect_tx(&sm.full_b[stage], S::kStageBytes);
                            tma_load_2d(&sm.B[stage][0], &tmap_d, h * STAGE_CH, t * TILE_N, &sm.full_b[stage]);
                        }
                    }
                }
            }
            if (!ok) {                                    // let the copies already issued land
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
        {
            uint32_t p = 0, accn = 0, steps = 0;
            bool ok = true;
            for (int64_t pair = blockIdx.x; pair < n_pairs && ok; pair += gridDim.x) {
                for (int g = 0; g < s && ok; ++g, ++steps) {
                    if (!warp_wait_bounded_suspended(&sm.res_ready, steps & 1, wc, 4000)) {
                        ok = false;
                        break;
                    }
                    // Each row tile takes all stages of a dictionary tile before the other takes the same ones: the
                    // accumulators then complete a whole tile's MMAs apart, and the epilogue drains them one
                    // after the other.
                    for (int t = 0; t < T && ok; ++t, ++accn, p += KH) {
#pragma unroll
                        for (int tile = 0; tile < 2; ++tile) {
                            ok = warp_wait_bounded_suspended(&sm.acc_empty[tile], (accn & 1) ^ 1, wc, 1000);
                            const uint32_t d_tmem = tmem_d + tile * TILE_N;
#pragma unroll
                            for (int h = 0; h < KH; ++h) {
                                const uint32_t ps = p + h;
                                const int stage = ps % STAGES;
                                if (tile == 0 && ok) ok = warp_wait_bounded_suspended(&sm.full_b[stage], (ps / STAGES) & 1, wc, 1000);
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
                umma_commit(&sm.drained);
                const unsigned long long t0 = globaltimer_ns();
                while (!mbar_try_wait(&sm.drained, 0))
                    if (globaltimer_ns() - t0 > 20000000ull) break;
            }
        }
    } else {
        // ------------------------------ epilogue ------------------------------
        constexpr int CH = D_ / 8;                          // channels per lane when eight lanes share a row
        const int q = warp & 3;                             // TMEM lane quarter
        const int half = warp >> 2;                         // column half drained by this warp
        const int own_tile = warp >> 2;                     // row tile whose rows this warp settles
        const int r_own = q * 32 + lane;                    // this lane's row in either tile
        const int l8 = lane & 7, grp = lane >> 3;
        const uint32_t taddr = tmem_base + (static_cast<uint32_t>(q * 32) << 16) + half * 128;
        double* Rd_cta = Rd_all + static_cast<int64_t>(blockIdx.x) * ROWS * D_;
        uint8_t* A_own = &sm.A[own_tile][0];
        const DictBounds db = dict_bounds(parts, n_parts, lane);
        uint32_t accn = 0;
        bool ok = true;
        for (int64_t pair = blockIdx.x; pair < n_pairs && ok; pair += gridDim.x) {
            float band = 0.f, norm = 0.f;                   // of row r_own of tile own_tile, scaled
            // A row's new residual to memory; its norm and band to the lane that has the row (pass p's, if set in `rows`).
            auto put_row = [&](const double (&R)[CH], int p, bool write, uint32_t rows) {
                const int r = q * 32 + 4 * p + grp;
                const Operand<CH> o = to_operand<CH>(R);
                if (write) {
                    double2* row = reinterpret_cast<double2*>(Rd_cta + static_cast<int64_t>(own_tile * TILE_M + r) * D_);
#pragma unroll
                    for (int k = 0; k < CH / 2; ++k) {
                        row[8 * k + l8] = make_double2(R[2 * k], R[2 * k + 1]);
                        // channels 2 (8 k + l8), +1: 16-byte chunk 2 k + l8 / 4 of the row, word l8 % 4 of it
                        *reinterpret_cast<uint32_t*>(A_own + swz_off(r, 2 * k + (l8 >> 2)) + (l8 & 3) * 4) = o.w[k];
                    }
                }
                const float n_o = __shfl_sync(FULL, o.norm, (lane & 3) * 8), e_o = __shfl_sync(FULL, o.err2, (lane & 3) * 8);
                if ((lane >> 2) == p && ((rows >> lane) & 1u)) {
                    norm = n_o;
                    band = row_band(n_o, e_o, db);
                }
            };
            // ---- R_0 = x ----
#pragma unroll 1
            for (int p = 0; p < 8; ++p) {
                const int r = q * 32 + 4 * p + grp;
                const int64_t m = pair * ROWS + own_tile * TILE_M + r;
                double R[CH];
                if (m < M) {
#pragma unroll
                    for (int k = 0; k < CH / 2; ++k) load_x2(X, x_dtype, m * ldx + 2 * (8 * k + l8), R[2 * k], R[2 * k + 1]);
                } else {
#pragma unroll
                    for (int k = 0; k < CH; ++k) R[k] = 0.0;
                }
                put_row(R, p, true, FULL);
            }
            fence_proxy_async_smem();
            mbar_arrive(&sm.res_ready);

            for (int g = 0; g < s && ok; ++g) {
                // ---- sweep: the largest keys of this thread's half of two rows ----
                Tops st[2] = {no_tops(), no_tops()};
                // the filter's bands of this thread's two rows: its own and the one the warp of the
                // other row tile left in shared memory
                float* band_x = reinterpret_cast<float*>(&sm.xchg[0][0]);
                band_x[own_tile * TILE_M + r_own] = band;
                epilogue_barrier();
                const float band_other = band_x[(own_tile ^ 1) * TILE_M + r_own];
                epilogue_barrier();
                const float fb_own = band > 0.f ? band * 1.0625f : -1.f;
                const float fb_other = band_other > 0.f ? band_other * 1.0625f : -1.f;
                const float fband[2] = {own_tile == 0 ? fb_own : fb_other, own_tile == 0 ? fb_other : fb_own};
                for (int t = 0; t < T && ok; ++t, ++accn) {
#pragma unroll 1
                    for (int a = 0; a < 2; ++a) {           // (rolled: one copy of the drain's code)
                        bool got = wait_bounded_suspended(&sm.acc_full[a], accn & 1, wc, 2000);
                        got = __all_sync(FULL, got);
                        if (!got) {
                            ok = false;
                            break;
                        }
                        tc_fence_after();
                        Tops qa = a ? st[1] : st[0];
                        drain<4>(taddr + a * TILE_N, qa, static_cast<uint32_t>(t), a ? fband[1] : fband[0], &sm.acc_empty[a], lane);
                        if (a)
                            st[1] = qa;
                        else
                            st[0] = qa;
                    }
                }
                // ---- bring the column halves together: warps 0-3 get row tile 0's, warps 4-7 row tile 1's ----
                auto post = [&](const Tops& o) {
                    sm.xchg[0][r_own] = o.k0;
                    sm.xchg[1][r_own] = o.k1;
                    sm.xchg[2][r_own] = o.k2;
                    sm.xchg[3][r_own] = o.k3;
                    sm.xchg[4][r_own] = o.i0 | (o.i1 << 8) | (o.i2 << 16);   // (at most 256 tiles)
                };
                Tops other = no_tops();
                auto take = [&]() {
                    const uint32_t ids = sm.xchg[4][r_own];
                    other = Tops{sm.xchg[0][r_own], sm.xchg[1][r_own], sm.xchg[2][r_own], sm.xchg[3][r_own],
                                 ids & 255u,        (ids >> 8) & 255u, ids >> 16};
                };
                if (half == 1) post(st[0]);
                if (epilogue_barrier_any(!ok || sm.abort != 0)) {
                    ok = false;
                    break;
                }
                if (half == 0) take();
                epilogue_barrier();
                if (half == 0) post(st[1]);
                epilogue_barrier();
                if (half == 1) take();
                epilogue_barrier();                         // (the exchange area is rewritten from here on)
                // The row's groups: the first three of either half, a bit in my_flags for each that is inside the band;
                // kUnknown: the fourth of a half is inside too, so there may be more than are known (NaN counts as inside).
                constexpr int kUnknown = 64;
                const Tops mine = own_tile ? st[1] : st[0];
                const float v0 = fmaxf(__uint_as_float(mine.k0 & kKeyMask), __uint_as_float(other.k0 & kKeyMask));
                int my_start[6], my_flags = 0, my_n1 = 0, my_first = 0;   // an all-zero sweep picks atom 0
                {
                    const uint32_t key[6] = {mine.k0, mine.k1, mine.k2, other.k0, other.k1, other.k2};
                    const uint32_t id[6] = {mine.i0, mine.i1, mine.i2, other.i0, other.i1, other.i2};
#pragma unroll
                    for (int i = 0; i < 6; ++i)             // (mine: the columns of this warp's half)
                        my_start[i] = static_cast<int>(id[i]) * TILE_N + (i < 3 ? half : half ^ 1) * 128 + static_cast<int>(key[i] & 31u) * G;
                    if (v0 > 0.f && N > 1) {
#pragma unroll
                        for (int i = 5; i >= 0; --i)
                            if (!(v0 - __uint_as_float(key[i] & kKeyMask) > band) && my_start[i] < N) {
                                my_flags |= 1 << i;
                                my_n1 = my_first = my_start[i];
                            }
                        if (!(v0 - __uint_as_float(mine.k3 & kKeyMask) > band) || !(v0 - __uint_as_float(other.k3 & kKeyMask) > band))
                            my_flags |= kUnknown;
                    }
                }

                // ---- the pick's atom within its group; a wave of passes' gathers in flight together ----
                bool open = false;                          // this lane's row is for fp64 to decide
                {
                    constexpr int CK = D_ / 64, WAVE = 32 / (G * CK);
#pragma unroll 1
                    for (int w0 = 0; w0 < 8; w0 += WAVE) {
                        GroupAtoms<D_> at[WAVE];
                        int n0[WAVE];
#pragma unroll
                        for (int u = 0; u < WAVE; ++u) {
                            n0[u] = __shfl_sync(FULL, my_first, 4 * (w0 + u) + grp);
                            at[u].load(dict, n0[u], N, l8);
                        }
#pragma unroll
                        for (int u = 0; u < WAVE; ++u) {
                            const int src = 4 * (w0 + u) + grp;
                            uint4 r[CK];
#pragma unroll
                            for (int j = 0; j < CK; ++j) r[j] = *reinterpret_cast<const uint4*>(A_own + swz_off(q * 32 + src, l8 + 8 * j));
                            const uint32_t in = inside(at[u].value(r, n0[u], N, l8), __shfl_sync(FULL, band, src));
                            if ((lane >> 2) == w0 + u && my_flags != 0) {
                                const uint32_t bits = (in >> (8 * (lane & 3))) & 255u;
                                if (bits != 0u) my_n1 = my_first + __ffs(bits) - 1;
                                open = __popc(bits) != 1 || (my_flags & (my_flags - 1)) != 0;   // (no value at all: a row that is not finite)
                            }
                        }
                    }
#pragma unroll 1
                    for (uint32_t left = __ballot_sync(FULL, open && (my_flags & kUnknown) == 0); left; left &= left - 1) {
                        const int src = __ffs(left) - 1;
                        int st6[6];
#pragma unroll
                        for (int i = 0; i < 6; ++i) st6[i] = __shfl_sync(FULL, my_start[i], src);
                        const int f = __shfl_sync(FULL, my_flags, src);
                        const int n = decide<D_>(D, N, Rd_cta + static_cast<int64_t>(own_tile * TILE_M + q * 32 + src) * D_, __popc(f), [&](int i) {
                            int k = f;
                            for (int j = 0; j < i; ++j) k &= k - 1;
                            const int at = __ffs(k) - 1;
                            return at == 0 ? st6[0] : at == 1 ? st6[1] : at == 2 ? st6[2] : at == 3 ? st6[3] : at == 4 ? st6[4] : st6[5];
                        }, lane);
                        if (lane == src) my_n1 = n;
                    }
                }

                // ---- settle the 32 rows of this warp, eight lanes per row, four rows per pass; the
                // next pass's residual rows and atoms are requested before this pass is worked on
                // (one copy of the code: it has to stay in the instruction cache next to the sweep) ----
                auto fetch = [&](int p, int& n, double (&R)[CH], float (&a)[CH]) {
                    const int src = 4 * p + grp;
                    n = __shfl_sync(FULL, my_n1, src);
                    const double* Rrow = Rd_cta + static_cast<int64_t>(own_tile * TILE_M + q * 32 + src) * D_;
#pragma unroll
                    for (int k = 0; k < CH / 2; ++k) {
                        const double2 v = reinterpret_cast<const double2*>(Rrow)[8 * k + l8];
                        R[2 * k] = v.x;
                        R[2 * k + 1] = v.y;
                    }
                    load_atom<CH>(D + static_cast<int64_t>(n) * D_, l8, a);
                };
                // Rows whose candidates are not all known are left for a second round: the eight warps search
                // the dictionary for each of them together (a single warp took 450 us for 4096 atoms, and
                // about one sweep of 37888 rows in eight has such a row).
                const uint32_t unknown = __ballot_sync(FULL, (my_flags & kUnknown) != 0);
                uint32_t todo = ~unknown;
#pragma unroll 1
                for (int round = 0; round < 2; ++round) {
                    if (round == 1) {
                        uint32_t* lists = &sm.xchg[0][0];   // 8 words of row masks, 256 thresholds
                        float* limit = reinterpret_cast<float*>(lists + 8);
                        Rescored* found = reinterpret_cast<Rescored*>(lists + 8 + ROWS);
                        if (lane == 0) lists[warp] = unknown;
                        if (my_flags & kUnknown) limit[warp * 32 + lane] = relative_limit(v0, band, norm, db);
                        if (!epilogue_barrier_any(unknown != 0)) break;
#pragma unroll 1
                        for (int w = 0; w < 8; ++w)
                            for (uint32_t left = lists[w]; left; left &= left - 1) {
                                const int i = __ffs(left) - 1;
                                const int64_t slot = (w >> 2) * TILE_M + (w & 3) * 32 + i;
                                const int nr = rescore_row<D_>(D, N, Rd_cta + slot * D_, limit[w * 32 + i], found, warp, lane);
                                if (w == warp && lane == i) my_n1 = nr;
                            }
                        epilogue_barrier();                 // (the next sweep's bands go to the same words)
                        todo = unknown;
                    }
                    int n;
                    double R[CH];
                    float a[CH];
                    fetch(0, n, R, a);
#pragma unroll 1
                    for (int p = 0; p < 8; ++p) {
                        int n_nx = 0;
                        double R_nx[CH];
                        float a_nx[CH];
                        if (p + 1 < 8) {
                            fetch(p + 1, n_nx, R_nx, a_nx);
                        } else {
#pragma unroll
                            for (int k = 0; k < CH; ++k) {
                                R_nx[k] = 0.0;
                                a_nx[k] = 0.f;
                            }
                        }
                        const int src = 4 * p + grp;
                        const int r = q * 32 + src;
                        const int64_t m = pair * ROWS + own_tile * TILE_M + r;
                        const bool has = (todo >> src) & 1u;
                        double ad[CH];
                        widen<CH>(a, ad);
                        const double c = group8_sum(slice_dot<CH>(R, ad));
#ifdef CSR_DEBUG_CHECKS
                        const bool was_open = __shfl_sync(FULL, open, src);
                        check_value<CH>(diag, R, a, c, __shfl_sync(FULL, v0, src), __shfl_sync(FULL, band, src), __shfl_sync(FULL, norm, src), db, l8,
                                        m < M && has && round == 0 && !was_open);
#endif
                        if (l8 == 0 && m < M && has) {
                            out_idx[m * ldc + g] = static_cast<uint16_t>(n);
                            const float cf = static_cast<float>(c);
                            if (coef_dtype == CSR_DTYPE_F16)
                                reinterpret_cast<__half*>(out_coef)[m * ldc + g] = __float2half_rn(cf);
                            else
                                reinterpret_cast<float*>(out_coef)[m * ldc + g] = cf;
                        }
                        if (g + 1 < s) {
                            if (has) {
#pragma unroll
                                for (int k = 0; k < CH; ++k) R[k] = fma(-c, ad[k], R[k]);
                            }
                            put_row(R, p, has, todo);
                        }
                        n = n_nx;
#pragma unroll
                        for (int k = 0; k < CH; ++k) {
                            R[k] = R_nx[k];
                            a[k] = a_nx[k];
                        }
                    }
                }
                if (g + 1 < s) {
                    fence_proxy_async_smem();
                    mbar_arrive(&sm.res_ready);
                }
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
}

// D (fp32, [N][d]) -> fp16 of `scale` times it, same layout, and each block's largest squared norms of an atom and of
// what the rounding took from one (see DictBounds).  The scale is the power of two that brings the largest of 32
// atoms spread over the dictionary to a norm in [1, 2): every block takes the same.  Atoms far larger than those
// overflow; the error's norm is then infinite, as it is for them, and every row is searched for in fp64.  Atoms
// that are not finite are left out of the norms: the sweep meets them as they are.  Also zeroes the words that the
// CTAs of a split row tile meet at and leave for one another.  One warp per atom.
template <int D_>
__global__ void __launch_bounds__(256)
dict_to_f16_kernel(const float* __restrict__ D, int N, uint32_t* __restrict__ out, DictPart* __restrict__ parts, uint4* __restrict__ zero,
                   int n_zero) {
    constexpr int PER = D_ / 64;                          // pairs of channels per lane
    __shared__ float red[2][8];
    __shared__ float first[8];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n_zero; i += gridDim.x * blockDim.x) zero[i] = make_uint4(0u, 0u, 0u, 0u);
    auto load = [&](int n, float2 (&v)[PER]) {
#pragma unroll
        for (int k = 0; k < PER; ++k) v[k] = __ldg(reinterpret_cast<const float2*>(D + static_cast<int64_t>(n) * D_) + lane + 32 * k);
    };
    float big = 0.f;                                      // largest magnitude, then norm relative to it: no overflow on the way
    {
        float2 v[4][PER];
#pragma unroll
        for (int j = 0; j < 4; ++j) load(static_cast<int>(static_cast<int64_t>(warp * 4 + j) * N / 32), v[j]);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            float m = 0.f, ss = 0.f;
#pragma unroll
            for (int k = 0; k < PER; ++k) m = fmaxf(m, fmaxf(fabsf(v[j][k].x), fabsf(v[j][k].y)));
            for (int o = 16; o; o >>= 1) m = fmaxf(m, __shfl_xor_sync(FULL, m, o));
            if (!(m > 0.f) || !(m <= 3.0e38f)) continue;
#pragma unroll
            for (int k = 0; k < PER; ++k) {
                const float x = v[j][k].x / m, y = v[j][k].y / m;
                ss = fmaf(x, x, fmaf(y, y, ss));
            }
            for (int o = 16; o; o >>= 1) ss += __shfl_xor_sync(FULL, ss, o);
            const float nrm = m * sqrtf(ss);
            if (nrm <= 3.0e38f) big = fmaxf(big, nrm);    // (NaN channels: not taken)
        }
    }
    if (lane == 0) first[warp] = big;
    __syncthreads();
#pragma unroll
    for (int w = 0; w < 8; ++w) big = fmaxf(big, first[w]);
    const int e = static_cast<int>(__float_as_uint(big) >> 23);           // biased exponent of the largest norm
    const float scale = e >= 2 && e <= 252 ? __uint_as_float(static_cast<uint32_t>(254 - e) << 23) : 1.f;
    float norm2 = 0.f, err2 = 0.f;
    for (int n = blockIdx.x * 8 + warp; n < N; n += gridDim.x * 8) {
        float2 v[PER];
        load(n, v);
        float nn = 0.f, ee = 0.f;
        bool finite = true;
#pragma unroll
        for (int k = 0; k < PER; ++k) {
            finite = finite && fabsf(v[k].x) <= 3.4028234e38f && fabsf(v[k].y) <= 3.4028234e38f;
            const float x = v[k].x * scale, y = v[k].y * scale;
            const __half2 h = __floats2half2_rn(x, y);
            const float2 w = __half22float2(h);
            nn = fmaf(x, x, fmaf(y, y, nn));
            ee = fmaf(x - w.x, x - w.x, fmaf(y - w.y, y - w.y, ee));
            out[static_cast<int64_t>(n) * (D_ / 2) + lane + 32 * k] = *reinterpret_cast<const uint32_t*>(&h);
        }
        for (int o = 16; o; o >>= 1) {
            nn += __shfl_xor_sync(FULL, nn, o);
            ee += __shfl_xor_sync(FULL, ee, o);
        }
        if (!__all_sync(FULL, finite)) continue;
        norm2 = fmaxf(norm2, nn);
        err2 = fmaxf(err2, ee == ee ? ee : __int_as_float(0x7f800000));
    }
    if (lane == 0) {
        red[0][warp] = norm2;
        red[1][warp] = err2;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
#pragma unroll
        for (int w = 1; w < 8; ++w) {
            norm2 = fmaxf(norm2, red[0][w]);
            err2 = fmaxf(err2, red[1][w]);
        }
        parts[blockIdx.x] = DictPart{norm2, err2, scale, 0.f};
    }
}

size_t align1k(size_t x) { return (x + 1023) / 1024 * 1024; }
int ctas_for(int64_t M) {
    const int64_t n_pairs = (M + ROWS - 1) / ROWS;
    const int64_t sms = sm_count();
    return (int)(n_pairs < sms ? n_pairs : sms);
}

template <int D_>
int run(const EncodeArgs& a, const CUtensorMap& map, const uint16_t* dict, const DictPart* parts, int n_parts, double* Rd, uint32_t* status, uint32_t* diag) {
    const size_t smem = sizeof(TcSmem<D_>);
    cudaError_t e = cudaFuncSetAttribute(encode_exact_tc_kernel<D_>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return fail(CSR_ERR_CUDA, "cudaFuncSetAttribute: %s", cudaGetErrorString(e));
    const int grid = ctas_for(a.M);
    encode_exact_tc_kernel<D_><<<grid, NT, smem, a.stream>>>(map, dict, parts, n_parts, a.D, a.X, a.x_dtype, a.ldx, a.M, a.N, a.s, a.out_idx,
                                                             a.out_coef, a.coef_dtype, a.ld_code, Rd, status, diag, options().wait_limit_ns);
    e = cudaGetLastError();
    if (e != cudaSuccess) return fail(CSR_ERR_CUDA, "encode_exact_tc launch: %s", cudaGetErrorString(e));
    return CSR_OK;
}

// How M rows are run: `pair_rows` of them as pairs of row tiles, one CTA each for the whole
// dictionary, then up to two launches of one row tile per CTA whose CTAs split the dictionary.
// A wave of pairs costs less than two waves of single row tiles (39 against 29 us an iteration at N = 1024, d = 128, plus
// 1.2 and 0.7 us per 256 atoms), and the last, partial wave is replaced wherever single tiles take less.  Up to one tile per
// SM they always do.  With more, a second launch follows, and it has to be short: its tiles' dictionary is cut into at least
// least_slices() slices each.  Measured at s = 6, d = 128 in us (warm L2, preparation included), two launches / pairs for
// 18944 + 128 k rows: N = 1024: k = 8 (16 slices) 230 / 238, 24 (six) 247 / 228; N = 4096: six 333 / 376, four 382 / 380,
// three 417 / 382; N = 8192: four 462 / 512, three 542 / 513; N = 16384: three 751 / 826, two 808 / 828; N = 32768: three
// 1459 / 1443, two 1549 / 1459.  d = 64: N = 1024 sixteen 179 / 196, ten 218 / 197; N = 2048 six 237 / 238, five 257 / 233; N = 4096
// four 307 / 323, three 313 / 292; N = 8192 three 398 / 423, two 419 / 425; N = 16384 two 662 / 714; N = 32768 two 1133 / 1314.
struct Plan {
    int64_t pair_rows;
    int64_t grid_rows[2];
};
int least_slices(int d, int N) { return N < 2048 ? 16 : N < 4096 ? 8 : N < 16384 ? 4 : d == 64 ? 2 : 3; }

Plan make_plan(int64_t M, int d, int N, bool pairs_only) {
    Plan p{M, {0, 0}};
    if (pairs_only) return p;
    const int64_t sms = sm_count(), wave = sms * ROWS;
    const int64_t rest = M % wave, tiles = (rest + TILE_M - 1) / TILE_M;
    const int64_t over = tiles > sms ? tiles - sms : 0;   // row tiles of the second launch
    if (tiles == 0 || (over > 0 && exact_grid_slices(over * TILE_M, N) < least_slices(d, N))) return p;
    p.pair_rows = M - rest;
    p.grid_rows[0] = over > 0 ? sms * TILE_M : rest;
    p.grid_rows[1] = rest - p.grid_rows[0];
    return p;
}
size_t pair_scratch_bytes(int64_t M, int d) { return (size_t)ctas_for(M) * ROWS * d * sizeof(double); }

}  // namespace

// [fp16 dictionary][its bounds][words of the two split launches][rows of the launch that is running]
size_t encode_exact_tc_scratch_bytes(int64_t M, int d, int N) {
    const Plan p = make_plan(M, d, N, false);
    size_t rows = pair_scratch_bytes(M, d), words = 0;    // (also what is needed where a split launch is refused)
    for (int64_t m : p.grid_rows) {
        if (m == 0) continue;
        const size_t b = exact_grid_scratch_bytes(m, d);
        if (b > rows) rows = b;
        words += exact_grid_word_bytes(m, N);
    }
    return align1k((size_t)N * d * 2) + align1k(kMaxDictParts * sizeof(DictPart)) + align1k(words) + rows;
}

int launch_encode_exact_tc(const EncodeArgs& a, void* scratch, uint32_t* status, uint32_t* diag, bool pairs_only) {
    if (a.M == 0) return CSR_OK;
    if ((reinterpret_cast<uintptr_t>(scratch) & 1023u) != 0)
        return fail(CSR_ERR_ALIGNMENT, "internal: exact-mode scratch not 1024-byte aligned");
    const Plan plan = make_plan(a.M, a.d, a.N, pairs_only);
    char* base = static_cast<char*>(scratch);
    void* dict = base;
    base += align1k((size_t)a.N * a.d * 2);
    DictPart* parts = reinterpret_cast<DictPart*>(base);
    base += align1k(kMaxDictParts * sizeof(DictPart));
    char* words = base;
    size_t n_words = 0;
    for (int64_t m : plan.grid_rows)
        if (m) n_words += exact_grid_word_bytes(m, a.N);
    char* rows = base + align1k(n_words);
    int n_parts = (a.N + 7) / 8;
    if (n_parts > kMaxDictParts) n_parts = kMaxDictParts;
    auto to_f16 = a.d == 128 ? dict_to_f16_kernel<128> : dict_to_f16_kernel<64>;
    to_f16<<<n_parts, 256, 0, a.stream>>>(a.D, a.N, static_cast<uint32_t*>(dict), parts, reinterpret_cast<uint4*>(words), (int)(n_words / 16));
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return fail(CSR_ERR_CUDA, "dict_to_f16 launch: %s", cudaGetErrorString(e));
    auto rows_from = [&](int64_t r0, int64_t m) {
        EncodeArgs b = a;
        b.X = static_cast<const char*>(a.X) + (size_t)r0 * a.ldx * dtype_size(a.x_dtype);
        b.out_idx = a.out_idx + r0 * a.ld_code;
        b.out_coef = static_cast<char*>(a.out_coef) + (size_t)r0 * a.ld_code * (a.coef_dtype == CSR_DTYPE_F16 ? 2 : 4);
        b.M = m;
        return b;
    };
    auto run_pairs = [&](const EncodeArgs& b) {
        CUtensorMap map;
        if (int rc = dict_map(&map, dict, a.N, a.d, TILE_N)) return rc;
        double* Rd = reinterpret_cast<double*>(rows);
        const uint16_t* copy = static_cast<const uint16_t*>(dict);
        return a.d == 128 ? run<128>(b, map, copy, parts, n_parts, Rd, status, diag) : run<64>(b, map, copy, parts, n_parts, Rd, status, diag);
    };
    if (plan.pair_rows)
        if (int rc = run_pairs(rows_from(0, plan.pair_rows))) return rc;
    int64_t r0 = plan.pair_rows;
    for (int64_t m : plan.grid_rows) {
        if (m == 0) continue;
        const EncodeArgs b = rows_from(r0, m);
        int rc = launch_encode_exact_grid(b, dict, parts, n_parts, rows, words, status, diag);
        if (rc == kGridLaunchRefused) rc = run_pairs(b);
        if (rc != CSR_OK) return rc;
        words += exact_grid_word_bytes(m, a.N);
        r0 += m;
    }
    return CSR_OK;
}

}  // namespace csr
