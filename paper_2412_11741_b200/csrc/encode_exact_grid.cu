// Correctness-mode matching pursuit (paper Eq. 2-4) on the tensor cores for up to one tile of 128
// rows per SM: the dictionary is split across the CTAs that share a row tile.
//
// A CTA of encode_exact_tc.cu holds two row tiles and sweeps the whole dictionary, so a call of a
// few rows leaves all but a few SMs idle and takes s whole sweeps all the same.  Here the grid is
// (row tiles) x (slices of the dictionary), at most one CTA per SM, and all s iterations run in one
// launch.  Per iteration
//   - every CTA loads its tile's 128 residual rows as fp16 (32 KB from the L2), multiplies them with
//     its slice by the same fp16 product per correlation, and every thread keeps the
//     largest keys of its half row (drain as in encode_exact_tc.cu);
//   - the keys go to a scratch array, tagged with the iteration, and are taken from there as they come;
//   - the rows of the tile are dealt out to its CTAs, eight lanes settle a row: the largest key
//     over all slices, everything inside the band re-scored in fp64, fp64 coefficient and residual
//     update; the new fp16 rows go back to the scratch array and the CTAs meet (counter in global memory, bounded
//     wait).
// The fp64 rows, bands and fp16 rows live in L2-resident scratch.  The dictionary stages of the next
// iteration are fetched while the rows are being settled.
//
// What bounds it: with few rows the chain of dependent steps, in cycles of an iteration at 128 rows, N = 8192: the rows' load
// 1800, the sweep 2500, the keys on their way 2100, their maximum and band 1800, fp64 3000, the meeting 3500; with many
// the settling (26000 of 128 rows, beside a sweep of 23000 at N = 4096).  128 rows, N = 8192, s = 16: 180 us with three bf16
// products per correlation, 158 us with one fp16 product, 147 us with the branch-free drain, keys taken as they come
// instead of behind a second meeting and fp64 for all atoms of the group at once.  (The rows as tagged words too, instead of the
// meeting: 192 us, and 299 us when every thread polled all of its words.)
// The grid is launched cooperatively whenever a row tile has more than one CTA, so all CTAs that
// wait for one another are resident.
#include "exact_tc_common.cuh"

namespace csr {
namespace {

using namespace exact_tc;

constexpr int NT = 320;
constexpr int EPI = 256;                                  // epilogue threads
constexpr int PRODUCER_WARP = 8;
constexpr int MMA_WARP = 9;
constexpr uint32_t TMEM_COLS = 512;
constexpr int UNIT = 64;                                  // atoms per TMA box; slices are whole units
constexpr int MAX_SLICES = TILE_M;                        // at most one CTA per row
constexpr int CAND = 16;                                  // groups a row may have inside the band before the whole dictionary is re-scored

// What a CTA leaves of its keys for the others: 16 bytes written and read at once, the last word the number of the
// iteration they are for, from 1.  The reader takes them as soon as they carry the number that it waits for: no fence and
// no second trip to the L2, as after a barrier.  They are written again only when every CTA of the tile has
// passed the meeting after the settling, that is, has read them.
struct Word {
    uint32_t x, y, z, tag;
};
__device__ __forceinline__ void put_word(Word* p, const Word& v) {
    asm volatile(
        "{\n"
        ".reg .b64 lo, hi;\n"
        ".reg .b128 t;\n"
        "mov.b64 lo, {%1, %2};\n"
        "mov.b64 hi, {%3, %4};\n"
        "mov.b128 t, {lo, hi};\n"
        "st.relaxed.gpu.global.b128 [%0], t;\n"
        "}\n" ::"l"(p),
        "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.tag)
        : "memory");
}
__device__ __forceinline__ Word get_word(const Word* p) {
    Word v;
    asm volatile(
        "{\n"
        ".reg .b64 lo, hi;\n"
        ".reg .b128 t;\n"
        "ld.relaxed.gpu.global.b128 t, [%4];\n"
        "mov.b128 {lo, hi}, t;\n"
        "mov.b64 {%0, %1}, lo;\n"
        "mov.b64 {%2, %3}, hi;\n"
        "}\n"
        : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.tag)
        : "l"(p)
        : "memory");
    return v;
}
// Keys of one row over one column half of a slice: the four largest and the groups of the first three, by their first atom.
struct Entry {
    uint32_t k[4];
    uint32_t n01, n2;
};
constexpr int ENTRY_WORDS = 2;

// Takes an entry once it carries `tag`.  Bounded like every wait; false: given up.
__device__ __forceinline__ bool take_entry(const Word* p, uint32_t tag, const WaitCtx& w, Entry& e) {
    unsigned long long t0 = 0;
    for (uint32_t it = 0;; ++it) {
        const Word a = get_word(p), b = get_word(p + 1);
        if (a.tag == tag && b.tag == tag) {
            e = Entry{{a.x, a.y, b.x, b.y}, a.z, b.z};
            return true;
        }
        bool out = w.limit_ns == 0 || it >= (1u << 28);
        if (!out && (it & 15u) == 0) {
            if (*w.abort) return false;
            const unsigned long long t = globaltimer_ns();
            if (t0 == 0) t0 = t;
            out = t - t0 > w.limit_ns;
        }
        if (out) {
            *w.abort = 1;
            atomicOr(w.status, kStatusTimeout);
            return false;
        }
    }
}

template <int D_>
struct GridSmem {
    static constexpr int kStages = 5;
    static constexpr int kATileBytes = TILE_M * D_ * 2;
    static constexpr int kStageBytes = TILE_N * STAGE_CH * 2;
    alignas(1024) uint8_t A[kATileBytes];
    alignas(1024) uint8_t B[kStages][kStageBytes];
    // of the rows settled here: the largest key, the groups inside the band by their first atoms, their number
    uint32_t top_key[TILE_M];
    uint16_t cand[TILE_M][CAND];
    int n_cand[TILE_M];
    uint32_t unknown[TILE_M / 32];                        // rows settled here whose candidates are not all known
    float limit[TILE_M];                                  // ... from which |correlation| / ||R|| on an atom can be the pick
    int found_n[TILE_M];                                  // ... and what the search of the whole dictionary found
    Rescored found[EPI / 32];
    uint64_t full_b[kStages];
    uint64_t empty_b[kStages];
    uint64_t acc_full[2];
    uint64_t acc_empty[2];
    uint64_t res_ready;
    uint64_t drained;
    uint32_t tmem_base;
    volatile uint32_t abort;
};

struct GridArgs {
    const float* D;
    const void* X;
    int x_dtype;
    int64_t ldx, M;
    int N, s;
    uint16_t* out_idx;
    void* out_coef;
    int coef_dtype;
    int64_t ldc;
    double* Rd;             // [tiles * 128][d] fp64 residual rows
    uint32_t* Rh;           // [tiles * 128][d / 2] the scaled rows as fp16, two channels per word
    float2* band;           // [tiles * 128] band and norm of the scaled rows
    const uint16_t* dict;   // [N][d] the dictionary's scaled fp16 copy
    const DictPart* parts;  // [n_parts] its bounds
    int n_parts;
    Word* entries;          // [tiles][128][2 * slices][ENTRY_WORDS], tags zero at launch
    uint32_t* counters;     // [tiles * 32], zero at launch
    int slices;
    uint32_t* status;
    uint32_t* diag;
    unsigned long long wait_limit_ns;
};

// The CTAs of a row tile meet: everything their epilogue threads wrote before is visible to all of
// them afterwards.  All 256 epilogue threads call; returns false to all when any has given up.
__device__ __forceinline__ bool meet(uint32_t* counter, uint32_t target, int slices, bool ok, const WaitCtx& w) {
    if (epilogue_barrier_any(!ok || *w.abort != 0)) return false;
    if (slices > 1) {
        if (threadIdx.x == 0) {
            // (release: what the CTA's other threads wrote before the barrier above goes with it)
            asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(counter) : "memory");
            uint32_t seen;
            unsigned long long t0 = 0;
            bool in = false;
            for (uint32_t it = 0; it < (1u << 28); ++it) {
                asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(counter) : "memory");
                if (seen >= target) {
                    in = true;
                    break;
                }
                if ((it & 63u) == 0) {
                    if (*w.abort) break;
                    const unsigned long long t = globaltimer_ns();
                    if (t0 == 0) t0 = t;
                    if (t - t0 > w.limit_ns || w.limit_ns == 0) break;
                }
            }
            if (!in) {
                *w.abort = 1;
                atomicOr(w.status, kStatusTimeout);
            }
        }
        if (epilogue_barrier_any(*w.abort != 0)) return false;
    }
    return true;
}

template <int D_>
__global__ void __launch_bounds__(NT, 1)
encode_exact_grid_kernel(const __grid_constant__ CUtensorMap tmap_d, const GridArgs a) {
    using S = GridSmem<D_>;
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    if ((smem_u32(smem_raw) & 1023u) != 0) {              // the swizzled tiles need this; never seen otherwise
        if (threadIdx.x == 0) atomicOr(a.status, kStatusLayout);
        return;
    }
    S& sm = *reinterpret_cast<S*>(smem_raw);
    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    const int slices = a.slices;
    const int tile = blockIdx.x / slices, slice = blockIdx.x % slices;
    const int units = (a.N + UNIT - 1) / UNIT;
    const int u0 = static_cast<int>(static_cast<int64_t>(units) * slice / slices);
    const int u1 = static_cast<int>(static_cast<int64_t>(units) * (slice + 1) / slices);
    const int n_first = u0 * UNIT, width = (u1 - u0) * UNIT;   // this CTA's atoms (slices <= units: never empty)
    const int T = (width + TILE_N - 1) / TILE_N;          // accumulator tiles of a sweep, the last 64 .. 256 wide
    constexpr int KH = D_ / STAGE_CH;
    constexpr int STAGES = S::kStages;
    const WaitCtx wc{&sm.abort, a.status, a.wait_limit_ns};

    if (threadIdx.x == 0) {
        for (int i = 0; i < STAGES; ++i) {
            mbar_init(&sm.full_b[i], 1);
            mbar_init(&sm.empty_b[i], 1);
        }
        for (int t = 0; t < 2; ++t) {
            mbar_init(&sm.acc_full[t], 1);
            mbar_init(&sm.acc_empty[t], 8);
        }
        mbar_init(&sm.res_ready, EPI);
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
            for (int g = 0; g < a.s && ok; ++g) {
                for (int t = 0; t < T && ok; ++t) {
                    const int w = min(TILE_N, width - t * TILE_N);
                    for (int h = 0; h < KH; ++h, ++p) {
                        const int stage = p % STAGES;
                        if (!wait_bounded_suspended(&sm.empty_b[stage], ((p / STAGES) & 1) ^ 1, wc, 2000)) {
                            ok = false;
                            break;
                        }
                        // atoms past N arrive as zeros and count as bytes
                        mbar_expect_tx(&sm.full_b[stage], static_cast<uint32_t>(w) * STAGE_CH * 2);
                        for (int u = 0; u < w / UNIT; ++u)
                            tma_load_2d(&sm.B[stage][u * (UNIT * STAGE_CH * 2)], &tmap_d, h * STAGE_CH, n_first + t * TILE_N + u * UNIT,
                                        &sm.full_b[stage]);
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
            uint32_t p = 0, accn = 0;
            bool ok = true;
            for (int g = 0; g < a.s && ok; ++g) {
                if (!warp_wait_bounded(&sm.res_ready, g & 1, wc)) {
                    ok = false;
                    break;
                }
                for (int t = 0; t < T && ok; ++t, ++accn, p += KH) {
                    const int acc = accn & 1;             // the accumulators take the tiles in turn
                    const uint32_t idesc = instr_desc_f16(TILE_M, min(TILE_N, width - t * TILE_N));
                    if (!warp_wait_bounded(&sm.acc_empty[acc], ((accn >> 1) & 1) ^ 1, wc)) {
                        ok = false;
                        break;
                    }
                    const uint32_t d_tmem = tmem_d + acc * TILE_N;
                    for (int h = 0; h < KH; ++h) {
                        const uint32_t ps = p + h;
                        const int stage = ps % STAGES;
                        if (!warp_wait_bounded(&sm.full_b[stage], (ps / STAGES) & 1, wc)) {
                            ok = false;
                            break;
                        }
                        tc_fence_after();
                        const uint64_t b0 = make_smem_desc(smem_u32(&sm.B[stage][0]));
                        const uint64_t a0 = make_smem_desc(smem_u32(&sm.A[h * (TILE_M * 128)]));
                        if (h < KH - 1)
                            umma_f16_block(d_tmem, a0, b0, idesc, h, &sm.empty_b[stage]);
                        else
                            umma_f16_block(d_tmem, a0, b0, idesc, h, &sm.empty_b[stage], &sm.acc_full[acc]);
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
        constexpr int CH = D_ / 8;                        // channels per lane when eight lanes share a row
        const int q = warp & 3, half = warp >> 2;         // TMEM lane quarter, column half
        const int r_own = q * 32 + lane;                  // the row of the tile whose correlations this thread sees
        const int l8 = lane & 7, grp = lane >> 3;
        const uint32_t taddr = tmem_base + (static_cast<uint32_t>(q * 32) << 16);
        const int64_t row_base = static_cast<int64_t>(tile) * TILE_M;
        const int rows_here = static_cast<int>(a.M - row_base < TILE_M ? a.M - row_base : TILE_M);   // >= 1
        // rows settled here: slice, slice + slices, ...; the k-th by warp k % 8, lane group k / 8 % 4, pass k / 32
        const int n_own = rows_here > slice ? (rows_here - slice + slices - 1) / slices : 0;
        const int n_ent = 2 * slices;                     // entries of a row
        const DictBounds db = dict_bounds(a.parts, a.n_parts, lane);
        uint32_t* counter = a.counters + tile * 32;
        uint32_t target = 0;
        bool ok = true;
        uint32_t accn = 0;
        // An fp64 row, its scaled form as fp16 and its band to the scratch arrays, by the eight lanes of a row (all lanes
        // of the warp call; only those with `has` write).
        auto put_row = [&](const double (&R)[CH], int64_t row, bool has) {
            const Operand<CH> o = to_operand<CH>(R);
            if (!has) return;
#pragma unroll
            for (int k = 0; k < CH / 2; ++k) {
                __stcg(reinterpret_cast<double2*>(a.Rd + row * D_) + 8 * k + l8, make_double2(R[2 * k], R[2 * k + 1]));
                __stcg(a.Rh + row * (D_ / 2) + 8 * k + l8, o.w[k]);
            }
            if (l8 == 0) __stcg(a.band + row, make_float2(row_band(o.norm, o.err2, db), o.norm));
        };
        auto put_code = [&](int64_t row, int g, int n, double c) {
            a.out_idx[row * a.ldc + g] = static_cast<uint16_t>(n);
            const float cf = static_cast<float>(c);
            if (a.coef_dtype == CSR_DTYPE_F16)
                reinterpret_cast<__half*>(a.out_coef)[row * a.ldc + g] = __float2half_rn(cf);
            else
                reinterpret_cast<float*>(a.out_coef)[row * a.ldc + g] = cf;
        };
        auto load_row = [&](int64_t row, double (&R)[CH]) {
#pragma unroll
            for (int c = 0; c < CH / 2; ++c) {
                const double2 x = __ldcg(reinterpret_cast<const double2*>(a.Rd + row * D_) + 8 * c + l8);
                R[2 * c] = x.x;
                R[2 * c + 1] = x.y;
            }
        };
        // ---- R_0 = x ----
        for (int k0 = 0; k0 < n_own; k0 += EPI / 8) {
            const int k = k0 + grp * 8 + warp;
            const bool has = k < n_own;
            const int64_t row = row_base + slice + (has ? k : 0) * slices;
            double R[CH];
#pragma unroll
            for (int c = 0; c < CH / 2; ++c) load_x2(a.X, a.x_dtype, row * a.ldx + 2 * (8 * c + l8), R[2 * c], R[2 * c + 1]);
            put_row(R, row, has);
        }
        ok = meet(counter, target += slices, slices, ok, wc);

        for (int g = 0; g < a.s && ok; ++g) {
            // ---- the residual into the operand tile (rows past M: zeros, once) ----
            constexpr int CPR = D_ / 8;                   // 16-byte chunks of a row
            constexpr int PER = TILE_M * CPR / EPI;
            uint4 v[PER];
#pragma unroll
            for (int u = 0; u < PER; ++u) {
                const int f = threadIdx.x + u * EPI;
                const int r = f / CPR, c = f % CPR;
                v[u] = make_uint4(0u, 0u, 0u, 0u);
                if (r < rows_here) v[u] = __ldcg(reinterpret_cast<const uint4*>(a.Rh + (row_base + r) * (D_ / 2)) + c);
            }
            const float band_own = r_own < rows_here ? __ldcg(&a.band[row_base + r_own].x) : 0.f;
#pragma unroll
            for (int u = 0; u < PER; ++u) {
                const int f = threadIdx.x + u * EPI;
                const int r = f / CPR, c = f % CPR;
                if (g == 0 || r < rows_here) *reinterpret_cast<uint4*>(&sm.A[swz_off(r, c)]) = v[u];
            }
            fence_proxy_async_smem();
            mbar_arrive(&sm.res_ready);

            // ---- sweep of this slice: the largest keys of this thread's half row ----
            Tops top = no_tops();
            const float fband = band_own > 0.f ? band_own * 1.0625f : -1.f;
            for (int t = 0; t < T; ++t, ++accn) {
                const int acc = accn & 1;
                bool got = wait_bounded(&sm.acc_full[acc], (accn >> 1) & 1, wc);
                got = __all_sync(FULL, got);
                if (!got) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                const int w = min(TILE_N, width - t * TILE_N);
                const uint32_t ta = taddr + acc * TILE_N + half * (w / 2);
                uint64_t* back = &sm.acc_empty[acc];
                const uint32_t id = static_cast<uint32_t>(t);
                if (w == TILE_N)
                    drain<4>(ta, top, id, fband, back, lane);
                else if (w == 3 * UNIT)
                    drain<3>(ta, top, id, fband, back, lane);
                else if (w == 2 * UNIT)
                    drain<2>(ta, top, id, fband, back, lane);
                else
                    drain<1>(ta, top, id, fband, back, lane);
            }
            if (ok && r_own < rows_here) {
                auto start = [&](uint32_t key, uint32_t id) {     // (an empty key's place is never used)
                    const int t = static_cast<int>(id), w = min(TILE_N, width - t * TILE_N);
                    return static_cast<uint32_t>(n_first + t * TILE_N + half * (w / 2) + static_cast<int>(key & 31u) * G) & 0xFFFFu;
                };
                Word* e = a.entries + ((row_base + r_own) * n_ent + 2 * slice + half) * ENTRY_WORDS;
                const uint32_t tag = static_cast<uint32_t>(g) + 1u;
                put_word(e, Word{top.k0, top.k1, start(top.k0, top.i0) | (start(top.k1, top.i1) << 16), tag});
                put_word(e + 1, Word{top.k2, top.k3, start(top.k2, top.i2), tag});
            }

            // ---- this CTA's rows: largest key over all slices, then what lies inside its band ----
            // (an entry per thread and trip, at most two trips: rows x 2 slices <= 2 (127 + slices))
            constexpr int TRIPS = 2;
            Entry mine[TRIPS];
            float2 band_of[TRIPS];
            if (threadIdx.x < TILE_M / 32) sm.unknown[threadIdx.x] = 0u;
            if (threadIdx.x < TILE_M) {
                sm.top_key[threadIdx.x] = 0u;
                sm.n_cand[threadIdx.x] = 0;
            }
#pragma unroll
            for (int u = 0; u < TRIPS; ++u) {
                const int f = threadIdx.x + u * EPI;
                mine[u] = Entry{{0u, 0u, 0u, 0u}, 0u, 0u};
                band_of[u] = f < n_own * n_ent ? __ldcg(a.band + row_base + slice + f / n_ent * slices) : make_float2(0.f, 0.f);
            }
            // (a warp that has at most one row keeps it at hand: what it needs next are only the atoms)
            double R[CH];
            if (n_own <= EPI / 32) load_row(row_base + slice + min(warp, max(n_own - 1, 0)) * slices, R);
#pragma unroll
            for (int u = 0; u < TRIPS; ++u) {
                const int f = threadIdx.x + u * EPI;
                if (ok && f < n_own * n_ent)
                    ok = take_entry(a.entries + ((row_base + slice + f / n_ent * slices) * n_ent + f % n_ent) * ENTRY_WORDS,
                                    static_cast<uint32_t>(g) + 1u, wc, mine[u]);
            }
            if (epilogue_barrier_any(!ok || sm.abort != 0)) {
                ok = false;
                break;
            }
#pragma unroll
            for (int u = 0; u < TRIPS; ++u) {
                const int f = threadIdx.x + u * EPI;
                const bool in = f < n_own * n_ent;
                // (where all of a warp's entries are one row's, their maximum goes there once)
                const int k = in ? f / n_ent : -1;
                const uint32_t top = mine[u].k[0];
                if (__all_sync(FULL, k == __shfl_sync(FULL, k, 0))) {
                    const uint32_t most = __reduce_max_sync(FULL, top);
                    if (lane == 0 && in) atomicMax(&sm.top_key[k], most);
                } else if (in) {
                    atomicMax(&sm.top_key[k], top);
                }
            }
            epilogue_barrier();
#pragma unroll
            for (int u = 0; u < TRIPS; ++u) {
                const int f = threadIdx.x + u * EPI;
                if (f >= n_own * n_ent) continue;
                const int k = f / n_ent;
                const float v0 = __uint_as_float(sm.top_key[k] & kKeyMask), band = band_of[u].x;
                if (!(v0 > 0.f) || a.N == 1 || v0 - __uint_as_float(mine[u].k[0] & kKeyMask) > band) continue;
                // four of a half slice inside the band: there may be more; a band above everything: anything may be the pick
                bool full = !(v0 > band) || (mine[u].k[3] != 0u && !(v0 - __uint_as_float(mine[u].k[3] & kKeyMask) > band));
#pragma unroll
                for (int i = 0; i < 3; ++i) {
                    const uint32_t key = mine[u].k[i];
                    const uint32_t n = i == 0 ? mine[u].n01 & 0xFFFFu : i == 1 ? mine[u].n01 >> 16 : mine[u].n2;
                    if (key != 0u && !(v0 - __uint_as_float(key & kKeyMask) > band) && n < static_cast<uint32_t>(a.N)) {
                        const int slot = atomicAdd(&sm.n_cand[k], 1);
                        if (slot < CAND)
                            sm.cand[k][slot] = static_cast<uint16_t>(n);
                        else
                            full = true;
                    }
                }
                if (full) {
                    atomicOr(&sm.unknown[k >> 5], 1u << (k & 31));
                    sm.limit[k] = relative_limit(v0, band, band_of[u].y, db);   // (every writer of a row writes the same)
                }
            }
            epilogue_barrier();

            // ---- settle them: a row per warp, its lane groups an atom each ... ----
            const bool single_rows = n_own <= EPI / 32;
            if (single_rows && warp < n_own && !((sm.unknown[0] >> warp) & 1u)) {
                const int64_t row = row_base + slice + warp * slices;
                const int cnt = min(sm.n_cand[warp], CAND);   // none: an all-zero sweep (or NaN, or one atom) picks atom 0
                double best = -1.0, c = 0.0;
                float at[CH];
                int n = 0;
                if (cnt == 0) {
                    load_atom<CH>(a.D, l8, at);
                    c = group8_sum(slice_dot<CH>(R, at));
                }
#pragma unroll 1
                for (int i = 0; i < cnt; ++i) {
                    const int n0 = sm.cand[warp][i];
                    float x[2][CH];
#pragma unroll
                    for (int h = 0; h < 2; ++h) load_atom<CH>(a.D + static_cast<int64_t>(min(n0 + 4 * h + grp, a.N - 1)) * D_, l8, x[h]);
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int nh = n0 + 4 * h + grp;
                        const double ch = group8_sum(slice_dot<CH>(R, x[h]));
                        if (nh < a.N && (fabs(ch) > best || (fabs(ch) == best && nh < n))) {
                            best = fabs(ch);
                            c = ch;
                            n = nh;
#pragma unroll
                            for (int k = 0; k < CH; ++k) at[k] = x[h][k];
                        }
                    }
                }
                // the lane group that has the pick (the lowest atom among equal values) goes on with it
                double top = best;
                int low = n;
#pragma unroll
                for (int o = 8; o < 32; o <<= 1) {
                    const double ob = __shfl_xor_sync(FULL, top, o);
                    const int on = __shfl_xor_sync(FULL, low, o);
                    if (ob > top || (ob == top && on < low)) {
                        top = ob;
                        low = on;
                    }
                }
                const uint32_t won = __ballot_sync(FULL, best == top && n == low);   // (nothing but NaN: every group has atom 0 and -1)
                const bool has = won != 0u && grp == (__ffs(won) - 1) / 8;
                if (top < 0.0 && cnt > 0) {
                    load_atom<CH>(a.D, l8, at);
                    c = group8_sum(slice_dot<CH>(R, at));
                }
                if (l8 == 0 && has) put_code(row, g, n, c);
                if (g + 1 < a.s) {
                    double ad[CH];
                    widen<CH>(at, ad);
#pragma unroll
                    for (int k = 0; k < CH; ++k) R[k] = fma(-c, ad[k], R[k]);
                    put_row(R, row, has);
                }
            }
            // ---- ... or eight lanes per row; rows with unknown candidates in a second round ----
#pragma unroll 1
            for (int round = single_rows ? 1 : 0; round < 2; ++round) {
                if (round == 1) {
                    epilogue_barrier();
                    if ((sm.unknown[0] | sm.unknown[1] | sm.unknown[2] | sm.unknown[3]) == 0u) break;
#pragma unroll 1
                    for (int w = 0; w < TILE_M / 32; ++w)
                        for (uint32_t left = sm.unknown[w]; left; left &= left - 1) {
                            const int k = w * 32 + __ffs(left) - 1;
                            const int nr = rescore_row<D_>(a.D, a.N, a.Rd + (row_base + slice + k * slices) * D_, sm.limit[k], sm.found, warp, lane);
                            if (threadIdx.x == 0) sm.found_n[k] = nr;
                        }
                    epilogue_barrier();
                }
#pragma unroll 1
                for (int k0 = 0; k0 < n_own; k0 += EPI / 8) {
                    const int k = k0 + grp * 8 + warp;
                    bool has = k < n_own;
                    if (round == 1) has = has && ((sm.unknown[k >> 5] >> (k & 31)) & 1u);
                    if (!__any_sync(FULL, has)) continue;
                    const int kk = k < n_own ? k : 0;         // (lane groups without a row repeat one and write nothing)
                    const int64_t row = row_base + slice + kk * slices;
                    load_row(row, R);
                    const bool open = (sm.unknown[kk >> 5] >> (kk & 31)) & 1u;
                    const int cnt = min(sm.n_cand[kk], CAND);   // none: an all-zero sweep (or NaN, or one atom) picks atom 0
                    int n = cnt > 0 ? sm.cand[kk][0] : 0;
                    [[maybe_unused]] bool single = false;
                    if (round == 1) {                     // searched for by all warps: nothing left to decide
                        n = has ? sm.found_n[kk] : 0;
                    } else {
                        // the pick's atom within its group; where that does not decide it, fp64 over all groups, a row at a time
                        if (open) has = false;
                        GroupAtoms<D_> ga;
                        ga.load(a.dict, n, a.N, l8);
                        uint4 r[D_ / 64];
#pragma unroll
                        for (int j = 0; j < D_ / 64; ++j) r[j] = *reinterpret_cast<const uint4*>(&sm.A[swz_off(slice + kk * slices, l8 + 8 * j)]);
                        const uint32_t bits = (inside(ga.value(r, n, a.N, l8), __ldcg(&a.band[row].x)) >> (8 * grp)) & 255u;
                        single = cnt == 1 && __popc(bits) == 1;
                        if (single) n += __ffs(bits) - 1;
#pragma unroll 1
                        for (uint32_t left = __ballot_sync(FULL, has && cnt > 0 && !single && l8 == 0); left; left &= left - 1) {
                            const int src = __ffs(left) - 1;
                            const int k2 = __shfl_sync(FULL, kk, src);
                            const int found = decide<D_>(a.D, a.N, a.Rd + (row_base + slice + k2 * slices) * D_, min(sm.n_cand[k2], CAND),
                                                         [&](int i) { return static_cast<int>(sm.cand[k2][i]); }, lane);
                            if (grp == (src >> 3)) n = found;
                        }
                    }
                    float at[CH];
                    load_atom<CH>(a.D + static_cast<int64_t>(n) * D_, l8, at);
                    double ad[CH];
                    widen<CH>(at, ad);
                    const double c = group8_sum(slice_dot<CH>(R, ad));
#ifdef CSR_DEBUG_CHECKS
                    const float2 bn = __ldcg(a.band + row);
                    check_value<CH>(a.diag, R, at, c, __uint_as_float(sm.top_key[kk] & kKeyMask), bn.x, bn.y, db, l8, has && single);
#endif
                    if (l8 == 0 && has) put_code(row, g, n, c);
                    if (g + 1 < a.s) {
#pragma unroll
                        for (int c2 = 0; c2 < CH; ++c2) R[c2] = fma(-c, ad[c2], R[c2]);
                        put_row(R, row, has);
                    }
                }
            }
            if (g + 1 < a.s) ok = meet(counter, target += slices, slices, ok, wc);
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

size_t align256(size_t x) { return (x + 255) / 256 * 256; }
int tiles_of(int64_t M) { return static_cast<int>((M + TILE_M - 1) / TILE_M); }

template <int D_>
int run(const CUtensorMap& map, const GridArgs& g, int grid, cudaStream_t stream) {
    const size_t smem = sizeof(GridSmem<D_>);
    cudaError_t e = cudaFuncSetAttribute(encode_exact_grid_kernel<D_>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return fail(CSR_ERR_CUDA, "cudaFuncSetAttribute: %s", cudaGetErrorString(e));
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    cfg.gridDim = dim3((unsigned)grid, 1, 1);
    cfg.blockDim = dim3(NT, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = g.slices > 1 ? 1 : 0;                  // a lone CTA per row tile waits for nobody
    e = cudaLaunchKernelEx(&cfg, encode_exact_grid_kernel<D_>, map, g);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return kGridLaunchRefused;                        // nothing ran: the caller takes the other engine
    }
    return CSR_OK;
}

}  // namespace

int exact_grid_slices(int64_t M, int N) {
    const int tiles = tiles_of(M), units = (N + UNIT - 1) / UNIT;
    if (tiles < 1 || tiles > sm_count()) return 0;
    int s = sm_count() / tiles;
    if (s > units) s = units;
    return s < MAX_SLICES ? s : MAX_SLICES;
}

size_t exact_grid_scratch_bytes(int64_t M, int d) {
    const size_t rows = (size_t)tiles_of(M) * TILE_M;
    return rows * d * 8 + rows * d * 2 + align256(rows * 8);
}
// [counters][entries]
size_t exact_grid_word_bytes(int64_t M, int N) {
    return (size_t)tiles_of(M) * 128 + (size_t)tiles_of(M) * TILE_M * 2 * exact_grid_slices(M, N) * ENTRY_WORDS * sizeof(Word);
}

int launch_encode_exact_grid(const EncodeArgs& a, void* dict_f16, const void* dict_parts, int n_parts, void* scratch, void* words,
                             uint32_t* status, uint32_t* diag) {
    const size_t rows = (size_t)tiles_of(a.M) * TILE_M;
    char* p = static_cast<char*>(scratch);
    GridArgs g;
    g.D = a.D;
    g.X = a.X;
    g.x_dtype = a.x_dtype;
    g.ldx = a.ldx;
    g.M = a.M;
    g.N = a.N;
    g.s = a.s;
    g.out_idx = a.out_idx;
    g.out_coef = a.out_coef;
    g.coef_dtype = a.coef_dtype;
    g.ldc = a.ld_code;
    g.Rd = reinterpret_cast<double*>(p);
    p += rows * a.d * 8;
    g.Rh = reinterpret_cast<uint32_t*>(p);
    p += rows * a.d * 2;
    g.band = reinterpret_cast<float2*>(p);
    p += align256(rows * 8);
    g.dict = static_cast<const uint16_t*>(dict_f16);
    g.parts = static_cast<const DictPart*>(dict_parts);
    g.n_parts = n_parts;
    g.counters = static_cast<uint32_t*>(words);
    g.entries = reinterpret_cast<Word*>(static_cast<char*>(words) + (size_t)tiles_of(a.M) * 128);
    g.slices = exact_grid_slices(a.M, a.N);
    g.status = status;
    g.diag = diag;
    g.wait_limit_ns = options().wait_limit_ns;
    CUtensorMap map;
    if (int rc = dict_map(&map, dict_f16, a.N, a.d, UNIT)) return rc;
    const int grid = tiles_of(a.M) * g.slices;
    return a.d == 128 ? run<128>(map, g, grid, a.stream) : run<64>(map, g, grid, a.stream);
}

}  // namespace csr
