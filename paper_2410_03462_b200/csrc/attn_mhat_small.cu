// Masked attention over the materialised mask on small graphs (N <= GRF_MASK_SMALL): many problems of few tiles each.
//
// attn_mhat.cu gathers key and value rows by 16-byte copies and gives every (block, problem) a CTA of its own.  On a grid of 196
// patches (768 problems, m = d = 64: 77 MB, 1536 CTAs of four tiles) that took 50.4 us: issuing one tile's copies took its warps
// 1000 to 2300 cycles, and every CTA started over (5900 cycles before its first product).  Here, 25.9 us:
//   * a block's key list is a run of whole aligned tiles of 64 keys (mask_structure_kernel fills the gaps, whose mask values are
//     zeros), so key, value and query tiles are boxes of consecutive rows: one instruction of the copy engine each;
//   * rows of keys that no row of the block reaches come with such a box, and an infinity or NaN in one (a padded node's row) would
//     meet the mask's zeros: every row of the block would be NaN.  So a group whose outputs hold a NaN goes over its problems a
//     second time and clears these rows in shared memory before it multiplies.  (Clearing them always: grid of 400, 200 problems
//     20.6 -> 21.8 us, cloud of 512, 600 problems, m = 64, a third of whose places are such keys, 51.5 -> 57.5; looking at the
//     outputs instead 20.6 -> 20.6, 51.5 -> 51.8; lattice of 484, 300 problems 22.8 -> 23.7, the grid of 196 24.7 -> 24.7.  Both passes
//     in one loop needed more registers than there are: 27.2);
//   * a CTA has an SM and its tensor memory to itself and stays with one block for many problems, of which it works on four at a
//     time, each with a group of row threads, an issuing warp, a score buffer and an accumulator of its own.  Nothing is exchanged
//     between groups, and while one waits for its products the others use the issue slots.
//   warps 0-15   four groups of 128 row threads (a query = a tensor-memory lane): P = S * Mhat, in place, row sums, outputs
//   warps 16-19  one for each group: copies the queries and a ring of two key and value tiles, issues S = Q K_tile^T and
//                O += P V_tile
// What bounds it is the length of a tile's chain: by cycle counters 2500 cycles a tile and group, of which 1000 are multiplications
// (16 warps share the issue slots), 700 the first product, 350 the second, the rest hand-overs; a problem's outputs take 2000.
// Slower designs of the same kernel: two blocks a CTA that share every tile, one warp for all first products (31.7; 26.9 with what
// follows from uniform registers, below); one block, six score buffers, the groups in turn over its tiles (30.4: the row sums of four
// groups meet in every epilogue); four problems with common issuing warps (29.4: a fixed order makes the groups wait together); the
// mask in shared memory (no change).
#include <type_traits>

#include "tc_common.cuh"

namespace {

using namespace grf_tc;

constexpr int BQ = GRF_PLAN_BLOCK, KT = GRF_MASK_TILE;
constexpr int GROUPS = 4;
constexpr int THREADS = 640;
constexpr int ISSUER = 16;              // first of four

template <int M, int D> struct SmallShape {
    static constexpr int NS = 2;                                // stages of a group
    static constexpr int K_BYTES = KT * M * 2, V_BYTES = KT * D * 2, STAGE = K_BYTES + V_BYTES;
    static constexpr int Q_BYTES = BQ * M * 2;
    static constexpr int K_ROW = M * 2;
    static constexpr uint64_t K_SWIZZLE = M == 64 ? 2u : M == 32 ? 4u : 6u, V_SWIZZLE = D == 64 ? 2u : 4u;
    static constexpr int O_COL = GROUPS * KT;                   // + D per group
    static constexpr size_t SMEM = GROUPS * ((size_t)NS * STAGE + Q_BYTES) + 1024;
    static_assert(STAGE % 1024 == 0 && K_BYTES % 1024 == 0 && Q_BYTES % 1024 == 0, "swizzle phase");
    static_assert(O_COL + GROUPS * D <= 512, "tensor memory");
};

// K-major operand of rows of ROW bytes, swizzled over the row: eight-row groups follow each other; 32 bytes along a row per step
template <int ROW> __device__ __forceinline__ uint64_t row_operand(uint32_t base, uint64_t swizzle)
{
    return swizzled_desc(base, 16, 8 * ROW, swizzle);
}

template <int M, int D>
__global__ void __launch_bounds__(THREADS, 1)
mhat_small_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_k,
                  const __grid_constant__ CUtensorMap map_v, int32_t G, int32_t nblocks, int32_t N, const int32_t* __restrict__ mk_off,
                  const int32_t* __restrict__ mk_cnt, const int32_t* __restrict__ mk_key, const uint4* __restrict__ mk_val,
                  __nv_bfloat16* __restrict__ out, float* __restrict__ den_out, int* __restrict__ error_word)
{
    using Sh = SmallShape<M, D>;
    constexpr int NS = Sh::NS;
    extern __shared__ unsigned char smem_dyn[];
    // per group: kv_full, kv_done per stage, q_full, s_full, p_full, acc_done, and one to drain
    constexpr int PER_GROUP = 2 * NS + 5;
    __shared__ __align__(8) unsigned long long bars[GROUPS * PER_GROUP];
    __shared__ uint32_t tmem_slot;
    __shared__ int abort_flag;
    __shared__ int nan_seen[GROUPS];        // in outputs of a group's problems

    // what the whole warp shares is read from one lane, so that the compiler keeps it (and what follows from it) in uniform
    // registers: a tensor-pipe instruction then costs its warp 25 cycles instead of 100
    auto uniform = [](int32_t x) { return __shfl_sync(0xffffffffu, x, 0); };
    const int tid = threadIdx.x, lane = tid & 31, warp = uniform(tid >> 5);
    const uint32_t stage_base = (smem_u32(smem_dyn) + 1023u) & ~1023u;
    const uint32_t q_base = stage_base + (uint32_t)(GROUPS * NS * Sh::STAGE);
    const uint32_t bar_base = smem_u32(bars);
    auto bar = [&](int x, int what) { return bar_base + 8u * (uint32_t)(x * PER_GROUP + what); };
    auto kv_full = [&](int x, int s) { return bar(x, s); };
    auto kv_done = [&](int x, int s) { return bar(x, NS + s); };
    auto q_full = [&](int x) { return bar(x, 2 * NS); };
    auto s_full = [&](int x) { return bar(x, 2 * NS + 1); };
    auto p_full = [&](int x) { return bar(x, 2 * NS + 2); };
    auto acc_done = [&](int x) { return bar(x, 2 * NS + 3); };
    auto drain = [&](int x) { return bar(x, 2 * NS + 4); };

    // which block, and which problems: CTAs are shared out over the blocks (a lane each) in proportion to their tiles, one more each
    // for a problem's start and end (with as many CTAs as shares and more, every block gets one at least: see the launch)
    const int32_t cnt = lane < nblocks ? __ldg(mk_cnt + lane) / KT : 0, place = lane < nblocks ? __ldg(mk_off + lane) : 0;
    int32_t seen = lane < nblocks ? cnt + 1 : 0;
#pragma unroll
    for (int o = 1; o <= GRF_MASK_SMALL / BQ; o <<= 1) {
        const int32_t y = __shfl_up_sync(0xffffffffu, seen, o);
        if (lane >= o) seen += y;
    }
    const int32_t to = (int32_t)gridDim.x * seen / __shfl_sync(0xffffffffu, seen, nblocks - 1);
    const int32_t blk = __popc(__ballot_sync(0xffffffffu, lane < nblocks && to <= (int32_t)blockIdx.x));
    const int32_t from = blk > 0 ? __shfl_sync(0xffffffffu, to, blk - 1) : 0;
    const int32_t g_first = (int32_t)blockIdx.x - from, g_step = __shfl_sync(0xffffffffu, to, blk) - from;
    const int32_t T = __shfl_sync(0xffffffffu, cnt, blk), off = __shfl_sync(0xffffffffu, place, blk);     // tiles, place in the mask
    const int32_t g_round = GROUPS * g_step;                    // from a group's problem to its next one

    // An issuing warp starts its first copies before anything else is ready.
    const int x_copy = warp - ISSUER, mine = g_first + x_copy * g_step;
    const uint32_t my_stages = stage_base + (uint32_t)(x_copy * NS * Sh::STAGE), my_q = q_base + (uint32_t)(x_copy * Sh::Q_BYTES);
    int32_t first_row = 0;                                      // of the first tile
    int32_t g_copy = T > 0 ? mine : G, t_copy = 0, copied = 0, asked = 0;       // next tile to copy; tiles and queries asked for
    auto copy_tile = [&]() {
        if (g_copy >= G) return;
        const int s = copied & (NS - 1);
        const uint32_t at = my_stages + (uint32_t)(s * Sh::STAGE);
        expect_tx_elected(kv_full(x_copy, s), (uint32_t)Sh::STAGE);
        tma_load3_elected(at, &map_k, first_row + t_copy * KT, g_copy, kv_full(x_copy, s));
        tma_load3_elected(at + Sh::K_BYTES, &map_v, first_row + t_copy * KT, g_copy, kv_full(x_copy, s));
        ++copied;
        if (++t_copy == T) { t_copy = 0; g_copy += g_round; }
    };
    auto copy_queries = [&](int32_t g) {
        expect_tx_elected(q_full(x_copy), (uint32_t)Sh::Q_BYTES);
        tma_load3_elected(my_q, &map_q, blk * BQ, g, q_full(x_copy));
        ++asked;
    };
    if (warp >= ISSUER) {
        if (lane == 0) {
            for (int y = 0; y < PER_GROUP; ++y) mbar_init(bar(x_copy, y), y == 2 * NS + 2 ? 4 : 1);     // (p_full: a warp each)
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        }
        __syncwarp();
        if (g_copy < G) {
            copy_queries(mine);
            first_row = uniform(__ldg(mk_key + off) & ~(KT - 1));
            for (int s = 0; s < NS; ++s) copy_tile();
        }
    }
    if (tid == 0) abort_flag = 0;
    if (tid < GROUPS) nan_seen[tid] = 0;
    if (warp == 0) tmem_alloc(&tmem_slot, 512u);
    fence_before_sync();
    __syncthreads();
    fence_after_sync();
    const uint32_t tmem_base = (uint32_t)uniform((int32_t)tmem_slot);
    auto score_col = [&](int x) { return tmem_base + (uint32_t)(x * KT); };
    auto acc_col = [&](int x) { return tmem_base + (uint32_t)(Sh::O_COL + x * D); };
    // The keys of every tile that no row of the block reaches: bits 32 h .. 32 h + 31 of tile t in lane 2 t + h.  (Their places hold
    // another key; rows behind the last key are zeros as they come.)
    auto unreached = [&]() {
        const int32_t first = __ldg(mk_key + off) & ~(KT - 1);
        uint32_t mine_bits = 0u;
        for (int32_t e = 0; e < 2 * T; ++e) {
            const int32_t k = first + e * 32 + lane;
            const uint32_t b = __ballot_sync(0xffffffffu, k < N && __ldg(mk_key + off + e * 32 + lane) != k);
            if (lane == e) mine_bits = b;
        }
        return mine_bits;
    };
    // After a group's last problem: whether it goes over them once more (the same answer in its five warps; all of their products
    // are complete, as the row threads have waited for every accumulator)
    auto once_more = [&](int x, uint32_t& gaps) {
        __syncwarp();
        asm volatile("bar.sync %0, 160;" ::"r"(1 + x) : "memory");
        if (nan_seen[x] == 0 || *(volatile int*)&abort_flag != 0) return false;
        gaps = unreached();
        return __any_sync(0xffffffffu, gaps != 0u) != 0;
    };
    if (warp < 16) {
        // ------------------------------------------------------------ row threads
        const int x = warp >> 2;
        const int rr = (warp & 3) * 32 + lane;                  // row of the block = tensor-memory lane
        const int32_t row = blk * BQ + rr;
        const uint32_t lane_field = (uint32_t)((warp & 3) * 32) << 16;
        const uint4* mrow = mk_val + ((size_t)(off / 16) * BQ + rr) * 2;       // keys 16y .. 16y+15 of this row: mrow[2 * y * BQ], and the next
        uint4 mk[KT / 8];
        auto load_mask = [&](int32_t t) {
#pragma unroll
            for (int c = 0; c < KT / 16; ++c) ld_nc_32bytes(mrow + (size_t)(t * (KT / 16) + c) * (2 * BQ), mk[2 * c], mk[2 * c + 1]);
        };
        bool ok = true;
        uint32_t par = 0u, acc_par = 0u;                         // of this group's present tile and problem
        const uint32_t s_addr = score_col(x) + lane_field, o_addr = acc_col(x) + lane_field;
        const bool whole = ((uintptr_t)out & 31u) == 0;          // whole sectors at once where the outputs allow it
        auto problems = [&](auto again) {
            if (T > 0) load_mask(0);
            for (int32_t g = g_first + x * g_step; g < G; g += g_round) {
                uint64_t den2[2] = {0ull, 0ull};                     // row sums, four partial sums in two packed pairs
                for (int32_t t = 0; t < T; ++t) {
                    if (!mbar_wait(s_full(x), par, &abort_flag)) ok = false;
                    ok = __all_sync(0xffffffffu, ok);
                    if (!ok) break;
                    par ^= 1u;
                    fence_after_sync();
                    uint32_t sv[2][16];
                    tmem_ld16_nowait(s_addr, sv[0]);
#pragma unroll
                    for (int c16 = 0; c16 < KT / 16; ++c16) {
                        tmem_ld_wait();
                        if (c16 + 1 < KT / 16) tmem_ld16_nowait(s_addr + (uint32_t)((c16 + 1) * 16), sv[(c16 + 1) & 1]);
                        const uint32_t (&sc)[16] = sv[c16 & 1];
                        uint32_t pw[8];
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            const uint4 mm = mk[2 * c16 + h];
                            const uint32_t mw[4] = {mm.x, mm.y, mm.z, mm.w};
#pragma unroll
                            for (int e = 0; e < 4; ++e) {
                                // two masked scores at a time; the denominator adds them in fp32, before the rounding to bf16
                                const uint64_t p2 = mul2(pack2(sc[8 * h + 2 * e], sc[8 * h + 2 * e + 1]),
                                                              pack2(mw[e] << 16, mw[e] & 0xffff0000u));
                                den2[e & 1] = add2(den2[e & 1], p2);
                                float p0, p1;
                                unpack2(p2, p0, p1);
                                const __nv_bfloat162 pb = __floats2bfloat162_rn(p0, p1);
                                pw[4 * h + e] = *reinterpret_cast<const uint32_t*>(&pb);
                            }
                        }
                        tmem_st8(s_addr + (uint32_t)(c16 * 8), pw);
                    }
                    tmem_st_wait();
                    fence_before_sync();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(p_full(x));
                    // the next tile's mask values travel while the products run
                    if (t + 1 < T) load_mask(t + 1);
                    else if (T > 1 && g + g_round < G) load_mask(0);
                }
                if (ok && T > 0) ok = mbar_wait(acc_done(x), acc_par, &abort_flag);
                acc_par ^= 1u;
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) break;
                fence_after_sync();
                float d0, d1, d2, d3;
                unpack2(den2[0], d0, d1);
                unpack2(den2[1], d2, d3);
                const float den = (d0 + d1) + (d2 + d3), inv = (den != 0.0f) ? 1.0f / den : 0.0f;
                __nv_bfloat16* dst = out + ((size_t)g * N + row) * D;
                bool not_a_number = den != den;
                uint32_t o[2][16];
#pragma unroll
                for (int e = 0; e < 16; ++e) o[0][e] = o[1][e] = 0u;
#pragma unroll
                for (int c = 0; c < D / 32; ++c) {
                    if (T > 0) {
                        tmem_ld16_nowait(o_addr + (uint32_t)(c * 32), o[0]);
                        tmem_ld16_nowait(o_addr + (uint32_t)(c * 32 + 16), o[1]);
                        tmem_ld_wait();
                    }
                    // what an unreached key does it does to every lane: each of the four warps looks at its share of the columns
#pragma unroll
                    for (int h = 0; h < 2 && !decltype(again)::value; ++h) {
                        if ((warp & (D / 16 - 1)) == 2 * c + h) {
                            float y[2] = {0.0f, 0.0f};
#pragma unroll
                            for (int e = 0; e < 16; ++e) y[e & 1] += __uint_as_float(o[h][e]);
                            not_a_number |= y[0] + y[1] != y[0] + y[1];
                        }
                    }
                    if (row < N) {
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            uint32_t w[8];
#pragma unroll
                            for (int e = 0; e < 8; ++e) {
                                const __nv_bfloat162 y = __floats2bfloat162_rn(__uint_as_float(o[h][2 * e]) * inv, __uint_as_float(o[h][2 * e + 1]) * inv);
                                w[e] = *reinterpret_cast<const uint32_t*>(&y);
                            }
                            if (whole) {
                                asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
                                             ::"l"(dst + c * 32 + h * 16), "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3]), "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7]) : "memory");
                            } else {
                                uint4* half = reinterpret_cast<uint4*>(dst + c * 32 + h * 16);
                                half[0] = make_uint4(w[0], w[1], w[2], w[3]);
                                half[1] = make_uint4(w[4], w[5], w[6], w[7]);
                            }
                        }
                    }
                }
                // (read before this group hands its next tile over, which is when the accumulator is written again)
                fence_before_sync();
                if (row < N && den_out) den_out[(size_t)g * N + row] = den;
                if (!decltype(again)::value && not_a_number) nan_seen[x] = 1;
            }
        };
        uint32_t gaps;
        problems(std::false_type());
        if (once_more(x, gaps)) problems(std::true_type());
    } else {
        // ------------------------------------------------------------ copies and products of one group (the whole warp in step)
        const int x = warp - ISSUER;
        constexpr uint32_t idesc_s = instr_desc(KT, false, false);     // both operands K-major
        constexpr uint32_t idesc_o = instr_desc(D, false, true);       // V is MN-major (rows of d values)
        constexpr uint32_t ATOM = 8u * D * 2u;                         // eight value rows
        // (an issuing warp shares its scheduler with four others, so its instructions count: operands by one addition each)
        const uint64_t k_op = row_operand<Sh::K_ROW>(my_stages, Sh::K_SWIZZLE), q_op = row_operand<Sh::K_ROW>(my_q, Sh::K_SWIZZLE);
        const uint64_t v_op = swizzled_desc(my_stages + Sh::K_BYTES, ATOM, ATOM, Sh::V_SWIZZLE);
        const uint32_t k_hi = (uint32_t)(k_op >> 32), q_hi = (uint32_t)(q_op >> 32), q_lo = (uint32_t)q_op, v_hi = (uint32_t)(v_op >> 32);
        const uint32_t score = score_col(x), acc = acc_col(x);
        bool ok = true;
        auto wait = [&](uint32_t b, uint32_t parity) { return __all_sync(0xffffffffu, mbar_wait(b, parity, &abort_flag)); };
        uint32_t i = 0;                                                // tiles so far
        // Clears the rows of unreached keys in the t-th tile of a problem (`at`: the first stage's; P pieces of 16 bytes each); a
        // swizzle moves pieces inside a row only.  Neighbouring lanes take the pieces of a row, so that they meet in no bank.
        uint32_t gaps = 0u;
        auto clear = [&](int32_t t, uint32_t at, auto pieces) {
            constexpr int P = decltype(pieces)::value, ROWS = 32 / P;              // of a row; rows at a time
            const uint32_t gap[2] = {__shfl_sync(0xffffffffu, gaps, 2 * t), __shfl_sync(0xffffffffu, gaps, 2 * t + 1)};
            const uint32_t to = at + (i & (NS - 1)) * Sh::STAGE + (uint32_t)lane * 16u;
#pragma unroll
            for (int y = 0; y < 2 * P; ++y)
                if (gap[y / P] >> (y % P * ROWS + lane / P) & 1u)
                    asm volatile("st.shared.v4.b32 [%0], {%1, %1, %1, %1};" ::"r"(to + (uint32_t)(y * 512)), "r"(0u) : "memory");
        };
        // S of tile i, the t-th of its problem
        auto scores = [&](int32_t t, auto again) {
            const int s = i & (NS - 1);
            if (t == 0 && !wait(q_full(x), (uint32_t)(asked - 1) & 1u)) return false;
            if (!wait(kv_full(x, s), (i / NS) & 1u)) return false;
            if (decltype(again)::value) {
                clear(t, my_stages, std::integral_constant<int, M / 8>());
                clear(t, my_stages + Sh::K_BYTES, std::integral_constant<int, D / 8>());
                fence_async_smem();                             // the products read through the asynchronous proxy
                __syncwarp();
            }
            fence_after_sync();
            const uint32_t k_lo = (uint32_t)k_op + (uint32_t)(s * (Sh::STAGE / 16));
            mma_bf16_ss_halves<false>(score, q_lo, q_hi, k_lo, k_hi, idesc_s);
#pragma unroll
            for (int y = 1; y < M / 16; ++y) mma_bf16_ss_halves<true>(score, q_lo + 2 * y, q_hi, k_lo + 2 * y, k_hi, idesc_s);
            mma_commit(s_full(x));
            return true;
        };
        auto problems = [&](auto again) {
            ok = scores(0, again);
            for (int32_t g = mine; g < G && ok; g += g_round) {
                const bool more = g + g_round < G;
                for (int32_t t = 0; t < T && ok; ++t, ++i) {
                    const bool last = t == T - 1;
                    const int s = i & (NS - 1);
                    // the next problem's queries, as soon as this one's last scores are there
                    if (last && more) {
                        if (!wait(s_full(x), i & 1u)) { ok = false; break; }
                        copy_queries(g + g_round);
                    }
                    if (!wait(p_full(x), i & 1u)) { ok = false; break; }
                    fence_after_sync();
                    const uint32_t v_lo = (uint32_t)v_op + (uint32_t)(s * (Sh::STAGE / 16));
                    mma_bf16_ts_halves(acc, score, v_lo, v_hi, idesc_o, t > 0 ? 1u : 0u);
#pragma unroll
                    for (int y = 1; y < KT / 16; ++y) mma_bf16_ts_halves(acc, score + y * 8, v_lo + y * (2 * ATOM / 16), v_hi, idesc_o, 1u);
                    mma_commit(kv_done(x, s));
                    if (last) mma_commit(acc_done(x));
                    // P has been read and the stage is free: the next scores, and a tile for the stage
                    if (last && !more) continue;
                    if (!wait(kv_done(x, s), (i / NS) & 1u)) { ok = false; break; }
                    ++i;
                    ok = scores(last ? 0 : t + 1, again);
                    --i;
                    copy_tile();
                }
            }
        };
        if (T > 0 && mine < G) problems(std::false_type());
        if (once_more(x, gaps) && ok && T > 0 && mine < G) {            // from the first one again
            g_copy = mine;
            t_copy = 0;
            copy_queries(mine);
            for (int s = 0; s < NS; ++s) copy_tile();
            problems(std::true_type());
        }
        if (!ok) {
            // products and copies under way end before the CTA does
            mma_commit(drain(x));
            mbar_drain(drain(x), 0u, 20000000ll);
            for (int32_t y = max(0, copied - NS); y < copied; ++y) mbar_drain(kv_full(x, y & (NS - 1)), (uint32_t)(y / NS) & 1u, 20000000ll);
            if (asked > 0) mbar_drain(q_full(x), (uint32_t)(asked - 1) & 1u, 20000000ll);
        }
        __syncwarp();
    }

    fence_before_sync();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem_base, 512u);
    if (tid == 0 && abort_flag) atomicExch(error_word, 1);
}

template <int M, int D>
int launch(grf_ctx* ctx, const grf_features* feat, int32_t G, int32_t N, const void* phiQ, const void* phiK, const void* V, void* out,
           float* den_out)
{
    using Sh = SmallShape<M, D>;
    const grf_mask_dev& K = feat->mask;
    CUtensorMap mq, mk, mv;
    if (!grf_make_row_box_map(&mq, phiQ, (uint32_t)G, (uint32_t)N, M, BQ) || !grf_make_row_box_map(&mk, phiK, (uint32_t)G, (uint32_t)N, M, KT) ||
        !grf_make_row_box_map(&mv, V, (uint32_t)G, (uint32_t)N, D, KT)) return 1;
    // a CTA per SM, but no more than there are problems; at least as many as all blocks' shares, of which each has one or more: so
    // every block gets a CTA
    const int64_t least = (int64_t)K.blocks * (K.longest / KT + 1), items = (int64_t)K.blocks * G;
    int64_t ctas = items < ctx->sm_count ? items : ctx->sm_count;
    if (ctas < least) ctas = least;
    GRF_CUDA_TRY(cudaFuncSetAttribute(mhat_small_kernel<M, D>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Sh::SMEM));
    {
        grf_launch_scope scope(ctx, 9);
        mhat_small_kernel<M, D><<<(unsigned)ctas, THREADS, Sh::SMEM, ctx->stream>>>(
            mq, mk, mv, G, K.blocks, N, (const int32_t*)K.off.ptr, (const int32_t*)K.cnt.ptr, (const int32_t*)K.key.ptr,
            (const uint4*)K.val.ptr, (__nv_bfloat16*)out, den_out, ctx->error_word);
    }
    return cudaGetLastError() == cudaSuccess ? GRF_OK : GRF_ERR_CUDA;
}

}  // namespace

int grf_mhat_small_launch(grf_ctx* ctx, const grf_features* feat, int32_t G, int32_t N, int32_t m, int32_t d, const void* phiQ,
                          const void* phiK, const void* V, void* out, float* den_out)
{
#define GRF_SMALL_CASE(MM, DD) if (m == MM && d == DD) return launch<MM, DD>(ctx, feat, G, N, phiQ, phiK, V, out, den_out);
    GRF_SMALL_CASE(16, 32) GRF_SMALL_CASE(16, 64) GRF_SMALL_CASE(32, 32) GRF_SMALL_CASE(32, 64) GRF_SMALL_CASE(64, 32) GRF_SMALL_CASE(64, 64)
#undef GRF_SMALL_CASE
    return GRF_ERR_INVALID;
}
