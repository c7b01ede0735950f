// Masked attention over the materialised mask on small graphs (N <= GRF_MASK_SMALL): many problems of few tiles each.
//
// attn_mhat.cu gathers key and value rows by 16-byte copies and gives every (block, problem) a CTA of its own.  On a grid of 196
// patches (768 problems, m = d = 64) that is 1536 CTAs of four tiles: 50 us for 77 MB, and neither more overlap between problems
// nor more copies ahead changed it: issuing one tile's copies took its warps 1000 to 2300 cycles, and every CTA started over (5900
// cycles before its first product).  Here
//   * a block's key list is a run of whole aligned tiles of 64 keys (mask_structure_kernel fills the gaps, whose mask values are
//     zeros), so key, value and query tiles are boxes of consecutive rows: one instruction of the copy engine each;
//   * a CTA has an SM and its tensor memory to itself and takes two blocks of one problem together, which share the key and value
//     tiles; it stays with its blocks for many problems, and its pipeline runs on from one problem to the next: queries in two
//     buffers, outputs of a problem written while the next one's first tiles are multiplied.
//   warps 0-15   row threads: for each of the two blocks two groups of 128 (a query = a tensor-memory lane), which take the
//                block's tiles in turn: P = S * Mhat, in place, and row sums; each writes half of the output columns
//   warp 16      copies: queries of a problem, then its key and value tiles, into a ring of stages
//   warp 17      issues S = Q K_tile^T for both blocks, three score buffers each
//   warps 18, 19 issue O += P V_tile, one block each
// Tensor memory: two blocks of three score buffers of 64 columns and D columns of output.
#include "tc_common.cuh"

namespace {

using namespace grf_tc;

constexpr int BQ = GRF_PLAN_BLOCK, KT = GRF_MASK_TILE;
constexpr int NB = 3;                   // score buffers per block
constexpr int DEN_SLOTS = 4;            // a group's row sums wait here for the other group's epilogue, which may be this far behind
constexpr int THREADS = 640;
constexpr int COPIER = 16, ISSUER_S = 17, ISSUER_O = 18;

template <int M, int D> struct SmallShape {
    static constexpr int NS = 6;
    static constexpr int K_BYTES = KT * M * 2, V_BYTES = KT * D * 2, STAGE = K_BYTES + V_BYTES;
    static constexpr int Q_BYTES = BQ * M * 2;                  // of one block
    static constexpr int K_ROW = M * 2;
    static constexpr uint64_t K_SWIZZLE = M == 64 ? 2u : M == 32 ? 4u : 6u, V_SWIZZLE = D == 64 ? 2u : 4u;
    static constexpr int O_COL = 2 * NB * KT;                   // + D per block
    static constexpr size_t SMEM = (size_t)NS * STAGE + 4 * Q_BYTES + 1024;
    static_assert(STAGE % 1024 == 0 && K_BYTES % 1024 == 0 && Q_BYTES % 1024 == 0, "swizzle phase");
    static_assert(O_COL + 2 * D <= 512, "tensor memory");
};

// K-major operand of rows of ROW bytes, swizzled over the row: eight-row groups follow each other; 32 bytes along a row per step
template <int ROW> __device__ __forceinline__ uint64_t row_operand(uint32_t base, int step, uint64_t swizzle)
{
    return swizzled_desc(base + (uint32_t)step * 32u, 16, 8 * ROW, swizzle);
}

__device__ __forceinline__ void st_32bytes(void* p, const uint32_t (&w)[8])
{
    asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
                 ::"l"(p), "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3]), "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7]) : "memory");
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
    // kv_full, kv_empty per stage; q_full, q_empty per query buffer; two drain barriers for each issuer; per block: s_full, p_full,
    // s_free per score buffer, acc_done, acc_free, den_ready per group and slot
    constexpr int PER_BLOCK = 3 * NB + 2 + 2 * DEN_SLOTS;
    __shared__ __align__(8) unsigned long long bars[2 * NS + 4 + 3 + 2 * PER_BLOCK];
    __shared__ uint32_t tmem_slot;
    __shared__ int abort_flag;
    __shared__ float den_part[2][2][DEN_SLOTS][BQ];

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t stage_base = (smem_u32(smem_dyn) + 1023u) & ~1023u;
    const uint32_t q_base = stage_base + (uint32_t)(NS * Sh::STAGE);
    const uint32_t bar_base = smem_u32(bars);
    auto kv_full = [&](int s) { return bar_base + 8u * (uint32_t)s; };
    auto kv_empty = [&](int s) { return bar_base + 8u * (uint32_t)(NS + s); };
    auto q_full = [&](int b) { return bar_base + 8u * (uint32_t)(2 * NS + b); };
    auto q_empty = [&](int b) { return bar_base + 8u * (uint32_t)(2 * NS + 2 + b); };
    auto drain = [&](int w) { return bar_base + 8u * (uint32_t)(2 * NS + 4 + w); };
    auto blk_bar = [&](int b, int x) { return bar_base + 8u * (uint32_t)(2 * NS + 7 + b * PER_BLOCK + x); };
    auto s_full = [&](int b, int i) { return blk_bar(b, i); };
    auto p_full = [&](int b, int i) { return blk_bar(b, NB + i); };
    auto s_free = [&](int b, int i) { return blk_bar(b, 2 * NB + i); };
    auto acc_done = [&](int b) { return blk_bar(b, 3 * NB); };
    auto acc_free = [&](int b) { return blk_bar(b, 3 * NB + 1); };
    auto den_ready = [&](int b, int grp, int k) { return blk_bar(b, 3 * NB + 2 + grp * DEN_SLOTS + k % DEN_SLOTS); };

    // which two blocks, and which problems: CTAs are shared out over the pairs of blocks in proportion to their tiles, one more
    // each for a problem's start and end (with as many CTAs as pairs and more, every pair gets one at least: see the launch)
    const int32_t pairs = (nblocks + 1) / 2;
    int32_t pair = 0, g_first = 0, g_step = 1;
    {
        int32_t total = 0, seen = 0, from = 0, to = 0;
        for (int32_t b = 0; b < nblocks; ++b) total += __ldg(mk_cnt + b) / KT + 1;
        for (pair = 0; pair < pairs; ++pair) {
            for (int32_t b = 2 * pair; b < min(nblocks, 2 * pair + 2); ++b) seen += __ldg(mk_cnt + b) / KT + 1;
            to = (int32_t)((int64_t)gridDim.x * seen / total);
            if ((int32_t)blockIdx.x < to) break;
            from = to;
        }
        g_first = (int32_t)blockIdx.x - from;
        g_step = to - from;
    }
    const int nb = min(2, nblocks - 2 * pair);                  // blocks of this CTA
    int32_t T[2] = {0, 0}, lo[2] = {0, 0}, off[2] = {0, 0};     // tiles, first tile, place in the mask
#pragma unroll
    for (int b = 0; b < 2; ++b)
        if (b < nb) {
            off[b] = __ldg(mk_off + 2 * pair + b);
            T[b] = __ldg(mk_cnt + 2 * pair + b) / KT;
            if (T[b] > 0) lo[b] = __ldg(mk_key + off[b]) / KT;
        }
    const int32_t t_lo = T[0] == 0 ? lo[1] : T[1] == 0 ? lo[0] : min(lo[0], lo[1]);
    const int32_t t_hi = max(T[0] > 0 ? lo[0] + T[0] : t_lo, T[1] > 0 ? lo[1] + T[1] : t_lo);
    const int32_t g_end = t_hi > t_lo ? G : 0;                  // no tiles: nothing to copy or multiply

    if (tid == 0) {
        for (int s = 0; s < NS; ++s) { mbar_init(kv_full(s), 1); mbar_init(kv_empty(s), (uint32_t)nb); }
        for (int b = 0; b < 2; ++b) {
            mbar_init(q_full(b), 1);
            mbar_init(q_empty(b), 1);
            for (int i = 0; i < NB; ++i) { mbar_init(s_full(b, i), 1); mbar_init(p_full(b, i), 4); mbar_init(s_free(b, i), 1); }
            mbar_init(acc_done(b), 1);
            mbar_init(acc_free(b), 8);
            for (int x = 0; x < DEN_SLOTS; ++x) { mbar_init(den_ready(b, 0, x), 4); mbar_init(den_ready(b, 1, x), 4); }
        }
        for (int w = 0; w < 3; ++w) mbar_init(drain(w), 1);
        abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == ISSUER_S) tmem_alloc(&tmem_slot, 512u);
    fence_before_sync();
    __syncthreads();
    fence_after_sync();
    const uint32_t tmem_base = tmem_slot;
    auto score_col = [&](int b, int i) { return tmem_base + (uint32_t)((b * NB + i) * KT); };

    if (warp < 16) {
        // ------------------------------------------------------------ row threads
        const int b = warp >> 3, grp = warp >> 2 & 1, other = grp ^ 1;
        const int rr = (warp & 3) * 32 + lane;                  // row of the block = tensor-memory lane
        const int32_t row = (2 * pair + b) * BQ + rr, tiles = b ? T[1] : T[0];
        const uint32_t lane_field = (uint32_t)((warp & 3) * 32) << 16;
        const uint4* mrow = mk_val + ((size_t)((b ? off[1] : off[0]) / 16) * BQ + rr) * 2;    // keys 16x .. 16x+15 of this row: mrow[2 * x * BQ], and the next
        const bool mine = b < nb;
        uint4 mk[KT / 8];
        auto load_mask = [&](int32_t t) {
#pragma unroll
            for (int c = 0; c < KT / 16; ++c) ld_nc_32bytes(mrow + (size_t)(t * (KT / 16) + c) * (2 * BQ), mk[2 * c], mk[2 * c + 1]);
        };
        bool ok = true;
        // outputs of problem number k: this group's half of the columns
        auto epilogue = [&](int k, int32_t g, float den) {
            if (ok && other < tiles) {
                ok = mbar_wait(den_ready(b, other, k), (uint32_t)(k / DEN_SLOTS) & 1u, &abort_flag);
                den += den_part[b][other][k % DEN_SLOTS][rr];
            }
            if (ok && tiles > 0) ok = mbar_wait(acc_done(b), (uint32_t)k & 1u, &abort_flag);
            ok = __all_sync(0xffffffffu, ok);
            fence_after_sync();
            uint32_t r[D / 2];
#pragma unroll
            for (int e = 0; e < D / 2; ++e) r[e] = 0u;
            if (ok && tiles > 0) {
#pragma unroll
                for (int c = 0; c < D / 32; ++c)
                    tmem_ld16_nowait(tmem_base + lane_field + (uint32_t)(Sh::O_COL + b * D + grp * (D / 2) + c * 16), *reinterpret_cast<uint32_t(*)[16]>(r + c * 16));
                tmem_ld_wait();
            }
            fence_before_sync();
            __syncwarp();
            if (lane == 0) mbar_arrive(acc_free(b));
            if (row < N && ok) {
                const float inv = (den != 0.0f) ? 1.0f / den : 0.0f;
                if (grp == 0 && den_out) den_out[(size_t)g * N + row] = den;
                __nv_bfloat16* dst = out + ((size_t)g * N + row) * D + grp * (D / 2);
#pragma unroll
                for (int c = 0; c < D / 32; ++c) {
                    uint32_t w[8];
#pragma unroll
                    for (int e = 0; e < 8; ++e) {
                        const __nv_bfloat162 h = __floats2bfloat162_rn(__uint_as_float(r[c * 16 + 2 * e]) * inv, __uint_as_float(r[c * 16 + 2 * e + 1]) * inv);
                        w[e] = *reinterpret_cast<const uint32_t*>(&h);
                    }
                    if (D == 64) {
                        st_32bytes(dst + c * 16, w);
                    } else {
                        reinterpret_cast<uint4*>(dst + c * 16)[0] = make_uint4(w[0], w[1], w[2], w[3]);
                        reinterpret_cast<uint4*>(dst + c * 16)[1] = make_uint4(w[4], w[5], w[6], w[7]);
                    }
                }
            }
        };
        int k = 0;
        bool due = false;                                        // the former problem's outputs are still to be written
        float den = 0.0f;
        if (mine && grp < tiles) load_mask(grp);
        for (int32_t g = mine ? g_first : G; g < G; g += g_step, ++k) {
            uint64_t den2[2] = {0ull, 0ull};                     // row sums, four partial sums in two packed pairs
            for (int32_t t = grp; t < tiles; t += 2) {
                const uint32_t i = (uint32_t)(k * tiles + t), use = i / NB, buf = i - use * NB;
                if (!mbar_wait(s_full(b, buf), use & 1u, &abort_flag)) ok = false;
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) break;
                fence_after_sync();
                const uint32_t s_addr = score_col(b, buf) + lane_field;
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
                            const uint64_t p2 = mul_f32x2(pack_f32x2(sc[8 * h + 2 * e], sc[8 * h + 2 * e + 1]),
                                                          pack_f32x2(mw[e] << 16, mw[e] & 0xffff0000u));
                            den2[e & 1] = add_f32x2(den2[e & 1], p2);
                            float p0, p1;
                            unpack_f32x2(p2, p0, p1);
                            const __nv_bfloat162 pb = __floats2bfloat162_rn(p0, p1);
                            pw[4 * h + e] = *reinterpret_cast<const uint32_t*>(&pb);
                        }
                    }
                    tmem_st8(s_addr + (uint32_t)(c16 * 8), pw);
                }
                // this group's next tile, of this problem or the next: its mask values travel while the products run
                if (t + 2 < tiles) load_mask(t + 2);
                else if (tiles > 2 && g + g_step < G) load_mask(grp);
                tmem_st_wait();
                fence_before_sync();
                __syncwarp();
                if (lane == 0) mbar_arrive(p_full(b, buf));
                // the former problem's outputs: by now its last product is complete
                if (due) { epilogue(k - 1, g - g_step, den); due = false; }
            }
            if (!ok) break;
            if (due) epilogue(k - 1, g - g_step, den);
            {
                float d0, d1, d2, d3;
                unpack_f32x2(den2[0], d0, d1);
                unpack_f32x2(den2[1], d2, d3);
                den = (d0 + d1) + (d2 + d3);
            }
            if (grp < tiles) {
                den_part[b][grp][k % DEN_SLOTS][rr] = den;
                __syncwarp();
                if (lane == 0) mbar_arrive(den_ready(b, grp, k));
            }
            due = true;
        }
        if (due && ok) epilogue(k - 1, g_first + (k - 1) * g_step, den);
    } else if (warp == COPIER) {
        // ------------------------------------------------------------ copies (the whole warp runs the loop in step)
        bool ok = true;
        int s = 0, n = 0;
        uint32_t use = 0;                                        // of stage s
        int32_t copied = 0, asked = 0;                           // tiles, problems' queries
        for (int32_t g = g_first; g < g_end && ok; g += g_step, ++n) {
            const int qb = n & 1;
            if (n >= 2 && !__all_sync(0xffffffffu, mbar_wait(q_empty(qb), (uint32_t)((n >> 1) - 1) & 1u, &abort_flag))) { ok = false; break; }
            expect_tx_elected(q_full(qb), (uint32_t)(nb * Sh::Q_BYTES));
            ++asked;
            for (int b = 0; b < nb; ++b)
                tma_load3_elected(q_base + (uint32_t)((qb * 2 + b) * Sh::Q_BYTES), &map_q, (2 * pair + b) * BQ, g, q_full(qb));
            for (int32_t t = t_lo; t < t_hi; ++t) {
                if (use > 0 && !__all_sync(0xffffffffu, mbar_wait(kv_empty(s), (use - 1) & 1u, &abort_flag))) { ok = false; break; }
                expect_tx_elected(kv_full(s), (uint32_t)Sh::STAGE);
                const uint32_t k_st = stage_base + (uint32_t)(s * Sh::STAGE);
                tma_load3_elected(k_st, &map_k, t * KT, g, kv_full(s));
                tma_load3_elected(k_st + Sh::K_BYTES, &map_v, t * KT, g, kv_full(s));
                ++copied;
                if (++s == NS) { s = 0; ++use; }
            }
        }
        if (!ok) {                                               // no copy outlives the CTA
            for (int x = 0; x < NS && x < copied; ++x) {
                if (--s < 0) { s = NS - 1; --use; }
                mbar_drain(kv_full(s), use & 1u, 20000000ll);
            }
            for (int x = max(0, asked - 2); x < asked; ++x) mbar_drain(q_full(x & 1), (uint32_t)(x >> 1) & 1u, 20000000ll);
        }
        __syncwarp();
    } else if (warp == ISSUER_S) {
        // ------------------------------------------------------------ S = Q K_tile^T (the whole warp runs the loop in step)
        constexpr uint32_t idesc_s = instr_desc(KT, false, false);     // both operands K-major
        bool ok = true;
        int s = 0, n = 0;
        uint32_t use = 0, count[2] = {0, 0};                           // uses of stage s; tiles of each block so far
        for (int32_t g = g_first; g < g_end && ok; g += g_step, ++n) {
            const int qb = n & 1;
            if (!__all_sync(0xffffffffu, mbar_wait(q_full(qb), (uint32_t)(n >> 1) & 1u, &abort_flag))) { ok = false; break; }
            for (int32_t t = t_lo; t < t_hi && ok; ++t) {
                if (!__all_sync(0xffffffffu, mbar_wait(kv_full(s), use & 1u, &abort_flag))) { ok = false; break; }
                const uint32_t k_st = stage_base + (uint32_t)(s * Sh::STAGE);
#pragma unroll
                for (int b = 0; b < 2; ++b) {
                    if (!ok || t < lo[b] || t >= lo[b] + T[b]) continue;
                    const uint32_t round = count[b] / NB, buf = count[b] - round * NB;
                    // the score buffer is free once the second product of the tile three back, which read its P, is complete
                    if (round > 0 && !__all_sync(0xffffffffu, mbar_wait(s_free(b, buf), (round - 1) & 1u, &abort_flag))) { ok = false; continue; }
                    fence_after_sync();
#pragma unroll
                    for (int x = 0; x < M / 16; ++x)
                        mma_bf16_ss(score_col(b, buf), row_operand<Sh::K_ROW>(q_base + (uint32_t)((qb * 2 + b) * Sh::Q_BYTES), x, Sh::K_SWIZZLE),
                                    row_operand<Sh::K_ROW>(k_st, x, Sh::K_SWIZZLE), idesc_s, x > 0 ? 1u : 0u);
                    mma_commit(s_full(b, buf));
                    ++count[b];
                }
                if (++s == NS) { s = 0; ++use; }
            }
            if (ok) mma_commit(q_empty(qb));
        }
        if (!ok) {
            mma_commit(drain(0));
            mbar_drain(drain(0), 0u, 20000000ll);
        }
        __syncwarp();
    } else {
        // ------------------------------------------------------------ O += P V_tile (the whole warp runs the loop in step)
        const int b = warp - ISSUER_O;
        const int32_t b_lo = b ? lo[1] : lo[0], b_hi = b_lo + (b ? T[1] : T[0]);
        constexpr uint32_t idesc_o = instr_desc(D, false, true);       // V is MN-major (rows of d values)
        constexpr uint32_t ATOM = 8u * D * 2u;                         // eight value rows
        bool ok = true;
        int s = 0, n = 0;
        uint32_t use = 0, count = 0;
        for (int32_t g = b < nb ? g_first : g_end; g < g_end && ok; g += g_step, ++n) {
            for (int32_t t = t_lo; t < t_hi; ++t) {
                if (!__all_sync(0xffffffffu, mbar_wait(kv_full(s), use & 1u, &abort_flag))) { ok = false; break; }
                if (t < b_lo || t >= b_hi) {                           // a tile of the other block alone
                    if (lane == 0) mbar_arrive(kv_empty(s));
                    __syncwarp();
                } else {
                    const uint32_t round = count / NB, buf = count - round * NB;
                    if (!__all_sync(0xffffffffu, mbar_wait(p_full(b, buf), round & 1u, &abort_flag))) { ok = false; break; }
                    // the former problem's outputs have been read
                    if (t == b_lo && n > 0 && !__all_sync(0xffffffffu, mbar_wait(acc_free(b), (uint32_t)(n - 1) & 1u, &abort_flag))) { ok = false; break; }
                    fence_after_sync();
                    const uint32_t v_st = stage_base + (uint32_t)(s * Sh::STAGE) + Sh::K_BYTES;
#pragma unroll
                    for (int x = 0; x < KT / 16; ++x)
                        mma_bf16_ts(tmem_base + (uint32_t)(Sh::O_COL + b * D), score_col(b, buf) + (uint32_t)x * 8u,
                                    swizzled_desc(v_st + (uint32_t)x * 2u * ATOM, ATOM, ATOM, Sh::V_SWIZZLE), idesc_o, (t > b_lo || x > 0) ? 1u : 0u);
                    mma_commit(kv_empty(s));
                    mma_commit(s_free(b, buf));
                    ++count;
                }
                if (++s == NS) { s = 0; ++use; }
            }
            if (ok && b_hi > b_lo) mma_commit(acc_done(b));
        }
        if (!ok) {
            mma_commit(drain(1 + b));
            mbar_drain(drain(1 + b), 0u, 20000000ll);
        }
        __syncwarp();
    }

    fence_before_sync();
    __syncthreads();
    if (warp == ISSUER_S) tmem_dealloc(tmem_base, 512u);
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
        !grf_make_row_box_map(&mv, V, (uint32_t)G, (uint32_t)N, D, KT)) return GRF_ERR_CUDA;
    GRF_CUDA_TRY(cudaFuncSetAttribute(mhat_small_kernel<M, D>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Sh::SMEM));
    const int32_t pairs = (K.blocks + 1) / 2;
    // a CTA per SM, but no more than there are problems; at least as many as all blocks' shares, of which a pair has one or more:
    // so every pair gets a CTA
    const int64_t least = (int64_t)K.blocks * (K.longest / KT + 1), items = (int64_t)pairs * G;
    int64_t ctas = items < ctx->sm_count ? items : ctx->sm_count;
    if (ctas < least) ctas = least;
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
