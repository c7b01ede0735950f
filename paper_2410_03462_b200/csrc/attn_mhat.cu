// Masked attention with the mask estimate materialised (Eqs. 1-2 with Mhat = Phi Psi^T, Sec. 3.3), bf16 storage.
//
// Instead of going through the per-node states of Eq. 12, the sparse product Mhat = Phi Psi^T is formed once per
// feature object and the attention is evaluated from its definition,
//     out_i = sum_j Mhat_ij (phi(q_i) . phi(k_j)) v_j / sum_j Mhat_ij (phi(q_i) . phi(k_j)),
// over the non-zeros of Mhat only.  On graphs whose node numbering keeps neighbours together, the rows of a block
// of 128 consecutive queries reach a few thousand keys between them and about a quarter of that block of Mhat is
// non-zero: dense enough for the tensor cores.  Per block the mask is stored densely (bf16) over the block's key
// list, and one CTA per (block, problem) runs a two-product pipeline over tiles of 64 keys:
//     S = phi(Q_blk) phi(K_tile)^T   (tcgen05, accumulator in tensor memory)
//     P = S * Mhat_tile              (row threads: tensor memory -> registers -> tensor memory, bf16)
//     O += P V_tile                  (tcgen05, P read from tensor memory)
// and the row sums of P (taken in fp32, before its rounding) give the denominators.  Key and value rows are gathered
// by key index with 16-byte asynchronous copies: value rows into the 128-byte-swizzled MN-major operand layout,
// key-feature rows into the unswizzled K-major layout.
//
// Building the mask (once per feature object): the key list of a block is the union of the rows of Psi^T over the
// block's node list (the block plan of Phi); the values are accumulated row by row, one warp per row, in ascending
// order of the node l, each lane owning distinct keys, so the sums are reproducible without atomics.
#include <type_traits>

#include "tc_common.cuh"

namespace {

using namespace grf_tc;

constexpr int BQ = GRF_PLAN_BLOCK;      // queries per block
constexpr int KT = GRF_MASK_TILE;       // keys per tile

// ---------------------------------------------------------------------------------------------------
// Structure of the mask: a cluster of CTAs per block of rows (see below), everything that does not depend on values.
//   keys       the union of Psi^T's rows over the block's node list, marked in a bitmap (a bit is looked at before it is
//              set: a block reaches each of its keys about thirty times), counted, and written as the block's key list,
//              padded to whole tiles with the last key (whose mask values there are zeros); on graphs of GRF_MASK_SMALL nodes
//              and fewer the list has a place for every key of the aligned tiles from the first to the last one reached, and
//              places of keys that no row of the block reaches are padding as well (a key of the block, zeros in the mask):
//              what such a key's rows of K and V hold must not matter;
//   positions  for every node of the list the accumulator (by position in the key list) of each of its keys, 16 bits each;
//              for every non-zero Phi_il of the block's rows where node l's positions begin.
// A warp takes 32 nodes at a time (lane x holds node x's extent in Psi^T) and fetches the keys of two nodes together.
// Blocks take their places in the lists by atomic additions, so the order of the blocks inside the arrays varies; nothing
// depends on it.  A block whose part does not fit the room that the host has made writes none of it: the totals tell
// the host how much is needed.  The last CTA to finish orders the blocks by decreasing key count.
// One kernel for all of this, at the N = 32768 cloud: 237 us in five kernels and two prefix sums before, 160 us with a CTA per
// block, 150 now (profiled: issue slots 75 % busy, 65 % of the warps there; the blocks with the longest lists end last).
// A cluster of C CTAs builds each block (one CTA a block leaves SMs idle where there are few): they share out the nodes, merge their
// key bitmaps through each other's shared memory, and share out list, positions and non-zeros; ranks and prefix sums are formed by
// each for itself (cheaper than asking).  Structure and values together, us, one CTA a block / cluster: clouds of 2048 (8 CTAs) 91 / 62, 4096 (8) 124 / 89,
// 6000 (4) 167 / 127, 9000 (4) 203 / 166, 22000 (2) 419 / 393.

constexpr int MS_THREADS = 768;

struct grf_mask_totals {                // zeroed before the launch; host[0..2] = entries, positions, longest list
    unsigned long long entries, positions;
    int32_t longest, finished;
};

// exclusive prefix sum of one value per thread over MS_THREADS threads; *total (shared) = the sum
__device__ __forceinline__ int32_t ms_scan(int32_t x, int32_t* warp_sums, int32_t* total)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int32_t inc = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int32_t y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
    }
    if (lane == 31) warp_sums[warp] = inc;
    __syncthreads();
    if (warp == 0) {
        int32_t w = lane < MS_THREADS / 32 ? warp_sums[lane] : 0;
        const int32_t own = w;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int32_t y = __shfl_up_sync(0xffffffffu, w, o);
            if (lane >= o) w += y;
        }
        warp_sums[lane] = w - own;
        if (lane == 31) *total = w;
    }
    __syncthreads();
    const int32_t r = inc - x + warp_sums[warp];
    __syncthreads();
    return r;
}

// bits set before each word of a bitmap; returns their number
__device__ __forceinline__ int32_t ms_ranks(const uint32_t* bits, int32_t* before, int32_t words, int32_t* warp_sums, int32_t* total)
{
    const int32_t per = (words + MS_THREADS - 1) / MS_THREADS;
    const int32_t w0 = min(words, (int32_t)threadIdx.x * per), w1 = min(words, w0 + per);
    int32_t mine = 0;
    for (int32_t x = w0; x < w1; ++x) mine += __popc(bits[x]);
    int32_t run = ms_scan(mine, warp_sums, total);
    for (int32_t x = w0; x < w1; ++x) { before[x] = run; run += __popc(bits[x]); }
    __syncthreads();
    return *total;
}

// Where the accumulator of position p lies: the 16-byte quarters of a group of sixteen change places from pair to pair of
// groups, so that lanes which read whole neighbouring groups meet in no bank.
__host__ __device__ __forceinline__ uint32_t mask_slot(uint32_t p) { return p ^ ((p >> 5 & 3u) << 2); }

// Cluster of CTAs on one block: barrier, and a word of another CTA's shared memory (the same place as `local` in this one's).
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ uint32_t cluster_ld(const void* local, uint32_t rank)
{
    uint32_t a, x;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_u32(local)), "r"(rank));
    asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(x) : "r"(a) : "memory");
    return x;
}

template <int C>
__global__ void __launch_bounds__(MS_THREADS, 2) __cluster_dims__(C, 1, 1)
mask_structure_kernel(int32_t N, int32_t Nk, int32_t R, const int32_t* __restrict__ phi_rowptr, const int32_t* __restrict__ phi_col,
                      const int32_t* __restrict__ plan_off, const int32_t* __restrict__ plan_cnt,
                      const int32_t* __restrict__ plan_col, const int32_t* __restrict__ t_rowptr,
                      const int32_t* __restrict__ t_col, int64_t key_room, int64_t pos_room, uint32_t* __restrict__ bits_out,
                      int32_t* node_off, int32_t* __restrict__ mk_off, int32_t* __restrict__ mk_cnt,
                      int32_t* __restrict__ mk_key, unsigned short* __restrict__ pos16, int32_t* __restrict__ phi_pos,
                      grf_mask_totals* totals, int32_t* host)
{
    extern __shared__ uint32_t smem_ms[];       // key bitmap, its ranks, node bitmap, its ranks
    __shared__ int32_t warp_sums[32];
    __shared__ int32_t total, last_cta;
    __shared__ unsigned long long base_keys, base_pos;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int32_t part = (int32_t)(blockIdx.x % C);                             // of the block's CTAs
    const int32_t blk = blockIdx.x / C, nblocks = gridDim.x / C;
    const int32_t wk = (Nk + 31) >> 5, wr = (R + 31) >> 5;
    uint32_t* kbits = smem_ms;
    int32_t* kbefore = reinterpret_cast<int32_t*>(smem_ms + wk);
    uint32_t* nbits = smem_ms + 2 * wk;
    int32_t* nbefore = reinterpret_cast<int32_t*>(smem_ms + 2 * wk + wr);
    for (int32_t x = tid; x < wk; x += MS_THREADS) kbits[x] = 0u;
    for (int32_t x = tid; x < wr; x += MS_THREADS) nbits[x] = 0u;
    __syncthreads();
    const int32_t uoff = plan_off[blk], ucnt = plan_cnt[blk];
    const int32_t* ulist = plan_col + uoff;

    // ---- nodes: bitmap, where their positions begin (the padding at the list's end repeats the last node; it gets a
    // place of its own that nobody uses)
    int32_t npos = 0;
    for (int32_t u0 = 0; u0 < ucnt; u0 += MS_THREADS) {
        const int32_t u = u0 + tid;
        int32_t len = 0;
        if (u < ucnt) {
            const int32_t l = __ldg(ulist + u);
            len = __ldg(t_rowptr + l + 1) - __ldg(t_rowptr + l);
            if (!(nbits[l >> 5] >> (l & 31) & 1u)) atomicOr(&nbits[l >> 5], 1u << (l & 31));
        }
        const int32_t at = ms_scan(len, warp_sums, &total);
        if (u < ucnt) node_off[uoff + u] = npos + at;
        npos += total;
        __syncthreads();
    }

    // ---- keys
    // nodes per warp and turn, at most 32: equal shares for all warps in as few turns as it takes (with 32 each, a list of
    // 166 nodes kept 6 warps busy and one of 908 took 5 of them a second turn)
    constexpr int32_t WARPS = C * MS_THREADS / 32;
    const int32_t turns = (ucnt + WARPS * 32 - 1) / (WARPS * 32);
    const int32_t turn = min(32, ((ucnt + turns * WARPS - 1) / max(1, turns * WARPS) + 1) & ~1);
    // (a node's number `of` comes with its extent, one load for 32 nodes, not with every key)
    auto each_key = [&](const int32_t* of, auto&& use) {
        for (int32_t u0 = (part * (MS_THREADS / 32) + warp) * turn; u0 < ucnt; u0 += turn * WARPS) {
            const int32_t n = min(turn, ucnt - u0);
            const int32_t my_l = lane < n ? __ldg(ulist + u0 + lane) : 0;
            const int32_t my_beg = lane < n ? __ldg(t_rowptr + my_l) : 0;
            const int32_t my_len = lane < n ? __ldg(t_rowptr + my_l + 1) - my_beg : 0;
            const int32_t my_of = of && lane < n ? of[u0 + lane] : 0;
            for (int32_t e0 = 0; e0 < n; e0 += 2) {
                int32_t j[2][4], beg[2], len[2], num[2];
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    beg[e] = __shfl_sync(0xffffffffu, my_beg, (e0 + e) & 31);
                    len[e] = e0 + e < n ? __shfl_sync(0xffffffffu, my_len, (e0 + e) & 31) : 0;
                    num[e] = __shfl_sync(0xffffffffu, my_of, (e0 + e) & 31);
#pragma unroll
                    for (int sl = 0; sl < 4; ++sl) j[e][sl] = sl * 32 + lane < len[e] ? __ldg(t_col + beg[e] + sl * 32 + lane) : -1;
                }
#pragma unroll
                for (int e = 0; e < 2; ++e) {
#pragma unroll
                    for (int sl = 0; sl < 4; ++sl)
                        if (j[e][sl] >= 0) use(num[e] + sl * 32 + lane, j[e][sl]);
                    for (int32_t x = 128 + lane; x < len[e]; x += 32) use(num[e] + x, __ldg(t_col + beg[e] + x));
                }
            }
        }
    };
    each_key(nullptr, [&](int32_t, int32_t k) {
        if (!(kbits[k >> 5] >> (k & 31) & 1u)) atomicOr(&kbits[k >> 5], 1u << (k & 31));
    });
    __syncthreads();
    {                                                           // what the block's other CTAs have marked (gathered where the ranks will be)
        cluster_arrive();
        cluster_wait();
        for (int32_t x = tid; x < wk; x += MS_THREADS) {
            uint32_t b = kbits[x];
#pragma unroll
            for (int r = 1; r < C; ++r) b |= cluster_ld(kbits + x, (uint32_t)((part + r) % C));
            kbefore[x] = (int32_t)b;
        }
        cluster_arrive();
        cluster_wait();
        for (int32_t x = tid; x < wk; x += MS_THREADS) kbits[x] = (uint32_t)kbefore[x];
        __syncthreads();
    }
    __shared__ uint32_t reached[GRF_MASK_SMALL / 32];
    const bool whole_tiles = Nk <= GRF_MASK_SMALL;
    if (whole_tiles) {                                          // a place for every key of the tiles from the first to the last one reached
        if (warp == 0) {
            if (lane < GRF_MASK_SMALL / 32) reached[lane] = lane < wk ? kbits[lane] : 0u;
            const uint32_t any = __ballot_sync(0xffffffffu, lane < wk && kbits[min(lane, wk - 1)] != 0u);
            if (any) {
                const int32_t first = (__ffs(any) - 1) & ~1, last = (31 - __clz(any)) | 1;       // two words a tile
                if (lane >= first && lane <= last && lane < wk) kbits[lane] = lane * 32 + 32 <= Nk ? 0xffffffffu : (1u << (Nk & 31)) - 1u;
            }
        }
        __syncthreads();
    }
    const int32_t keys = ms_ranks(kbits, kbefore, wk, warp_sums, &total);
    ms_ranks(nbits, nbefore, wr, warp_sums, &total);
    const int32_t padded = (keys + KT - 1) / KT * KT;
    if (tid == 0 && part == 0) {
        base_keys = atomicAdd(&totals->entries, (unsigned long long)padded);
        base_pos = atomicAdd(&totals->positions, (unsigned long long)npos);
        atomicMax(&totals->longest, padded);
        mk_cnt[blk] = padded;
        mk_off[blk] = (int32_t)base_keys;
    }
    __syncthreads();
    {                                                           // the places that the first CTA has taken
        cluster_arrive();
        cluster_wait();
        if (part > 0 && tid == 0) {
            const uint32_t* keys_at = reinterpret_cast<const uint32_t*>(&base_keys);
            const uint32_t* pos_at = reinterpret_cast<const uint32_t*>(&base_pos);
            base_keys = cluster_ld(keys_at, 0) | (unsigned long long)cluster_ld(keys_at + 1, 0) << 32;
            base_pos = cluster_ld(pos_at, 0) | (unsigned long long)cluster_ld(pos_at + 1, 0) << 32;
        }
        __syncthreads();
        cluster_arrive();                                       // waited for at the end: no CTA leaves while another one reads it
    }
    if ((int64_t)base_keys + padded <= key_room) {
        int32_t* list = mk_key + base_keys;
        // the key that stands at key k's place: itself, or the nearest one before it that is reached, or else the first one
        auto standing = [&](int32_t k) {
            if (!whole_tiles) return k;
            int32_t x = k >> 5;
            uint32_t b = reached[x] & (0xffffffffu >> (31 - (k & 31)));
            while (b == 0u && x > 0) b = reached[--x];
            if (b) return (x << 5) + 31 - __clz(b);
            while (reached[x] == 0u) ++x;
            return (x << 5) + __ffs(reached[x]) - 1;
        };
        const int32_t per = (wk + C * MS_THREADS - 1) / (C * MS_THREADS);
        const int32_t w0 = min(wk, (part * MS_THREADS + tid) * per), w1 = min(wk, w0 + per);
        for (int32_t x = w0; x < w1; ++x) {
            uint32_t b = kbits[x];
            int32_t o = kbefore[x];
            while (b) {
                const int k = (x << 5) + __ffs(b) - 1;
                b &= b - 1;
                const int32_t key = standing(k);
                if (o == keys - 1)
                    for (int32_t e = keys; e < padded; ++e) list[e] = key;
                list[o++] = key;
            }
        }
    }
    if (bits_out && part == 0) {                // for the kernel that looks positions up row by row
        uint32_t* dst = bits_out + (size_t)blk * 2 * wk;
        for (int32_t x = tid; x < wk; x += MS_THREADS) { dst[x] = kbits[x]; dst[wk + x] = (uint32_t)kbefore[x]; }
    }
    if ((int64_t)base_pos + npos <= pos_room && padded <= 65536) {
        unsigned short* pos = pos16 + base_pos;
        each_key(node_off + uoff, [&](int32_t at, int32_t k) {
            pos[at] = (unsigned short)mask_slot((uint32_t)(kbefore[k >> 5] + __popc(kbits[k >> 5] & ((1u << (k & 31)) - 1u))));
        });
        const int32_t r0 = blk * BQ, r1 = min(N, r0 + BQ);
        const int32_t end = phi_rowptr[r1];
        for (int32_t p0 = phi_rowptr[r0] + part * (4 * MS_THREADS) + tid; p0 < end; p0 += C * 4 * MS_THREADS) {
            int32_t at[4];                      // four in flight: two dependent loads each
#pragma unroll
            for (int q = 0; q < 4; ++q) at[q] = p0 + q * MS_THREADS < end ? __ldg(phi_col + p0 + q * MS_THREADS) : -1;
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (at[q] >= 0)
                    at[q] = node_off[uoff + nbefore[at[q] >> 5] + __popc(nbits[at[q] >> 5] & ((1u << (at[q] & 31)) - 1u))];
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (p0 + q * MS_THREADS < end) phi_pos[p0 + q * MS_THREADS] = (int32_t)base_pos + at[q];
        }
    }

    __syncthreads();
    cluster_wait();
    if (part > 0) return;
    // ---- the last block's first CTA: sizes to the host, blocks by decreasing key count (ties: lower index first) behind the counts
    __threadfence();
    __syncthreads();
    if (tid == 0) last_cta = atomicAdd(&totals->finished, 1) == nblocks - 1;
    __syncthreads();
    if (!last_cta) return;
    __threadfence();
    // (compared out of shared memory, in place of the bitmap: a block has four words of it and more)
    int32_t* counts = reinterpret_cast<int32_t*>(smem_ms);
    for (int32_t i = tid; i < nblocks; i += MS_THREADS) counts[i] = __ldcg(mk_cnt + i);
    __syncthreads();
    for (int32_t i = tid; i < nblocks; i += MS_THREADS) {
        const int32_t c = counts[i];
        int32_t rank = 0;
        for (int32_t j = 0; j < nblocks; ++j) {
            const int32_t cj = counts[j];
            rank += (cj > c || (cj == c && j < i)) ? 1 : 0;
        }
        mk_cnt[nblocks + rank] = i;
    }
    if (tid == 0) {
        const volatile grf_mask_totals* t = totals;
        const unsigned long long e = t->entries, p = t->positions;
        host[0] = e > 0x7fffffffull ? -1 : (int32_t)e;
        host[1] = p > 0x7fffffffull ? -1 : (int32_t)p;
        host[2] = t->longest;
    }
}

// ---------------------------------------------------------------------------------------------------
// Mask values: Mhat_ij = sum_l Phi_il Psi_jl for the rows i of one block and the keys j of its list.
// A CTA takes MASK_ROWS rows of one block (the blocks with the longest key lists first), one warp per row at a
// time.  The warp keeps the row's accumulators (fp32, one per key of a segment of the list) in shared memory; for
// every non-zero Phi_il, taken in ascending l, its lanes add Phi_il * Psi_jl at the position of key j, found from
// the bitmap of the block's keys and the number of set bits before each bitmap word.  Keys of one l are distinct,
// so no two lanes meet at one position, and the warp is synchronised between two l: the order of every sum is
// fixed.  The keys of four nodes are fetched together and the next four are on their way while these are added.
// Lists longer than a segment take further passes.

// A segment of a row's accumulators -> the mask blocks, sixteen keys per lane at a time: 32 bytes, a whole sector, at
// [group of 16 keys][row of the block] (in groups of 8 the half sectors cost 90 us of 660).  Cleared for the next row
// as they are read.
// SLOTS: the accumulators lie where mask_slot says.
template <bool SLOTS>
__device__ __forceinline__ void store_mask_row(float* acc, int32_t len, int lane, __nv_bfloat16* __restrict__ mk_val,
                                               int32_t first_key, int32_t first_acc, int32_t rr)
{
    for (int32_t c = lane; c < len / 16; c += 32) {
        float4* a4 = reinterpret_cast<float4*>(acc + c * 16);
        const int turn = SLOTS ? ((first_acc / 16 + c) >> 1) & 3 : 0;
        uint32_t w[8];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const float4 x = a4[q ^ turn];
            a4[q ^ turn] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            const __nv_bfloat162 lo = __floats2bfloat162_rn(x.x, x.y), hi = __floats2bfloat162_rn(x.z, x.w);
            w[2 * q] = *reinterpret_cast<const uint32_t*>(&lo);
            w[2 * q + 1] = *reinterpret_cast<const uint32_t*>(&hi);
        }
        asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
                     ::"l"(mk_val + ((size_t)(first_key / 16 + c) * BQ + rr) * 16), "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3]),
                       "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7]) : "memory");
    }
}

constexpr int MASK_SEG = 4096;          // accumulators per warp
constexpr int MASK_WARPS = 4;
constexpr int MASK_ROWS = 8;            // rows of a block per CTA

struct MaskGroup {                      // the keys of four nodes l, up to 128 each: lane x holds keys x, x+32, x+64, x+96
    int32_t j[4][4];
    float v[4][4];
    int32_t beg[4], end[4];
};

__global__ void __launch_bounds__(MASK_WARPS * 32)
mask_values_kernel(int32_t N, int32_t Nk, const int32_t* __restrict__ phi_rowptr, const int32_t* __restrict__ phi_col,
                   const float* __restrict__ phi_val, const int32_t* __restrict__ t_rowptr,
                   const int32_t* __restrict__ t_col, const float* __restrict__ t_val,
                   const int32_t* __restrict__ mk_off, const int32_t* __restrict__ mk_cnt,
                   const uint32_t* __restrict__ bits, __nv_bfloat16* __restrict__ mk_val)
{
    extern __shared__ uint32_t smem_mask[];     // bitmap, set bits before each word, accumulators
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    constexpr int GROUPS = BQ / MASK_ROWS;
    const int32_t nblocks = (N + BQ - 1) / BQ;
    const int32_t blk = mk_cnt[nblocks + blockIdx.x / GROUPS];     // blocks by decreasing key count
    const int32_t rg = blockIdx.x % GROUPS;
    const int32_t words = (Nk + 31) >> 5;
    const int32_t words_al = (words + 1) & ~1;
    uint32_t* bitmap = smem_mask;
    int32_t* before_word = reinterpret_cast<int32_t*>(smem_mask + words_al);
    // (the accumulators are read as float4: they start at a multiple of 16 bytes)
    float* acc = reinterpret_cast<float*>(smem_mask + 2 * (size_t)words_al) + (size_t)warp * MASK_SEG;
    const int32_t off = mk_off[blk], cnt = mk_cnt[blk];
    // the block's bitmap and prefix counts as the key-set kernel left them
    const uint32_t* src = bits + (size_t)blk * 2 * words;
    for (int32_t x = tid; x < words; x += MASK_WARPS * 32) {
        bitmap[x] = src[x];
        before_word[x] = (int32_t)src[words + x];
    }
    for (int32_t x = lane; x < MASK_SEG; x += 32) acc[x] = 0.0f;
    __syncthreads();
    const int32_t r0 = blk * BQ;
    for (int32_t seg0 = 0; seg0 < cnt; seg0 += MASK_SEG) {
        const int32_t seglen = min(MASK_SEG, cnt - seg0);       // a multiple of the tile, hence of 16
        auto position = [&](int32_t j) {
            const int32_t ps = before_word[j >> 5] + __popc(bitmap[j >> 5] & ((1u << (j & 31)) - 1u)) - seg0;
            return (ps >= 0 && ps < seglen) ? ps : -1;
        };
        for (int32_t rr = rg * MASK_ROWS + warp; rr < (rg + 1) * MASK_ROWS; rr += MASK_WARPS) {
            const int32_t r = r0 + rr;
            if (r < N) {
                const int32_t pbeg = phi_rowptr[r], pend = phi_rowptr[r + 1];
                for (int32_t p0 = pbeg; p0 < pend; p0 += 32) {
                    // 32 non-zeros of the row at a time: lane x holds node l_x, Phi_il and the extent of row l_x of Psi^T
                    const int32_t n = min(32, pend - p0);
                    const int32_t my_l = lane < n ? __ldg(phi_col + p0 + lane) : 0;
                    const float my_phi = lane < n ? __ldg(phi_val + p0 + lane) : 0.0f;
                    const int32_t my_beg = lane < n ? __ldg(t_rowptr + my_l) : 0;
                    const int32_t my_end = lane < n ? __ldg(t_rowptr + my_l + 1) : 0;
                    auto fetch = [&](int32_t e0, MaskGroup& gq) {
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            gq.beg[e] = e0 + e < n ? __shfl_sync(0xffffffffu, my_beg, (e0 + e) & 31) : 0;
                            gq.end[e] = e0 + e < n ? __shfl_sync(0xffffffffu, my_end, (e0 + e) & 31) : 0;
#pragma unroll
                            for (int sl = 0; sl < 4; ++sl) {
                                const int32_t q = gq.beg[e] + sl * 32 + lane;
                                const bool valid = q < gq.end[e];
                                gq.j[e][sl] = valid ? __ldg(t_col + q) : -1;
                                gq.v[e][sl] = valid ? __ldg(t_val + q) : 0.0f;
                            }
                        }
                    };
                    auto add = [&](int32_t e0, MaskGroup& gq) {
#pragma unroll
                        for (int e = 0; e < 4; ++e)
#pragma unroll
                            for (int sl = 0; sl < 4; ++sl) gq.j[e][sl] = gq.j[e][sl] >= 0 ? position(gq.j[e][sl]) : -1;
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            const float phi = __shfl_sync(0xffffffffu, my_phi, (e0 + e) & 31);
                            float a[4];
                            // one node's keys are distinct: a lane's four additions go side by side
#pragma unroll
                            for (int sl = 0; sl < 4; ++sl) a[sl] = gq.j[e][sl] >= 0 ? acc[gq.j[e][sl]] : 0.0f;
#pragma unroll
                            for (int sl = 0; sl < 4; ++sl)
                                if (gq.j[e][sl] >= 0) acc[gq.j[e][sl]] = fmaf(phi, gq.v[e][sl], a[sl]);
                            for (int32_t q = gq.beg[e] + 128 + lane; q < gq.end[e]; q += 32) {   // nodes with more than 128 keys
                                const int32_t ps = position(__ldg(t_col + q));
                                if (ps >= 0) acc[ps] = fmaf(phi, __ldg(t_val + q), acc[ps]);
                            }
                            __syncwarp();
                        }
                    };
                    MaskGroup ga, gb;
                    fetch(0, ga);
                    for (int32_t e0 = 0; e0 < n; e0 += 8) {
                        if (e0 + 4 < n) fetch(e0 + 4, gb);
                        add(e0, ga);
                        if (e0 + 4 < n) {
                            if (e0 + 8 < n) fetch(e0 + 8, ga);
                            add(e0 + 4, gb);
                        }
                    }
                }
            }
            store_mask_row<false>(acc, seglen, lane, mk_val, off + seg0, seg0, rr);
            __syncwarp();
        }
    }
}

// ---------------------------------------------------------------------------------------------------
// The same sums with the positions looked up once per (block, node) instead of once per (row, node): a node of a
// block's list is used by nine of the block's rows on average, and the look-up (two shared-memory reads and a
// population count per key) was most of the work of every addition.
//
// Bound by the load/store unit: per 32 multiply-adds two accesses of the accumulators (2.6 wavefronts each) and the
// position and value loads.  So every row makes one pass over its nodes: a warp's accumulators are as long as the block's
// key list, and the CTA runs as many of its warps as then fit its shared memory (a list beyond an eighth of it is
// taken in segments).  Rows are handed to the warps by a counter.  N = 32768 cloud, 297 M multiply-adds: 853 -> 557 us
// (fixed segments of 4096 keys made two passes of half the rows; four shuffles per node were 14 % of the unit's work; half
// sectors in the output 10 %; 422 -> 222 M warp instructions).  The unit is busy 76 % of the time
// (124 M wavefronts); 40 M of them are bank conflicts in shared memory, the others would take it 0.29 ms.
constexpr int MVP_WARPS = 16;
constexpr int MVP_MIN_WARPS = 8;
constexpr int MVP_ROOM = 212 * 256;      // accumulators (fp32) of a CTA at most: what an SM's shared memory holds

struct MaskPosGroup {                   // the keys of two nodes l, up to 128 each: lane x holds keys x, x+32, x+64, x+96
    int32_t ps[2][4];
    float v[2][4], phi[2];
};

// nodes: (Phi_il, length of row l of Psi^T, start of its values, start of node l's positions) of the 32 non-zeros a warp works on: read back
// as one broadcast each, which costs the load/store unit a quarter of what four shuffles do
template <bool SEGMENTED>
__device__ __forceinline__ void mask_row_pass(int32_t pbeg, int32_t pend, int32_t seg0, int32_t seglen, int lane, float* acc,
                                              int4* nodes, const int32_t* __restrict__ phi_col,
                                              const float* __restrict__ phi_val, const int32_t* __restrict__ phi_pos,
                                              const int32_t* __restrict__ t_rowptr, const float* __restrict__ t_val,
                                              const unsigned short* __restrict__ pos16)
{
    auto place = [&](int32_t ps) { return SEGMENTED ? ((uint32_t)(ps - seg0) < (uint32_t)seglen ? ps - seg0 : -1) : ps; };
    for (int32_t p0 = pbeg; p0 < pend; p0 += 32) {
        const int32_t n = min(32, pend - p0);
        int4 mine = make_int4(0, 0, 0, 0);
        if (lane < n) {
            const int32_t l = __ldg(phi_col + p0 + lane);
            mine.x = __float_as_int(__ldg(phi_val + p0 + lane));
            mine.w = __ldg(phi_pos + p0 + lane);
            mine.z = __ldg(t_rowptr + l);
            mine.y = __ldg(t_rowptr + l + 1) - mine.z;
        }
        __syncwarp();
        nodes[lane] = mine;
        __syncwarp();
        const bool any_long = __any_sync(0xffffffffu, mine.y > 128);
        auto fetch = [&](int32_t e0, MaskPosGroup& gq) {
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const int4 nd = nodes[e0 + e];
                gq.phi[e] = __int_as_float(nd.x);
                const unsigned short* pp = pos16 + (uint32_t)nd.w + lane;
                const float* vp = t_val + (uint32_t)nd.z + lane;
#pragma unroll
                for (int sl = 0; sl < 4; ++sl) {
                    const bool valid = sl * 32 + lane < nd.y;
                    gq.ps[e][sl] = valid ? (int32_t)__ldg(pp + sl * 32) : -1;
                    gq.v[e][sl] = valid ? __ldg(vp + sl * 32) : 0.0f;
                }
            }
        };
        auto add = [&](int32_t e0, MaskPosGroup& gq) {
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const float phi = gq.phi[e];
                float a[4];
                int32_t ps[4];
                // one node's keys are distinct: a lane's four additions go side by side
#pragma unroll
                for (int sl = 0; sl < 4; ++sl) {
                    ps[sl] = place(gq.ps[e][sl]);
                    if (ps[sl] >= 0) a[sl] = acc[ps[sl]];
                }
#pragma unroll
                for (int sl = 0; sl < 4; ++sl)
                    if (ps[sl] >= 0) acc[ps[sl]] = fmaf(phi, gq.v[e][sl], a[sl]);
                if (any_long) {                                             // nodes with more than 128 keys
                    const int4 nd = nodes[e0 + e];
                    for (int32_t x = 128 + lane; x < nd.y; x += 32) {
                        const int32_t y = place((int32_t)__ldg(pos16 + (uint32_t)nd.w + x));
                        if (y >= 0) acc[y] = fmaf(phi, __ldg(t_val + (uint32_t)nd.z + x), acc[y]);
                    }
                }
                __syncwarp();
            }
        };
        MaskPosGroup g[3];
        fetch(0, g[0]);
        fetch(2, g[1]);
        for (int32_t e0 = 0; e0 < n; e0 += 6) {
#pragma unroll
            for (int u = 0; u < 3; ++u) {
                if (e0 + 2 * u < n) {
                    if (e0 + 2 * u + 4 < n) fetch(e0 + 2 * u + 4, g[(u + 2) % 3]);
                    add(e0 + 2 * u, g[u]);
                }
            }
        }
    }
}

__global__ void __launch_bounds__(MVP_WARPS * 32)
mask_values_pos_kernel(int32_t N, int32_t rows_per_cta, int32_t room, const int32_t* __restrict__ phi_rowptr,
                       const int32_t* __restrict__ phi_col, const float* __restrict__ phi_val,
                       const int32_t* __restrict__ phi_pos, const int32_t* __restrict__ t_rowptr,
                       const float* __restrict__ t_val, const unsigned short* __restrict__ pos16,
                       const int32_t* __restrict__ mk_off, const int32_t* __restrict__ mk_cnt,
                       __nv_bfloat16* __restrict__ mk_val)
{
    extern __shared__ __align__(16) float smem_acc[];         // the warps' accumulators, `room` floats in all
    __shared__ int32_t next_row;
    __shared__ int4 nodes[MVP_WARPS][32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int32_t groups = BQ / rows_per_cta;
    const int32_t nblocks = (N + BQ - 1) / BQ;
    const int32_t blk = mk_cnt[nblocks + blockIdx.x / groups];     // blocks by decreasing key count
    const int32_t rr0 = (blockIdx.x % groups) * rows_per_cta;
    const int32_t off = mk_off[blk], cnt = mk_cnt[blk];
    if (cnt == 0) return;
    // warps that run and accumulators of each (a multiple of 16: they leave sixteen at a time)
    const int32_t nw = min(MVP_WARPS, max(MVP_MIN_WARPS, room / cnt));
    const int32_t seg = min(cnt, room / nw & ~15);
    if (tid == 0) next_row = 0;
    __syncthreads();
    if (warp >= nw) return;
    float* acc = smem_acc + (size_t)warp * seg;
    for (int32_t x = lane; x < seg; x += 32) acc[x] = 0.0f;
    __syncwarp();
    const int32_t r0 = blk * BQ;
    for (;;) {
        int32_t rr = 0;
        if (lane == 0) rr = atomicAdd(&next_row, 1);
        rr = __shfl_sync(0xffffffffu, rr, 0);
        if (rr >= rows_per_cta) break;
        rr += rr0;
        const int32_t r = r0 + rr;
        const int32_t pbeg = r < N ? phi_rowptr[r] : 0, pend = r < N ? phi_rowptr[r + 1] : 0;
        for (int32_t seg0 = 0; seg0 < cnt; seg0 += seg) {
            const int32_t seglen = min(seg, cnt - seg0);           // a multiple of 16
            if (seg == cnt)
                mask_row_pass<false>(pbeg, pend, 0, cnt, lane, acc, nodes[warp], phi_col, phi_val, phi_pos, t_rowptr, t_val, pos16);
            else
                mask_row_pass<true>(pbeg, pend, seg0, seglen, lane, acc, nodes[warp], phi_col, phi_val, phi_pos, t_rowptr, t_val, pos16);
            store_mask_row<true>(acc, seglen, lane, mk_val, off + seg0, seg0, rr);
            __syncwarp();
        }
    }
}

// Dense rows of the mask for checking and export: out[x][j] = Mhat[rows[x]][j] (zeros elsewhere), one CTA per row.
__global__ void __launch_bounds__(256)
mask_rows_kernel(int32_t Nk, const int32_t* __restrict__ rows, const int32_t* __restrict__ mk_off,
                 const int32_t* __restrict__ mk_cnt, const int32_t* __restrict__ mk_key,
                 const __nv_bfloat16* __restrict__ mk_val, float* __restrict__ out)
{
    const int32_t r = rows[blockIdx.x];
    float* o = out + (size_t)blockIdx.x * Nk;
    for (int32_t j = threadIdx.x; j < Nk; j += 256) o[j] = 0.0f;
    __syncthreads();
    const int32_t blk = r / BQ, rr = r % BQ;
    const int32_t off = mk_off[blk], cnt = mk_cnt[blk];
    // padding entries repeat another key with the value 0: skip an entry whose predecessor has the same key, in lists of whole
    // aligned tiles one that holds another key than its place's
    const int32_t first = cnt > 0 ? mk_key[off] & ~(KT - 1) : 0;
    for (int32_t e = threadIdx.x; e < cnt; e += 256) {
        const int32_t j = mk_key[off + e];
        if (Nk <= GRF_MASK_SMALL ? j != first + e : e > 0 && mk_key[off + e - 1] == j) continue;
        o[j] = __bfloat162float(mk_val[((size_t)((off + e) / 16) * BQ + rr) * 16 + ((off + e) & 15)]);
    }
}

// ---------------------------------------------------------------------------------------------------
// The attention kernel.  One CTA = 128 queries of one head; the block's keys come in tiles of 64.
//   warps 0-3, 4-7  two groups of row threads (one query = one tensor-memory lane each): a group multiplies the
//                   scores of every other tile by the mask, in place (fp32 scores -> bf16 pairs), and sums its rows
//   warp 8          issues S_t = Q K_t^T into one of three score buffers
//   warp 9          issues O += P_t V_t once the rows of tile t are masked, and frees the tile's stage and buffer
//   warps 10-13     producers: a quarter of every tile's key-feature and value rows each, by 16-byte async copies
// An instruction of the tensor pipe costs its issuing warp 25 cycles with operands in uniform registers (100 with operands that
// the compiler takes for per-thread: 306 us instead of 282 on the N = 32768 cloud), so the two products have a warp each; three
// score buffers let the first product run two tiles ahead of the masking.
// (A round trip to tensor memory is about 230 cycles and the hand-overs add several hundred per tile: what bounds
// the kernel is the length of that chain, not a pipe.)

// M features of the keys, D values: 64, or 32 with half as long value rows.
template <int M, int D> struct MhShape {
    // key/value stages in flight: two CTAs' rings then leave the SM the larger part of its L1, which serves the mask
    // values and the rows that neighbouring keys share (eight stages were 8 % slower at the point cloud, 25 % at the grid)
    // (m = 64, d = 64, 8 problems at 32768 points: four stages 398 us, five 421, six 469; d = 32: 379, 369, 370;
    // m = 32, d = 64: four 293, five 282, six 282)
    static constexpr int NS = M <= 32 || D == 32 ? 5 : 4;
    static constexpr int NB = 3;                          // score buffers
    static constexpr int V_BYTES = KT * D * 2;            // 64 value rows of 128 or 64 bytes, swizzled over that length
    static constexpr uint32_t V_SWIZZLE = D == 64 ? 2u : 4u;
    static constexpr int K_BYTES = KT * M * 2;            // [M/8][KT keys][8] bf16: K-major, unswizzled
    static constexpr int STAGE = V_BYTES + K_BYTES;
    static constexpr int Q_BYTES = BQ * M * 2;            // [M/8][128 rows][8] bf16
    static constexpr int S_COLS = KT;                     // one score buffer; P (bf16 pairs) reuses its first half
    static constexpr int O_COL = NB * S_COLS;
    static constexpr int TMEM_COLS = 256;                 // 3 score buffers + the output accumulator
    static constexpr size_t SMEM = (size_t)NS * STAGE + Q_BYTES + 1024;
    static_assert(STAGE % 1024 == 0, "stages must keep the swizzle phase");
    static_assert(O_COL + D <= TMEM_COLS, "tensor memory");
};

constexpr int MH_THREADS = 448;

constexpr int MH_ISSUER_S = 8, MH_ISSUER_O = 9, MH_PRODUCER0 = 10;

template <int M, int D>
__global__ void __launch_bounds__(MH_THREADS, 2)
mhat_attention_kernel(int32_t G, int32_t nblocks, int32_t N, const int32_t* __restrict__ mk_off,
                      const int32_t* __restrict__ mk_cnt, const int32_t* __restrict__ mk_key,
                      const uint4* __restrict__ mk_val, const __nv_bfloat16* __restrict__ phiQ,
                      const __nv_bfloat16* __restrict__ phiK, const __nv_bfloat16* __restrict__ Vg,
                      __nv_bfloat16* __restrict__ out, float* __restrict__ den_out, int* __restrict__ error_word)
{
    using Sh = MhShape<M, D>;
    constexpr int NS = Sh::NS, NB = Sh::NB;
    extern __shared__ unsigned char smem_dyn[];
    // kv_full, kv_empty per stage; s_full, p_full per score buffer; acc_done; den_ready; one drain barrier per issuer
    __shared__ __align__(8) unsigned long long bars[2 * NS + 2 * NB + 4];
    __shared__ uint32_t tmem_slot;
    __shared__ int abort_flag;
    __shared__ float den_odd[BQ];                  // row sums of the odd tiles, handed to the first group

    // what the whole warp shares is read from one lane, so that the compiler keeps it (and what follows from it) in uniform registers:
    // a tensor-pipe instruction then costs its warp a quarter of the cycles
    auto uniform = [](int32_t x) { return __shfl_sync(0xffffffffu, x, 0); };
    const int tid = threadIdx.x, lane = tid & 31, warp = uniform(tid >> 5);
    const int32_t g = (int32_t)(blockIdx.x % (uint32_t)G);
    const int32_t blk = uniform(mk_cnt[nblocks + (int32_t)(blockIdx.x / (uint32_t)G)]);   // blocks by decreasing key count
    const uint32_t stage_base = (smem_u32(smem_dyn) + 1023u) & ~1023u;
    unsigned char* stage_generic = smem_dyn + (stage_base - smem_u32(smem_dyn));
    const uint32_t q_base = stage_base + (uint32_t)NS * Sh::STAGE;
    const uint32_t bar_base = smem_u32(bars);
    auto kv_full = [&](int s) { return bar_base + 8u * (uint32_t)s; };
    auto kv_empty = [&](int s) { return bar_base + 8u * (uint32_t)(NS + s); };
    auto s_full = [&](int b) { return bar_base + 8u * (uint32_t)(2 * NS + b); };
    auto p_full = [&](int b) { return bar_base + 8u * (uint32_t)(2 * NS + NB + b); };
    const uint32_t acc_done = bar_base + 8u * (uint32_t)(2 * NS + 2 * NB);
    const uint32_t den_ready = acc_done + 8u;
    const uint32_t drain_s = acc_done + 16u, drain_o = acc_done + 24u;

    if (tid == 0) {
        for (int s = 0; s < NS; ++s) { mbar_init(kv_full(s), 128); mbar_init(kv_empty(s), 1); }
        for (int b = 0; b < NB; ++b) { mbar_init(s_full(b), 1); mbar_init(p_full(b), 4); }
        mbar_init(acc_done, 1);
        mbar_init(den_ready, 4);
        mbar_init(drain_s, 1);
        mbar_init(drain_o, 1);
        abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == MH_ISSUER_S) tmem_alloc(&tmem_slot, (uint32_t)Sh::TMEM_COLS);
    // the block's queries in the K-major operand layout: 16-byte chunk c of row r at (c * 128 + r) * 16
    if (tid < BQ) {
        const int32_t row = blk * BQ + tid;
        const uint4* qp = reinterpret_cast<const uint4*>(phiQ + ((size_t)g * N + min(row, N - 1)) * M);
#pragma unroll
        for (int c = 0; c < M / 8; ++c) {
            const uint4 x = row < N ? __ldg(qp + c) : make_uint4(0u, 0u, 0u, 0u);
            *reinterpret_cast<uint4*>(stage_generic + (size_t)NS * Sh::STAGE + ((size_t)c * BQ + tid) * 16) = x;
        }
    }
    fence_async_smem();
    fence_before_sync();
    __syncthreads();
    fence_after_sync();
    const uint32_t tmem_base = (uint32_t)uniform((int32_t)tmem_slot);

    const int32_t off = uniform(mk_off[blk]);
    const int32_t T = uniform(mk_cnt[blk] / KT);                   // key tiles of this block

    if (warp < 8) {
        // ------------------------------------------------------------ row threads: P = S * Mhat, row sums, epilogue
        const int grp = warp >> 2;                               // 0: even tiles, 1: odd tiles
        const int rr = (warp & 3) * 32 + lane;                   // row of the block = tensor-memory lane
        const int32_t row = blk * BQ + rr;
        const uint32_t lane_field = (uint32_t)((warp & 3) * 32) << 16;
        const uint4* mrow = mk_val + ((size_t)(off / 16) * BQ + rr) * 2;   // keys 16x .. 16x+15 of this row: mrow[2 * x * BQ], and the next
        uint64_t den2[2] = {0ull, 0ull};                         // row sums, four partial sums in two packed pairs
        uint4 mk[KT / 8];
        auto load_mask = [&](int32_t t) {
#pragma unroll
            for (int c = 0; c < KT / 16; ++c) ld_nc_32bytes(mrow + (size_t)(t * (KT / 16) + c) * (2 * BQ), mk[2 * c], mk[2 * c + 1]);
        };
        if (grp < T) load_mask(grp);
        bool ok = true;
        int buf = grp;                                           // t % NB and the parity of t / NB, kept in step
        uint32_t par = 0u;
        for (int32_t t = grp; t < T; t += 2) {
            if (!mbar_wait(s_full(buf), par, &abort_flag)) ok = false;
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            fence_after_sync();
            const uint32_t s_addr = tmem_base + lane_field + (uint32_t)(buf * Sh::S_COLS);
#pragma unroll
            for (int c16 = 0; c16 < KT / 16; ++c16) {
                uint32_t sv[16];
                tmem_ld16(s_addr + (uint32_t)(c16 * 16), sv);
                uint32_t pw[8];
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const uint4 mm = mk[2 * c16 + h];
                    const uint32_t mw[4] = {mm.x, mm.y, mm.z, mm.w};
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        // two masked scores at a time; the denominator adds them in fp32, before the rounding to bf16
                        const uint64_t p2 = mul2(pack2(sv[8 * h + 2 * e], sv[8 * h + 2 * e + 1]),
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
            if (lane == 0) mbar_arrive(p_full(buf));
            // this group's next tile: its mask values travel while the products run
            if (t + 2 < T) load_mask(t + 2);
            buf += 2;
            if (buf >= NB) { buf -= NB; par ^= 1u; }
        }
        float den;
        {
            float d0, d1, d2, d3;
            unpack2(den2[0], d0, d1);
            unpack2(den2[1], d2, d3);
            den = (d0 + d1) + (d2 + d3);
        }
        if (grp == 1) {
            // hand the odd tiles' row sums to the first group, which writes the block's outputs
            den_odd[rr] = den;
            __syncwarp();
            if (lane == 0) mbar_arrive(den_ready);
        } else {
            if (ok && !mbar_wait(den_ready, 0u, &abort_flag)) ok = false;
            den += den_odd[rr];
            if (ok && T > 0) ok = mbar_wait(acc_done, 0u, &abort_flag);
            ok = __all_sync(0xffffffffu, ok);
            fence_after_sync();
            const bool live = row < N;
            const float inv = (den != 0.0f) ? 1.0f / den : 0.0f;
            if (live && ok && den_out) den_out[(size_t)g * N + row] = den;
            __nv_bfloat16* orow = out + ((size_t)g * N + row) * D;
#pragma unroll
            for (int c0 = 0; c0 < D; c0 += 16) {
                uint32_t r[16];
#pragma unroll
                for (int e = 0; e < 16; ++e) r[e] = 0u;
                if (ok && T > 0) tmem_ld16(tmem_base + lane_field + (uint32_t)(Sh::O_COL + c0), r);
                if (live && ok) {
                    uint32_t w[8];
#pragma unroll
                    for (int e = 0; e < 8; ++e) {
                        __nv_bfloat162 h = __floats2bfloat162_rn(__uint_as_float(r[2 * e]) * inv, __uint_as_float(r[2 * e + 1]) * inv);
                        w[e] = *reinterpret_cast<uint32_t*>(&h);
                    }
                    uint4* dst = reinterpret_cast<uint4*>(orow + c0);
                    dst[0] = make_uint4(w[0], w[1], w[2], w[3]);
                    dst[1] = make_uint4(w[4], w[5], w[6], w[7]);
                }
            }
        }
    } else if (warp >= MH_PRODUCER0) {
        // ------------------------------------------------------------ producers: warp w takes keys 16w .. 16w+15 of every tile
        // Lanes x and x + 16 hold key x of the warp's sixteen.  Rows travel as 16-byte pieces.  Value rows: D / 8
        // consecutive lanes copy one row, into the swizzle that the second product's operand descriptor names (128-byte
        // rows: piece c of row r at c ^ (r & 7); 64-byte rows: at c ^ (r / 2 & 3)).  Key-feature rows: piece c of key y
        // goes to (c * 64 + y) * 16; lanes 0-15 copy the even pieces, lanes 16-31 the odd ones.  A warp's copies of
        // one tile arrive on the stage's barrier by themselves as they land (the barrier counts all 128 producer
        // threads), so a producer never waits for its own copies; the issuing threads run the proxy fence between
        // their wait on that barrier and the product that reads the stage.  Key indices are read three tiles ahead.
        const int pw = warp - MH_PRODUCER0;
        const __nv_bfloat16* Kg = phiK + (size_t)g * N * M;
        const __nv_bfloat16* Vh = Vg + (size_t)g * N * D;
        const int ky = pw * 16 + (lane & 15);                   // this lane's key within the tile
        constexpr int VP = D / 8;                               // pieces of a value row
        const int vc = lane % VP;                               // its piece of a value row
        bool ok = true;
        const int32_t* kp = mk_key + off + ky;
        int32_t k1 = T > 0 ? __ldg(kp) : 0, k2 = T > 1 ? __ldg(kp + KT) : 0, k3 = T > 2 ? __ldg(kp + 2 * KT) : 0;
        for (int32_t t = 0; t < T; ++t) {
            const int s = t % NS;
            const int32_t k = k1;
            k1 = k2; k2 = k3;
            if (t + 3 < T) k3 = __ldg(kp + (size_t)(t + 3) * KT);
            if (t >= NS && !mbar_wait(kv_empty(s), (uint32_t)(t / NS - 1) & 1u, &abort_flag)) ok = false;
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            const uint32_t v_st = stage_base + (uint32_t)s * Sh::STAGE, k_st = v_st + Sh::V_BYTES;
#pragma unroll
            for (int i = 0; i < VP / 2; ++i) {
                const int y = lane / VP + (32 / VP) * i;        // key of the warp's sixteen
                const int32_t kv = __shfl_sync(0xffffffffu, k, y);
                const int r = pw * 16 + y;
                const int piece = D == 64 ? vc ^ (r & 7) : vc ^ (r >> 1 & 3);
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;"
                             ::"r"(v_st + (uint32_t)(r * (D * 2) + piece * 16)), "l"(Vh + (size_t)kv * D + vc * 8) : "memory");
            }
#pragma unroll
            for (int c2 = 0; c2 < M / 16; ++c2) {
                const int c = 2 * c2 + (lane >> 4);
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;"
                             ::"r"(k_st + (uint32_t)(c * KT + ky) * 16u), "l"(Kg + (size_t)k * M + c * 8) : "memory");
            }
            // every thread's arrival on the stage's barrier happens when its own copies above have landed
            asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(kv_full(s)) : "memory");
        }
        asm volatile("cp.async.wait_all;" ::: "memory");         // also after giving up: no copy outlives the CTA
    } else if (warp == MH_ISSUER_S) {
        // ------------------------------------------------------------ S_t = Q K_t^T (the whole warp runs the loop in step)
        constexpr uint32_t idesc_s = instr_desc(KT, false, false);     // both operands K-major
        bool ok = true;
        int buf = 0, s = 0, back = 0;                                  // back: the stage of the tile NB back
        uint32_t par = 0u, par_back = 0u;
        // operands by one addition each: an issuing warp's instructions count
        const uint64_t q_op = operand_desc(q_base, BQ * 16, 128), k_op = operand_desc(stage_base + Sh::V_BYTES, KT * 16, 128);
        const uint32_t q_hi = (uint32_t)(q_op >> 32), k_hi = (uint32_t)(k_op >> 32);
        for (int32_t t = 0; t < T; ++t) {
            if (!__all_sync(0xffffffffu, mbar_wait(kv_full(s), par, &abort_flag))) { ok = false; break; }
            // the score buffer is free once the second product of the tile three back, which read its P, is complete
            if (t >= NB) {
                if (!__all_sync(0xffffffffu, mbar_wait(kv_empty(back), par_back, &abort_flag))) { ok = false; break; }
                if (++back == NS) { back = 0; par_back ^= 1u; }
            }
            fence_async_smem();                                        // the copies wrote through the generic proxy
            fence_after_sync();
            const uint32_t q_lo = (uint32_t)q_op, k_lo = (uint32_t)k_op + (uint32_t)(s * (Sh::STAGE / 16));
            const uint32_t to = tmem_base + (uint32_t)(buf * Sh::S_COLS);
            mma_bf16_ss_halves<false>(to, q_lo, q_hi, k_lo, k_hi, idesc_s);
#pragma unroll
            for (int k = 1; k < M / 16; ++k) mma_bf16_ss_halves<true>(to, q_lo + k * 2 * BQ, q_hi, k_lo + k * 2 * KT, k_hi, idesc_s);
            mma_commit(s_full(buf));
            if (++buf == NB) buf = 0;
            if (++s == NS) { s = 0; par ^= 1u; }
        }
        if (!ok) {
            mma_commit(drain_s);
            mbar_drain(drain_s, 0u, 20000000ll);
        }
        __syncwarp();
    } else {
        // ------------------------------------------------------------ O += P_t V_t (the whole warp runs the loop in step)
        constexpr uint32_t idesc_o = instr_desc(D, false, true);       // V is MN-major (rows of d values)
        constexpr uint32_t ATOM = 8u * D * 2u;                         // eight value rows
        bool ok = true;
        int buf = 0, s = 0;
        uint32_t par = 0u, par_s = 0u;
        const uint64_t v_op = swizzled_desc(stage_base, ATOM, ATOM, Sh::V_SWIZZLE);
        const uint32_t v_hi = (uint32_t)(v_op >> 32);
        for (int32_t t = 0; t < T; ++t) {
            if (!__all_sync(0xffffffffu, mbar_wait(p_full(buf), par, &abort_flag))) { ok = false; break; }
            // (complete since the first product of this tile ran; waited on here for this thread's own view of the stage)
            if (!__all_sync(0xffffffffu, mbar_wait(kv_full(s), par_s, &abort_flag))) { ok = false; break; }
            fence_async_smem();
            fence_after_sync();
            const uint32_t p_op = tmem_base + (uint32_t)(buf * Sh::S_COLS);
            const uint32_t v_lo = (uint32_t)v_op + (uint32_t)(s * (Sh::STAGE / 16)), acc = tmem_base + (uint32_t)Sh::O_COL;
            mma_bf16_ts_halves(acc, p_op, v_lo, v_hi, idesc_o, t > 0 ? 1u : 0u);
#pragma unroll
            for (int ks = 1; ks < KT / 16; ++ks) mma_bf16_ts_halves(acc, p_op + ks * 8, v_lo + ks * (2 * ATOM / 16), v_hi, idesc_o, 1u);
            mma_commit(kv_empty(s));                                   // frees the stage and the score buffer
            if (++buf == NB) { buf = 0; par ^= 1u; }
            if (++s == NS) { s = 0; par_s ^= 1u; }
        }
        if (ok && T > 0) mma_commit(acc_done);
        if (!ok) {
            mma_commit(drain_o);
            mbar_drain(drain_o, 0u, 20000000ll);
        }
        __syncwarp();
    }

    fence_before_sync();
    __syncthreads();
    if (warp == MH_ISSUER_S) tmem_dealloc(tmem_base, (uint32_t)Sh::TMEM_COLS);
    if (tid == 0 && abort_flag) atomicExch(error_word, 1);
}

}  // namespace

void grf_mask_invalidate(grf_features* feat)
{
    grf_mask_dev& K = feat->mask;
    K.ready = K.requested = K.refused = K.no_room = K.lists_ready = K.structure_ready = false;
}
// Phi's and Psi's values changed, their structure did not (re-modulation): key lists and positions stay
void grf_mask_values_stale(grf_features* feat) { feat->mask.ready = feat->mask.requested = false; }

namespace {
int reserve_with_headroom(grf_buf* b, size_t bytes)
{
    return b->bytes >= bytes ? GRF_OK : grf_buf_reserve(b, bytes + bytes / 8 + 256);
}

// The values of the mask from the present values of Phi and Psi^T, over key lists (and positions) that are in place.
int launch_mask_values(grf_ctx* ctx, grf_features* feat, bool by_position)
{
    grf_mask_dev& K = feat->mask;
    const int32_t N = feat->phi.rows, Nk = feat->psi.rows, nblocks = feat->plan_blocks;
    const size_t words = ((size_t)Nk + 31) / 32;
    if (by_position) {
        // accumulators for sixteen rows of the longest list, up to an SM's shared memory; few blocks: fewer rows per CTA
        const int64_t want = (int64_t)MVP_WARPS * (K.longest > 0 ? K.longest : KT);
        const int32_t room = (int32_t)(want < MVP_ROOM ? want : MVP_ROOM);
        const int32_t rows_per_cta = nblocks * 4 >= 2 * ctx->sm_count ? 32 : 16;
        const size_t smem_acc = (size_t)room * sizeof(float);
        GRF_CUDA_TRY(cudaFuncSetAttribute(mask_values_pos_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_acc));
        grf_launch_scope scope(ctx, 8);
        mask_values_pos_kernel<<<nblocks * (BQ / rows_per_cta), MVP_WARPS * 32, smem_acc, ctx->stream>>>(
            N, rows_per_cta, room, (const int32_t*)feat->phi.rowptr.ptr, (const int32_t*)feat->phi.col.ptr,
            (const float*)feat->phi.val.ptr, (const int32_t*)K.phi_pos.ptr, (const int32_t*)feat->psit.rowptr.ptr,
            (const float*)feat->psit.val.ptr, (const unsigned short*)K.pos16.ptr, (const int32_t*)K.off.ptr,
            (const int32_t*)K.cnt.ptr, (__nv_bfloat16*)K.val.ptr);
    } else {
        const size_t smem_values = ((words + 1) & ~(size_t)1) * 8 + (size_t)MASK_WARPS * MASK_SEG * sizeof(float);
        GRF_CUDA_TRY(cudaFuncSetAttribute(mask_values_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_values));
        grf_launch_scope scope(ctx, 8);
        mask_values_kernel<<<nblocks * (BQ / MASK_ROWS), MASK_WARPS * 32, smem_values, ctx->stream>>>(
            N, Nk, (const int32_t*)feat->phi.rowptr.ptr, (const int32_t*)feat->phi.col.ptr, (const float*)feat->phi.val.ptr,
            (const int32_t*)feat->psit.rowptr.ptr, (const int32_t*)feat->psit.col.ptr, (const float*)feat->psit.val.ptr,
            (const int32_t*)K.off.ptr, (const int32_t*)K.cnt.ptr, (const uint32_t*)K.bits.ptr, (__nv_bfloat16*)K.val.ptr);
    }
    return cudaGetLastError() == cudaSuccess ? GRF_OK : GRF_ERR_CUDA;
}
}  // namespace

void grf_mask_release(grf_features* feat)
{
    grf_mask_dev& K = feat->mask;
    grf_buf_release(&K.off); grf_buf_release(&K.cnt); grf_buf_release(&K.key); grf_buf_release(&K.bits); grf_buf_release(&K.val); grf_buf_release(&K.node_off);
    grf_buf_release(&K.totals); grf_buf_release(&K.pos16); grf_buf_release(&K.phi_pos);
    grf_mask_invalidate(feat);
}

// The structure kernel, and a wait for its sizes.  Its arrays have room from earlier builds; where that was not enough
// (once for a feature object, as a rule) it runs again with what it has found to be needed.
static int prepare_mask_lists(grf_ctx* ctx, grf_features* feat)
{
    grf_mask_dev& K = feat->mask;
    const int32_t N = feat->phi.rows, Nk = feat->psi.rows, R = feat->psit.rows, nblocks = feat->plan_blocks;
    const size_t words = ((size_t)Nk + 31) / 32, smem = (words + ((size_t)R + 31) / 32) * 8;
    GRF_TRY(grf_buf_reserve(&K.cnt, sizeof(int32_t) * 2 * (size_t)nblocks));
    GRF_TRY(grf_buf_reserve(&K.off, sizeof(int32_t) * (size_t)nblocks));
    GRF_TRY(grf_buf_reserve(&K.totals, sizeof(grf_mask_totals)));
    GRF_TRY(reserve_with_headroom(&K.node_off, sizeof(int32_t) * (size_t)(feat->plan_entries > 0 ? feat->plan_entries : 1)));
    GRF_TRY(reserve_with_headroom(&K.phi_pos, sizeof(int32_t) * (size_t)(feat->phi.nnz + 1)));
    K.by_position = true;
    if (!K.key.ptr) {
        // a first guess, so that the kernel need not run twice: 3 keys per node-list entry (1.8 to 2.8 were counted on clouds
        // of 2048 to 32768 points), and a mean row of Psi^T of positions for each; not where that is a lot of memory for a guess
        const int64_t most = (int64_t)nblocks * ((Nk + KT - 1) / KT * KT), guess = 3 * feat->plan_entries;
        const double positions = 1.125 * (double)feat->plan_entries * (double)feat->psi.nnz / R;
        if (positions < (double)(128 << 20)) {
            GRF_TRY(grf_buf_reserve(&K.key, sizeof(int32_t) * (size_t)((guess < most ? guess : most) + KT)));
            GRF_TRY(grf_buf_reserve(&K.pos16, sizeof(unsigned short) * ((size_t)positions + 256)));
        }
    }
    for (int attempt = 0; attempt < 3; ++attempt) {
        const int64_t key_room = (int64_t)(K.key.bytes / sizeof(int32_t));
        const int64_t pos_room = K.by_position ? (int64_t)(K.pos16.bytes / sizeof(unsigned short)) : -1;
        GRF_CUDA_TRY(cudaMemsetAsync(K.totals.ptr, 0, sizeof(grf_mask_totals), ctx->stream));
        {
            auto launch = [&](auto cluster) {
                constexpr int C = decltype(cluster)::value;
                GRF_CUDA_TRY(cudaFuncSetAttribute(mask_structure_kernel<C>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
                grf_launch_scope scope(ctx, 8);
                mask_structure_kernel<C><<<nblocks * C, MS_THREADS, smem, ctx->stream>>>(
                    N, Nk, R, (const int32_t*)feat->phi.rowptr.ptr, (const int32_t*)feat->phi.col.ptr,
                    (const int32_t*)feat->plan_off.ptr, (const int32_t*)feat->plan_cnt.ptr, (const int32_t*)feat->plan_col.ptr,
                    (const int32_t*)feat->psit.rowptr.ptr, (const int32_t*)feat->psit.col.ptr, key_room, pos_room,
                    K.by_position ? nullptr : (uint32_t*)K.bits.ptr, (int32_t*)K.node_off.ptr, (int32_t*)K.off.ptr,
                    (int32_t*)K.cnt.ptr, (int32_t*)K.key.ptr, (unsigned short*)K.pos16.ptr, (int32_t*)K.phi_pos.ptr,
                    (grf_mask_totals*)K.totals.ptr, ctx->pinned + 5);
                return GRF_OK;
            };
            // about as many CTAs per block as find room at once, two on an SM; two also where a block finds room for one only, as
            // the halves fill the SMs more evenly.  Structure and values, us, with 1 / 2 / 4 / 8 CTAs a block: clouds of 9000 points
            // 203 / - / 165 / 178, 14000 - / 257 / 250 / -, 22000 419 / 393 / 396 / -, 32768 575 / 565 / 582 / -, 60000 1092 / 1091 / 1090
            const int64_t room = 2 * (int64_t)ctx->sm_count / nblocks;
            if (room >= 8) GRF_TRY(launch(std::integral_constant<int, 8>()));
            else if (room >= 2) GRF_TRY(launch(std::integral_constant<int, 4>()));
            else GRF_TRY(launch(std::integral_constant<int, 2>()));
        }
        GRF_CUDA_TRY(cudaGetLastError());
        GRF_CUDA_TRY(cudaStreamSynchronize(ctx->stream));      // the sizes of the key lists are known only now
        K.blocks = nblocks;
        K.entries = ctx->pinned[5];
        K.positions = ctx->pinned[6];
        K.longest = ctx->pinned[7];
        // (a negative sum means that it passed 2^31); no locality: the S/z route serves this object
        K.refused = K.entries < 0 || (size_t)K.entries * BQ * sizeof(__nv_bfloat16) > ((size_t)8 << 30);
        if (K.refused) break;
        // positions are looked up once per (block, node) when they fit 16 bits and their number an int32; otherwise once
        // per (row, node), in the blocks' key bitmaps
        const bool by_position = K.positions >= 0 && K.longest <= 65536;
        if (by_position == K.by_position && K.entries <= key_room && (!by_position || K.positions <= pos_room)) break;
        K.by_position = by_position;
        GRF_TRY(reserve_with_headroom(&K.key, (size_t)K.entries * 4));
        if (by_position) GRF_TRY(reserve_with_headroom(&K.pos16, sizeof(unsigned short) * (size_t)K.positions));
        else GRF_TRY(grf_buf_reserve(&K.bits, sizeof(uint32_t) * 2 * (size_t)nblocks * words));
    }
    K.lists_ready = true;
    return GRF_OK;
}

// Shared memory of the structure kernel (two bitmaps and their ranks) and of the row-by-row values kernel (the key bitmap,
// its ranks and the accumulators).
static bool mask_fits_smem(const grf_features* feat)
{
    const size_t words = ((size_t)feat->psi.rows + 31) / 32, node_words = ((size_t)feat->psit.rows + 31) / 32;
    return ((words + 1) & ~(size_t)1) * 8 + (size_t)MASK_WARPS * MASK_SEG * sizeof(float) <= 200 * 1024 &&
           (words + node_words) * 8 <= 200 * 1024;
}

// Forms the mask of the present features (or only its values, where the key lists still hold).
static int build_mask(grf_ctx* ctx, grf_features* feat)
{
    grf_mask_dev& K = feat->mask;
    K.ready = false;
    if (K.structure_ready && feat->plan_ready && !feat->plan_stale) {
        // same walks, new coefficients: the key lists and positions still hold
        GRF_TRY(launch_mask_values(ctx, feat, K.by_position));
        grf_built_by(ctx, feat);
        K.ready = true;
        return GRF_OK;
    }
    K.structure_ready = false;
    if (!mask_fits_smem(feat)) return GRF_ERR_TOO_LARGE;
    GRF_TRY(grf_ensure_block_plan(ctx, feat, false));         // the node lists only
    if (!feat->plan_ready) return GRF_ERR_TOO_LARGE;          // rows of a block share too little
    if (!K.lists_ready) GRF_TRY(prepare_mask_lists(ctx, feat));
    if (K.refused) return GRF_ERR_TOO_LARGE;
    GRF_TRY(reserve_with_headroom(&K.val, (size_t)K.entries * BQ * sizeof(__nv_bfloat16)));
    GRF_TRY(launch_mask_values(ctx, feat, K.by_position));
    grf_built_by(ctx, feat);
    K.structure_ready = true;
    K.ready = true;
    return GRF_OK;
}

extern "C" int grf_features_materialise(grf_ctx* ctx, grf_features* feat)
{
    if (!ctx || !feat) return GRF_ERR_INVALID;
    GRF_CUDA_TRY(cudaSetDevice(ctx->device));
    GRF_TRY(grf_wait_built(ctx, feat));
    feat->mask.requested = false;
    GRF_TRY(build_mask(ctx, feat));
    feat->mask.requested = true;
    feat->mask.no_room = false;
    return GRF_OK;
}

static bool mhat_shape(int32_t m, int32_t d, int dtype)
{
    return dtype == GRF_DTYPE_BF16 && (d == 64 || d == 32) && (m == 16 || m == 32 || m == 64);
}

// Which association of the product serves a batch of grf_masked_linear_attn: the per-node states of Eq. 12, or the
// mask formed first.  The choice depends on the features' sizes and the batch only (never on earlier calls), so equal
// calls give equal bits.  Times in nanoseconds, fitted on a B200 to clouds, grids and expanders of 2^6 .. 2^17 nodes:
//   states   the cheaper gather, 15 000 for launches, and per problem 0.04 per non-zero at m = 32 (a key's rows into a
//            state, z into a denominator; 0.67 of that at m = 16, 1.67 at m = 64; measured at 32768 points, 8 problems,
//            all kernels: 2.0, 2.4, 4.4 ms at d = 64 and 1.8, 2.6, 4.6 ms at d = 32, which is therefore charged alike;
//            by the mask 1.03, 1.05, 1.22 and 1.02, 1.04, 1.20);
//   mask     per problem: 2.5 per 64-key tile at m = 32 (0.8 of that at m = 16, 1.4 at m = 64) and 15 per block; once:
//            0.0011 per multiply-add of Phi Psi^T (non-zeros of Phi times the mean row of Psi^T, again for every further
//            segment of the lists), 0.004 per mask entry, 60 000 for launches and the wait (0.07 ms measured at 2048
//            points, 0.14 at 4096, 0.20 at 8192, 0.41 at 16384, 0.74 at 32768).
// The number of keys is not known before the lists are made, which is a quarter of the mask's cost, so it is estimated for
// the decision: 2.5 per node-list entry where the rows of a block share their nodes (1.8 to 2.8 on clouds of 2048 to 32768
// points), otherwise as many distinct keys as the blocks' nodes would draw at random.  With the lists there, the known
// number may still turn the call back to the states if what is left to do costs more.
// The mask is charged as if this call had to form it, although frozen features keep it: a batch too small for that keeps
// to the states.
int grf_linear_by_mask(grf_ctx* ctx, const grf_features* cfeat, int32_t G, int32_t N, int32_t m, int32_t d, int dtype,
                       bool* by_mask)
{
    *by_mask = false;
    grf_features* feat = const_cast<grf_features*>(cfeat);     // the mask is a cache inside the object, like the block plan
    grf_mask_dev& K = feat->mask;
    if (!ctx->use_tensor_cores || ctx->states_only || !mhat_shape(m, d, dtype)) return GRF_OK;
    if (feat->psi.rows != N || !mask_fits_smem(feat)) return GRF_OK;
    GRF_TRY(grf_features_sizes(feat));
    const double rows = grf_gather_rows_ns(feat, G, m, d);
    if (rows < GRF_PLAN_WORTH_NS) return GRF_OK;
    GRF_TRY(grf_ensure_block_plan(ctx, feat, false));
    if (!feat->plan_ready || K.refused || K.no_room) return GRF_OK;
    const double state_scale = (m + 16) / 48.0, mask_scale = (m + 48) / 80.0;
    const double nnz = 0.5 * ((double)feat->phi.nnz + (double)feat->psi.nnz);
    const double tiles = grf_gather_tiles_ns(feat, G, m);
    const double states = 15000.0 + (tiles < rows ? tiles : rows) + state_scale * G * 0.04 * nnz;
    const double macs = (double)feat->phi.nnz * (double)feat->psi.nnz / feat->psit.rows;
    const double build = 60000.0 + 0.0011 * macs;
    auto rest = [&](double entries) {                           // values and attention for lists of so many keys in all
        const double lists = entries / feat->plan_blocks / (MVP_ROOM / MVP_MIN_WARPS);      // mean list, in accumulator segments
        return (lists > 1.0 ? 0.0011 * macs * (lists - 1.0) : 0.0) + 0.004 * entries * BQ +
               G * (2.5 * mask_scale * entries / KT + 15.0 * feat->plan_blocks);
    };
    const double list = (double)feat->plan_entries / feat->plan_blocks;
    const double drawn = N * (1.0 - exp(-list * (double)feat->psi.nnz / feat->psit.rows / N));
    const double shared = 2.5 * list < N ? 2.5 * list : N;
    const double keys = 1.8 * (double)feat->plan_entries > (double)feat->phi.nnz ? drawn : shared;
    if (build + rest(keys * feat->plan_blocks) > states) return GRF_OK;
    // Memory for the mask is the library's own wish: without it the states serve the call, and later ones on these features
    auto without_mask = [&](int rc) {
        if (rc != GRF_ERR_NOMEM) return rc;
        cudaDeviceSynchronize();                                // the structure kernel may still be writing to what goes
        grf_mask_release(feat);
        K.no_room = true;
        return (int)GRF_OK;
    };
    if (!K.lists_ready) {
        GRF_TRY(without_mask(prepare_mask_lists(ctx, feat)));
        if (K.no_room) return GRF_OK;
    }
    if (K.refused || (int64_t)G * K.blocks > 0x7fffffffll || (int64_t)G * N > 0x7fffffffll) return GRF_OK;
    if (0.75 * build + rest((double)K.entries) > states) return GRF_OK;
    if (!K.ready) {
        const int rc = build_mask(ctx, feat);
        if (rc == GRF_ERR_TOO_LARGE) { K.refused = true; return GRF_OK; }
        GRF_TRY(without_mask(rc));
        if (K.no_room) return GRF_OK;
    }
    *by_mask = true;
    return GRF_OK;
}

extern "C" int grf_mask_stats(const grf_features* feat, int32_t* blocks, int64_t* key_entries, int64_t* bytes)
{
    if (!feat || !feat->mask.ready || !feat->mask.requested) return GRF_ERR_INVALID;
    if (blocks) *blocks = feat->mask.blocks;
    if (key_entries) *key_entries = feat->mask.entries;
    if (bytes) *bytes = feat->mask.entries * (int64_t)(BQ * sizeof(__nv_bfloat16) + sizeof(int32_t));
    return GRF_OK;
}

extern "C" int grf_mask_rows(grf_ctx* ctx, const grf_features* feat, int32_t n, const int32_t* rows, float* out)
{
    if (!ctx || !feat || n <= 0 || !rows || !out) return GRF_ERR_INVALID;
    if (!feat->mask.ready || !feat->mask.requested) return GRF_ERR_INVALID;
    GRF_CUDA_TRY(cudaSetDevice(ctx->device));
    GRF_TRY(grf_wait_built(ctx, feat));
    const grf_mask_dev& K = feat->mask;
    {
        grf_launch_scope scope(ctx, 8);
        mask_rows_kernel<<<n, 256, 0, ctx->stream>>>(feat->psi.rows, rows, (const int32_t*)K.off.ptr, (const int32_t*)K.cnt.ptr,
                                                     (const int32_t*)K.key.ptr, (const __nv_bfloat16*)K.val.ptr, out);
    }
    return cudaGetLastError() == cudaSuccess ? GRF_OK : GRF_ERR_CUDA;
}

template <int M, int D>
static int launch_mhat(grf_ctx* ctx, const grf_features* feat, int32_t G, int32_t N, const void* phiQ, const void* phiK,
                       const void* V, void* out, float* den_out)
{
    using Sh = MhShape<M, D>;
    const grf_mask_dev& K = feat->mask;
    // at most two CTAs per SM: each holds half of the SM's tensor memory
    const size_t smem = Sh::SMEM > 78 * 1024 ? Sh::SMEM : 78 * 1024;
    GRF_CUDA_TRY(cudaFuncSetAttribute(mhat_attention_kernel<M, D>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    {
        grf_launch_scope scope(ctx, 9);
        mhat_attention_kernel<M, D><<<(unsigned)K.blocks * (unsigned)G, MH_THREADS, smem, ctx->stream>>>(
            G, K.blocks, N, (const int32_t*)K.off.ptr, (const int32_t*)K.cnt.ptr, (const int32_t*)K.key.ptr,
            (const uint4*)K.val.ptr, (const __nv_bfloat16*)phiQ, (const __nv_bfloat16*)phiK, (const __nv_bfloat16*)V,
            (__nv_bfloat16*)out, den_out, ctx->error_word);
    }
    return cudaGetLastError() == cudaSuccess ? GRF_OK : GRF_ERR_CUDA;
}

template <int M>
static int launch_mhat_values(grf_ctx* ctx, const grf_features* feat, int32_t G, int32_t N, int32_t d, const void* phiQ,
                              const void* phiK, const void* V, void* out, float* den_out)
{
    return d == 32 ? launch_mhat<M, 32>(ctx, feat, G, N, phiQ, phiK, V, out, den_out)
                   : launch_mhat<M, 64>(ctx, feat, G, N, phiQ, phiK, V, out, den_out);
}

int grf_mhat_launch(grf_ctx* ctx, const grf_features* feat, int32_t G, int32_t N, int32_t m, int32_t d, const void* phiQ,
                    const void* phiK, const void* V, void* out, float* den_out)
{
    if (N <= GRF_MASK_SMALL && G <= (1 << 30)) {
        const int rc = grf_mhat_small_launch(ctx, feat, G, N, m, d, phiQ, phiK, V, out, den_out);
        if (rc <= 0) return rc;                                 // (the kernel below gathers rows and needs no tensor maps)
    }
    if (m == 16) return launch_mhat_values<16>(ctx, feat, G, N, d, phiQ, phiK, V, out, den_out);
    if (m == 32) return launch_mhat_values<32>(ctx, feat, G, N, d, phiQ, phiK, V, out, den_out);
    return launch_mhat_values<64>(ctx, feat, G, N, d, phiQ, phiK, V, out, den_out);
}

extern "C" int grf_masked_attn_mhat(grf_ctx* ctx, const grf_features* feat, int32_t G, int32_t N, int32_t m, int32_t d,
                                    int dtype, const void* phiQ, const void* phiK, const void* V, void* out, float* den_out)
{
    if (!ctx || !feat || !phiQ || !phiK || !V || !out || G <= 0 || N <= 0) return GRF_ERR_INVALID;
    if (!mhat_shape(m, d, dtype) || d != 64) return GRF_ERR_INVALID;
    if (!feat->mask.ready || !feat->mask.requested || feat->phi.rows != N || feat->psi.rows != N) return GRF_ERR_INVALID;
    if ((int64_t)G * N > 0x7fffffffll || (int64_t)G * feat->mask.blocks > 0x7fffffffll) return GRF_ERR_TOO_LARGE;
    if (((uintptr_t)phiQ | (uintptr_t)phiK | (uintptr_t)V | (uintptr_t)out) & 15u) return GRF_ERR_INVALID;
    GRF_CUDA_TRY(cudaSetDevice(ctx->device));
    GRF_TRY(grf_wait_built(ctx, feat));
    return grf_mhat_launch(ctx, feat, G, N, m, d, phiQ, phiK, V, out, den_out);
}
