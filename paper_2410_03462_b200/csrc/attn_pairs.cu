// The states of Eq. 12 used where they are made: for every node l and problem, S_l and z_l are formed from l's keys (a row of
// Psi^T) and multiplied at once with the queries of all rows i that have a non-zero Phi_il, so no state ever leaves the SM.
// Each (row, node) pair leaves a record, phi(q_i)^T S_l (fp32), and phi(q_i)^T z_l; a second kernel adds every row's records,
// times Phi_il, in ascending l, and divides.  The records replace the gather of whole states: 4 d bytes written and 4 d read per
// pair instead of m d elements read, and the m d multiply-adds of a pair run on a tile that is in registers (bf16: tensor
// cores, fp32: plain ALUs).  Measured, whole attention, stored states / pairs: expander of 2^18 nodes, 4 problems, m = 32,
// d = 64, bf16 24.1 / 8.9 ms (records 5.2, sums 3.3, regrouping 0.33); cloud of 5003, 3 problems, fp32 687 / 437 us (322, 82, 24).
//
// Records lie in the order of the nodes (Phi's entries regrouped by column), so that a node writes one contiguous run, and are
// read row by row, whole records at a time in any order: 3.8 GB of 256-byte records on a B200 take 0.51 ms written in order and
// 0.64 read at random, but 0.66 (whole rows per instruction) to 1.23 ms (fragments) written at random.  What a row adds, and in
// which order, depends on Phi alone, so results do not depend on the order inside a node's run, which the regrouping leaves to
// chance.
#include <cfloat>
#include <type_traits>

#include "grf_internal.cuh"
#include "packed.cuh"

namespace {

// ---------------------------------------------------------------------------------------------------
// Regrouping of Phi's entries by column: entry p of column l takes place slot[p] = start of l's run + its rank there.

// A CTA takes 1024 entries.  Additions to one count come one after the other, 2.4 ns each, so a column that most rows use would be
// waited for (7200 entries: 17 us); a CTA therefore counts its entries in shared memory first, each column in the place that its
// hash names, and adds once per place.  Columns that find their place taken add for themselves.  us, all of the regrouping, one addition
// per entry / this: 8060 nodes, one in 7200 of their rows 34.7 / 25.3, 30000, one in 23800 65.5 / 39.8, without such nodes 17.3 / 17.2;
// with the sample's own: cloud of 5003 40.2 / 36.8, expander of 2^18 468 / 469.
__global__ void __launch_bounds__(256)
pair_ranks_kernel(int64_t nnz, const int32_t* __restrict__ col, int32_t* __restrict__ counts, int32_t* __restrict__ rank)
{
    constexpr int PLACES = 1024;
    __shared__ int32_t column[PLACES], sum[PLACES];
    for (int x = threadIdx.x; x < PLACES; x += 256) { column[x] = -1; sum[x] = 0; }
    __syncthreads();
    const int64_t p0 = ((int64_t)blockIdx.x * 256 + threadIdx.x) * 4;
    const int n = p0 < nnz ? (int)min((int64_t)4, nnz - p0) : 0;
    int32_t c[4], place[4], r[4];
    if (n == 4) {                               // col and rank start on whole cache lines
        const int4 c4 = __ldg(reinterpret_cast<const int4*>(col + p0));
        c[0] = c4.x; c[1] = c4.y; c[2] = c4.z; c[3] = c4.w;
    } else {
#pragma unroll
        for (int e = 0; e < 4; ++e) c[e] = e < n ? __ldg(col + p0 + e) : 0;
    }
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        place[e] = (int32_t)(((uint32_t)c[e] * 2654435769u) >> 22);
        if (e >= n) continue;
        const int32_t holder = atomicCAS(column + place[e], -1, c[e]);
        if (holder == -1 || holder == c[e]) {
            r[e] = atomicAdd(sum + place[e], 1);
        } else {
            r[e] = atomicAdd(counts + c[e], 1);
            place[e] = -1;
        }
    }
    __syncthreads();
    for (int x = threadIdx.x; x < PLACES; x += 256)
        if (sum[x] > 0) sum[x] = atomicAdd(counts + column[x], sum[x]);
    __syncthreads();
#pragma unroll
    for (int e = 0; e < 4; ++e)
        if (e < n && place[e] >= 0) r[e] += sum[place[e]];
    if (n == 4) {
        *reinterpret_cast<int4*>(rank + p0) = make_int4(r[0], r[1], r[2], r[3]);
    } else {
#pragma unroll
        for (int e = 0; e < 4; ++e)
            if (e < n) rank[p0 + e] = r[e];
    }
}

// The first blocks take a row of Phi per warp, the others a node per thread: nodes with more than `limit` keys and queries are
// listed for the kernels of long nodes (below), in any order, those with more than `huge` from the list's end.
__global__ void __launch_bounds__(256)
pair_slots_kernel(int32_t N, int32_t R, int32_t row_blocks, const int32_t* __restrict__ rowptr, const int32_t* __restrict__ col,
                  const int32_t* __restrict__ start, const int32_t* __restrict__ t_rowptr, int32_t limit, int32_t huge,
                  int32_t* __restrict__ slot, int32_t* __restrict__ query, int32_t* __restrict__ long_count,
                  int32_t* __restrict__ long_nodes)
{
    if ((int32_t)blockIdx.x >= row_blocks) {
        const int32_t l = ((int32_t)blockIdx.x - row_blocks) * 256 + (int32_t)threadIdx.x;
        if (l >= R) return;
        const int32_t nq = start[l + 1] - start[l], nk = t_rowptr[l + 1] - t_rowptr[l];
        if (nq == 0 || nk <= limit - nq) return;
        if (nk > huge - nq) long_nodes[R - 1 - atomicAdd(long_count + 1, 1)] = l;
        else long_nodes[atomicAdd(long_count, 1)] = l;
        return;
    }
    const int lane = threadIdx.x & 31;
    const int32_t i = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (i >= N) return;
    const int32_t end = rowptr[i + 1];
    for (int32_t p = rowptr[i] + lane; p < end; p += 32) {
        const int32_t t = __ldg(start + __ldg(col + p)) + slot[p];
        slot[p] = t;
        query[t] = i;
    }
}

// ---------------------------------------------------------------------------------------------------
// Asynchronous copies and fragments

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
// 16 bytes; zeros where there is nothing to read
__device__ __forceinline__ void copy16(uint32_t dst, const void* src, bool valid)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(valid ? 16 : 0) : "memory");
}
// ... nothing where j < 0
__device__ __forceinline__ void copy16_row(uint32_t dst, const void* src, int32_t j)
{
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ge.s32 p, %2, 0;\n\t@p cp.async.cg.shared.global [%0], [%1], 16;\n\t}"
                 ::"r"(dst), "l"(src), "r"(j) : "memory");
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int PENDING> __device__ __forceinline__ void copy_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(PENDING) : "memory"); }

__device__ __forceinline__ void ldmatrix4(uint32_t addr, uint32_t (&r)[4])
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void ldmatrix4_trans(uint32_t addr, uint32_t (&r)[4])
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void mma_16816(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1)
{
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi)
{
    const __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t*>(&h);
}

// Where 16-byte piece p of row r lies among rows of ROW bytes: at p ^ turn, so that rows which one ldmatrix reads (eight, the
// same piece) meet in no bank.
template <int ROW> __device__ __forceinline__ constexpr int piece_turn(int r)
{
    return ROW >= 128 ? r & 7 : ROW == 64 ? (r >> 1) & 3 : (r >> 2) & 1;
}

struct PairArgs {
    int32_t R, N, d;
    const int32_t *t_rowptr, *t_col;        // Psi^T
    const float* t_val;
    const int32_t *start, *query;           // Phi's entries by column
    const void *phiQ, *phiK, *V;
    float *rec, *den;                       // [problem][nnz][width], [problem][nnz]
    int64_t nnz;
    int32_t width;                          // columns of a record: columns col0 .. col0 + width - 1 of V
    int32_t col0;
    int32_t slices;                         // of DS columns each, side by side in a record
    int32_t long_limit;                     // keys and queries of a node beyond which it is one of the long ones
    int32_t items;                          // problems times slices
    const int32_t *long_count, *long_nodes; // long ones and very long ones; their nodes from the front and from the end (R places)
};

// Long nodes.  A node is one warp's work, at 0.7 us a chunk (bf16) once the other warps of its SM have finished: a hub that all
// 2^15 nodes of an expander visit kept its warp busy for 1.4 ms a problem where all other nodes take 0.14.  So a node with many
// keys and queries is the work of a CTA, one with very many that of a cluster: the warps share its keys, add their parts of S and z
// up in shared memory (a CTA's warps first, then the CTAs), and share its queries.  The shares depend on the node and the
// whole batch alone, so the bits do not depend on the parts that it is taken in or the workspace.
// Whole attention, us, whole states / one warp a node / this: expanders with a hub, 4 problems, m = 32, d = 64, bf16: 2^15 nodes
// 2099 / 6060 / 1224 (eight hubs 3272 / 6910 / 1302), 2^17 9380 / 26400 / 4697; 2 problems, 2^13 321 / 489 / 176; graph grown by
// preferential attachment, 2^15 2254 / 1804 / 1416, 2^17 10146 / 6365 / 5092; fp32, 3 problems: 5003 1161 / 1435 / 349, 2^15 10813 /
// 25422 / 2436.
constexpr int PAIR_WARPS = 8, PAIR_CLUSTER = 8;
// Keys and queries of a node beyond which it is long, or a cluster's.  Sharing a node costs adding its parts up, so it pays where
// the node would be what the call waits for: beyond an eighth, or a quarter, of what an SM has to do for the whole batch on average, within
// 128 .. 512 and 2048 .. 8192; and never below twice what a warp has to do in a problem (few nodes in all: warps go without work, so
// that does not matter).  us, whole attention (with one addition per entry in the regrouping, 10 to 25 us more than now), 512 and 8192
// throughout / this / whole states, rows of 20 entries in columns N x^4, x uniform:
// fp32, 1 problem, m = 32, d = 64, 8060 nodes 286 / 175 / 136, 20000 349 / 292 / 316, 2697, m = 64 134 / 101 / 93; 2 problems, 30000 716 /
// 634 / 914, 4 problems 1168 / 1185 / 6744 (at 128 and 2048 1551); bf16, 8060, 1 problem 123 / 101 / 85, 3 problems, m = 16, d = 32 124 / 116 / 118.
// (What is left to whole states on one problem: their gather finds the few states that most rows use in L1.)
struct PairLimits { int32_t longer, huge; };
PairLimits pair_limits(int64_t entries, int32_t R, int32_t G_all)
{
    const int64_t share = entries * G_all / 148, twice = (int64_t)R * G_all < 512 ? 0 : 2 * entries / (R < 16384 ? R : 16384);
    auto within = [](int64_t x, int64_t least, int64_t most) { return x < least ? least : x > most ? most : x; };
    const int64_t from = within(share / 8, 128, 512), longer = from > twice ? from : twice, huge = within(share / 4, 2048, 8192);
    return {(int32_t)longer, (int32_t)(huge > longer ? huge : longer)};
}

__device__ __forceinline__ uint32_t cluster_rank()
{
    uint32_t r;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ float cluster_ld(const float* local, uint32_t rank)
{
    uint32_t a;
    float x;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_addr(local)), "r"(rank));
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(x) : "r"(a) : "memory");
    return x;
}

// the share of n rows, in whole chunks, that a warp of `ctas` CTAs has
__device__ __forceinline__ void pair_share(int32_t& first, int32_t& n, int32_t ctas, int chunk)
{
    const int32_t warps = ctas * PAIR_WARPS, who = (ctas > 1 ? (int32_t)cluster_rank() * PAIR_WARPS : 0) + (int32_t)(threadIdx.x >> 5);
    const int32_t per = ((n + warps - 1) / warps + chunk - 1) / chunk * chunk;
    const int32_t skip = min((int64_t)n, (int64_t)who * per);
    first += skip;
    n = min(per, n - skip);
}

// Sums COUNT values per lane over the warps of a CTA or of the cluster's CTAs, in their order; all receive them.  `area` is the
// first warp's room of `stride` floats, the others' follow; a warp may write to its own again afterwards.  (value(i) names value
// i: unrolled, so that values stay in registers)
template <int COUNT, typename Value>
__device__ __forceinline__ void pair_add_up(float* area, int stride, int32_t ctas, Value&& value)
{
    constexpr int EACH = (COUNT + PAIR_WARPS - 1) / PAIR_WARPS;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float* own = area + (size_t)warp * stride + lane;
#pragma unroll
    for (int i = 0; i < COUNT; ++i) own[i * 32] = value(i);
    __syncthreads();
    float sum[EACH];
#pragma unroll
    for (int e = 0; e < EACH; ++e) {
        const int at = min(e * PAIR_WARPS + warp, COUNT - 1) * 32 + lane;
        sum[e] = area[at];
#pragma unroll
        for (int w = 1; w < PAIR_WARPS; ++w) sum[e] += area[(size_t)w * stride + at];
    }
    __syncthreads();
    auto spread = [&]() {
#pragma unroll
        for (int e = 0; e < EACH; ++e)
            if (e * PAIR_WARPS + warp < COUNT) area[(e * PAIR_WARPS + warp) * 32 + lane] = sum[e];
    };
    spread();
    if (ctas > 1) {
        cluster_sync();
#pragma unroll
        for (int e = 0; e < EACH; ++e) {
            const int at = min(e * PAIR_WARPS + warp, COUNT - 1) * 32 + lane;
            sum[e] = 0.0f;
            for (int32_t r = 0; r < ctas; ++r) sum[e] += cluster_ld(area + at, (uint32_t)r);
        }
        cluster_sync();
        spread();
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < COUNT; ++i) value(i) = area[i * 32 + lane];
    __syncthreads();
}

// The long nodes' kernels: clusters take the very long ones, then every CTA for itself the others, all in turn.  They need nothing
// of the kernel for the other nodes, so they may start as soon as that one's last CTAs have (it says so by pair_let_next_start);
// before they end they wait for it to be complete, so that what follows finds all records.  Without long nodes this kernel costs a
// launch 1.2 us (4.5 when it starts behind the other one: fp32 cloud of 5003, 3 problems, 509.7 -> 511.1 and 514.2).
__device__ __forceinline__ void pair_let_next_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
template <typename Node>
__device__ __forceinline__ void pair_long_nodes(const PairArgs& A, Node&& node)
{
    const int64_t huge = (int64_t)__ldg(A.long_count + 1) * A.items, end = (int64_t)__ldg(A.long_count) * A.items;
    for (int64_t x = blockIdx.x / PAIR_CLUSTER; x < huge; x += gridDim.x / PAIR_CLUSTER) {
        node(__ldg(A.long_nodes + (A.R - 1 - x / A.items)), (int32_t)(x % A.items), PAIR_CLUSTER);
        __syncthreads();
    }
    for (int64_t x = blockIdx.x; x < end; x += gridDim.x) {
        node(__ldg(A.long_nodes + x / A.items), (int32_t)(x % A.items), 1);
        __syncthreads();
    }
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

// ---------------------------------------------------------------------------------------------------
// bf16.  A warp takes a node and problem by itself (the long ones' kernel: all warps of a CTA).  Keys and queries come in chunks of 32 rows through a ring of two slots
// (the next chunk's copies are under way while one is used; three slots and twelve warps an SM instead of sixteen: 678 us against
// 621 at 2^15 nodes, 4 problems).
//   keys      S^T (DS columns b x M features a) += V^T (b x keys) . (Psi phi(K)) (keys x a): both operands by transposing
//             ldmatrix from the rows as they lie; Psi_jl enters in registers, in fp32, and the product is rounded to bf16 (once:
//             the tensor-core builds of whole states round Psi_jl as well, which is why their outputs are further from fp64).
//             z is added up in fp32 from the same rounded products.
//   S         rounded to bf16, as the stored states are: the accumulators' layout is the second product's operand layout
//   queries   records (queries x b) = phi(Q) . S; z rides along as three bf16 columns that add up to its fp32 value
// Inside a record columns stand in the order that lets a thread store four: position 16 u + 4 q + 2 h + e holds column
// 16 u + 8 h + 2 q + e.
// mma.sync and not tcgen05: a node has about sixty keys and queries, half a tile of the latter.  What bounds it is the length of
// a warp's chain of instructions at sixteen warps an SM (2^15 nodes: 621 us, without the stores 480, without the copies 485,
// without either 359; tensor pipe 22 % busy).

constexpr int PB_CHUNK = 32, PB_RING = 2;
template <int M, int DS> struct PairShape {
    static constexpr int KROW = M * 2, VROW = DS * 2;
    static constexpr int SLOT = PB_CHUNK * (KROW + VROW);       // a chunk of queries takes the place of the keys
    static constexpr int WARP_BYTES = PB_RING * (SLOT + PB_CHUNK * 4);
    static constexpr int WARPS = 4;
    static constexpr int CTAS = 4;
};

// TOGETHER: by all warps of `ctas` CTAs
template <int M, int DS, bool TOGETHER>
__device__ __forceinline__ void pair_node_bf16(const PairArgs& A, int32_t l, int32_t item, unsigned char* smem_pairs, int32_t ctas = 1)
{
    using Sh = PairShape<M, DS>;
    constexpr int BT = DS / 16, AT = M / 8;                     // 16-column tiles of V, 8-feature tiles
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int32_t slice = item % A.slices, g = item / A.slices;
    int32_t q_beg = __ldg(A.start + l), nq = __ldg(A.start + l + 1) - q_beg;
    if (!TOGETHER && nq == 0) return;
    int32_t k_beg = __ldg(A.t_rowptr + l), nk = __ldg(A.t_rowptr + l + 1) - k_beg;
    if (!TOGETHER && nk > A.long_limit - nq) return;
    if (TOGETHER) {
        pair_share(k_beg, nk, ctas, PB_CHUNK);
        pair_share(q_beg, nq, ctas, PB_CHUNK);
    }
    const int32_t c0 = A.col0 + slice * DS;
    const bool with_den = c0 == 0;
    const __nv_bfloat16* Kg = (const __nv_bfloat16*)A.phiK + (size_t)g * A.N * M;
    const __nv_bfloat16* Vg = (const __nv_bfloat16*)A.V + (size_t)g * A.N * A.d + c0;
    const __nv_bfloat16* Qg = (const __nv_bfloat16*)A.phiQ + (size_t)g * A.N * M;
    unsigned char* ring = smem_pairs + (size_t)warp * Sh::WARP_BYTES;
    float* psi_ring = reinterpret_cast<float*>(ring + PB_RING * Sh::SLOT);
    const uint32_t ring_addr = smem_addr(ring);

    const int32_t kc = (nk + PB_CHUNK - 1) / PB_CHUNK, chunks = kc + (nq + PB_CHUNK - 1) / PB_CHUNK;
    // what names the rows of a chunk is read one chunk before its copies are issued
    int32_t row_next = -1;
    float psi_next = 0.0f;
    auto fetch_rows = [&](int32_t c) {
        row_next = -1;
        psi_next = 0.0f;
        if (c < kc) {
            const int32_t x = c * PB_CHUNK + lane;
            if (x < nk) { row_next = __ldg(A.t_col + k_beg + x); psi_next = __ldg(A.t_val + k_beg + x); }
        } else {
            const int32_t x = (c - kc) * PB_CHUNK + lane;
            if (x < nq) row_next = __ldg(A.query + q_beg + x);
        }
    };
    auto issue = [&](int32_t c, int slot) {
        if (c < chunks) {
            const int32_t row = row_next;
            const uint32_t base = ring_addr + (uint32_t)slot * Sh::SLOT;
            const bool keys = c < kc;
            if (keys) psi_ring[slot * PB_CHUNK + lane] = psi_next;
            if (c + 1 < chunks) fetch_rows(c + 1);
            const __nv_bfloat16* feat = keys ? Kg : Qg;
            constexpr int KP = M / 8, VP = DS / 8;              // pieces of a row
            constexpr int KR = 32 / KP, VR = 32 / VP;           // rows per copy instruction
            {
                const int r = lane / KP, p = lane % KP;
                const __nv_bfloat16* src = feat + p * 8;
#pragma unroll
                for (int x = 0; x < KP; ++x) {
                    const int32_t j = __shfl_sync(0xffffffffu, row, x * KR + r);
                    const int turn = piece_turn<Sh::KROW>(x * KR) ^ piece_turn<Sh::KROW>(r);       // of row x * KR + r
                    copy16_row(base + (uint32_t)(x * KR * Sh::KROW + r * Sh::KROW + ((p ^ turn) << 4)), src + (int64_t)j * M, j);
                }
            }
            if (keys) {
                const int r = lane / VP, p = lane % VP;
                const __nv_bfloat16* src = Vg + p * 8;
                const uint32_t vb = base + PB_CHUNK * Sh::KROW;
#pragma unroll
                for (int x = 0; x < VP; ++x) {
                    const int32_t j = __shfl_sync(0xffffffffu, row, x * VR + r);
                    const int turn = piece_turn<Sh::VROW>(x * VR) ^ piece_turn<Sh::VROW>(r);
                    copy16_row(vb + (uint32_t)(x * VR * Sh::VROW + r * Sh::VROW + ((p ^ turn) << 4)), src + (int64_t)j * A.d, j);
                }
                // rows behind the last key, up to the end of its product: zeros
                const int n = min(PB_CHUNK, nk - c * PB_CHUNK);
                if (n & 15) {
                    const uint4 zero = make_uint4(0u, 0u, 0u, 0u);
                    unsigned char* at = ring + slot * Sh::SLOT;
                    const int rows = 16 - (n & 15);
                    for (int x = lane; x < rows * KP; x += 32) *reinterpret_cast<uint4*>(at + n * Sh::KROW + x * 16) = zero;
                    for (int x = lane; x < rows * VP; x += 32) *reinterpret_cast<uint4*>(at + PB_CHUNK * Sh::KROW + n * Sh::VROW + x * 16) = zero;
                }
            }
        }
        copy_commit();
    };

    float S[BT][AT][4];
    float z[AT][2];                                             // a quarter of the keys of feature 8 t + (lane / 4), even and odd ones
#pragma unroll
    for (int t = 0; t < AT; ++t)
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            z[t][e & 1] = 0.0f;
#pragma unroll
            for (int b = 0; b < BT; ++b) S[b][t][e] = 0.0f;
        }

    fetch_rows(0);
    if (!TOGETHER || kc > 0) issue(0, 0);
    const int mi = lane >> 3, mr = lane & 7, fq = lane & 3, fr = lane >> 2;     // ldmatrix: matrix, row; fragment: quarter, row
    // this lane's row in the three kinds of ldmatrix: keys (8-key halves, then features), values (columns, then keys), queries
    const uint32_t k_lane = (uint32_t)(((mi & 1) * 8 + mr) * Sh::KROW + (((mi >> 1) ^ piece_turn<Sh::KROW>(mr)) << 4));
    const uint32_t v_lane = (uint32_t)(((mi >> 1) * 8 + mr) * Sh::VROW + (((mi & 1) ^ piece_turn<Sh::VROW>(mr)) << 4));
    int slot = 0;
    for (int32_t c = 0; c < kc; ++c) {
        copy_wait<0>();
        __syncwarp();
        if (!TOGETHER || c + 1 < kc) issue(c + 1, slot ^ 1);    // the slot that chunk c - 1 has left
        const uint32_t kbase = ring_addr + (uint32_t)slot * Sh::SLOT, vbase = kbase + PB_CHUNK * Sh::KROW;
        const int32_t n = min(PB_CHUNK, nk - c * PB_CHUNK);
#pragma unroll
        for (int ks = 0; ks < PB_CHUNK / 16; ++ks) {
            if (ks * 16 < n) {
                const float2 p0 = *reinterpret_cast<const float2*>(psi_ring + slot * PB_CHUNK + ks * 16 + 2 * fq);
                const float2 p1 = *reinterpret_cast<const float2*>(psi_ring + slot * PB_CHUNK + ks * 16 + 8 + 2 * fq);
                uint32_t kb[AT][2], va[BT][4];
#pragma unroll
                for (int b = 0; b < BT; ++b) ldmatrix4_trans(vbase + (v_lane ^ (uint32_t)(b << 5)) + ks * 16 * Sh::VROW, va[b]);
#pragma unroll
                for (int t = 0; t < AT; t += 2) {
                    uint32_t r[4];
                    ldmatrix4_trans(kbase + (k_lane ^ (uint32_t)(t << 4)) + ks * 16 * Sh::KROW, r);
#pragma unroll
                    for (int y = 0; y < 4; ++y) {
                        const float2 p = (y & 1) ? p1 : p0;
                        kb[t + (y >> 1)][y & 1] = pack_bf16(__uint_as_float(r[y] << 16) * p.x, __uint_as_float(r[y] & 0xffff0000u) * p.y);
                    }
                }
#pragma unroll
                for (int t = 0; t < AT; ++t)
#pragma unroll
                    for (int y = 0; y < 2; ++y) { z[t][0] += __uint_as_float(kb[t][y] << 16); z[t][1] += __uint_as_float(kb[t][y] & 0xffff0000u); }
#pragma unroll
                for (int b = 0; b < BT; ++b)
#pragma unroll
                    for (int t = 0; t < AT; ++t) mma_16816(S[b][t], va[b], kb[t][0], kb[t][1]);
            }
        }
        slot ^= 1;
    }
    if (TOGETHER) {                             // in place of the ring, which holds nothing now
        constexpr int SV = BT * AT * 4, ZV = AT * 2;
        static_assert((SV + ZV) * 128 <= Sh::WARP_BYTES, "parts of S and z");
        __syncwarp();
        pair_add_up<SV + ZV>(reinterpret_cast<float*>(smem_pairs), Sh::WARP_BYTES / 4, ctas, [&](int i) -> float& {
            return i < SV ? S[i / (AT * 4)][i / 4 % AT][i % 4] : z[(i - SV) / 2][i % 2];
        });
        issue(kc, slot);
    }

    // S in the second product's operand layout; z's three columns
    uint32_t sb[BT][AT][2];
#pragma unroll
    for (int b = 0; b < BT; ++b)
#pragma unroll
        for (int t = 0; t < AT; ++t) {
            sb[b][t][0] = pack_bf16(S[b][t][0], S[b][t][1]);
            sb[b][t][1] = pack_bf16(S[b][t][2], S[b][t][3]);
        }
    uint32_t zb[AT];
#pragma unroll
    for (int t = 0; t < AT; ++t) {
        float x = z[t][0] + z[t][1];
        x += __shfl_xor_sync(0xffffffffu, x, 1);
        x += __shfl_xor_sync(0xffffffffu, x, 2);
        float w[2];
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const float y = __shfl_sync(0xffffffffu, x, (2 * fq + e) * 4);      // feature 8 t + 2 fq + e
            const float hi = __bfloat162float(__float2bfloat16_rn(y)), rest = fabsf(hi) <= 3.4e38f ? y - hi : 0.0f;
            const float mid = __bfloat162float(__float2bfloat16_rn(rest));
            w[e] = fr == 0 ? hi : fr == 1 ? mid : fr == 2 ? rest - mid : 0.0f;
        }
        zb[t] = pack_bf16(w[0], w[1]);
    }

    float* rec = A.rec + ((size_t)g * A.nnz + q_beg) * A.width + slice * DS;
    float* den = A.den + (size_t)g * A.nnz + q_beg;
    for (int32_t c = kc; c < chunks; ++c) {
        copy_wait<0>();
        __syncwarp();
        issue(c + 1, slot ^ 1);
        const uint32_t qbase = ring_addr + (uint32_t)slot * Sh::SLOT;
        const int32_t x0 = (c - kc) * PB_CHUNK;
#pragma unroll
        for (int half = 0; half < PB_CHUNK / 16; ++half) {
            const int32_t first = x0 + half * 16;
            if (first < nq) {
                uint32_t qa[M / 16][4];
#pragma unroll
                for (int s = 0; s < M / 16; ++s)
                    ldmatrix4(qbase + (k_lane ^ (uint32_t)(s << 5)) + half * 16 * Sh::KROW, qa[s]);
                const int32_t r0 = first + fr, r1 = r0 + 8;
                float *to0 = rec + (size_t)r0 * A.width + fq * 4, *to1 = to0 + 8 * (size_t)A.width;
#pragma unroll
                for (int b = 0; b < BT; ++b) {
                    float lo[4] = {0.0f, 0.0f, 0.0f, 0.0f}, hi[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
                    for (int s = 0; s < M / 16; ++s) {
                        mma_16816(lo, qa[s], sb[b][2 * s][0], sb[b][2 * s + 1][0]);
                        mma_16816(hi, qa[s], sb[b][2 * s][1], sb[b][2 * s + 1][1]);
                    }
                    if (r0 < nq) __stcs(reinterpret_cast<float4*>(to0 + b * 16), make_float4(lo[0], lo[1], hi[0], hi[1]));
                    if (r1 < nq) __stcs(reinterpret_cast<float4*>(to1 + b * 16), make_float4(lo[2], lo[3], hi[2], hi[3]));
                }
                if (with_den) {
                    float w[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
                    for (int s = 0; s < M / 16; ++s) mma_16816(w, qa[s], zb[2 * s], zb[2 * s + 1]);
                    // columns 0, 1 in the first lane of a quad, 2 in the second
                    const float w0 = __shfl_down_sync(0xffffffffu, w[0], 1), w1 = __shfl_down_sync(0xffffffffu, w[2], 1);
                    if (fq == 0) {
                        if (r0 < nq) den[r0] = w[0] + (w[1] + w0);
                        if (r1 < nq) den[r1] = w[2] + (w[3] + w1);
                    }
                }
            }
        }
        slot ^= 1;
    }
    copy_wait<0>();
}

template <int M, int DS>
__global__ void __launch_bounds__(PairShape<M, DS>::WARPS * 32, PairShape<M, DS>::CTAS)
pair_records_bf16_kernel(const __grid_constant__ PairArgs A)
{
    extern __shared__ __align__(128) unsigned char smem_pairs[];
    pair_let_next_start();
    const int32_t l = blockIdx.x * PairShape<M, DS>::WARPS + (threadIdx.x >> 5);
    if (l < A.R) pair_node_bf16<M, DS, false>(A, l, blockIdx.y, smem_pairs);
}

template <int M, int DS>
__global__ void __launch_bounds__(PAIR_WARPS * 32, 2) __cluster_dims__(PAIR_CLUSTER, 1, 1)
pair_long_bf16_kernel(const __grid_constant__ PairArgs A)
{
    extern __shared__ __align__(128) unsigned char smem_pairs[];
    pair_long_nodes(A, [&](int32_t l, int32_t item, int32_t ctas) {
        pair_node_bf16<M, DS, true>(A, l, item, smem_pairs, ctas);
    });
}

// ---------------------------------------------------------------------------------------------------
// fp32.  The same walk over a node's keys and queries on the plain ALUs, chunks of 8 keys or 16 queries.  The 32 lanes are 4
// groups along the features times 8 along the columns; a lane keeps M / 4 x DS / 8 sums of S in registers and multiplies with
// them there.  What bounds it is the register write-back of shared-memory loads (four cycles of the SM for a 16-byte load by a
// warp, broadcast or not) beside the FMA pipe: per key and 64 multiply-adds a lane four such loads, 16 cycles of each; per
// query two and six shuffles, 14 cycles.

constexpr int PF_KEYS = 8, PF_QUERIES = 16, PF_RING = 2;
template <int M, int DS> struct PairShapeF {
    static constexpr int KEY_FLOATS = PF_KEYS * (M + DS), QUERY_FLOATS = PF_QUERIES * M;
    static constexpr int SLOT = KEY_FLOATS > QUERY_FLOATS ? KEY_FLOATS : QUERY_FLOATS;
    static constexpr int S_FLOATS = M;                          // z, for the queries
    static constexpr int WARP_FLOATS = PF_RING * (SLOT + PF_KEYS) + S_FLOATS;
    static constexpr int PART_FLOATS = M * DS + (M + 31) / 32 * 32;                     // a warp's part of S and z, for long nodes
    static constexpr int LONG_FLOATS = WARP_FLOATS > PART_FLOATS ? WARP_FLOATS : PART_FLOATS;
    static constexpr int WARPS = 2;
    static constexpr int FIT = 227 * 1024 / (WARPS * WARP_FLOATS * 4 + 1024), CTAS = FIT < 6 ? FIT : 6;
};
// query rows: piece p of row r (sixteen lanes read the same piece of sixteen rows for the denominators)
template <int M> __device__ __forceinline__ int query_at(int r, int p)
{
    return r * M + ((p ^ (r & (M / 4 - 1))) << 2);
}

template <int M, int DS, bool TOGETHER>
__device__ __forceinline__ void pair_node_f32(const PairArgs& A, int32_t l, int32_t item, float* smem_pairs, int32_t ctas = 1)
{
    using Sh = PairShapeF<M, DS>;
    constexpr int MA = M / 4, NB = DS / 8;                      // features and columns of a lane
    constexpr int NQ = NB / 4;                                  // 16-byte pieces of its columns: 4 x at 32 y + 4 bg
    static_assert(NB % 4 == 0 && MA % 4 == 0, "whole pieces");
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int32_t slice = item % A.slices, g = item / A.slices;
    int32_t q_beg = __ldg(A.start + l), nq = __ldg(A.start + l + 1) - q_beg;
    if (!TOGETHER && nq == 0) return;
    int32_t k_beg = __ldg(A.t_rowptr + l), nk = __ldg(A.t_rowptr + l + 1) - k_beg;
    if (!TOGETHER && nk > A.long_limit - nq) return;
    if (TOGETHER) {
        pair_share(k_beg, nk, ctas, PF_KEYS);
        pair_share(q_beg, nq, ctas, PF_QUERIES);
    }
    const int32_t c0 = A.col0 + slice * DS;
    const bool with_den = c0 == 0;
    const float* Kg = (const float*)A.phiK + (size_t)g * A.N * M;
    const float* Vg = (const float*)A.V + (size_t)g * A.N * A.d + c0;
    const float* Qg = (const float*)A.phiQ + (size_t)g * A.N * M;
    constexpr int STRIDE = TOGETHER ? Sh::LONG_FLOATS : Sh::WARP_FLOATS;
    float* ring = smem_pairs + (size_t)warp * STRIDE;
    float* psi_ring = ring + PF_RING * Sh::SLOT;
    float* z_tile = psi_ring + PF_RING * PF_KEYS;

    const int32_t kc = (nk + PF_KEYS - 1) / PF_KEYS, chunks = kc + (nq + PF_QUERIES - 1) / PF_QUERIES;
    int32_t row_next = -1;
    float psi_next = 0.0f;
    auto fetch_rows = [&](int32_t c) {                          // lanes 0 .. 15
        row_next = -1;
        psi_next = 0.0f;
        if (c < kc) {
            const int32_t x = c * PF_KEYS + lane;
            if (lane < PF_KEYS && x < nk) { row_next = __ldg(A.t_col + k_beg + x); psi_next = __ldg(A.t_val + k_beg + x); }
        } else {
            const int32_t x = (c - kc) * PF_QUERIES + lane;
            if (lane < PF_QUERIES && x < nq) row_next = __ldg(A.query + q_beg + x);
        }
    };
    auto issue = [&](int32_t c, int slot) {
        if (c < chunks) {
            const int32_t row = row_next;
            float* base = ring + slot * Sh::SLOT;
            const bool keys = c < kc;
            if (keys && lane < PF_KEYS) psi_ring[slot * PF_KEYS + lane] = psi_next;
            if (c + 1 < chunks) fetch_rows(c + 1);
            constexpr int KP = M / 4, VP = DS / 4;
            if (keys) {
#pragma unroll
                for (int x = 0; x < PF_KEYS * KP / 32; ++x) {
                    const int idx = x * 32 + lane, r = idx / KP, p = idx % KP;
                    const int32_t j = __shfl_sync(0xffffffffu, row, r);
                    copy16(smem_addr(base + r * M + p * 4), Kg + (size_t)max(j, 0) * M + p * 4, j >= 0);
                }
#pragma unroll
                for (int x = 0; x < PF_KEYS * VP / 32; ++x) {
                    const int idx = x * 32 + lane, r = idx / VP, p = idx % VP;
                    const int32_t j = __shfl_sync(0xffffffffu, row, r);
                    copy16(smem_addr(base + PF_KEYS * M + r * DS + p * 4), Vg + (size_t)max(j, 0) * A.d + p * 4, j >= 0);
                }
            } else {
#pragma unroll
                for (int x = 0; x < PF_QUERIES * KP / 32; ++x) {
                    const int idx = x * 32 + lane, r = idx / KP, p = idx % KP;
                    const int32_t j = __shfl_sync(0xffffffffu, row, r);
                    copy16_row(smem_addr(base + query_at<M>(r, p)), Qg + (int64_t)j * M + p * 4, j);
                }
            }
        }
        copy_commit();
    };

    const int ag = lane >> 3, bg = lane & 7;
    constexpr int ZL = (M + 31) / 32;                           // features of z per lane
    uint64_t S[MA][NB / 2];                                     // pairs of columns
    float z[ZL];
#pragma unroll
    for (int a = 0; a < MA; ++a)
#pragma unroll
        for (int b = 0; b < NB / 2; ++b) S[a][b] = 0ull;
#pragma unroll
    for (int y = 0; y < ZL; ++y) z[y] = 0.0f;

    fetch_rows(0);
    if (!TOGETHER || kc > 0) issue(0, 0);
    int slot = 0;
    for (int32_t c = 0; c < kc; ++c) {
        copy_wait<0>();
        __syncwarp();
        if (!TOGETHER || c + 1 < kc) issue(c + 1, slot ^ 1);
        float* kt = ring + slot * Sh::SLOT;
        const float* vt = kt + PF_KEYS * M;
        const int32_t n4 = min(PF_KEYS, (nk - c * PF_KEYS + 3) & ~3);
        // Psi_jl phi(k_j) in place, and z (rows behind the last key are zeros)
#pragma unroll
        for (int y = 0; y < ZL; ++y) {
            const int a = y * 32 + lane;
            if (M >= 32 || lane < M) {
#pragma unroll
                for (int32_t j = 0; j < PF_KEYS; ++j) {
                    const float x = psi_ring[slot * PF_KEYS + j] * kt[j * M + a];
                    kt[j * M + a] = x;
                    z[y] += x;
                }
            }
        }
        __syncwarp();
#pragma unroll 4
        for (int32_t j = 0; j < n4; ++j) {
            float k[MA];
            uint64_t v[NB / 2];
#pragma unroll
            for (int a = 0; a < MA; a += 4) {
                const float4 x = *reinterpret_cast<const float4*>(kt + j * M + ag * MA + a);
                k[a] = x.x; k[a + 1] = x.y; k[a + 2] = x.z; k[a + 3] = x.w;
            }
#pragma unroll
            for (int b = 0; b < NQ; ++b) {
                const ulonglong2 x = *reinterpret_cast<const ulonglong2*>(vt + j * DS + b * 32 + bg * 4);
                v[2 * b] = x.x; v[2 * b + 1] = x.y;
            }
#pragma unroll
            for (int a = 0; a < MA; ++a) {
                const uint64_t k2 = pack2(k[a], k[a]);
#pragma unroll
                for (int b = 0; b < NB / 2; ++b) S[a][b] = fma2(k2, v[b], S[a][b]);
            }
        }
        slot ^= 1;
    }
    if (TOGETHER) {
        constexpr int SV = MA * NB;
        static_assert((SV + ZL) * 32 <= Sh::LONG_FLOATS, "parts of S and z");
        float part[SV + ZL];
#pragma unroll
        for (int i = 0; i < SV; i += 2) {
            unpack2(S[i / NB][i % NB / 2], part[i], part[i + 1]);
        }
#pragma unroll
        for (int y = 0; y < ZL; ++y) part[SV + y] = z[y];
        __syncwarp();
        pair_add_up<SV + ZL>(smem_pairs, STRIDE, ctas, [&](int i) -> float& { return part[i]; });
#pragma unroll
        for (int i = 0; i < SV; i += 2) S[i / NB][i % NB / 2] = pack2(part[i], part[i + 1]);
#pragma unroll
        for (int y = 0; y < ZL; ++y) z[y] = part[SV + y];
        issue(kc, slot);
    }
#pragma unroll
    for (int y = 0; y < ZL; ++y)
        if (M >= 32 || lane < M) z_tile[y * 32 + lane] = z[y];
    __syncwarp();

    float* rec = A.rec + ((size_t)g * A.nnz + q_beg) * A.width + slice * DS;
    float* den = A.den + (size_t)g * A.nnz + q_beg;
    for (int32_t c = kc; c < chunks; ++c) {
        copy_wait<0>();
        __syncwarp();
        issue(c + 1, slot ^ 1);
        const float* qt = ring + slot * Sh::SLOT;
        const int32_t x0 = (c - kc) * PF_QUERIES;
        const int32_t n = min(PF_QUERIES, nq - x0);
        // A lane multiplies with its features; the four lanes of a column group add up, each ending with a quarter of the
        // columns: what a lane gives away at a step is what its partner keeps.
#pragma unroll 2
        for (int32_t i = 0; i < n; ++i) {
            float q[MA];
#pragma unroll
            for (int a = 0; a < MA; a += 4) {
                const float4 x = *reinterpret_cast<const float4*>(qt + query_at<M>(i, ag * (MA / 4) + a / 4));
                q[a] = x.x; q[a + 1] = x.y; q[a + 2] = x.z; q[a + 3] = x.w;
            }
            uint64_t t[NB / 2];
#pragma unroll
            for (int b = 0; b < NB / 2; ++b) t[b] = 0ull;
#pragma unroll
            for (int a = 0; a < MA; ++a) {
                const uint64_t q2 = pack2(q[a], q[a]);
#pragma unroll
                for (int b = 0; b < NB / 2; ++b) t[b] = fma2(q2, S[a][b], t[b]);
            }
            float u[NB], w[NB / 2], x[NB / 4];
#pragma unroll
            for (int b = 0; b < NB / 2; ++b) unpack2(t[b], u[2 * b], u[2 * b + 1]);
#pragma unroll
            for (int b = 0; b < NB / 2; ++b) {
                const float give = (ag & 1) ? u[b] : u[NB / 2 + b], keep = (ag & 1) ? u[NB / 2 + b] : u[b];
                w[b] = keep + __shfl_xor_sync(0xffffffffu, give, 8);
            }
#pragma unroll
            for (int b = 0; b < NB / 4; ++b) {
                const float give = (ag & 2) ? w[b] : w[NB / 4 + b], keep = (ag & 2) ? w[NB / 4 + b] : w[b];
                x[b] = keep + __shfl_xor_sync(0xffffffffu, give, 16);
            }
            // columns NB / 2 (ag & 1) + NB / 4 (ag / 2) .. of the lane's own NB
            constexpr int HALF = NB / 2, QUARTER = NB / 4;
            const int first = (ag & 1) * HALF + (ag >> 1) * QUARTER;
            float* to = rec + (size_t)(x0 + i) * A.width + (first >> 2) * 32 + bg * 4 + (first & 3);
            if (QUARTER == 2) __stcs(reinterpret_cast<float2*>(to), make_float2(x[0], x[QUARTER - 1]));
            else __stcs(to, x[0]);
        }
        if (with_den) {                                          // lanes x and x + 16 take half of query x's features each
            const int r = lane & 15, h = lane >> 4;
            float w = 0.0f;
#pragma unroll
            for (int p = 0; p < M / 8; ++p) {
                const float4 q = *reinterpret_cast<const float4*>(qt + query_at<M>(r, h * (M / 8) + p));
                const float4 x = *reinterpret_cast<const float4*>(z_tile + (h * (M / 8) + p) * 4);
                w = fmaf(q.x, x.x, w); w = fmaf(q.y, x.y, w); w = fmaf(q.z, x.z, w); w = fmaf(q.w, x.w, w);
            }
            w += __shfl_xor_sync(0xffffffffu, w, 16);
            if (lane < 16 && x0 + r < nq) den[x0 + r] = w;
        }
        slot ^= 1;
    }
    copy_wait<0>();
}

template <int M, int DS>
__global__ void __launch_bounds__(PairShapeF<M, DS>::WARPS * 32, PairShapeF<M, DS>::CTAS)
pair_records_f32_kernel(const __grid_constant__ PairArgs A)
{
    extern __shared__ __align__(128) unsigned char smem_pairs[];
    pair_let_next_start();
    const int32_t l = blockIdx.x * PairShapeF<M, DS>::WARPS + (threadIdx.x >> 5);
    if (l < A.R) pair_node_f32<M, DS, false>(A, l, blockIdx.y, reinterpret_cast<float*>(smem_pairs));
}

template <int M, int DS>
__global__ void __launch_bounds__(PAIR_WARPS * 32, 1) __cluster_dims__(PAIR_CLUSTER, 1, 1)
pair_long_f32_kernel(const __grid_constant__ PairArgs A)
{
    extern __shared__ __align__(128) unsigned char smem_pairs[];
    pair_long_nodes(A, [&](int32_t l, int32_t item, int32_t ctas) {
        pair_node_f32<M, DS, true>(A, l, item, reinterpret_cast<float*>(smem_pairs), ctas);
    });
}

// ---------------------------------------------------------------------------------------------------
// out_i = sum_l Phi_il rec_il / sum_l Phi_il den_il: a warp per (row, problem), W / 4 lanes per record, 128 / W records side by
// side.  Bound by the delivery of records, from HBM where a problem's do not fit L2.

__device__ __forceinline__ void put_pair(float* dst, float x, float y) { *reinterpret_cast<float2*>(dst) = make_float2(x, y); }
__device__ __forceinline__ void put_pair(__nv_bfloat16* dst, float x, float y) { *reinterpret_cast<uint32_t*>(dst) = pack_bf16(x, y); }

// sum += phi * y with what the addition rounds off carried to the next one (Kahan).  The other route adds over l for every
// feature by itself and lets the features' roundings average out; here a row's sum is one chain, and plain fp32 additions made
// the fp32 outputs of m = 64 a quarter less exact (1.3e-7 against 1.05e-7 of fp64).
__device__ __forceinline__ void add_carried(float& sum, float& lost, float phi, float y)
{
    const float x = fmaf(phi, y, -lost), t = sum + x;
    lost = fabsf(t) <= FLT_MAX ? (t - sum) - x : 0.0f;          // an infinite sum rounds nothing off (inf - inf would make it NaN)
    sum = t;
}

template <typename T, int W>
__global__ void __launch_bounds__(256, sizeof(T) == 2 || W < 64 ? 3 : 2)
pair_sums_kernel(int32_t N, int32_t d, int32_t col0, int64_t nnz, const int32_t* __restrict__ rowptr, const float* __restrict__ val,
                 const int32_t* __restrict__ slot, const float* __restrict__ rec, const float* __restrict__ den_rec,
                 T* __restrict__ out, float* __restrict__ den)
{
    constexpr int LPR = W / 4, SIDE = 32 / LPR, CHAINS = 8 / SIDE;       // eight chains of sums: by an entry's place in its row
    const int lane = threadIdx.x & 31, sub = lane / LPR, pl = lane % LPR;
    const int32_t i = blockIdx.x * 8 + (threadIdx.x >> 5), g = blockIdx.y;
    if (i >= N) return;
    const float* base = rec + (size_t)g * nnz * W + pl * 4;
    const int32_t beg = __ldg(rowptr + i), end = __ldg(rowptr + i + 1);
    using Sum = typename std::conditional<sizeof(T) == 2, float, double>::type;
    float a[CHAINS][4], lost[CHAINS][4], dn;
    Sum dsum = 0;
#pragma unroll
    for (int c = 0; c < CHAINS; ++c)
#pragma unroll
        for (int e = 0; e < 4; ++e) a[c][e] = lost[c][e] = 0.0f;
    for (int32_t p0 = beg; p0 < end; p0 += 32) {
        const int32_t n = min(32, end - p0);
        const int32_t my_t = lane < n ? __ldg(slot + p0 + lane) : 0;
        const float my_phi = lane < n ? __ldg(val + p0 + lane) : 0.0f;
        if (col0 == 0 && lane < n) dsum += (Sum)my_phi * (Sum)__ldg(den_rec + (size_t)g * nnz + my_t);
#pragma unroll
        for (int32_t j = 0; j < 32; j += 16) {                  // sixteen records of the row under way
            if (j >= n) break;
            float4 x[2 * CHAINS];
#pragma unroll
            for (int c = 0; c < 2 * CHAINS; ++c) {
                const int32_t t = __shfl_sync(0xffffffffu, my_t, j + c * SIDE + sub);
                x[c] = j + c * SIDE + sub < n ? __ldcs(reinterpret_cast<const float4*>(base + (size_t)t * W)) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            }
#pragma unroll
            for (int c = 0; c < CHAINS; ++c) {
                const float phi = __shfl_sync(0xffffffffu, my_phi, j + c * SIDE + sub);
                const float phi8 = __shfl_sync(0xffffffffu, my_phi, j + 8 + c * SIDE + sub);
                const float y[4] = {x[c].x, x[c].y, x[c].z, x[c].w};
                const float y8[4] = {x[c + CHAINS].x, x[c + CHAINS].y, x[c + CHAINS].z, x[c + CHAINS].w};
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    if (sizeof(T) == 2) {
                        a[c][e] += fmaf(phi8, y8[e], phi * y[e]);
                    } else {
                        add_carried(a[c][e], lost[c][e], phi, y[e]);
                        add_carried(a[c][e], lost[c][e], phi8, y8[e]);
                    }
                }
            }
        }
    }
    if (col0 == 0) {
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) dsum += __shfl_xor_sync(0xffffffffu, dsum, o);
        dn = (float)dsum;
        if (lane == 0 && den) den[(size_t)g * N + i] = dn;
    } else {
        dn = den[(size_t)g * N + i];
    }
    // the eight chains meet in the same order whatever the width: neighbours first
    Sum s[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        Sum w[CHAINS];
#pragma unroll
        for (int c = 0; c < CHAINS; ++c) {
            w[c] = sizeof(T) == 2 ? (Sum)a[c][e] : (Sum)a[c][e] - (Sum)lost[c][e];
#pragma unroll
            for (int o = LPR; o < 32; o <<= 1) w[c] += __shfl_xor_sync(0xffffffffu, w[c], o);
        }
        s[e] = CHAINS == 4 ? (w[0] + w[1 % CHAINS]) + (w[2 % CHAINS] + w[3 % CHAINS]) : CHAINS == 2 ? w[0] + w[1 % CHAINS] : w[0];
    }
    if (sub != 0) return;
    const Sum inv = dn != 0.0f ? (Sum)1 / (Sum)dn : (Sum)0;
    T* row = out + ((size_t)g * N + i) * d + col0;
    if (sizeof(T) == 2) {                                       // the records' order of columns (see above)
        T* dst = row + (pl >> 2) * 16 + (pl & 3) * 2;
        put_pair(dst, (float)(s[0] * inv), (float)(s[1] * inv));
        put_pair(dst + 8, (float)(s[2] * inv), (float)(s[3] * inv));
    } else {
        put_pair(row + pl * 4, (float)(s[0] * inv), (float)(s[1] * inv));
        put_pair(row + pl * 4 + 2, (float)(s[2] * inv), (float)(s[3] * inv));
    }
}

template <int M, int DS>
int launch_records(grf_ctx* ctx, const PairArgs& A, bool bf16)
{
    auto launch = [&](auto kernel, auto long_kernel, int warps, size_t warp_bytes, size_t long_bytes, int long_ctas) {
        GRF_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(warps * warp_bytes)));
        GRF_CUDA_TRY(cudaFuncSetAttribute(long_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(PAIR_WARPS * long_bytes)));
        kernel<<<dim3(grf_ceil_div(A.R, warps), A.items), warps * 32, warps * warp_bytes, ctx->stream>>>(A);
        const int ctas = ctx->sm_count * long_ctas / PAIR_CLUSTER * PAIR_CLUSTER;
        cudaLaunchAttribute beside = {};
        beside.id = cudaLaunchAttributeProgrammaticStreamSerialization;
        beside.val.programmaticStreamSerializationAllowed = 1;
        cudaLaunchConfig_t config = {};
        config.gridDim = dim3(ctas > 0 ? ctas : PAIR_CLUSTER);
        config.blockDim = dim3(PAIR_WARPS * 32);
        config.dynamicSmemBytes = PAIR_WARPS * long_bytes;
        config.stream = ctx->stream;
        config.attrs = &beside;
        config.numAttrs = 1;
        GRF_CUDA_TRY(cudaLaunchKernelEx(&config, long_kernel, A));
        return cudaGetLastError() == cudaSuccess ? GRF_OK : GRF_ERR_CUDA;
    };
    if (bf16) {
        using Sh = PairShape<M, DS>;
        return launch(pair_records_bf16_kernel<M, DS>, pair_long_bf16_kernel<M, DS>, Sh::WARPS, Sh::WARP_BYTES, Sh::WARP_BYTES, 2);
    }
    if constexpr (DS >= 32) {
        using Sh = PairShapeF<M, DS>;
        return launch(pair_records_f32_kernel<M, DS>, pair_long_f32_kernel<M, DS>, Sh::WARPS, Sh::WARP_FLOATS * sizeof(float),
                      Sh::LONG_FLOATS * sizeof(float), 1);
    }
    return GRF_ERR_INVALID;
}

template <int M>
int launch_records_m(grf_ctx* ctx, PairArgs& A, int32_t G, bool bf16)
{
    // M x DS sums are held in registers: at most 2048 a warp
    const int32_t ds = M == 64 && A.width > 32 ? 32 : A.width;
    A.slices = A.width / ds;
    A.items = G * A.slices;
    switch (ds) {
        case 16: return launch_records<M, 16>(ctx, A, bf16);
        case 32: return launch_records<M, 32>(ctx, A, bf16);
        default:
            if constexpr (M <= 32) return launch_records<M, 64>(ctx, A, bf16);
            return GRF_ERR_INVALID;
    }
}

template <typename T>
void launch_sums(grf_ctx* ctx, const PairArgs& A, int32_t G, const grf_csr_dev& phi, const int32_t* slot, void* out, float* den)
{
    const dim3 grid(grf_ceil_div(A.N, 8), G);
    auto launch = [&](auto w) {
        constexpr int W = decltype(w)::value;
        pair_sums_kernel<T, W><<<grid, 256, 0, ctx->stream>>>(A.N, A.d, A.col0, A.nnz, (const int32_t*)phi.rowptr.ptr,
                                                              (const float*)phi.val.ptr, slot, A.rec, A.den, (T*)out, den);
    };
    if (A.width == 64) launch(std::integral_constant<int, 64>());
    else if (A.width == 32) launch(std::integral_constant<int, 32>());
    else launch(std::integral_constant<int, 16>());
}

size_t pair_bytes(int64_t nnz, int32_t width) { return (size_t)nnz * ((size_t)width + 1) * sizeof(float) + 512; }

}  // namespace

// The records of a launch lie in the caller's workspace, or in the context's own scratch of at most PAIR_SCRATCH bytes where
// that takes the whole batch, or more problems, in one launch: fp32 cloud of 5003 points, 3
// problems of 104 MB of records: 374 us one by one (a workspace of 125 MB), 323 together.
constexpr size_t PAIR_SCRATCH = (size_t)512 << 20;
// and of more where the workspace holds not even the narrowest records of one problem.
constexpr size_t PAIR_MOST = (size_t)1 << 30;

static int32_t least_width(int dtype) { return dtype == GRF_DTYPE_BF16 ? 16 : 32; }

namespace {
struct PairRoom { int32_t width; int64_t chunk; size_t scratch; };     // columns of a record, problems a launch (0: no room), own scratch (0: the workspace)
PairRoom pair_room(int64_t nnz, int32_t G, int32_t d, int dtype, size_t workspace_bytes, bool own_scratch = true)
{
    const size_t whole = pair_bytes(nnz, d);
    int64_t in_ws = (int64_t)(workspace_bytes / whole), in_scratch = own_scratch ? (int64_t)(PAIR_SCRATCH / whole) : 0;
    if (in_ws > G) in_ws = G;
    if (in_scratch > G) in_scratch = G;
    PairRoom r = {d, in_ws, 0};
    if (in_scratch > in_ws) {
        r.chunk = in_scratch;
        r.scratch = whole * (size_t)in_scratch;
    } else if (in_ws == 0) {
        while (r.width > least_width(dtype) && pair_bytes(nnz, r.width) > workspace_bytes) r.width >>= 1;
        r.chunk = (int64_t)(workspace_bytes / pair_bytes(nnz, r.width));
        if (r.chunk == 0 && own_scratch) { r.chunk = 1; r.scratch = pair_bytes(nnz, r.width); }
        if (r.chunk > G) r.chunk = G;
    }
    if (r.chunk > 16000) r.chunk = 16000;                       // the grid's second dimension, two slices a problem
    return r;
}
}  // namespace

// Estimated times in nanoseconds of a batch with `nnz` non-zeros each in Phi and Psi: by pairs, and by whole states with the
// plain gather.  Fitted on a B200 to expanders of 2^10 .. 2^18 nodes and clouds of 1024 .. 8192 points; us measured, states / pairs:
//   bf16  m = 32, d = 64: expander of 1024, 2 problems 100 / 58, 8192, 3 problems 401 / 227, 2^18, 4 problems 24100 / 8930;
//         m = 16, d = 64: 8192 235 / 213, 200000 8765 / 7365, 50000 (records of 32 columns) 1774 / 1839;  m = 64, d = 32: 533 / 201
//   fp32  m = 32, d = 64: cloud of 1024, 1 problem 71 / 74, 4 problems 174 / 134, 5003, 3 problems 687 / 441;
//         m = d = 64: 8192, 4 problems 2784 / 1696;  m = 16, d = 32: 487 / 454;  lattice of 400, 4 problems 36 / 40
// (the fixed part of the pairs is six launches: regrouping Phi's entries by column takes three).
double grf_pairs_ns(double nnz, int32_t G, int32_t m, int32_t d, int dtype, size_t workspace_per_problem)
{
    double each;
    if (dtype == GRF_DTYPE_BF16) {
        // narrower records where the workspace of a batch holds no whole ones: more passes
        const PairRoom r = pair_room((int64_t)nnz, G, d, dtype, workspace_per_problem * (size_t)G);
        const int32_t w = r.width, ds = m == 64 && w > 32 ? 32 : w;
        each = d / ds * (0.008 + 0.00075 * m + 0.0006 * ds + 0.000008 * m * ds) + d / w * (0.009 + 0.00075 * w);
    } else {
        each = 0.05 + 0.00012 * m * d + 0.0011 * d;
    }
    return 45000.0 + 0.022 * nnz + G * nnz * each;
}
double grf_states_by_rows_ns(double nnz, int32_t nodes, int32_t G, int32_t m, int32_t d, int dtype)
{
    if (dtype == GRF_DTYPE_BF16) {
        const double out_of_l2 = nodes < 400000 ? nodes / 400000.0 : 1.0;       // the gather's slices: 1.4 times the time at 2^17 nodes, 1.7 at 2^18
        return 45000.0 + G * nnz * ((1.0 + out_of_l2) * 0.2 * ((double)m * d + 256.0) / 2304.0 + 0.03 + 0.001 * m);
    }
    return 30000.0 + G * nnz * (0.03 + 0.000265 * m * d);
}

bool grf_pairs_shape(const grf_ctx* ctx, int32_t m, int32_t d)
{
    return ctx->use_tensor_cores && !ctx->tiles_only && (m == 16 || m == 32 || m == 64) && (d == 32 || d == 64);
}

bool grf_pairs_fit(int64_t nnz, int dtype) { return nnz > 0 && pair_bytes(nnz, least_width(dtype)) <= PAIR_MOST; }

int grf_pairs_attn(grf_ctx* ctx, const grf_features* feat, int32_t G, int32_t G_all, int32_t N, int32_t m, int32_t d, int dtype, const void* phiQ,
                   const void* phiK, const void* V, void* out, float* den_out, void* workspace, size_t workspace_bytes)
{
    const bool bf16 = dtype == GRF_DTYPE_BF16;
    const size_t es = bf16 ? 2 : 4;
    const int64_t nnz = feat->phi.nnz;
    const int32_t R = feat->phi.cols;
    PairRoom room = pair_room(nnz, G, d, dtype, workspace_bytes);
    if (room.scratch > 0) {
        const int rc = grf_buf_reserve(&ctx->pair_scratch, room.scratch);
        if (rc == GRF_ERR_NOMEM) room = pair_room(nnz, G, d, dtype, workspace_bytes, false);     // narrower records, fewer problems: the same bits
        if (rc != GRF_OK && (rc != GRF_ERR_NOMEM || room.chunk == 0)) return rc;
    }
    const int32_t width = room.width;
    const int64_t chunk = room.chunk;
    float* records = (float*)(room.scratch > 0 ? ctx->pair_scratch.ptr : workspace);

    // Phi's entries by column
    const int32_t counts_len = (R + 3) & ~3;
    GRF_TRY(grf_buf_reserve(&ctx->t_cursor, sizeof(int32_t) * (3 * (size_t)counts_len + 8)));
    GRF_TRY(grf_reserve_buckets(ctx, nnz + 4));
    float* den = den_out;
    if (!den && width < d) GRF_TRY(grf_den_scratch(ctx, (int64_t)G * N, &den));
    int32_t *counts = (int32_t*)ctx->t_cursor.ptr, *long_count = counts + counts_len, *start = long_count + 4;
    int32_t* long_nodes = start + counts_len + 4;
    const PairLimits limits = pair_limits(nnz + feat->psit.nnz, R, G_all);
    int32_t *slot = (int32_t*)ctx->t_tmp.ptr, *query = slot + ((nnz + 3) & ~(int64_t)3);
    GRF_CUDA_TRY(cudaMemsetAsync(counts, 0, sizeof(int32_t) * ((size_t)counts_len + 2), ctx->stream));
    {
        grf_launch_scope scope(ctx, 3);
        pair_ranks_kernel<<<grf_ceil_div(nnz, 1024), 256, 0, ctx->stream>>>(nnz, (const int32_t*)feat->phi.col.ptr, counts, slot);
    }
    if (R <= GRF_SCAN_DIRECT_MAX) {
        grf_scan_jobs jobs = {};
        jobs.job[0] = {counts, start, nullptr, nullptr};
        GRF_TRY(grf_scan_jobs_launch(ctx, ctx->stream, jobs, 1, R));
    } else {
        GRF_TRY(grf_exclusive_scan(ctx, counts, start, R, 1));
    }
    {
        grf_launch_scope scope(ctx, 3);
        const int row_blocks = grf_ceil_div(N, 8);
        pair_slots_kernel<<<row_blocks + grf_ceil_div(R, 256), 256, 0, ctx->stream>>>(
            N, R, row_blocks, (const int32_t*)feat->phi.rowptr.ptr, (const int32_t*)feat->phi.col.ptr, start,
            (const int32_t*)feat->psit.rowptr.ptr, limits.longer, limits.huge, slot, query, long_count, long_nodes);
    }

    for (int64_t g0 = 0; g0 < G; g0 += chunk) {
        const int32_t gc = (int32_t)(G - g0 < chunk ? G - g0 : chunk);
        PairArgs A = {};
        A.R = R; A.N = N; A.d = d;
        A.t_rowptr = (const int32_t*)feat->psit.rowptr.ptr; A.t_col = (const int32_t*)feat->psit.col.ptr;
        A.t_val = (const float*)feat->psit.val.ptr;
        A.start = start; A.query = query;
        A.long_limit = limits.longer; A.long_count = long_count; A.long_nodes = long_nodes;
        A.phiQ = (const char*)phiQ + (size_t)g0 * N * m * es;
        A.phiK = (const char*)phiK + (size_t)g0 * N * m * es;
        A.V = (const char*)V + (size_t)g0 * N * d * es;
        A.nnz = nnz; A.width = width;
        A.rec = records;
        A.den = A.rec + (size_t)gc * nnz * width;
        for (A.col0 = 0; A.col0 < d; A.col0 += width) {
            {
                grf_launch_scope scope(ctx, 4, 2);
                GRF_TRY(m == 16 ? launch_records_m<16>(ctx, A, gc, bf16)
                                : m == 32 ? launch_records_m<32>(ctx, A, gc, bf16) : launch_records_m<64>(ctx, A, gc, bf16));
            }
            grf_launch_scope scope(ctx, 5);
            void* o = (char*)out + (size_t)g0 * N * d * es;
            float* dn = den ? den + (size_t)g0 * N : nullptr;
            if (bf16) launch_sums<__nv_bfloat16>(ctx, A, gc, feat->phi, slot, o, dn);
            else launch_sums<float>(ctx, A, gc, feat->phi, slot, o, dn);
            GRF_CUDA_TRY(cudaGetLastError());
        }
    }
    return GRF_OK;
}
