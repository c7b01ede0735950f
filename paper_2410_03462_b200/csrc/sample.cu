// Walk sampler and feature assembly (Alg. 1 steps 1-2; Sec. 3.3, Eqs. 9-10).
//
// One warp owns one feature row (ensemble e, source node i); its lanes are walkers.  Every decision
// of a walk is integer (Philox words against a threshold, multiply-high neighbour pick), the load is
// fp32 with a fixed operation order, so the walks do not depend on the launch geometry.  Deposits
// stay in shared memory: the warp sorts their keys by (column, walk, step) with a bitonic network (in
// registers and shuffles for rows of up to 512 deposits), adds equal columns in that order and writes the
// merged row once.
#include "grf_internal.cuh"

namespace {

constexpr uint32_t PHILOX_M0 = 0xD2511F53u, PHILOX_M1 = 0xCD9E8D57u;
constexpr uint32_t PHILOX_W0 = 0x9E3779B9u, PHILOX_W1 = 0xBB67AE85u;

// Philox4x32 with 10 rounds (Salmon et al., SC'11).
__device__ __forceinline__ void philox4x32_10(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3,
                                               uint32_t k0, uint32_t k1, uint32_t (&out)[4])
{
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        const uint32_t hi0 = __umulhi(PHILOX_M0, c0), lo0 = PHILOX_M0 * c0;
        const uint32_t hi1 = __umulhi(PHILOX_M1, c2), lo1 = PHILOX_M1 * c2;
        c0 = hi1 ^ c1 ^ k0;
        c1 = lo1;
        c2 = hi0 ^ c3 ^ k1;
        c3 = lo0;
        k0 += PHILOX_W0;
        k1 += PHILOX_W1;
    }
    out[0] = c0; out[1] = c1; out[2] = c2; out[3] = c3;
}

// factor of the load for a hop along an edge of weight w out of a node of degree deg (Eq. 9)
__device__ __forceinline__ float hop_weight(float w, int32_t deg, float inv_keep)
{
    return __fmul_rn(__fmul_rn(w, (float)deg), inv_keep);
}

// State of one walker.
struct Walker {
    int32_t v, beg, deg;     // where it stands, and that node's edges
    float load;

    // edges: the records of edge_records_kernel, or null: then the CSR arrays are read
    __device__ __forceinline__ void hop(uint32_t r_next, const grf_walk_params& P, const int32_t* __restrict__ rowptr,
                                        const int32_t* __restrict__ col, const float* __restrict__ w,
                                        const int4* __restrict__ edges)
    {
        const int32_t eidx = beg + (int32_t)__umulhi(r_next, (uint32_t)deg);
        if (edges) {
            const int4 r = __ldg(edges + eidx);
            v = r.x; load = __fmul_rn(load, __int_as_float(r.y)); beg = r.z; deg = r.w;
        } else {
            load = __fmul_rn(load, hop_weight(__ldg(w + eidx), deg, P.inv_keep));
            v = __ldg(col + eidx);
            beg = __ldg(rowptr + v);
            deg = __ldg(rowptr + v + 1) - beg;
        }
    }
};

// One 16-byte record per edge u -> v: v, the factor of the hop's load, and where v's own edges are.  A hop of a warp's 32
// walkers then costs one gather instead of four, and fewer instructions.  Eight lanes per row.  (How many edges a graph has
// is known on the device only: the records have the room that earlier graphs needed, and a larger graph is walked through
// its CSR arrays until its number has reached the host.)
// It also clears what the walk kernel counts into, and tells the host how many edges there are if they found no room.
__global__ void __launch_bounds__(256)
edge_records_kernel(int32_t N, int64_t room, float inv_keep, const int32_t* __restrict__ rowptr, const int32_t* __restrict__ col,
                    const float* __restrict__ w, int4* __restrict__ edges, int32_t* __restrict__ col_counts,
                    int32_t* __restrict__ long_count, int32_t* __restrict__ host_edges)
{
    const int32_t E = rowptr[N];
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        if (E > room) *host_edges = E;
        *long_count = 0;
    }
    const int32_t u = blockIdx.x * 32 + (threadIdx.x >> 3);
    if (u >= N) return;
    if ((threadIdx.x & 7) == 0) col_counts[u] = 0;
    if (E > room) return;
    const int32_t beg = rowptr[u], end = rowptr[u + 1];
    for (int32_t p = beg + (threadIdx.x & 7); p < end; p += 8) {
        const int32_t v = col[p], vb = rowptr[v];
        edges[p] = make_int4(v, __float_as_int(hop_weight(w[p], end - beg, inv_keep)), vb, rowptr[v + 1] - vb);
    }
}

// the smaller of v and x, or the larger where `larger` is set: one comparison, one selection
__device__ __forceinline__ uint32_t min_or_max(uint32_t v, uint32_t x, bool larger)
{
    uint32_t r;
    asm("{\n\t.reg .pred p, q;\n\t"
        "setp.ne.u32 q, %3, 0;\n\t"
        "setp.lt.xor.u32 p, %1, %2, q;\n\t"
        "selp.u32 %0, %1, %2, p;\n\t}"
        : "=r"(r) : "r"(v), "r"(x), "r"((uint32_t)larger));
    return r;
}

// Bitonic sort of 32 * E keys held E per lane (key x = lane * E + r sits in register r of its lane): partners closer than E
// are registers of the same lane, the others are reached with one shuffle.  Every merge starts by comparing x with its
// mirror image in the block, so all comparators point the same way: two instructions per pair in a lane, three per key
// across lanes.
//
// Then, from the same registers, the places among the first cnt keys where a new column (key >> seq_bits) begins: written
// in order to heads, their number returned.
template <int E>
__device__ __forceinline__ int32_t sort_in_registers(uint32_t* keys, int lane, int32_t cnt, int32_t seq_bits,
                                                     unsigned short* heads)
{
    uint32_t v[E];
#pragma unroll
    for (int r = 0; r < E; ++r) v[r] = keys[r * 32 + lane];          // any order will do
#pragma unroll
    for (int k = 2; k <= 32 * E; k <<= 1) {
        if (k <= E) {
#pragma unroll
            for (int r = 0; r < E; ++r)
                if ((r & (k >> 1)) == 0) {
                    const int x = r ^ (k - 1);
                    const uint32_t mn = min(v[r], v[x]), mx = max(v[r], v[x]);
                    v[r] = mn; v[x] = mx;
                }
        } else {
            const int lm = k / E - 1;                                 // mirrored lane, mirrored register
            const bool larger = (lane & (k / E / 2)) != 0;
            uint32_t p[E];
#pragma unroll
            for (int r = 0; r < E; ++r) p[r] = __shfl_xor_sync(0xffffffffu, v[E - 1 - r], lm);
#pragma unroll
            for (int r = 0; r < E; ++r) v[r] = min_or_max(v[r], p[r], larger);
        }
#pragma unroll
        for (int j = k >> 2; j > 0; j >>= 1) {
            if (j >= E) {
                const bool larger = (lane & (j / E)) != 0;
#pragma unroll
                for (int r = 0; r < E; ++r) v[r] = min_or_max(v[r], __shfl_xor_sync(0xffffffffu, v[r], j / E), larger);
            } else {
#pragma unroll
                for (int r = 0; r < E; ++r)
                    if ((r & j) == 0) {
                        const uint32_t mn = min(v[r], v[r | j]), mx = max(v[r], v[r | j]);
                        v[r] = mn; v[r | j] = mx;
                    }
            }
        }
    }
    __syncwarp();
#pragma unroll
    for (int r = 0; r < E; ++r) keys[lane * E + r] = v[r];
    uint32_t before = __shfl_up_sync(0xffffffffu, v[E - 1], 1) >> seq_bits;
    if (lane == 0) before = 0xffffffffu;                    // no column is that large: the first key is a head
    uint32_t head = 0;
    int32_t mine = 0;
#pragma unroll
    for (int r = 0; r < E; ++r) {
        const uint32_t c = v[r] >> seq_bits;
        if (c != before && lane * E + r < cnt) { head |= 1u << r; ++mine; }
        before = c;
    }
    int32_t inc = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int32_t y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
    }
    int32_t at = inc - mine;
#pragma unroll
    for (int r = 0; r < E; ++r)
        if (head >> r & 1u) heads[at++] = (unsigned short)(lane * E + r);
    return __shfl_sync(0xffffffffu, inc, 31);
}

// shared memory of one warp: keys, the deposits' values by sequence number, the starts of the distinct columns
__host__ __device__ __forceinline__ size_t walk_smem_bytes(int32_t key_slots, int32_t cap)
{
    return ((size_t)key_slots * 4 + (size_t)cap * 4 + (size_t)key_slots * 2 + 15) & ~(size_t)15;
}

// One warp per row; what bounds it is instruction issue, the ALU pipe first (2 290 warp instructions per row of 240
// deposits: hops 650, Philox 360, sort 680, sums 600).
//   walks   lanes are walkers, all at the same step; one block of random words serves two hops, a hop is one gather (the
//           records above), and steps behind the last non-zero coefficient are not taken.
//   sort    the deposits' keys (column, walk, step).  The first deposit of every walk lies at the source, so without
//           KEEP only walk 0's is sorted (it holds the source's place in the row): 32 walks of a cloud leave 208 keys
//           instead of 240, which fit the 256-key network.
//   sums    the distinct columns are found first, then every lane adds one column's deposits in sorted order (the
//           source's first deposits are added where their walk begins), so a column with many deposits delays 31 others
//           once, not once per 32 deposits.
// N = 20011 cloud (40 022 rows, 32 walks of up to 12 hops): 200 us before these three, 130 with them.  (Sums over values laid
// out in sorted order first, which spares the key look-ups, cost as much as they saved.)
//
// KEEP: the row's deposits themselves are kept as well (for grf_remodulate): every prefix deposits whatever its
// coefficient, the sorted list of (step, load) pairs of the row goes to a staging area of stride P.cap, and every
// merged entry records where its deposits begin in that list.  The values are computed by the same operations in
// the same order as without KEEP.
template <bool KEEP>
__global__ void __launch_bounds__(256)
walk_merge_kernel(const __grid_constant__ grf_walk_params P,
                  const int32_t* __restrict__ rowptr, const int32_t* __restrict__ col, const float* __restrict__ w,
                  const int4* __restrict__ edge_records, int64_t edge_room, int32_t stage_stride, int32_t* __restrict__ stage_col, float* __restrict__ stage_val,
                  int32_t* __restrict__ counts, int32_t counts_stride, int32_t* __restrict__ stage_dep_start,
                  unsigned char* __restrict__ stage_dep_t, float* __restrict__ stage_dep_load, int32_t* __restrict__ dep_counts)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    const int warps = blockDim.x >> 5;
    const int32_t row = blockIdx.x * warps + warp;
    if (row >= 2 * P.N) return;
    const int32_t e = row >= P.N ? 1 : 0;
    const int32_t i = row - e * P.N;

    const int32_t key_slots = max(32, 1 << P.seq_bits);   // the sort pads a row to at least one key per lane
    unsigned char* mine = smem_raw + (size_t)warp * walk_smem_bytes(key_slots, P.cap);
    uint32_t* keys = reinterpret_cast<uint32_t*>(mine);
    float* vals = reinterpret_cast<float*>(keys + key_slots);
    unsigned short* heads = reinterpret_cast<unsigned short*>(vals + P.cap);
    const uint32_t lt_mask = (1u << lane) - 1u;
    const int32_t Lp1 = P.max_len + 1;
    const int32_t steps = KEEP ? P.max_len : P.last_step[e];
    // value of a deposit before the first hop: (f_0 * 1) / n
    const float first = __fmul_rn(__fmul_rn(P.f[e][0], 1.0f), P.inv_n);
    const bool at_source = !KEEP && P.f[e][0] != 0.0f;

    const int4* edges = __ldg(rowptr + P.N) <= edge_room ? edge_records : nullptr;
    const int32_t src_beg = __ldg(rowptr + i), src_deg = __ldg(rowptr + i + 1) - src_beg;

    // ---- walks: lanes are walkers, all at the same step t
    int32_t cnt = 0;
    if (at_source) {
        if (lane == 0) keys[0] = (uint32_t)i << P.seq_bits;
        cnt = 1;
    }
    for (int32_t k0 = 0; k0 < P.n_walks; k0 += 32) {
        const int32_t k = k0 + lane;
        Walker wk;
        wk.v = i; wk.beg = src_beg; wk.deg = src_deg; wk.load = 1.0f;
        bool alive = k < P.n_walks;
        float* my_vals = vals + k * Lp1;
        uint32_t word_key = (uint32_t)(k * Lp1);                 // the deposit's sequence number
        auto deposit = [&](int32_t t, uint32_t mask) {
            const float ft = P.f[e][t];
            if (KEEP || ft != 0.0f) {
                if (alive) {
                    keys[cnt + __popc(mask & lt_mask)] = ((uint32_t)wk.v << P.seq_bits) | (word_key + (uint32_t)t);
                    my_vals[t] = KEEP ? wk.load : __fmul_rn(__fmul_rn(ft, wk.load), P.inv_n);
                }
                cnt += __popc(mask);
            }
        };
        if (KEEP) deposit(0, __ballot_sync(0xffffffffu, alive));
        // a block of random words serves two hops: words 0 and 2 are the halting coins, 1 and 3 pick the neighbours
        for (int32_t t = 0; t < steps; t += 2) {
            uint32_t words[4];
            philox4x32_10((uint32_t)i, (uint32_t)k, (uint32_t)(t >> 1), (uint32_t)e, P.key0, P.key1, words);
            alive = alive && words[0] >= P.halt_threshold && wk.deg != 0;
            uint32_t mask = __ballot_sync(0xffffffffu, alive);
            if (mask == 0u) break;
            if (alive) wk.hop(words[1], P, rowptr, col, w, edges);
            deposit(t + 1, mask);
            if (t + 1 >= steps) break;
            alive = alive && words[2] >= P.halt_threshold && wk.deg != 0;
            mask = __ballot_sync(0xffffffffu, alive);
            if (mask == 0u) break;
            if (alive) wk.hop(words[3], P, rowptr, col, w, edges);
            deposit(t + 2, mask);
        }
    }
    __syncwarp();

    // ---- sort the row's deposits by (column, walk, step)
    int32_t Psort = 32;
    while (Psort < cnt) Psort <<= 1;
    for (int32_t x = cnt + lane; x < Psort; x += 32) keys[x] = 0xffffffffu;
    __syncwarp();
    int32_t r = 0;                                        // distinct columns
    if (Psort <= 512) {
        switch (Psort) {
            case 32: r = sort_in_registers<1>(keys, lane, cnt, P.seq_bits, heads); break;
            case 64: r = sort_in_registers<2>(keys, lane, cnt, P.seq_bits, heads); break;
            case 128: r = sort_in_registers<4>(keys, lane, cnt, P.seq_bits, heads); break;
            case 256: r = sort_in_registers<8>(keys, lane, cnt, P.seq_bits, heads); break;
            default: r = sort_in_registers<16>(keys, lane, cnt, P.seq_bits, heads); break;
        }
    } else {
        for (int32_t k = 2; k <= Psort; k <<= 1)
            for (int32_t j = k >> 1; j > 0; j >>= 1) {
                for (int32_t idx = lane; idx < (Psort >> 1); idx += 32) {
                    const int32_t a = ((idx & ~(j - 1)) << 1) | (idx & (j - 1));
                    const int32_t b = a | j;
                    const uint32_t ka = keys[a], kb = keys[b];
                    const bool up = (a & k) == 0;
                    if ((ka > kb) == up) { keys[a] = kb; keys[b] = ka; }
                }
                __syncwarp();
            }
        for (int32_t base = 0; base < cnt; base += 32) {
            const int32_t p = base + lane;
            const bool head = p < cnt && (p == 0 || (keys[p - 1] >> P.seq_bits) != (keys[p] >> P.seq_bits));
            const uint32_t hm = __ballot_sync(0xffffffffu, head);
            if (head) heads[r + __popc(hm & lt_mask)] = (unsigned short)p;
            r += __popc(hm);
        }
    }
    __syncwarp();
    const uint32_t seq_mask = (1u << P.seq_bits) - 1u;
    const size_t out_base = (size_t)row * stage_stride;
    const size_t dep_base = (size_t)row * P.cap;
    if (KEEP)
        for (int32_t p = lane; p < cnt; p += 32) {
            stage_dep_t[dep_base + p] = (unsigned char)((int32_t)(keys[p] & seq_mask) % Lp1);
            stage_dep_load[dep_base + p] = vals[keys[p] & seq_mask];
        }

    // ---- add every column's deposits in sorted order; one lane per distinct column
    // value of the deposit with sequence number seq = walk * (max_len + 1) + t
    auto term = [&](uint32_t seq) {
        if (!KEEP) return vals[seq];
        const int32_t t = (int32_t)seq % Lp1;
        return __fmul_rn(__fmul_rn(P.f[e][t], vals[seq]), P.inv_n);
    };
    for (int32_t d = lane; d < r; d += 32) {
        const int32_t p = heads[d], end = d + 1 < r ? heads[d + 1] : cnt;
        const uint32_t c = keys[p] >> P.seq_bits;
        float s;
        if (at_source && c == (uint32_t)i) {
            s = first;                                   // walk 0 begins
            int32_t begun = Lp1;                         // sequence number at which the next walk begins
            for (int32_t q = p + 1; q < end; ++q) {
                const int32_t seq = (int32_t)(keys[q] & seq_mask);
                for (; begun <= seq; begun += Lp1) s = __fadd_rn(s, first);
                s = __fadd_rn(s, vals[seq]);
            }
            for (; begun < P.cap; begun += Lp1) s = __fadd_rn(s, first);
        } else {
            s = term(keys[p] & seq_mask);
            for (int32_t q = p + 1; q < end; ++q) s = __fadd_rn(s, term(keys[q] & seq_mask));
        }
        stage_col[out_base + d] = (int32_t)c;
        stage_val[out_base + d] = s;
        if (KEEP) stage_dep_start[out_base + d] = p;
        if (e == 1) atomicAdd(counts + 2 * (size_t)counts_stride + c, 1);      // entries per column of Psi
    }
    if (lane == 0) {
        counts[(size_t)e * counts_stride + i] = r;
        if (KEEP) dep_counts[(size_t)e * counts_stride + i] = cnt;
    }
}

// Kept deposits: moves every row's sorted (step, load) list from the staging area to its place and turns the
// entries' in-row start positions into absolute offsets (dep_ptr has one more element than the matrix has entries).
__global__ void __launch_bounds__(256)
compact_deposits_kernel(int32_t N, int32_t stage_stride, int32_t cap,
                        const int32_t* __restrict__ stage_dep_start, const unsigned char* __restrict__ stage_dep_t,
                        const float* __restrict__ stage_dep_load,
                        const int32_t* __restrict__ rowptr_phi, const int32_t* __restrict__ rowptr_psi,
                        const int32_t* __restrict__ dep_rowptr2,
                        int32_t* __restrict__ ptr_phi, unsigned char* __restrict__ t_phi, float* __restrict__ load_phi,
                        int32_t* __restrict__ ptr_psi, unsigned char* __restrict__ t_psi, float* __restrict__ load_psi)
{
    const int lane = threadIdx.x & 31;
    const int32_t row = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (row >= 2 * N) return;
    const int32_t e = row >= N ? 1 : 0;
    const int32_t i = row - e * N;
    const int32_t* rp = e ? rowptr_psi : rowptr_phi;
    const int32_t* drp = dep_rowptr2 + (size_t)e * (N + 1);
    int32_t* optr = e ? ptr_psi : ptr_phi;
    unsigned char* ot = e ? t_psi : t_phi;
    float* ol = e ? load_psi : load_phi;
    const int32_t beg = rp[i], len = rp[i + 1] - beg;
    const int32_t dbeg = drp[i], dlen = drp[i + 1] - dbeg;
    for (int32_t x = lane; x < len; x += 32) optr[beg + x] = dbeg + stage_dep_start[(size_t)row * stage_stride + x];
    for (int32_t x = lane; x < dlen; x += 32) {
        ot[dbeg + x] = stage_dep_t[(size_t)row * cap + x];
        ol[dbeg + x] = stage_dep_load[(size_t)row * cap + x];
    }
    if (i == N - 1 && lane == 0) optr[rp[N]] = drp[N];
}

// Re-modulation (Alg. 1 step 2 with new "learnable mask parameters (f_i)"): every entry's value is rebuilt from its
// kept deposits as sum (f_t * load) * (1/n), the products and the sum taken in the sampler's operations and order.
struct grf_remod_params { float f[2][GRF_MAX_WALK_LEN + 1]; float inv_n; };
__global__ void index_as_float_kernel(int32_t n, float* __restrict__ out)
{
    const int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = (float)i;
}

__global__ void float_to_index_kernel(int32_t n, const float* __restrict__ in, int32_t* __restrict__ out)
{
    const int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = (int32_t)in[i];
}

// out[x] = src[perm[x]]: Psi^T's values from Psi's
__global__ void gather_values_kernel(int32_t n, const int32_t* __restrict__ perm, const float* __restrict__ src,
                                     float* __restrict__ out)
{
    const int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = src[perm[i]];
}

__global__ void __launch_bounds__(256)
remodulate_kernel(const __grid_constant__ grf_remod_params P, int32_t e, int64_t nnz, const int32_t* __restrict__ dep_ptr,
                  const unsigned char* __restrict__ dep_t, const float* __restrict__ dep_load, float* __restrict__ val)
{
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= nnz) return;
    const int32_t beg = dep_ptr[p], end = dep_ptr[p + 1];
    float s = 0.0f;
    for (int32_t q = beg; q < end; ++q) {
        const float term = __fmul_rn(__fmul_rn(P.f[e][dep_t[q]], dep_load[q]), P.inv_n);
        s = q == beg ? term : __fadd_rn(s, term);
    }
    val[p] = s;
}

// Copies each merged row from the fixed-stride staging area to its place in the CSR arrays, and Psi's entries at once into
// their column's bucket of Psi^T (in arrival order; the buckets are ordered afterwards).
__global__ void __launch_bounds__(256)
place_rows_kernel(int32_t N, int32_t stage_stride, const int32_t* __restrict__ stage_col,
                  const float* __restrict__ stage_val,
                  const int32_t* __restrict__ rowptr_phi, const int32_t* __restrict__ rowptr_psi,
                  int32_t* __restrict__ col_phi, float* __restrict__ val_phi,
                  int32_t* __restrict__ col_psi, float* __restrict__ val_psi, int32_t* __restrict__ cursor,
                  int2* __restrict__ buckets)
{
    const int lane = threadIdx.x & 31;
    const int32_t row = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (row >= 2 * N) return;
    // the rows of Psi first: their scatter takes longer
    const int32_t e = row >= N ? 0 : 1;
    const int32_t i = row - (1 - e) * N;
    const int32_t* rp = e ? rowptr_psi : rowptr_phi;
    const int32_t beg = rp[i], len = rp[i + 1] - beg;
    const size_t src = (size_t)(e * N + i) * stage_stride;
    for (int32_t x = lane; x < len; x += 32) {
        const int32_t c = stage_col[src + x];
        const float v = stage_val[src + x];
        (e ? col_psi : col_phi)[beg + x] = c;
        (e ? val_psi : val_phi)[beg + x] = v;
        if (e) buckets[atomicAdd(cursor + c, 1)] = make_int2(i, __float_as_int(v));
    }
}

__global__ void __launch_bounds__(256)
debug_walks_kernel(const __grid_constant__ grf_walk_params P,
                   const int32_t* __restrict__ rowptr, const int32_t* __restrict__ col, const float* __restrict__ w,
                   int32_t* __restrict__ traj, float* __restrict__ load)
{
    const int64_t total = 2ll * P.N * P.n_walks;
    const int64_t id = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (id >= total) return;
    const int32_t k = (int32_t)(id % P.n_walks);
    const int64_t row = id / P.n_walks;
    const int32_t e = row >= P.N ? 1 : 0;
    const int32_t i = (int32_t)(row - (int64_t)e * P.N);
    const int32_t Lp1 = P.max_len + 1;
    int32_t* tr = traj + id * Lp1;
    float* ld = load + id * Lp1;
    Walker wk;
    wk.v = i; wk.beg = rowptr[i]; wk.deg = rowptr[i + 1] - wk.beg; wk.load = 1.0f;
    uint32_t words[4] = {0, 0, 0, 0};
    int32_t t = 0;
    for (;; ++t) {
        tr[t] = wk.v; ld[t] = wk.load;
        if (t == P.max_len) break;
        if ((t & 1) == 0) philox4x32_10((uint32_t)i, (uint32_t)k, (uint32_t)(t >> 1), (uint32_t)e, P.key0, P.key1, words);
        if (((t & 1) ? words[2] : words[0]) < P.halt_threshold || wk.deg == 0) break;
        wk.hop((t & 1) ? words[3] : words[1], P, rowptr, col, w, nullptr);
    }
    for (++t; t < Lp1; ++t) { tr[t] = -1; ld[t] = 0.0f; }
}

// Consistency of a device-resident CSR graph: row pointers start at 0 and never decrease, column indices lie in
// [0, N).  A thread reads col only inside its own row's extent after checking that the extent lies inside
// [0, rowptr[N]], the length the caller vouches for.  Any violation sets *bad.
__global__ void __launch_bounds__(256)
check_graph_kernel(int32_t N, const int32_t* __restrict__ rowptr, const int32_t* __restrict__ col, int* __restrict__ bad)
{
    const int32_t E = rowptr[N];
    if (blockIdx.x == 0 && threadIdx.x == 0 && (rowptr[0] != 0 || E < 0)) *bad = 1;
    for (int32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < N; i += gridDim.x * blockDim.x) {
        const int32_t beg = rowptr[i], end = rowptr[i + 1];
        if (beg < 0 || end < beg || end > E) { *bad = 1; continue; }
        for (int32_t p = beg; p < end; ++p) {
            const int32_t c = col[p];
            if (c < 0 || c >= N) *bad = 1;
        }
    }
}

}  // namespace

int grf_walk_params_init(grf_walk_params* p, int32_t N, uint64_t seed, int32_t n_walks, float p_halt,
                         int32_t max_len, const float* f_phi, const float* f_psi)
{
    if (N <= 0 || n_walks < 1 || max_len < 0 || max_len > GRF_MAX_WALK_LEN || !f_phi) return GRF_ERR_INVALID;
    if (!(p_halt >= 0.0f) || !(p_halt < 1.0f)) return GRF_ERR_INVALID;
    const int64_t cap = (int64_t)n_walks * (max_len + 1);
    if (cap > 16384) return GRF_ERR_TOO_LARGE;
    int bits = 1;
    while ((1ll << bits) < cap) ++bits;
    if (((int64_t)N << bits) > (1ll << 32)) return GRF_ERR_TOO_LARGE;
    p->N = N; p->n_walks = n_walks; p->max_len = max_len;
    p->key0 = (uint32_t)seed; p->key1 = (uint32_t)(seed >> 32);
    double thr = (double)p_halt * 4294967296.0;   // halt iff word < floor(p_halt * 2^32)
    if (thr > 4294967295.0) thr = 4294967295.0;
    p->halt_threshold = (uint32_t)thr;            // conversion truncates: floor for values >= 0
    p->inv_keep = 1.0f / (1.0f - p_halt);
    p->inv_n = 1.0f / (float)n_walks;
    p->cap = (int32_t)cap;
    p->seq_bits = bits;
    if (!f_psi) f_psi = f_phi;
    for (int t = 0; t <= GRF_MAX_WALK_LEN; ++t) {
        p->f[0][t] = t <= max_len ? f_phi[t] : 0.0f;
        p->f[1][t] = t <= max_len ? f_psi[t] : 0.0f;
    }
    for (int e = 0; e < 2; ++e) {
        p->last_step[e] = max_len;
        while (p->last_step[e] > 0 && p->f[e][p->last_step[e]] == 0.0f) --p->last_step[e];
    }
    return GRF_OK;
}

// Row pointers of Phi, Psi and Psi^T (and the scatter cursors of the latter) from the counts; totals to the object's size slot.
static int sample_row_pointers(grf_ctx* ctx, grf_features* feat, int32_t N, int32_t stride_counts, int32_t* cursor)
{
    const int32_t* counts = (const int32_t*)ctx->counts.ptr;
    int32_t* out[3] = {(int32_t*)feat->phi.rowptr.ptr, (int32_t*)feat->psi.rowptr.ptr, (int32_t*)feat->psit.rowptr.ptr};
    if (N <= GRF_SCAN_DIRECT_MAX) {
        grf_scan_jobs jobs = {};
        for (int x = 0; x < 3; ++x)
            jobs.job[x] = {counts + (size_t)x * stride_counts, out[x], x == 2 ? cursor : nullptr, x == 2 ? nullptr : feat->sizes.host + x};
        return grf_scan_jobs_launch(ctx, ctx->stream, jobs, 3, N);
    }
    for (int x = 0; x < 3; ++x) GRF_TRY(grf_exclusive_scan(ctx, counts + (size_t)x * stride_counts, out[x], N, 1));
    GRF_CUDA_TRY(cudaMemcpyAsync(cursor, out[2], (size_t)N * sizeof(int32_t), cudaMemcpyDeviceToDevice, ctx->stream));
    for (int x = 0; x < 2; ++x)
        GRF_CUDA_TRY(cudaMemcpyAsync(feat->sizes.host + x, out[x] + N, sizeof(int32_t), cudaMemcpyDeviceToHost, ctx->stream));
    return GRF_OK;
}

// Up to this many entries per matrix the arrays of an object that is sampled again are made for the largest sample there can
// be, so that nothing has to be known about it before the kernels are queued, and grf_sample does not wait.  The first sample
// of an object waits and takes what it needs: features that are frozen (one object per layer and head) hold their non-zeros,
// where the bound is several times as much (cloud of 4096 points: 41 MB against 10).  Where the bound is 0.2 MB an object at
// most, it is not worth the wait (10 us of 86 for the first pass on a lattice of 64 nodes).
constexpr int64_t SAMPLE_WHOLE_ENTRIES = 4 << 20, SAMPLE_SMALL_ENTRIES = 8 << 10;

static int sample_into(grf_ctx* ctx, grf_features* feat, const grf_walk_params& P,
                       const int32_t* rowptr, const int32_t* col, const float* w)
{
    const int32_t N = P.N;
    const int32_t stride = P.cap < N ? P.cap : N;   // a row cannot hold more distinct columns than N
    const size_t rows2 = 2 * (size_t)N;
    const int64_t most = (int64_t)N * stride;
    const bool whole = most <= (feat->sampled ? SAMPLE_WHOLE_ENTRIES : SAMPLE_SMALL_ENTRIES) && !ctx->keep_walks;
    const int32_t stride_counts = (N + 3) & ~3;
    GRF_TRY(grf_buf_reserve(&ctx->stage_col, rows2 * stride * sizeof(int32_t)));
    GRF_TRY(grf_buf_reserve(&ctx->stage_val, rows2 * stride * sizeof(float)));
    GRF_TRY(grf_buf_reserve(&ctx->counts, 3 * (size_t)stride_counts * sizeof(int32_t)));
    GRF_TRY(grf_buf_reserve(&ctx->t_cursor, sizeof(int32_t) * (3 * (size_t)N + 1)));
    grf_csr_dev* const mats[3] = {&feat->phi, &feat->psi, &feat->psit};
    for (grf_csr_dev* m : mats) {
        if (whole) {
            GRF_TRY(grf_csr_reserve(m, N, N, most));
        } else {                                    // columns and values when their number is known
            m->rows = m->cols = N;
            GRF_TRY(grf_buf_reserve(&m->rowptr, sizeof(int32_t) * ((size_t)N + 1)));
        }
    }
    if (whole) GRF_TRY(grf_reserve_buckets(ctx, most));
    int32_t* counts = (int32_t*)ctx->counts.ptr;
    int32_t *long_count = (int32_t*)ctx->t_cursor.ptr, *cursor = long_count + 1, *long_list = cursor + N;

    // Room for the edge records by the last graph that is known to have found none: the kernels compare it with their own
    // graph's edges and read the CSR arrays where it is too small.  (An earlier sample may be writing the number just now;
    // either value will do.)
    const int64_t edges_seen = *(volatile const int32_t*)(ctx->pinned + grf_ctx::PINNED_EDGES);
    if (edges_seen > (int64_t)(ctx->edge_records.bytes / sizeof(int4)))
        (void)grf_buf_reserve(&ctx->edge_records, sizeof(int4) * ((size_t)edges_seen + (size_t)edges_seen / 8 + 64));
    int4* edges = (int4*)ctx->edge_records.ptr;
    const int64_t edge_room = (int64_t)(ctx->edge_records.bytes / sizeof(int4));

    const bool keep = ctx->keep_walks;
    feat->kept.valid = false;
    feat->kept.perm_valid = false;
    int32_t* dep_scan[2] = {nullptr, nullptr};
    if (keep) {
        GRF_TRY(grf_buf_reserve(&ctx->stage_dep_start, rows2 * stride * sizeof(int32_t)));
        GRF_TRY(grf_buf_reserve(&ctx->stage_dep_t, rows2 * (size_t)P.cap));
        GRF_TRY(grf_buf_reserve(&ctx->stage_dep_load, rows2 * (size_t)P.cap * sizeof(float)));
        GRF_TRY(grf_buf_reserve(&ctx->dep_counts, 2 * (size_t)stride_counts * sizeof(int32_t)));
        GRF_TRY(grf_buf_reserve(&ctx->dep_rowptr2, 2 * ((size_t)N + 1) * sizeof(int32_t)));
        for (int e = 0; e < 2; ++e) dep_scan[e] = (int32_t*)ctx->dep_rowptr2.ptr + (size_t)e * (N + 1);
    }

    const size_t per_warp = walk_smem_bytes(1 << P.seq_bits < 32 ? 32 : 1 << P.seq_bits, P.cap);
    int warps = (int)((200u * 1024u) / per_warp);
    if (warps > 8) warps = 8;
    if (warps < 1) warps = 1;
    const size_t smem = per_warp * warps;
    static_assert(sizeof(grf_walk_params) <= 4096, "kernel parameter block too large");
    GRF_CUDA_TRY(cudaFuncSetAttribute(keep ? walk_merge_kernel<true> : walk_merge_kernel<false>,
                                      cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    {
        grf_launch_scope scope(ctx, 0, 2);
        edge_records_kernel<<<grf_ceil_div(N, 32), 256, 0, ctx->stream>>>(
            N, edge_room, P.inv_keep, rowptr, col, w, edges, counts + 2 * (size_t)stride_counts, long_count,
            ctx->pinned + grf_ctx::PINNED_EDGES);
        if (keep)
            walk_merge_kernel<true><<<grf_ceil_div(rows2, warps), warps * 32, smem, ctx->stream>>>(
                P, rowptr, col, w, edges, edge_room, stride, (int32_t*)ctx->stage_col.ptr, (float*)ctx->stage_val.ptr,
                counts, stride_counts, (int32_t*)ctx->stage_dep_start.ptr, (unsigned char*)ctx->stage_dep_t.ptr,
                (float*)ctx->stage_dep_load.ptr, (int32_t*)ctx->dep_counts.ptr);
        else
            walk_merge_kernel<false><<<grf_ceil_div(rows2, warps), warps * 32, smem, ctx->stream>>>(
                P, rowptr, col, w, edges, edge_room, stride, (int32_t*)ctx->stage_col.ptr, (float*)ctx->stage_val.ptr,
                counts, stride_counts, nullptr, nullptr, nullptr, nullptr);
    }
    GRF_CUDA_TRY(cudaGetLastError());
    GRF_TRY(sample_row_pointers(ctx, feat, N, stride_counts, cursor));
    if (keep)
        for (int e = 0; e < 2; ++e) {
            GRF_TRY(grf_exclusive_scan(ctx, (const int32_t*)ctx->dep_counts.ptr + (size_t)e * stride_counts, dep_scan[e], N, 1));
            GRF_CUDA_TRY(cudaMemcpyAsync(feat->sizes.host + 2 + e, dep_scan[e] + N, sizeof(int32_t), cudaMemcpyDeviceToHost, ctx->stream));
        }
    GRF_CUDA_TRY(cudaEventRecord(feat->sizes.ready, ctx->stream));
    feat->sizes_pending = true;
    {
        // expected deposits of a walk: 1 + keep + ... + keep^max_len
        double deposits = 0.0, reached = 1.0;
        for (int32_t t = 0; t <= P.max_len; ++t) { deposits += reached; reached /= P.inv_keep; }
        deposits *= P.n_walks;
        feat->expected_entries = (double)N * (deposits < N ? deposits : N);
    }
    feat->plan_stale = true;       // the block plan of Phi is built by the first attention call that needs it
    feat->plan_ready = false;
    grf_mask_invalidate(feat);
    if (!whole) {
        // column/value arrays, grown with head-room so that resampling rarely reallocates
        GRF_TRY(grf_settle_sizes(feat));
        for (grf_csr_dev* m : mats)
            if (!m->col.ptr || !m->val.ptr || m->col.bytes < (size_t)m->nnz * 4 || m->val.bytes < (size_t)m->nnz * 4)
                GRF_TRY(grf_csr_reserve(m, N, N, m->nnz + m->nnz / 8 + 64));
        GRF_TRY(grf_reserve_buckets(ctx, feat->psi.nnz));
    }
    int2* buckets = (int2*)ctx->t_tmp.ptr;
    {
        grf_launch_scope scope(ctx, 2);
        place_rows_kernel<<<grf_ceil_div(rows2, 8), 256, 0, ctx->stream>>>(
            N, stride, (const int32_t*)ctx->stage_col.ptr, (const float*)ctx->stage_val.ptr,
            (const int32_t*)feat->phi.rowptr.ptr, (const int32_t*)feat->psi.rowptr.ptr,
            (int32_t*)feat->phi.col.ptr, (float*)feat->phi.val.ptr,
            (int32_t*)feat->psi.col.ptr, (float*)feat->psi.val.ptr, cursor, buckets);
    }
    {
        grf_launch_scope scope(ctx, 3, 2);
        GRF_TRY(grf_order_buckets(ctx->stream, N, N, (const int32_t*)feat->psit.rowptr.ptr, buckets, long_count, long_list,
                                  (int32_t*)feat->psit.col.ptr, (float*)feat->psit.val.ptr));
    }
    GRF_CUDA_TRY(cudaGetLastError());
    if (keep) {
        grf_kept_walks& K = feat->kept;
        const int64_t nnz_e[2] = {feat->phi.nnz, feat->psi.nnz};
        for (int e = 0; e < 2; ++e) {
            K.deposits[e] = feat->sizes.host[2 + e];
            const size_t dcap = (size_t)K.deposits[e] + (size_t)K.deposits[e] / 8 + 64;
            if (K.dep_ptr[e].bytes < ((size_t)nnz_e[e] + 1) * 4)
                GRF_TRY(grf_buf_reserve(&K.dep_ptr[e], ((size_t)nnz_e[e] + (size_t)nnz_e[e] / 8 + 65) * 4));
            if (K.dep_t[e].bytes < (size_t)K.deposits[e]) GRF_TRY(grf_buf_reserve(&K.dep_t[e], dcap));
            if (K.dep_load[e].bytes < (size_t)K.deposits[e] * 4) GRF_TRY(grf_buf_reserve(&K.dep_load[e], dcap * 4));
        }
        {
            grf_launch_scope scope(ctx, 2);
            compact_deposits_kernel<<<grf_ceil_div(rows2, 8), 256, 0, ctx->stream>>>(
                N, stride, P.cap, (const int32_t*)ctx->stage_dep_start.ptr, (const unsigned char*)ctx->stage_dep_t.ptr,
                (const float*)ctx->stage_dep_load.ptr, (const int32_t*)feat->phi.rowptr.ptr,
                (const int32_t*)feat->psi.rowptr.ptr, (const int32_t*)ctx->dep_rowptr2.ptr,
                (int32_t*)K.dep_ptr[0].ptr, (unsigned char*)K.dep_t[0].ptr, (float*)K.dep_load[0].ptr,
                (int32_t*)K.dep_ptr[1].ptr, (unsigned char*)K.dep_t[1].ptr, (float*)K.dep_load[1].ptr);
        }
        GRF_CUDA_TRY(cudaGetLastError());
        K.n_walks = P.n_walks; K.max_len = P.max_len; K.valid = true;
        K.perm_valid = false;
    }
    feat->sampled = true;
    return GRF_OK;
}

extern "C" int grf_sample(grf_ctx* ctx, int32_t N, const int32_t* rowptr, const int32_t* col, const float* w,
                          uint64_t seed, int32_t n_walks, float p_halt, int32_t max_len,
                          const float* f_phi, const float* f_psi, grf_features** inout)
{
    if (!ctx || !rowptr || !col || !w || !inout) return GRF_ERR_INVALID;
    grf_walk_params P;
    GRF_TRY(grf_walk_params_init(&P, N, seed, n_walks, p_halt, max_len, f_phi, f_psi));
    GRF_CUDA_TRY(cudaSetDevice(ctx->device));
    if (ctx->check_graphs) {
        // debugging aid: one pass over the graph and one wait for the device before any walk is taken
        GRF_CUDA_TRY(cudaMemsetAsync(ctx->error_word + 1, 0, sizeof(int), ctx->stream));
        check_graph_kernel<<<grf_ceil_div(N, 256) > 1184 ? 1184 : grf_ceil_div(N, 256), 256, 0, ctx->stream>>>(
            N, rowptr, col, ctx->error_word + 1);
        GRF_CUDA_TRY(cudaMemcpyAsync(ctx->pinned + 9, ctx->error_word + 1, sizeof(int), cudaMemcpyDeviceToHost, ctx->stream));
        GRF_CUDA_TRY(cudaStreamSynchronize(ctx->stream));
        if (ctx->pinned[9] != 0) return GRF_ERR_BADGRAPH;
    }
    grf_features* feat = *inout;
    if (!feat) GRF_TRY(grf_features_new(&feat, ctx->device));
    const int rc = sample_into(ctx, feat, P, rowptr, col, w);
    if (rc != GRF_OK) {
        if (*inout) grf_features_clear(feat);       // some of its arrays may be the new sample's already
        else grf_features_free(feat);
        return rc;
    }
    *inout = feat;
    return GRF_OK;
}

extern "C" int grf_debug_walks(grf_ctx* ctx, int32_t N, const int32_t* rowptr, const int32_t* col, const float* w,
                               uint64_t seed, int32_t n_walks, float p_halt, int32_t max_len,
                               int32_t* traj, float* load)
{
    if (!ctx || !rowptr || !col || !w || !traj || !load) return GRF_ERR_INVALID;
    grf_walk_params P;
    float ones[GRF_MAX_WALK_LEN + 1];
    for (float& x : ones) x = 1.0f;
    GRF_TRY(grf_walk_params_init(&P, N, seed, n_walks, p_halt, max_len, ones, ones));
    GRF_CUDA_TRY(cudaSetDevice(ctx->device));
    const int64_t total = 2ll * N * n_walks;
    {
        grf_launch_scope scope(ctx, 0);
        debug_walks_kernel<<<grf_ceil_div(total, 256), 256, 0, ctx->stream>>>(P, rowptr, col, w, traj, load);
    }
    GRF_CUDA_TRY(cudaGetLastError());
    return GRF_OK;
}

extern "C" int grf_ctx_keep_walks(grf_ctx* ctx, int enable)
{
    if (!ctx) return GRF_ERR_INVALID;
    ctx->keep_walks = enable != 0;
    return GRF_OK;
}

extern "C" int grf_remodulate(grf_ctx* ctx, grf_features* feat, int32_t max_len, const float* f_phi, const float* f_psi)
{
    if (!ctx || !feat || !f_phi) return GRF_ERR_INVALID;
    GRF_TRY(grf_features_sizes(feat));
    grf_kept_walks& K = feat->kept;
    if (!K.valid || max_len != K.max_len) return GRF_ERR_INVALID;
    GRF_CUDA_TRY(cudaSetDevice(ctx->device));
    if (!f_psi) f_psi = f_phi;
    grf_remod_params P;
    for (int t = 0; t <= GRF_MAX_WALK_LEN; ++t) {
        P.f[0][t] = t <= max_len ? f_phi[t] : 0.0f;
        P.f[1][t] = t <= max_len ? f_psi[t] : 0.0f;
    }
    P.inv_n = 1.0f / (float)K.n_walks;
    grf_csr_dev* mats[2] = {&feat->phi, &feat->psi};
    for (int e = 0; e < 2; ++e) {
        if (mats[e]->nnz == 0) continue;
        grf_launch_scope scope(ctx, 2);
        remodulate_kernel<<<grf_ceil_div(mats[e]->nnz, 256), 256, 0, ctx->stream>>>(
            P, e, mats[e]->nnz, (const int32_t*)K.dep_ptr[e].ptr, (const unsigned char*)K.dep_t[e].ptr,
            (const float*)K.dep_load[e].ptr, (float*)mats[e]->val.ptr);
    }
    GRF_CUDA_TRY(cudaGetLastError());
    // Psi^T carries copies of Psi's values in another order, which does not change with the coefficients: the first
    // re-modulation regroups the entries' own indices (exact in fp32 below 2^24 entries) and keeps the result; from then
    // on the new values are fetched through it
    const int64_t nnz_psi = feat->psi.nnz;
    if (nnz_psi > 0 && nnz_psi < (1ll << 24)) {
        const int blocks = grf_ceil_div(nnz_psi, 256);
        if (!K.perm_valid) {
            if (K.psit_perm.bytes < (size_t)nnz_psi * 4) GRF_TRY(grf_buf_reserve(&K.psit_perm, ((size_t)nnz_psi + (size_t)nnz_psi / 8 + 64) * 4));
            {
                grf_launch_scope scope(ctx, 2);
                index_as_float_kernel<<<blocks, 256, 0, ctx->stream>>>((int32_t)nnz_psi, (float*)K.psit_perm.ptr);
            }
            GRF_TRY(grf_transpose_launch(ctx, feat->psi.rows, feat->psi.cols, nnz_psi, (const int32_t*)feat->psi.rowptr.ptr,
                                         (const int32_t*)feat->psi.col.ptr, (const float*)K.psit_perm.ptr,
                                         (int32_t*)feat->psit.rowptr.ptr, (int32_t*)feat->psit.col.ptr,
                                         (float*)feat->psit.val.ptr));
            {
                grf_launch_scope scope(ctx, 2);
                float_to_index_kernel<<<blocks, 256, 0, ctx->stream>>>((int32_t)nnz_psi, (const float*)feat->psit.val.ptr,
                                                                       (int32_t*)K.psit_perm.ptr);
            }
            K.perm_valid = true;
        }
        grf_launch_scope scope(ctx, 2);
        gather_values_kernel<<<blocks, 256, 0, ctx->stream>>>((int32_t)nnz_psi, (const int32_t*)K.psit_perm.ptr,
                                                              (const float*)feat->psi.val.ptr, (float*)feat->psit.val.ptr);
    } else {
        GRF_TRY(grf_transpose_launch(ctx, feat->psi.rows, feat->psi.cols, feat->psi.nnz, (const int32_t*)feat->psi.rowptr.ptr,
                                     (const int32_t*)feat->psi.col.ptr, (const float*)feat->psi.val.ptr,
                                     (int32_t*)feat->psit.rowptr.ptr, (int32_t*)feat->psit.col.ptr,
                                     (float*)feat->psit.val.ptr));
    }
    GRF_CUDA_TRY(cudaGetLastError());
    // the structure is the same: the block plan's node lists and the mask's key lists stay; the gather kernel's
    // coefficient table and the mask's values hold the old values
    feat->plan_coef_ready = feat->plan_settled = false;
    grf_mask_values_stale(feat);
    return GRF_OK;
}
