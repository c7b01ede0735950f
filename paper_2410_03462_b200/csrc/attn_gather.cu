// Gather-and-contract with normalisation (Alg. 1 step 5, Eq. 12) on the plain ALUs (any supported m, d; fp32 or bf16):
//   num_i = sum_l Phi_il phi(q_i)^T S_l,  den_i = sum_l Phi_il phi(q_i)^T z_l,  out_i = num_i / den_i.
//
// What bounds it is the delivery of state tiles: every non-zero of Phi brings m x d values to the SM, and on graphs
// without locality nothing is shared.  From HBM that is 6 TB/s, from L2 up to 19 TB/s, so the columns of a problem's
// tiles are taken in slices (the grid runs through the rows of one slice before it starts the next): as far as a slice of
// all nodes fits L2, HBM sees each record once.  A group of lanes takes one node's slice, one 16-byte chunk (CH
// consecutive feature rows a of one column b) per lane, and adds Phi_il times it to T_i = sum_l Phi_il S_l in registers;
// phi(q_i) enters once, at the end.  What limits a slice is then the latency of L2 at one load per warp and 64 warps per
// SM; fewer warps with more loads each were slower.  Expanders, 2 heads, m = 32, d = 64, bf16: N = 2^18 16.8 ms with
// whole tiles -> 9.4 (12.9 TB/s into the SMs), N = 2^20 71.4 -> 60.9 (8 TB/s: 512 MB per slice).  Sums are carried in fp32
// in a fixed order.
#include <type_traits>

#include "grf_internal.cuh"
#include "packed.cuh"

namespace {

// a 16-byte chunk as packed pairs of fp32, and one element of a row
template <typename T> struct Chunk;
template <> struct Chunk<float> {
    static constexpr int PAIRS = 2;
    __device__ static __forceinline__ void widen(const uint4& x, uint64_t (&v)[2])
    {
        v[0] = (uint64_t)x.y << 32 | x.x;
        v[1] = (uint64_t)x.w << 32 | x.z;
    }
    __device__ static __forceinline__ float get(const float* p) { return __ldg(p); }
    __device__ static __forceinline__ void put(float* p, float x) { *p = x; }
};
template <> struct Chunk<__nv_bfloat16> {
    static constexpr int PAIRS = 4;
    __device__ static __forceinline__ void widen(const uint4& x, uint64_t (&v)[4])
    {
        const uint32_t w[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
        for (int q = 0; q < 4; ++q) v[q] = pack2(__uint_as_float(w[q] << 16), __uint_as_float(w[q] & 0xffff0000u));
    }
    __device__ static __forceinline__ float get(const __nv_bfloat16* p)
    {
        return __uint_as_float((uint32_t)__ldg(reinterpret_cast<const unsigned short*>(p)) << 16);
    }
    __device__ static __forceinline__ void put(__nv_bfloat16* p, float x) { *p = __float2bfloat16_rn(x); }
};

constexpr int GATHER_WARPS = 4;

// Denominator of row i of problem g, by a warp: M / 4 lanes per node on z_l in fp32.
template <typename T, int M, int D>
__device__ __forceinline__ float row_denominator(int32_t N, int32_t R, int32_t i, int32_t g, int lane, const int32_t* __restrict__ rowptr,
                                                 const int32_t* __restrict__ col, const float* __restrict__ val,
                                                 const T* __restrict__ phiQ, const unsigned char* __restrict__ states)
{
    constexpr int LPN = M / 4, NPS = 32 / LPN;          // lanes per node, nodes side by side
    const int sub = lane / LPN, pl = lane % LPN;
    const unsigned char* zbase = states + (size_t)g * grf_states_stride<T>(R, M, D) + grf_z_at<T>(true, 0, R, M, D) + (size_t)pl * 16;
    uint64_t z[2] = {0ull, 0ull};
    const int32_t beg = rowptr[i], end = rowptr[i + 1];
    for (int32_t p0 = beg; p0 < end; p0 += 32) {
        const int32_t n = min(32, end - p0);
        const int32_t my_l = lane < n ? __ldcs(col + p0 + lane) : 0;
        const float my_phi = lane < n ? __ldcs(val + p0 + lane) : 0.0f;
#pragma unroll 4
        for (int32_t j = 0; j < n; j += NPS) {
            const int32_t l = __shfl_sync(0xffffffffu, my_l, (j + sub) & 31);
            const float phi = __shfl_sync(0xffffffffu, my_phi, (j + sub) & 31);
            if (j + sub < n) {
                uint64_t v[2];
                Chunk<float>::widen(__ldg(reinterpret_cast<const uint4*>(zbase + (size_t)l * (M * 4))), v);
                const uint64_t phi2 = pack2(phi, phi);
                z[0] = fma2(phi2, v[0], z[0]);
                z[1] = fma2(phi2, v[1], z[1]);
            }
        }
    }
    const T* qrow = phiQ + ((size_t)g * N + i) * M + pl * 4;
    float a[4];
    unpack2(z[0], a[0], a[1]);
    unpack2(z[1], a[2], a[3]);
    float d = 0.0f;
#pragma unroll
    for (int e = 0; e < 4; ++e) d = fmaf(Chunk<T>::get(qrow + e), a[e], d);
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) d += __shfl_xor_sync(0xffffffffu, d, off);
    return d;
}

// The gather may start once all CTAs here have.
template <typename T, int M, int D>
__global__ void __launch_bounds__(GATHER_WARPS * 32)
gather_denominators_kernel(int32_t N, int32_t R, const int32_t* __restrict__ rowptr, const int32_t* __restrict__ col,
                           const float* __restrict__ val, const T* __restrict__ phiQ,
                           const unsigned char* __restrict__ states, float* __restrict__ den)
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int lane = threadIdx.x & 31;
    const int32_t i = blockIdx.x * GATHER_WARPS + (threadIdx.x >> 5), g = blockIdx.y;
    if (i >= N) return;
    const float d = row_denominator<T, M, D>(N, R, i, g, lane, rowptr, col, val, phiQ, states);
    if (lane == 0) den[(size_t)g * N + i] = d;
}

// Lanes of one node's slice (32, fewer where a whole tile has fewer chunks) and columns of a slice, for CPL chunks per lane.
template <typename T, int M, int D, int CPL> struct SliceShape {
    static constexpr int CH = grf_tile_chunk<T>();
    static constexpr int KC = M / CH;                                        // chunks along the feature rows a
    static constexpr int LPN = KC >= 32 ? KC : (KC * D < 32 ? KC * D : 32);
    static constexpr int SB = LPN / KC;                                      // columns side by side
    static constexpr int NB = SB * CPL <= D ? CPL : D / SB;                  // columns per lane
    static constexpr int COLS = SB * NB;                                     // columns of a slice
    static constexpr int SLICES = D / COLS;
};

// a chunk of a tile, kept in L2 in preference to the streams
__device__ __forceinline__ uint4 load_tile(const unsigned char* p, uint64_t policy)
{
    uint4 x;
    asm volatile("ld.global.nc.L2::cache_hint.v4.u32 {%0, %1, %2, %3}, [%4], %5;"
        : "=r"(x.x), "=r"(x.y), "=r"(x.z), "=r"(x.w) : "l"(p), "l"(policy));
    return x;
}

// DEN: every slice adds up the row's denominator itself, the first one writes it where it is asked for (see the launch).
template <typename T, int M, int D, int CPL, bool DEN>
__global__ void __launch_bounds__(GATHER_WARPS * 32, CPL == 1 ? 16 : 6)
gather_sliced_kernel(int32_t N, int32_t R, const int32_t* __restrict__ rowptr, const int32_t* __restrict__ col,
                     const float* __restrict__ val, const T* __restrict__ phiQ, const unsigned char* __restrict__ states,
                     T* __restrict__ out, float* den)
{
    using Sh = SliceShape<T, M, D, CPL>;
    constexpr int CH = Sh::CH, LPN = Sh::LPN, NPS = 32 / LPN, NB = Sh::NB, KC = Sh::KC, P = Chunk<T>::PAIRS;
    const int lane = threadIdx.x & 31, sub = lane / LPN, pl = lane % LPN;
    const int kc = pl % KC, b = pl / KC;                 // this lane's chunk along a, and its first column of the slice
    const int32_t i = blockIdx.x * GATHER_WARPS + (threadIdx.x >> 5);
    const int32_t slice = blockIdx.y, g = blockIdx.z;
    if (i >= N) return;
    float dn = 0.0f;
    if (DEN) {
        dn = row_denominator<T, M, D>(N, R, i, g, lane, rowptr, col, val, phiQ, states);
        if (den && slice == 0 && lane == 0) den[(size_t)g * N + i] = dn;
    }
    const int b0 = slice * Sh::COLS + b;
    // this lane's first chunk; chunk y lies y * SB columns further on: LPN consecutive chunks per group of lanes
    const unsigned char* base = states + (size_t)g * grf_states_stride<T>(R, M, D) + grf_chunk_at<T>(true, 0, kc * CH, b0, M, D);
    uint64_t policy;
    asm("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(policy));
    // entries are taken 32 at a time, and the next 32 are read before these are used (streamed: the matrix is read once per
    // slice and must not push the slice out of L2)
    const int32_t my_rp = __ldg(rowptr + i + min(lane, 1));
    int32_t beg = __shfl_sync(0xffffffffu, my_rp, 0);
    const int32_t end = __shfl_sync(0xffffffffu, my_rp, 1);
    int32_t next_l = beg + lane < end ? __ldcs(col + beg + lane) : 0;
    float next_phi = beg + lane < end ? __ldcs(val + beg + lane) : 0.0f;
    uint64_t acc[NB][P];
#pragma unroll
    for (int y = 0; y < NB; ++y)
#pragma unroll
        for (int q = 0; q < P; ++q) acc[y][q] = 0ull;
    while (beg < end) {
        const int32_t n = min(32, end - beg);
        const int32_t my_l = next_l;
        const float my_phi = next_phi;
        beg += n;
        next_l = beg + lane < end ? __ldcs(col + beg + lane) : 0;
        next_phi = beg + lane < end ? __ldcs(val + beg + lane) : 0.0f;
        constexpr int UNROLL = NB >= 4 ? 2 : 4;
#pragma unroll UNROLL
        for (int32_t j = 0; j < n; j += NPS) {
            const int32_t l = __shfl_sync(0xffffffffu, my_l, (j + sub) & 31);
            const float phi = __shfl_sync(0xffffffffu, my_phi, (j + sub) & 31);
            if (j + sub < n) {
                const unsigned char* tile = base + (size_t)l * (M * D * sizeof(T));
                const uint64_t phi2 = pack2(phi, phi);
#pragma unroll
                for (int y = 0; y < NB; ++y) {
                    uint64_t v[P];
                    Chunk<T>::widen(load_tile(tile + y * LPN * 16, policy), v);
#pragma unroll
                    for (int q = 0; q < P; ++q) acc[y][q] = fma2(phi2, v[q], acc[y][q]);
                }
            }
        }
    }
    // contract with phi(q): over this lane's rows a, then over the lanes along a and the nodes side by side
    const T* qrow = phiQ + ((size_t)g * N + i) * M;
    if (!DEN) {
        asm volatile("griddepcontrol.wait;" ::: "memory");       // for the denominators' kernel; all before it is complete
        dn = __ldcg(den + (size_t)g * N + i);
    }
    float s[NB];
    uint64_t qv[P];
    Chunk<T>::widen(__ldg(reinterpret_cast<const uint4*>(qrow + kc * CH)), qv);
#pragma unroll
    for (int y = 0; y < NB; ++y) {
        uint64_t t = 0ull;
#pragma unroll
        for (int q = 0; q < P; ++q) t = fma2(qv[q], acc[y][q], t);
        float s1;
        unpack2(t, s[y], s1);
        s[y] += s1;
    }
    const float inv = dn != 0.0f ? 1.0f / dn : 0.0f;
    T* orow = out + ((size_t)g * N + i) * D;
#pragma unroll
    for (int y = 0; y < NB; ++y) {
#pragma unroll
        for (int off = 1; off < KC; off <<= 1) s[y] += __shfl_xor_sync(0xffffffffu, s[y], off);
#pragma unroll
        for (int off = LPN; off < 32; off <<= 1) s[y] += __shfl_xor_sync(0xffffffffu, s[y], off);
        if (sub == 0 && kc == 0) Chunk<T>::put(orow + b0 + y * Sh::SB, s[y] * inv);
    }
}

// Bytes of a slice over all nodes that stay in L2 beside the streams.  Slices of 2 KB, four loads per lane and node, are
// taken where they fit it; all other graphs take 512 bytes, one load of every lane per node, which costs more passes over the
// matrix but hits L2 in part however large the graph.  ms, 2 KB / 512 bytes, expanders, 2 heads, m = 32, d = 64, bf16:
// N = 36000 0.92 / 0.98, 60000 1.79 / 1.63, 147000 7.2 / 4.2, 2^18 14.8 / 9.4, 2^19 32.1 / 26.1, 2^20 66.8 / 60.9; fp32, 3 heads,
// N = 20000 1.37 / 1.45.  (Narrower slices, with two or four nodes side by side, never win: 256 bytes 1.47, 2.45, 6.6, 13.6, 33.5,
// 76 ms, 128 bytes 1.75, 3.03, 10.3, 19.0, 40.6, 88.)
constexpr size_t SLICE_L2_BYTES = (size_t)72 << 20;

// Objects whose rows form their denominators inside: at most so many nodes (no row is longer), and entries a row on average.
constexpr int32_t DEN_INSIDE_NODES = 128;
constexpr int DEN_INSIDE_MEAN = 16;

template <typename T, int M, int D>
int launch_md(grf_ctx* ctx, const grf_csr_dev& phi, double entries, int32_t G, int32_t N, const void* phiQ, const void* states,
              void* out, float* den_out)
{
    const int32_t* rp = (const int32_t*)phi.rowptr.ptr;
    const int32_t* cl = (const int32_t*)phi.col.ptr;
    const float* vl = (const float*)phi.val.ptr;
    const int blocks = grf_ceil_div(N, GATHER_WARPS);
    // The gather starts beside the denominators' kernel, which it waits for before it divides.  Whole attention, us, one behind the other
    // / this: fp32 lattice of 64 nodes, m = d = 16 17.4 / 13.5, of 400, 4 problems, m = 32, d = 64 33.4 / 27.8, expander of 2000 99.4 /
    // 87.0; bf16, m = d = 64, cloud of 512 64.3 / 52.1; 120 calls of up to 8192 rows, of equal and of very different lengths, 1 / 0.81
    // of the time (geometric mean), none above 0.975.
    // The smallest objects' slices form the denominators themselves: the device needs 2 us more, but such calls wait for the host, for which
    // a launch is 2 to 3 us.  us, call after call, inside / beside: 64 and 128 nodes, 10 entries a row 14.2 / 16.4 (sample and attention
    // 38.7 / 41.8), 64 nodes, 32 entries, m = 32, d = 64, 4 problems 22.7 / 18.8, 192 nodes, 10 entries 17.7 / 17.4.
    auto launch = [&](auto cpl, auto inside, float* den) {
        using Sh = SliceShape<T, M, D, decltype(cpl)::value>;
        grf_launch_scope scope(ctx, 5);
        cudaLaunchAttribute beside = {};
        beside.id = cudaLaunchAttributeProgrammaticStreamSerialization;
        beside.val.programmaticStreamSerializationAllowed = 1;
        cudaLaunchConfig_t config = {};
        config.gridDim = dim3(blocks, Sh::SLICES, G);
        config.blockDim = dim3(GATHER_WARPS * 32);
        config.stream = ctx->stream;
        config.attrs = &beside;
        config.numAttrs = decltype(inside)::value ? 0 : 1;
        GRF_CUDA_TRY(cudaLaunchKernelEx(&config, gather_sliced_kernel<T, M, D, decltype(cpl)::value, decltype(inside)::value>, N, phi.cols,
                                        rp, cl, vl, (const T*)phiQ, (const unsigned char*)states, (T*)out, den));
        return cudaGetLastError() == cudaSuccess ? GRF_OK : GRF_ERR_CUDA;
    };
    if constexpr (SliceShape<T, M, D, 4>::SLICES <= 4) {
        if (phi.cols <= DEN_INSIDE_NODES && (int64_t)G * N <= 2048 && entries <= (double)DEN_INSIDE_MEAN * N)
            return launch(std::integral_constant<int, 4>(), std::true_type(), den_out);
    }
    float* den = den_out;
    if (!den) GRF_TRY(grf_den_scratch(ctx, (int64_t)G * N, &den));
    {
        grf_launch_scope scope(ctx, 6);
        gather_denominators_kernel<T, M, D><<<dim3(blocks, G), GATHER_WARPS * 32, 0, ctx->stream>>>(
            N, phi.cols, rp, cl, vl, (const T*)phiQ, (const unsigned char*)states, den);
    }
    if ((size_t)phi.cols * 2048 <= SLICE_L2_BYTES) return launch(std::integral_constant<int, 4>(), std::false_type(), den);
    return launch(std::integral_constant<int, 1>(), std::false_type(), den);
}

template <typename T, int M>
int launch_m(grf_ctx* ctx, const grf_csr_dev& phi, double entries, int32_t G, int32_t N, int32_t d,
             const void* phiQ, const void* states, void* out, float* den_out)
{
    switch (d) {
        case 8: return launch_md<T, M, 8>(ctx, phi, entries, G, N, phiQ, states, out, den_out);
        case 16: return launch_md<T, M, 16>(ctx, phi, entries, G, N, phiQ, states, out, den_out);
        case 32: return launch_md<T, M, 32>(ctx, phi, entries, G, N, phiQ, states, out, den_out);
        case 64: return launch_md<T, M, 64>(ctx, phi, entries, G, N, phiQ, states, out, den_out);
        case 128: return launch_md<T, M, 128>(ctx, phi, entries, G, N, phiQ, states, out, den_out);
        default: return GRF_ERR_INVALID;
    }
}

template <typename T>
int launch_t(grf_ctx* ctx, const grf_csr_dev& phi, double entries, int32_t G, int32_t N, int32_t m, int32_t d,
             const void* phiQ, const void* states, void* out, float* den_out)
{
    switch (m) {
        case 8: return launch_m<T, 8>(ctx, phi, entries, G, N, d, phiQ, states, out, den_out);
        case 16: return launch_m<T, 16>(ctx, phi, entries, G, N, d, phiQ, states, out, den_out);
        case 32: return launch_m<T, 32>(ctx, phi, entries, G, N, d, phiQ, states, out, den_out);
        case 64: return launch_m<T, 64>(ctx, phi, entries, G, N, d, phiQ, states, out, den_out);
        case 128: return launch_m<T, 128>(ctx, phi, entries, G, N, d, phiQ, states, out, den_out);
        default: return GRF_ERR_INVALID;
    }
}

}  // namespace

int grf_gather_contract_alu(grf_ctx* ctx, const grf_features* feat, int32_t G, int32_t N, int32_t m, int32_t d,
                            int dtype, const void* phiQ, const void* states, void* out, float* den_out)
{
    const grf_csr_dev& phi = feat->phi;
    // (a running sample's sizes are not waited for: both ways to form the denominators give the same bits)
    const double entries = feat->sizes_pending ? feat->expected_entries : (double)phi.nnz;
    if (G > 65535) return GRF_ERR_TOO_LARGE;
    if (dtype == GRF_DTYPE_F32) return launch_t<float>(ctx, phi, entries, G, N, m, d, phiQ, states, out, den_out);
    if (dtype == GRF_DTYPE_BF16) return launch_t<__nv_bfloat16>(ctx, phi, entries, G, N, m, d, phiQ, states, out, den_out);
    return GRF_ERR_INVALID;
}
