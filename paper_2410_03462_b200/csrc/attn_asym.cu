// Masked attention with asymmetric graph random features (App. "Asymmetric graph random features", Alg. 2):
// with f^(2) = delta_0 the key-side features are the identity, the mask estimate is Phi itself and
//     out_i = sum_l Phi_il A_il v_l / sum_l Phi_il A_il,   A_il = phi(q_i) . phi(k_l)   (linear)
//                                                           A_il = exp(q_i . k_l)         (softmax)
// over the nodes l that the walkers out of node i visited: m + d multiply-adds per non-zero of Phi, no
// per-node states at all.
//
// One warp per query and two problems (they share the row's indices and mask values), non-zeros 32 at a time.  What bounds the
// kernel is the number of cache lines that its loads touch (one per key row and one per value row at the least):
//   scores   M / CH lanes take one key row, 16 bytes each, so an instruction reads 32 CH / M whole rows (a lane per key
//            touched M / CH lines more often than needed: 4 per key at m = 32, bf16); the partial dot products of the
//            instructions are summed and spread over the lanes by one exchange per halving, which leaves every lane one key;
//   values   D / CH lanes take one value row, 16 bytes each, so an instruction adds 32 CH / D rows; the groups are summed once
//            per query.
// The exponentials are taken relative to a running maximum of the scores, which cancels in the quotient; sums are carried
// in fp32 in a fixed order, so results are run-to-run identical.
// Batches of 32 non-zeros, and steps of value rows within a last batch that are whole, take loads without conditions: a
// conditional load also zeroes its registers, and at d >= 8 m these instructions made the kernel slower than a lane per key and
// a warp per value row.  N = 32768 cloud, 8 problems, bf16, softmax, us: lane per key / whole rows, conditional / now: m = 32,
// d = 64 669 / 580 / 493; m = 16, d = 128 671 / 718 / 610; linear: 629 / 519 / 463 and 637 / 715 / 570.  Bound by
// instructions and latency, at the 32 warps per SM that 64 registers allow (80 registers: 531, 48 spill).
#include <type_traits>

#include "grf_internal.cuh"
#include "packed.cuh"

namespace {

// sixteen bytes of a row as packed pairs of fp32, and back
template <typename T> struct Row;
template <> struct Row<float> {
    static constexpr int CH = 4;
    __device__ static __forceinline__ void widen(const uint4& x, uint64_t (&v)[2])
    {
        v[0] = pack2(__uint_as_float(x.x), __uint_as_float(x.y));
        v[1] = pack2(__uint_as_float(x.z), __uint_as_float(x.w));
    }
    __device__ static __forceinline__ void store(float* p, const float (&v)[4]) { *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]); }
};
template <> struct Row<__nv_bfloat16> {
    static constexpr int CH = 8;
    __device__ static __forceinline__ void widen(const uint4& x, uint64_t (&v)[4])
    {
        const uint32_t w[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
        for (int q = 0; q < 4; ++q) v[q] = pack2(__uint_as_float(w[q] << 16), __uint_as_float(w[q] & 0xffff0000u));
    }
    __device__ static __forceinline__ void store(__nv_bfloat16* p, const float (&v)[8])
    {
        uint32_t w[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            __nv_bfloat162 h = __floats2bfloat162_rn(v[2 * q], v[2 * q + 1]);
            w[q] = *reinterpret_cast<uint32_t*>(&h);
        }
        *reinterpret_cast<uint4*>(p) = make_uint4(w[0], w[1], w[2], w[3]);
    }
};

// sixteen bytes, or zeros where there is no row to read
template <typename T> __device__ __forceinline__ uint4 row_piece(const T* p, bool valid)
{
    return valid ? __ldg(reinterpret_cast<const uint4*>(p)) : make_uint4(0u, 0u, 0u, 0u);
}

constexpr int ASYM_WARPS = 8;
constexpr int ASYM_GH = 2;      // problems per warp: they share the row's indices and mask values

template <typename T, int M, int D, bool SOFTMAX>
__global__ void __launch_bounds__(ASYM_WARPS * 32, 4)
asym_attention_kernel(int32_t G, int32_t N, const int32_t* __restrict__ rowptr, const int32_t* __restrict__ col,
                      const float* __restrict__ val, const T* __restrict__ Q, const T* __restrict__ K,
                      const T* __restrict__ V, T* __restrict__ out, float* __restrict__ den_out)
{
    constexpr int CH = Row<T>::CH, P = CH / 2, GH = ASYM_GH;
    constexpr int KL = M / CH, KPI = 32 / KL;        // lanes per key row, key rows per instruction
    constexpr int VL = D / CH, VPI = 32 / VL;        // lanes per value row, value rows per instruction
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int32_t i = blockIdx.x * ASYM_WARPS + warp;
    const int32_t g0 = blockIdx.y * GH;
    if (i >= N) return;
    const int ks = lane % KL, vs = lane % VL, vg = lane / VL;
    // within a batch of 32 non-zeros this lane owns number (lane % KL) * KPI + lane / KL: the one whose score the exchange
    // below leaves here
    const int own = ks * KPI + lane / KL;

    uint64_t q[GH][P], acc[GH][P];
    float den[GH], run_max[GH];                      // this lane's share of the denominators; softmax: running maxima
    const T* Kh[GH];
    const T* Vh[GH];
#pragma unroll
    for (int h = 0; h < GH; ++h) {
        const int32_t g = min(g0 + h, G - 1);        // a problem beyond the batch repeats the last one and is not written
        Row<T>::widen(row_piece(Q + ((size_t)g * N + i) * M + ks * CH, true), q[h]);
        Kh[h] = K + (size_t)g * N * M + ks * CH;
        Vh[h] = V + (size_t)g * N * D + vs * CH;
        den[h] = 0.0f; run_max[h] = -INFINITY;
#pragma unroll
        for (int e = 0; e < P; ++e) acc[h][e] = 0ull;
    }

    const int32_t beg = rowptr[i], end = rowptr[i + 1];
    // full: all 32 non-zeros are there, and no load or weight is conditional
    auto batch = [&](int32_t p0, int32_t n, auto full) {
        constexpr bool FULL = decltype(full)::value;
        const bool valid = FULL || own < n;
        const int32_t l = valid ? __ldg(col + p0 + own) : 0;
        const float phi = valid ? __ldg(val + p0 + own) : 0.0f;
        float w[GH];
#pragma unroll
        for (int h = 0; h < GH; ++h) {
            // number it * KPI + lane / KL of the batch belongs to lane (lane / KL) * KL + it
            float part[KL];
            constexpr int KB = KL < 4 ? KL : 4;                      // loads on their way together
#pragma unroll
            for (int i0 = 0; i0 < KL; i0 += KB) {
                uint4 x[KB];
#pragma unroll
                for (int u = 0; u < KB; ++u) {
                    const int32_t lk = __shfl_sync(0xffffffffu, l, (lane / KL) * KL + i0 + u);
                    x[u] = row_piece(Kh[h] + (size_t)lk * M, FULL || (i0 + u) * KPI + lane / KL < n);
                }
#pragma unroll
                for (int u = 0; u < KB; ++u) {
                    uint64_t k[P], s2 = 0ull;
                    Row<T>::widen(x[u], k);
#pragma unroll
                    for (int e = 0; e < P; ++e) s2 = fma2(k[e], q[h][e], s2);
                    float lo, hi;
                    unpack2(s2, lo, hi);
                    part[i0 + u] = lo + hi;
                }
            }
            // sum over the KL lanes of a key row; lane ks keeps the sum of instruction ks
#pragma unroll
            for (int off = KL / 2; off > 0; off >>= 1) {
                const bool upper = (ks & off) != 0;
#pragma unroll
                for (int x = 0; x < off; ++x) {
                    const float keep = upper ? part[x + off] : part[x], give = upper ? part[x] : part[x + off];
                    part[x] = keep + __shfl_xor_sync(0xffffffffu, give, off);
                }
            }
            const float s = part[0];
            if (SOFTMAX) {
                float bmax = valid ? s : -INFINITY;
#pragma unroll
                for (int off = 1; off < 32; off <<= 1) bmax = fmaxf(bmax, __shfl_xor_sync(0xffffffffu, bmax, off));
                const float new_max = fmaxf(run_max[h], bmax);
                if (new_max > run_max[h]) {
                    const float rescale = __expf(run_max[h] - new_max);     // 0 on the first batch (run_max = -inf)
                    const uint64_t r2 = pack2(rescale, rescale);
#pragma unroll
                    for (int e = 0; e < P; ++e) acc[h][e] = mul2(acc[h][e], r2);
                    den[h] *= rescale;
                    run_max[h] = new_max;
                }
                w[h] = valid ? phi * __expf(s - new_max) : 0.0f;
            } else {
                w[h] = phi * s;
            }
            den[h] += w[h];
        }
        // the batch's value rows, VPI at a time
        constexpr int VB = 32 / VPI < 4 ? 32 / VPI : 4;              // loads of a problem on their way together
        auto values = [&](int t0, auto whole) {
#pragma unroll
            for (int h = 0; h < GH; ++h) {
                uint4 x[VB];
                float wt[VB];
#pragma unroll
                for (int u = 0; u < VB; ++u) {
                    const int b = t0 + u * VPI + vg, src = (b % KPI) * KL + b / KPI;     // the lane that owns number b
                    const int32_t lv = __shfl_sync(0xffffffffu, l, src & 31);
                    wt[u] = __shfl_sync(0xffffffffu, w[h], src & 31);
                    x[u] = row_piece(Vh[h] + (size_t)lv * D, decltype(whole)::value || b < n);
                }
#pragma unroll
                for (int u = 0; u < VB; ++u) {
                    uint64_t v[P];
                    Row<T>::widen(x[u], v);
                    const uint64_t w2 = pack2(wt[u], wt[u]);
#pragma unroll
                    for (int e = 0; e < P; ++e) acc[h][e] = fma2(w2, v[e], acc[h][e]);
                }
            }
        };
        int t0 = 0;
        for (; t0 + VPI * VB <= (FULL ? 32 : n); t0 += VPI * VB) values(t0, std::true_type());
        if (!FULL && t0 < n) values(t0, std::false_type());
    };
    int32_t p0 = beg;
    for (; p0 + 32 <= end; p0 += 32) batch(p0, 32, std::true_type());
    if (p0 < end) batch(p0, end - p0, std::false_type());
#pragma unroll
    for (int h = 0; h < GH; ++h) {
        float dn = den[h];
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) dn += __shfl_xor_sync(0xffffffffu, dn, off);
        if (g0 + h >= G) break;
        const float inv = dn != 0.0f ? 1.0f / dn : 0.0f;
        float o[CH];
#pragma unroll
        for (int e = 0; e < P; ++e) unpack2(acc[h][e], o[2 * e], o[2 * e + 1]);
#pragma unroll
        for (int e = 0; e < CH; ++e) {
#pragma unroll
            for (int off = VL; off < 32; off <<= 1) o[e] += __shfl_xor_sync(0xffffffffu, o[e], off);
            o[e] *= inv;
        }
        if (vg == 0) Row<T>::store(out + ((size_t)(g0 + h) * N + i) * D + vs * CH, o);
        // with the softmax kernel the reported denominator is relative to exp(max score of the row)
        if (lane == 0 && den_out) den_out[(size_t)(g0 + h) * N + i] = dn;
    }
}

template <typename T, int M, int D>
int launch_md(grf_ctx* ctx, const grf_csr_dev& phi, int32_t G, int32_t N, int kernel, const void* Q, const void* K,
              const void* V, void* out, float* den_out)
{
    const dim3 grid(grf_ceil_div(N, ASYM_WARPS), grf_ceil_div(G, ASYM_GH));
    grf_launch_scope scope(ctx, 5);
    if (kernel == GRF_KERNEL_SOFTMAX)
        asym_attention_kernel<T, M, D, true><<<grid, ASYM_WARPS * 32, 0, ctx->stream>>>(
            G, N, (const int32_t*)phi.rowptr.ptr, (const int32_t*)phi.col.ptr, (const float*)phi.val.ptr, (const T*)Q,
            (const T*)K, (const T*)V, (T*)out, den_out);
    else
        asym_attention_kernel<T, M, D, false><<<grid, ASYM_WARPS * 32, 0, ctx->stream>>>(
            G, N, (const int32_t*)phi.rowptr.ptr, (const int32_t*)phi.col.ptr, (const float*)phi.val.ptr, (const T*)Q,
            (const T*)K, (const T*)V, (T*)out, den_out);
    return GRF_OK;
}

template <typename T, int M>
int launch_m(grf_ctx* ctx, const grf_csr_dev& phi, int32_t G, int32_t N, int32_t d, int kernel, const void* Q,
             const void* K, const void* V, void* out, float* den_out)
{
    switch (d) {
        case 8: return launch_md<T, M, 8>(ctx, phi, G, N, kernel, Q, K, V, out, den_out);
        case 16: return launch_md<T, M, 16>(ctx, phi, G, N, kernel, Q, K, V, out, den_out);
        case 32: return launch_md<T, M, 32>(ctx, phi, G, N, kernel, Q, K, V, out, den_out);
        case 64: return launch_md<T, M, 64>(ctx, phi, G, N, kernel, Q, K, V, out, den_out);
        case 128: return launch_md<T, M, 128>(ctx, phi, G, N, kernel, Q, K, V, out, den_out);
    }
    return GRF_ERR_INVALID;
}

template <typename T>
int launch_t(grf_ctx* ctx, const grf_csr_dev& phi, int32_t G, int32_t N, int32_t m, int32_t d, int kernel,
             const void* Q, const void* K, const void* V, void* out, float* den_out)
{
    switch (m) {
        case 8: return launch_m<T, 8>(ctx, phi, G, N, d, kernel, Q, K, V, out, den_out);
        case 16: return launch_m<T, 16>(ctx, phi, G, N, d, kernel, Q, K, V, out, den_out);
        case 32: return launch_m<T, 32>(ctx, phi, G, N, d, kernel, Q, K, V, out, den_out);
        case 64: return launch_m<T, 64>(ctx, phi, G, N, d, kernel, Q, K, V, out, den_out);
        case 128: return launch_m<T, 128>(ctx, phi, G, N, d, kernel, Q, K, V, out, den_out);
    }
    return GRF_ERR_INVALID;
}

}  // namespace

extern "C" int grf_masked_attn_asym(grf_ctx* ctx, const grf_features* feat, int32_t G, int32_t N, int32_t m, int32_t d,
                                    int dtype, int kernel, const void* Q, const void* K, const void* V, void* out,
                                    float* den_out)
{
    if (!ctx || !feat || !Q || !K || !V || !out) return GRF_ERR_INVALID;
    if (G <= 0 || G > 65535 || N <= 0) return GRF_ERR_INVALID;
    if (kernel != GRF_KERNEL_LINEAR && kernel != GRF_KERNEL_SOFTMAX) return GRF_ERR_INVALID;
    if (dtype != GRF_DTYPE_F32 && dtype != GRF_DTYPE_BF16) return GRF_ERR_INVALID;
    if (feat->phi.rows != N || feat->phi.cols != N) return GRF_ERR_INVALID;       // the mask estimate is Phi: N x N
    if ((((uintptr_t)Q | (uintptr_t)K | (uintptr_t)V | (uintptr_t)out) & 15) != 0) return GRF_ERR_INVALID;
    GRF_CUDA_TRY(cudaSetDevice(ctx->device));
    const int rc = dtype == GRF_DTYPE_F32
                       ? launch_t<float>(ctx, feat->phi, G, N, m, d, kernel, Q, K, V, out, den_out)
                       : launch_t<__nv_bfloat16>(ctx, feat->phi, G, N, m, d, kernel, Q, K, V, out, den_out);
    if (rc != GRF_OK) return rc;
    return cudaGetLastError() == cudaSuccess ? GRF_OK : GRF_ERR_CUDA;
}
