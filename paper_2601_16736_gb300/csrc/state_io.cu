// Export and import of the optimizer state in the canonical layout: [n][59]
// FP32 m and v in the column order xyz, scale, rot, opacity, sh, and the step
// counts t [n].
//
// Both directions are bound by HBM: each state row and each canonical row
// moves once.  The two layouts agree on the row order and differ in the order
// and width of the columns, so a CTA takes 64 consecutive rows, whose state
// rows are one contiguous run and whose canonical rows are another, and
// exchanges them in shared memory: the state side moves as 16-B chunks (one
// lane per chunk, whole 128-B lines per warp), the canonical side as float4.
// One thread per canonical value (4-B canonical accesses, 2-B state accesses,
// two exponent bytes fetched per FP16 value) left the loads too narrow to fill
// the memory system.
// The tile: 64 rows of m and v are 30 KB of shared memory, which lets 7 CTAs
// share an SM.  An import has its whole tile in flight (cp.async), an export
// four or five 16-B loads a thread.  At 1 234 567 rows, before and after
// (import, export; the floor is the bytes at the copy bandwidth):
//   FP16 block  376 -> 140 us, 275 -> 134 us (floor 131)
//   FP32        474 -> 178,    429 -> 183    (174)
//   BF16        443 -> 132,    403 -> 133    (131)
//   hybrid      702 -> 144,    582 -> 148    (141)

#include "step_common.cuh"

namespace gs {
namespace {

constexpr int kIoRows = 64;
// Canonical floats of the tile's m rows; its v rows start 4 banks further on,
// so that the m and v chunks that a warp takes together fall on other banks.
constexpr int kIoFloats = kIoRows * kNumCols, kIoV = kIoFloats + 4;

// A format's 16-B chunks of an m or v row.  chunk_t: the chunk of the m row
// with the step count.
//   load(c, w, x)   the chunk's values into the canonical row x
//   make(c, x, t)   the chunk from the canonical row x (t: the step count,
//                   used by chunk_t of the m row; 0 in the v row)
template <int kPrec>
struct Codec;

template <>
struct Codec<GS_MOM_FP32> {
    static constexpr int kChunks = kRowBytesF32 / 16, kChunkT = 14;
    static __device__ __forceinline__ void load(int c, uint4 w, float *x)
    {
        float *p = c < 12 ? x + 11 + 4 * c : c == 12 ? x + 6 : x;
        if (c < 14) {
            p[0] = __uint_as_float(w.x);
            p[1] = __uint_as_float(w.y);
            p[2] = __uint_as_float(w.z);
            p[3] = __uint_as_float(w.w);
        } else if (c == 14) {
            x[4] = __uint_as_float(w.x);
            x[5] = __uint_as_float(w.y);
            x[10] = __uint_as_float(w.z);
        }
    }
    static __device__ __forceinline__ uint32_t count(uint4 w) { return w.w; }
    static __device__ __forceinline__ uint4 make(int c, const float *x, uint32_t t)
    {
        if (c == 15) return make_uint4(0u, 0u, 0u, 0u);
        if (c == 14) return make_uint4(__float_as_uint(x[4]), __float_as_uint(x[5]), __float_as_uint(x[10]), t);
        const float *p = c < 12 ? x + 11 + 4 * c : c == 12 ? x + 6 : x;
        return make_uint4(__float_as_uint(p[0]), __float_as_uint(p[1]), __float_as_uint(p[2]), __float_as_uint(p[3]));
    }
};

// 8 BF16 values of a chunk <-> FP32, to nearest
__device__ __forceinline__ void bf16_words(uint4 w, float *y)
{
    unpack_bf16x2(w.x, y[0], y[1]);
    unpack_bf16x2(w.y, y[2], y[3]);
    unpack_bf16x2(w.z, y[4], y[5]);
    unpack_bf16x2(w.w, y[6], y[7]);
}

template <>
struct Codec<GS_MOM_BF16> {
    static constexpr int kChunks = kRowBytesBf16 / 16, kChunkT = 7;
    static __device__ __forceinline__ void load(int c, uint4 w, float *x)
    {
        float y[8];
        bf16_words(w, y);
        if (c < 6) {
#pragma unroll
            for (int q = 0; q < 8; ++q) x[11 + 8 * c + q] = y[q];
        } else if (c == 6) {
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                x[6 + q] = y[q];
                x[q] = y[4 + q];
            }
        } else {
            x[4] = y[0];
            x[5] = y[1];
            x[10] = y[2];
        }
    }
    static __device__ __forceinline__ uint32_t count(uint4 w) { return w.z; }
    static __device__ __forceinline__ uint4 make(int c, const float *x, uint32_t t)
    {
        if (c == 7) return make_uint4(pack_bf16x2(x[4], x[5]), pack_bf16x2(x[10], 0.f), t, 0u);
        const float *p = c < 6 ? x + 11 + 8 * c : x + 6, *p2 = c < 6 ? p + 4 : x;
        return make_uint4(pack_bf16x2(p[0], p[1]), pack_bf16x2(p[2], p[3]), pack_bf16x2(p2[0], p2[1]),
                          pack_bf16x2(p2[2], p2[3]));
    }
};

template <>
struct Codec<GS_MOM_BF16_HYBRID> {
    static constexpr int kChunks = kRowBytesHyb / 16, kChunkT = 0;
    static __device__ __forceinline__ void load(int c, uint4 w, float *x)
    {
        if (c >= 4) {                          // SH columns 8 (c - 4) ..; 0-2 live in the FP32 part
            float y[8];
            bf16_words(w, y);
            float *p = x + 11 + 8 * (c - 4);
#pragma unroll
            for (int q = 0; q < 8; ++q)
                if (c > 4 || q >= 3) p[q] = y[q];
            return;
        }
        const uint32_t u[4] = {w.x, w.y, w.z, w.w};
        float *p = c == 0 ? x + 11 : c == 1 ? x + 6 : x;       // DC; rotation; xyz and scale
#pragma unroll
        for (int q = 0; q < 3; ++q) (c == 3 ? q < 2 ? x + 4 : x + 8 : p)[q] = __uint_as_float(u[q]);
        if (c == 1 || c == 2) p[3] = __uint_as_float(u[3]);
    }
    static __device__ __forceinline__ uint32_t count(uint4 w) { return w.w; }
    static __device__ __forceinline__ uint4 make(int c, const float *x, uint32_t t)
    {
        if (c >= 4) {
            const float *p = x + 11 + 8 * (c - 4);
            const bool rest = c > 4;
            return make_uint4(rest ? pack_bf16x2(p[0], p[1]) : 0u, pack_bf16x2(rest ? p[2] : 0.f, p[3]),
                              pack_bf16x2(p[4], p[5]), pack_bf16x2(p[6], p[7]));
        }
        const float *p = c == 0 ? x + 11 : c == 1 ? x + 6 : x;
        if (c == 3) return make_uint4(__float_as_uint(x[4]), __float_as_uint(x[5]), __float_as_uint(x[10]), 0u);
        return make_uint4(__float_as_uint(p[0]), __float_as_uint(p[1]), __float_as_uint(p[2]),
                          c == 0 ? t : __float_as_uint(p[3]));
    }
};

// FP16-block chunks: 0-5 the SH groups, 6 the eight exponent bytes and the
// rotation, 7 xyz + scale + opacity and t.  Chunk and exponent group have the
// same number, and the 8 chunks of a row are 8 neighbouring lanes, which pass
// the exponents around by shuffles.
template <>
struct Codec<GS_MOM_FP16_BLOCK> {
    static constexpr int kChunks = kRowBytesF16B / 16, kChunkT = 7;
    static __device__ __forceinline__ float decode_scale(int c, uint4 w)
    {
        const uint32_t lo = __shfl_sync(0xffffffffu, w.x, 6, 8), hi = __shfl_sync(0xffffffffu, w.y, 6, 8);
        return dec_scale(((c < 4 ? lo : hi) >> (8 * (c & 3))) & 0xffu);
    }
    static __device__ __forceinline__ void load(int c, uint4 w, float d, float *x)
    {
        const uint32_t u[4] = {w.x, w.y, w.z, w.w};
        if (c < 6) {
            decode_w<8>(u, d, x + 11 + 8 * c);
        } else if (c == 6) {
            decode_w<4>(u + 2, d, x + 6);
        } else {
            float y[7];
            decode_w<7>(u, d, y);
#pragma unroll
            for (int q = 0; q < 6; ++q) x[q] = y[q];
            x[10] = y[6];
        }
    }
    static __device__ __forceinline__ uint32_t count(uint4 w) { return w.w >> 16; }
    // The group's values as FP16 words under its exponent (returned), to
    // nearest; a positive second moment stays positive.
    static __device__ __forceinline__ uint32_t encode(int c, const float *x, bool second, uint32_t *w)
    {
        float y[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) y[q] = 0.f;
        const int n = c < 6 ? 8 : c == 6 ? 4 : 6;
        const float *p = c < 6 ? x + 11 + 8 * c : c == 6 ? x + 6 : x;
#pragma unroll
        for (int q = 0; q < 8; ++q)
            if (q < n) y[q] = p[q];
        if (c == 7) y[6] = x[10];
        const uint32_t e = group_exponent(y, 8);
        const float s = e ? enc_scale(e) : 0.f;
#pragma unroll
        for (int q = 0; q < 8; q += 2) {
            uint32_t h = e ? h2_rn(y[q] * s, y[q + 1] * s) : 0u;
            if (second) {
                if ((h & 0x7fffu) == 0u && y[q] > 0.f) h = (h & 0xffff0000u) | 1u;
                if ((h & 0x7fff0000u) == 0u && y[q + 1] > 0.f) h = (h & 0xffffu) | 1u << 16;
            }
            w[q / 2] = h;
        }
        return e;
    }
};

__device__ __forceinline__ uint4 *state_chunks(void *m, int64_t r0, int c2)
{
    return static_cast<uint4 *>(m) + r0 * c2;
}

template <int kPrec>
__global__ void __launch_bounds__(kThreads) export_kernel(void *state, int32_t n, float *__restrict__ m_out,
                                                          float *__restrict__ v_out, uint32_t *__restrict__ t_out)
{
    using C = Codec<kPrec>;
    constexpr int kC2 = 2 * C::kChunks, kPer = kIoRows * kC2 / kThreads, kU = kPer < 5 ? kPer : kPer % 4 ? kPer : 4;
    static_assert(kIoRows * kC2 % kThreads == 0 && kPer % kU == 0, "whole chunks per thread");
    __shared__ __align__(16) float x[kIoV + kIoFloats];
    __shared__ uint32_t ts[kIoRows];
    pdl_wait();
    const int tid = threadIdx.x;
    const int64_t r0 = (int64_t)blockIdx.x * kIoRows;
    const int nrow = (int)min((int64_t)kIoRows, (int64_t)n - r0);
    const uint4 *in = state_chunks(state, r0, kC2);
#pragma unroll 1
    for (int u0 = 0; u0 < kPer; u0 += kU) {
        uint4 w[kU];
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            const int q = tid + (u0 + u) * kThreads, c2 = q % kC2;
            const bool want = c2 >= C::kChunks ? v_out != nullptr : m_out || (t_out && c2 == C::kChunkT);
            w[u] = make_uint4(0u, 0u, 0u, 0u);
            if (q < nrow * kC2 && want) w[u] = __ldcs(in + q);
        }
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            const int q = tid + (u0 + u) * kThreads;
            const int r = q / kC2, c2 = q - r * kC2;
            const bool second = c2 >= C::kChunks;
            const int c = second ? c2 - C::kChunks : c2;
            float *row = x + (second ? kIoV : 0) + r * kNumCols;
            if constexpr (kPrec == GS_MOM_FP16_BLOCK) {
                const float d = C::decode_scale(c, w[u]);
                C::load(c, w[u], d, row);
            } else {
                C::load(c, w[u], row);
            }
            if (!second && c == C::kChunkT) ts[r] = C::count(w[u]);
        }
    }
    __syncthreads();
    const int nf = nrow * kNumCols;
    if (m_out) store_canonical(m_out + r0 * kNumCols, nf, x);
    if (v_out) store_canonical(v_out + r0 * kNumCols, nf, x + kIoV);
    if (t_out && tid < nrow) t_out[r0 + tid] = ts[tid];
    pdl_release();
}

// A part that is NULL keeps the stored one.
template <int kPrec>
__global__ void __launch_bounds__(kThreads) import_kernel(void *state, int32_t n, const float *__restrict__ m_in,
                                                          const float *__restrict__ v_in,
                                                          const uint32_t *__restrict__ t_in)
{
    using C = Codec<kPrec>;
    constexpr int kC2 = 2 * C::kChunks, kPer = kIoRows * kC2 / kThreads;
    __shared__ __align__(16) float x[kIoV + kIoFloats];
    __shared__ uint32_t ts[kIoRows];
    pdl_wait();
    const int tid = threadIdx.x;
    const int64_t r0 = (int64_t)blockIdx.x * kIoRows;
    const int nrow = (int)min((int64_t)kIoRows, (int64_t)n - r0);
    uint4 *out = state_chunks(state, r0, kC2);
    const int nf = nrow * kNumCols;
    if (m_in) load_canonical(m_in + r0 * kNumCols, nf, x);
    if (v_in) load_canonical(v_in + r0 * kNumCols, nf, x + kIoV);
    if (tid < nrow) ts[tid] = t_in ? t_in[r0 + tid] : m_in ? C::count(out[tid * kC2 + C::kChunkT]) : 0u;
    cp_async_wait();
    __syncthreads();
#pragma unroll 1
    for (int u = 0; u < kPer; ++u) {
        const int q = tid + u * kThreads;
        const int r = q / kC2, c2 = q - r * kC2;
        const bool second = c2 >= C::kChunks, has = second ? v_in != nullptr : m_in != nullptr;
        const int c = second ? c2 - C::kChunks : c2;
        const float *row = x + (second ? kIoV : 0) + r * kNumCols;
        const bool mine = r < nrow && has;
        uint4 w = make_uint4(0u, 0u, 0u, 0u);
        if constexpr (kPrec == GS_MOM_FP16_BLOCK) {
            uint32_t h[4] = {0u, 0u, 0u, 0u}, e = 0u;
            if (mine) e = C::encode(c, row, second, h);
            uint32_t lo = c < 4 ? e << (8 * c) : 0u, hi = c < 4 ? 0u : e << (8 * (c - 4));
#pragma unroll
            for (int o = 4; o > 0; o >>= 1) {
                lo |= __shfl_xor_sync(0xffffffffu, lo, o);
                hi |= __shfl_xor_sync(0xffffffffu, hi, o);
            }
            w = c == 6 ? make_uint4(lo, hi, h[0], h[1]) : make_uint4(h[0], h[1], h[2], h[3]);
            if (c == 7 && !second && r < nrow) w.w |= min(ts[r], 65535u) << 16;
        } else if (mine) {
            w = C::make(c, row, second ? 0u : ts[r]);
        }
        if (mine) {
            __stcs(out + q, w);
        } else if (r < nrow && !second && c == C::kChunkT && t_in) {       // t alone
            if constexpr (kPrec == GS_MOM_FP16_BLOCK)
                reinterpret_cast<uint16_t *>(out + q)[7] = (uint16_t)min(ts[r], 65535u);
            else
                reinterpret_cast<uint32_t *>(out + q)[kPrec == GS_MOM_BF16 ? 2 : 3] = ts[r];
        }
    }
    pdl_release();
}

template <int kPrec>
cudaError_t export_t(const StateView &st, int32_t n, float *m, float *v, uint32_t *t, cudaStream_t s)
{
    const unsigned grid = (unsigned)(((int64_t)n + kIoRows - 1) / kIoRows);
    return launch_pdl(export_kernel<kPrec>, grid, kThreads, s, st.m, n, m, v, t);
}

template <int kPrec>
cudaError_t import_t(const StateView &st, int32_t n, const float *m, const float *v, const uint32_t *t, cudaStream_t s)
{
    const unsigned grid = (unsigned)(((int64_t)n + kIoRows - 1) / kIoRows);
    return launch_pdl(import_kernel<kPrec>, grid, kThreads, s, st.m, n, m, v, t);
}

}  // namespace

cudaError_t launch_export(const StateView &st, int32_t n, float *m_out, float *v_out, uint32_t *t_out,
                          cudaStream_t s)
{
    if (n <= 0) return cudaSuccess;
    switch (st.prec) {
    case GS_MOM_FP32: return export_t<GS_MOM_FP32>(st, n, m_out, v_out, t_out, s);
    case GS_MOM_BF16: return export_t<GS_MOM_BF16>(st, n, m_out, v_out, t_out, s);
    case GS_MOM_BF16_HYBRID: return export_t<GS_MOM_BF16_HYBRID>(st, n, m_out, v_out, t_out, s);
    case GS_MOM_FP16_BLOCK: return export_t<GS_MOM_FP16_BLOCK>(st, n, m_out, v_out, t_out, s);
    default: return launch_export_fp8(st, n, m_out, v_out, t_out, s);
    }
}

cudaError_t launch_import(const StateView &st, int32_t n, const float *m_in, const float *v_in,
                          const uint32_t *t_in, cudaStream_t s)
{
    if (n <= 0) return cudaSuccess;
    switch (st.prec) {
    case GS_MOM_FP32: return import_t<GS_MOM_FP32>(st, n, m_in, v_in, t_in, s);
    case GS_MOM_BF16: return import_t<GS_MOM_BF16>(st, n, m_in, v_in, t_in, s);
    case GS_MOM_BF16_HYBRID: return import_t<GS_MOM_BF16_HYBRID>(st, n, m_in, v_in, t_in, s);
    case GS_MOM_FP16_BLOCK: return import_t<GS_MOM_FP16_BLOCK>(st, n, m_in, v_in, t_in, s);
    default: return launch_import_fp8(st, n, m_in, v_in, t_in, s);
    }
}

}  // namespace gs
