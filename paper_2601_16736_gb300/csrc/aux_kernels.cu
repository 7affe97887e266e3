// Kernels around the fused step: the standalone visibility filter with
// global compaction, the FP64 bias-correction table, optimizer-state
// re-indexing across row-set changes, and the attribute gather that
// accompanies a re-index.

#include <algorithm>

#include "step_common.cuh"

namespace gs {
namespace {

__device__ __forceinline__ void record_error(int32_t *err, int32_t code)
{
    if (err) atomicCAS(err, 0, code);
}

// ---------------------------------------------------------------- visibility
struct CamArg {
    float c[kCamFloats];
};

// One thread per row decides V (frustum test of the mean); each CTA compacts
// its visible rows with warp ballots, reserves a contiguous range of the
// output list with one atomicAdd, and writes them in ascending row order.
__global__ void __launch_bounds__(kThreads) visibility_kernel(const float *__restrict__ xyz, int32_t n,
                                                              const CamArg cam, uint8_t *__restrict__ mask,
                                                              int32_t *__restrict__ list,
                                                              unsigned long long *__restrict__ count)
{
    __shared__ int32_t s_cnt[kThreads / 32];
    __shared__ unsigned long long s_base;
    pdl_wait();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t row = (int64_t)blockIdx.x * kThreads + tid;
    const float *c = cam.c;
    bool vis = false;
    if (row < n) {
        const float *p = xyz + row * 3;
        vis = frustum_visible(p[0], p[1], p[2], c);
        mask[row] = vis ? 1 : 0;
    }
    if (!count) return;
    const unsigned b = __ballot_sync(0xffffffffu, vis);
    if (lane == 0) s_cnt[warp] = __popc(b);
    __syncthreads();
    if (tid == 0) {
        int tot = 0;
        for (int q = 0; q < kThreads / 32; ++q) tot += s_cnt[q];
        s_base = tot ? atomicAdd(count, (unsigned long long)tot) : 0ull;
    }
    __syncthreads();
    if (list && vis) {
        int off = 0;
        for (int q = 0; q < warp; ++q) off += s_cnt[q];
        off += __popc(b & ((1u << lane) - 1u));
        list[s_base + off] = (int32_t)row;
    }
    pdl_release();
}

// The count starts from zero.  A kernel in the launch chain rather than a memset:
// the filter's CTAs are then already resident when the zero is written.
__global__ void zero_count_kernel(unsigned long long *count)
{
    pdl_release();
    pdl_wait();
    *count = 0ull;
}

// Eight consecutive rows per thread, for 16-B aligned means: six float4
// loads carry the rows' 24 values, two 32-bit stores their mask bytes.  The
// CTA's visible rows are placed by an exclusive scan of the per-thread
// counts, so the list stays ascending within the CTA's 2048 rows; one
// atomicAdd per CTA reserves its range of the list (8 rows per thread halves
// those atomics against 4, 10 % faster over 6 M means).
constexpr int kVisRpt = 8;

__global__ void __launch_bounds__(kThreads) visibility4_kernel(const float *__restrict__ xyz, int32_t n,
                                                               const CamArg cam, uint8_t *__restrict__ mask,
                                                               int32_t *__restrict__ list,
                                                               unsigned long long *__restrict__ count)
{
    __shared__ int32_t s_warp[kThreads / 32];
    __shared__ unsigned long long s_base;
    pdl_wait();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t r0 = ((int64_t)blockIdx.x * kThreads + tid) * kVisRpt;
    const float *c = cam.c;
    unsigned vis = 0;                      // bit j: row r0 + j is visible
    if (r0 + kVisRpt <= n) {
        const float4 *p = reinterpret_cast<const float4 *>(xyz + r0 * 3);
        float4 q4[3 * kVisRpt / 4];
#pragma unroll
        for (int u = 0; u < 3 * kVisRpt / 4; ++u) q4[u] = __ldcs(p + u);
        const float *q = reinterpret_cast<const float *>(q4);
        uint32_t mw[kVisRpt / 4];
#pragma unroll
        for (int u = 0; u < kVisRpt / 4; ++u) mw[u] = 0u;
#pragma unroll
        for (int j = 0; j < kVisRpt; ++j) {
            const bool v = frustum_visible(q[3 * j], q[3 * j + 1], q[3 * j + 2], c);
            vis |= v ? 1u << j : 0u;
            mw[j / 4] |= (v ? 1u : 0u) << (8 * (j % 4));
        }
#pragma unroll
        for (int u = 0; u < kVisRpt / 4; ++u) __stcs(reinterpret_cast<uint32_t *>(mask + r0) + u, mw[u]);
    } else {
        for (int j = 0; j < kVisRpt && r0 + j < n; ++j) {
            const float *q = xyz + (r0 + j) * 3;
            const bool v = frustum_visible(q[0], q[1], q[2], c);
            vis |= v ? 1u << j : 0u;
            mask[r0 + j] = v ? 1 : 0;
        }
    }
    if (!count) return;
    const int mine = __popc(vis);
    int incl = mine;                       // inclusive scan of the counts within the warp
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, incl, d);
        if (lane >= d) incl += y;
    }
    if (lane == 31) s_warp[warp] = incl;
    __syncthreads();
    if (tid == 0) {
        int tot = 0;
        for (int q = 0; q < kThreads / 32; ++q) tot += s_warp[q];
        s_base = tot ? atomicAdd(count, (unsigned long long)tot) : 0ull;
    }
    __syncthreads();
    if (list && vis) {
        int off = incl - mine;
        for (int q = 0; q < warp; ++q) off += s_warp[q];
        int32_t *dst = list + s_base + off;
        for (int j = 0; j < kVisRpt; ++j)
            if (vis & (1u << j)) *dst++ = (int32_t)(r0 + j);
    }
    pdl_release();
}

// --------------------------------------------------------------- bias table
// 1 - beta^k in FP64 for k = 0 .. len-1 (beta^k by binary exponentiation),
// plus the FP32 factors the step consumes: 1/(1 - b1^k), 1/sqrt(1 - b2^k).
__device__ double pow_int(double b, uint32_t e)
{
    double p = 1.0;
    while (e) {
        if (e & 1u) p *= b;
        b *= b;
        e >>= 1;
    }
    return p;
}

__global__ void bias_table_kernel(double beta1, double beta2, int32_t len, double *t1, double *t2,
                                  float2 *fac)
{
    const int32_t k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= len) return;
    const double d1 = 1.0 - pow_int(beta1, (uint32_t)k);
    const double d2 = 1.0 - pow_int(beta2, (uint32_t)k);
    t1[k] = d1;
    t2[k] = d2;
    fac[k] = (k == 0) ? make_float2(0.0f, 0.0f) : make_float2((float)(1.0 / d1), (float)(1.0 / sqrt(d2)));
}

// ------------------------------------------------------------------ reindex
// One thread per (output row, 16-B chunk of its state rows): kChunks chunks
// of the m and v rows (FP32: slots 0-59 incl. the counter; BF16: the whole
// 128-B row incl. the counter at byte 120; hybrid: the whole 160-B row).
// Copied from row src[j], or zeroed for a fresh row.
template <int kChunks, int kRowBytes>
__global__ void reindex_kernel(const StateView in, int32_t n_in, const StateView out, int32_t n_out,
                               const int32_t *__restrict__ src, const uint8_t *__restrict__ reset, int32_t *err)
{
    pdl_wait();
    const int64_t gid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t j = gid / kChunks;
    const int c = (int)(gid - j * kChunks);
    if (j >= n_out) return;
    int32_t s = src[j];
    if (s >= n_in) {
        if (c == 0) record_error(err, GS_ERR_INVALID_ARG);
        s = -1;
    }
    const bool fresh = s < 0 || (reset && reset[j]);
    uint4 mv = make_uint4(0u, 0u, 0u, 0u), vv = mv;
    if (!fresh) {      // each row is read once and written once: stream past L2
        mv = __ldcs(reinterpret_cast<const uint4 *>(static_cast<const char *>(in.m) + (size_t)s * (2 * kRowBytes) + 16 * c));
        vv = __ldcs(reinterpret_cast<const uint4 *>(static_cast<const char *>(in.v) + (size_t)s * (2 * kRowBytes) + 16 * c));
    }
    __stcs(reinterpret_cast<uint4 *>(static_cast<char *>(out.m) + (size_t)j * (2 * kRowBytes) + 16 * c), mv);
    __stcs(reinterpret_cast<uint4 *>(static_cast<char *>(out.v) + (size_t)j * (2 * kRowBytes) + 16 * c), vv);
    pdl_release();
}

// ----------------------------------------------------------- attribute gather
// One CTA per 128 output rows, in one launch for all five groups.  The source
// rows are copied into shared memory by cp.async (16 B for the SH and rotation
// rows, 4 B for the small groups, whose rows need not be 16-B aligned), so a
// CTA has its whole 30 KB in flight without holding it in registers, and leave
// as contiguous runs of the output arrays in float4.  Bound by HBM: 236 B read
// and written per row.  Rows whose source is negative keep what the output
// array held; out-of-range sources are recorded and not read.  6 M rows: 443 us
// against 549 for two launches that kept four items a thread in registers (the
// copy bandwidth gives 419); 100 k rows: 10 us against 15.
constexpr int kGatherRows = 128;

// kW floats per row (1 or 3) of the tile: into shared memory, and out of it.
template <int kW>
__device__ __forceinline__ void gather_small_in(const float *__restrict__ in, const int32_t *s_src, int nrow, float *x)
{
    for (int q = threadIdx.x; q < nrow * kW; q += kThreads) {
        const int j = q / kW, c = q - j * kW;
        const int32_t s = s_src[j];
        if (s >= 0) cp_async4(x + q, in + (int64_t)s * kW + c);
    }
}
template <int kW>
__device__ __forceinline__ void gather_small_out(float *__restrict__ out, const int32_t *s_src, int nrow, bool all,
                                                 const float *x)
{
    const int nf = nrow * kW, nv = all && !((uintptr_t)out & 15u) ? nf / 4 : 0;
    for (int q = threadIdx.x; q < nv; q += kThreads)
        st4(out + 4 * q, *reinterpret_cast<const float4 *>(x + 4 * q));
    for (int q = 4 * nv + threadIdx.x; q < nf; q += kThreads)
        if (s_src[q / kW] >= 0) __stcs(out + q, x[q]);
}

__global__ void __launch_bounds__(kThreads) gather_kernel(const gs_attrs in, int32_t n_in, const gs_attrs out,
                                                          const int32_t *__restrict__ src, int32_t n_new, int32_t *err)
{
    __shared__ __align__(16) float sh[kGatherRows * 48], rot[kGatherRows * 4], xyz[kGatherRows * 3],
        scale[kGatherRows * 3], op[kGatherRows];
    __shared__ int32_t s_src[kGatherRows];
    pdl_wait();
    const int tid = threadIdx.x;
    const int64_t r0 = (int64_t)blockIdx.x * kGatherRows;
    const int nrow = (int)min((int64_t)kGatherRows, (int64_t)n_new - r0);
    int32_t s0 = 0;
    if (tid < nrow) {
        s0 = src[r0 + tid];
        if (s0 >= n_in) {
            record_error(err, GS_ERR_INVALID_ARG);
            s0 = -1;
        }
        s_src[tid] = s0;
    }
    const bool all = !__syncthreads_or(s0 < 0);
    for (int q = tid; q < nrow * 12; q += kThreads) {
        const int j = q / 12, c = q - 12 * j;
        const int32_t s = s_src[j];
        if (s >= 0) cp_async16(sh + 4 * q, in.sh + (int64_t)s * 48 + 4 * c);
    }
    if (tid < nrow && s0 >= 0) cp_async16(rot + 4 * tid, in.rot + (int64_t)s0 * 4);
    gather_small_in<3>(in.xyz, s_src, nrow, xyz);
    gather_small_in<3>(in.scale, s_src, nrow, scale);
    gather_small_in<1>(in.opacity, s_src, nrow, op);
    cp_async_wait();
    __syncthreads();
    for (int q = tid; q < nrow * 12; q += kThreads)
        if (all || s_src[q / 12] >= 0) st4(out.sh + r0 * 48 + 4 * q, *reinterpret_cast<const float4 *>(sh + 4 * q));
    if (tid < nrow && s0 >= 0) st4(out.rot + (r0 + tid) * 4, *reinterpret_cast<const float4 *>(rot + 4 * tid));
    gather_small_out<3>(out.xyz + r0 * 3, s_src, nrow, all, xyz);
    gather_small_out<3>(out.scale + r0 * 3, s_src, nrow, all, scale);
    gather_small_out<1>(out.opacity + r0, s_src, nrow, all, op);
    pdl_release();
}

// ------------------------------------------------------------- row copy
// The memory traffic of a step over listed rows, without the update: each
// byte a visible row's step reads is read, each byte it writes is written
// back with the value read.  Items are kind-major (SH chunks, then
// moment-row chunks, then the four small groups) so warps stay convergent.
struct CopyRowsArgs {
    gs_attrs a;
    gs_grads g;
    char *m;
    int32_t row_bytes, chunks;              // bytes of an m or v row; 16-B chunks used of each
    const int32_t *rows;
    int64_t nl;
    int32_t n;
    int32_t *err;
    uint32_t zero;                          // 0, passed at run time (see below)
};

// The gradients are read and their bits folded into the stored values
// through a mask that is zero at run time: the stores write back exactly
// what was read, but the compiler cannot prove the gradient loads dead (a
// load whose result is never used is removed, and the copy would then move
// fewer bytes than the step).
__device__ __forceinline__ uint32_t grad_bits4(const float *p, uint32_t zero)
{
    const float4 g = __ldcs(reinterpret_cast<const float4 *>(p));
    return (__float_as_uint(g.x) ^ __float_as_uint(g.y) ^ __float_as_uint(g.z) ^ __float_as_uint(g.w)) & zero;
}
__device__ __forceinline__ float4 xor4(float4 x, uint32_t b)
{
    return make_float4(__uint_as_float(__float_as_uint(x.x) ^ b), __uint_as_float(__float_as_uint(x.y) ^ b),
                       __uint_as_float(__float_as_uint(x.z) ^ b), __uint_as_float(__float_as_uint(x.w) ^ b));
}

__global__ void __launch_bounds__(kThreads) copy_rows_kernel(const CopyRowsArgs c)
{
    pdl_wait();
    const int64_t nl = c.nl, e_sh = 12 * nl, e_m = e_sh + (int64_t)c.chunks * nl, e_st = e_m + (int64_t)c.chunks * nl;
    const int64_t total = e_st + 4 * nl;
    for (int64_t w = (int64_t)blockIdx.x * kThreads + threadIdx.x; w < total; w += (int64_t)gridDim.x * kThreads) {
        int64_t j;
        int i;
        if (w < e_sh) {
            j = w / 12;
            i = (int)(w - 12 * j);
        } else if (w < e_st) {
            const int64_t q = w < e_m ? w - e_sh : w - e_m;   // m rows, then v rows, chunks of a row adjacent
            j = q / c.chunks;
            i = (int)(q - j * c.chunks);
        } else {
            const int64_t q = w - e_st;
            i = (int)(q / nl);                   // 0 xyz, 1 rot, 2 scale, 3 opacity
            j = q - (int64_t)i * nl;
        }
        const int32_t r32 = c.rows[j];
        if (r32 < 0 || r32 >= c.n) {
            if (w < e_sh && i == 0) record_error(c.err, GS_ERR_INVALID_ARG);
            continue;
        }
        const int64_t r = r32;
        if (w < e_sh) {
            float4 *t = reinterpret_cast<float4 *>(c.a.sh + r * 48) + i;
            const uint32_t b = grad_bits4(c.g.sh + r * 48 + 4 * i, c.zero);
            __stcs(t, xor4(*t, b));
        } else if (w < e_st) {
            uint4 *t = reinterpret_cast<uint4 *>(c.m + (2 * r + (w < e_m ? 0 : 1)) * c.row_bytes) + i;
            __stcs(t, *t);
        } else if (i == 1) {
            float4 *t = reinterpret_cast<float4 *>(c.a.rot + r * 4);
            const uint32_t b = grad_bits4(c.g.rot + r * 4, c.zero);
            __stcs(t, xor4(*t, b));
        } else {
            float *t = i == 0 ? c.a.xyz + r * 3 : i == 2 ? c.a.scale + r * 3 : c.a.opacity + r;
            const float *g = i == 0 ? c.g.xyz + r * 3 : i == 2 ? c.g.scale + r * 3 : c.g.opacity + r;
            const int k = i == 3 ? 1 : 3;
            for (int u = 0; u < k; ++u) {
                const uint32_t b = __float_as_uint(__ldcs(g + u)) & c.zero;
                __stcs(t + u, __uint_as_float(__float_as_uint(t[u]) ^ b));
            }
        }
    }
    pdl_release();
}

// ------------------------------------------------------------ active rows
// The ascending list of rows with tau > tau_act (opacity > 1/255) in two
// passes over blocks of kActRows rows: per-block counts, then the ordered
// write.  In the second pass every block adds up the counts of the blocks
// before it (a few thousand ints, read from L2) to find its offset, so no
// separate scan is needed; the last block also writes the total.  Rows of a
// block are taken as kActRpt strided passes of the CTA (coalesced loads, all
// in flight at once), which is also their ascending order.
constexpr int kActRpt = 16;
constexpr int kActRows = kThreads * kActRpt;
constexpr int kActWarps = kThreads / 32;

__global__ void __launch_bounds__(kThreads) active_count_kernel(const float *__restrict__ tau, int32_t n,
                                                                float tau_act, int32_t *__restrict__ blk)
{
    __shared__ int32_t warp_sum[kActWarps];
    pdl_wait();
    const int64_t r0 = (int64_t)blockIdx.x * kActRows;
    float x[kActRpt];
#pragma unroll
    for (int j = 0; j < kActRpt; ++j) {
        const int64_t r = r0 + j * kThreads + threadIdx.x;
        x[j] = r < n ? __ldg(tau + r) : -INFINITY;      // kept in L2 for the write pass
    }
    int c = 0;
#pragma unroll
    for (int j = 0; j < kActRpt; ++j) c += x[j] > tau_act ? 1 : 0;
    c = __reduce_add_sync(0xffffffffu, c);
    if ((threadIdx.x & 31) == 0) warp_sum[threadIdx.x >> 5] = c;
    __syncthreads();
    if (threadIdx.x == 0) {
        int s = 0;
        for (int w = 0; w < kActWarps; ++w) s += warp_sum[w];
        blk[blockIdx.x] = s;
    }
    pdl_release();
}

// rows == NULL: count only (only the last block runs, to write the total).
__global__ void __launch_bounds__(kThreads) active_write_kernel(const float *__restrict__ tau, int32_t n,
                                                                float tau_act, const int32_t *__restrict__ blk,
                                                                int32_t *__restrict__ rows, long long *total)
{
    __shared__ int32_t cnt[kActRpt * kActWarps];      // per (pass, warp), then its exclusive offset
    __shared__ int32_t part[kActWarps];
    pdl_wait();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const bool last = blockIdx.x == gridDim.x - 1;
    if (!rows && !last) return;
    const int64_t r0 = (int64_t)blockIdx.x * kActRows;
    float x[kActRpt];
#pragma unroll
    for (int j = 0; j < kActRpt; ++j) {
        const int64_t r = r0 + j * kThreads + threadIdx.x;
        x[j] = r < n ? __ldcs(tau + r) : -INFINITY;
    }
    int before = 0;                                      // counts of the blocks before this one
    for (int b = threadIdx.x; b < (int)blockIdx.x; b += kThreads) before += blk[b];
    before = __reduce_add_sync(0xffffffffu, before);
    unsigned bal[kActRpt];
#pragma unroll
    for (int j = 0; j < kActRpt; ++j) {
        bal[j] = __ballot_sync(0xffffffffu, x[j] > tau_act);
        if (lane == 0) cnt[j * kActWarps + warp] = __popc(bal[j]);
    }
    if (lane == 0) part[warp] = before;
    __syncthreads();
    if (warp == 0) {                                     // exclusive scan of the kActRpt*kActWarps counts
        constexpr int kPer = kActRpt * kActWarps / 32;
        int v[kPer], sum = 0;
#pragma unroll
        for (int q = 0; q < kPer; ++q) {
            v[q] = cnt[lane * kPer + q];
            sum += v[q];
        }
        int incl = sum;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, incl, d);
            if (lane >= d) incl += y;
        }
        int base = 0;
        for (int w = 0; w < kActWarps; ++w) base += part[w];
        int run = base + incl - sum;
#pragma unroll
        for (int q = 0; q < kPer; ++q) {
            cnt[lane * kPer + q] = run;
            run += v[q];
        }
        if (last && lane == 31 && total) *total = run;
    }
    __syncthreads();
    if (!rows) return;
    const unsigned lt = (1u << lane) - 1u;
#pragma unroll
    for (int j = 0; j < kActRpt; ++j)
        if (bal[j] & (1u << lane))
            rows[cnt[j * kActWarps + warp] + __popc(bal[j] & lt)] = (int32_t)(r0 + j * kThreads + threadIdx.x);
    pdl_release();
}

unsigned blocks_for(int64_t n_threads) { return (unsigned)((n_threads + kThreads - 1) / kThreads); }

}  // namespace

cudaError_t launch_visibility(const float *xyz, int32_t n, const float cam[kCamFloats], uint8_t *mask, int32_t *list,
                              unsigned long long *count, cudaStream_t s)
{
    if (count) {
        const cudaError_t e = launch_pdl(zero_count_kernel, 1u, 1u, s, count);
        if (e != cudaSuccess) return e;
    }
    if (n <= 0) return cudaSuccess;
    CamArg c;
    memcpy(c.c, cam, sizeof(c.c));
    if (((uintptr_t)xyz & 15u) == 0 && ((uintptr_t)mask & 3u) == 0)
        return launch_pdl(visibility4_kernel, blocks_for(((int64_t)n + kVisRpt - 1) / kVisRpt), kThreads, s, xyz, n, c,
                          mask, list, count);
    return launch_pdl(visibility_kernel, blocks_for(n), kThreads, s, xyz, n, c, mask, list, count);
}

cudaError_t launch_bias_table(double beta1, double beta2, int32_t len, double *t1, double *t2, float2 *fac,
                              cudaStream_t s)
{
    bias_table_kernel<<<blocks_for(len), kThreads, 0, s>>>(beta1, beta2, len, t1, t2, fac);
    return cudaGetLastError();
}

namespace {

template <int kChunks, int kRowBytes>
cudaError_t launch_reindex_t(const StateView &in, int32_t n_in, const StateView &out, int32_t n_out, const int32_t *src,
                             const uint8_t *reset, int32_t *err, cudaStream_t s)
{
    return launch_pdl(reindex_kernel<kChunks, kRowBytes>, blocks_for((int64_t)n_out * kChunks), kThreads, s, in, n_in,
                      out, n_out, src, reset, err);
}

}  // namespace

cudaError_t launch_reindex(const StateView &in, int32_t n_in, const StateView &out, int32_t n_out,
                           const int32_t *src, const uint8_t *reset, int32_t *err, cudaStream_t s)
{
    if (n_out <= 0) return cudaSuccess;
    switch (in.prec) {
    case GS_MOM_FP8E4M3: return launch_reindex_fp8(in, n_in, out, n_out, src, reset, err, s);
    case GS_MOM_FP32:      // whole 256-B rows (the last 16 B are padding): a warp moves two rows
        return launch_reindex_t<16, kRowBytesF32>(in, n_in, out, n_out, src, reset, err, s);
    case GS_MOM_BF16: return launch_reindex_t<8, kRowBytesBf16>(in, n_in, out, n_out, src, reset, err, s);
    case GS_MOM_BF16_HYBRID: return launch_reindex_t<10, kRowBytesHyb>(in, n_in, out, n_out, src, reset, err, s);
    case GS_MOM_FP16_BLOCK: return launch_reindex_t<8, kRowBytesF16B>(in, n_in, out, n_out, src, reset, err, s);
    default: return cudaErrorNotSupported;
    }
}

cudaError_t launch_gather_attrs(const gs_attrs &in, int32_t n_in, const gs_attrs &out, const int32_t *src,
                                int32_t n_new, int32_t *err, cudaStream_t s)
{
    if (n_new <= 0) return cudaSuccess;
    const unsigned grid = (unsigned)(((int64_t)n_new + kGatherRows - 1) / kGatherRows);
    return launch_pdl(gather_kernel, grid, kThreads, s, in, n_in, out, src, n_new, err);
}

cudaError_t launch_copy_rows(const gs_attrs &a, const gs_grads &g, void *m, int32_t row_bytes,
                             int32_t used_bytes, const int32_t *rows, int64_t n_listed, int32_t n, int32_t *err,
                             cudaStream_t s)
{
    if (n_listed <= 0) return cudaSuccess;
    CopyRowsArgs c{a, g, static_cast<char *>(m), row_bytes, used_bytes / 16, rows, n_listed,
                   n, err, 0u};
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const int64_t items = (16 + 2 * (int64_t)c.chunks) * n_listed;
    const unsigned grid = (unsigned)std::min<int64_t>((items + kThreads - 1) / kThreads, 8 * (int64_t)sms);
    return launch_pdl(copy_rows_kernel, grid, kThreads, s, c);
}

int64_t active_rows_scratch(int64_t n) { return std::max<int64_t>(1, (n + kActRows - 1) / kActRows); }

cudaError_t launch_active_rows(const float *tau, int32_t n, float tau_act, int32_t *blk, int32_t *rows,
                               long long *n_active, cudaStream_t s)
{
    if (n <= 0) return cudaMemsetAsync(n_active, 0, sizeof(long long), s);
    const int32_t nblk = (int32_t)((n + kActRows - 1) / kActRows);
    cudaError_t e = launch_pdl(active_count_kernel, (unsigned)nblk, kThreads, s, tau, n, tau_act, blk);
    if (e != cudaSuccess) return e;
    return launch_pdl(active_write_kernel, (unsigned)nblk, kThreads, s, tau, n, tau_act,
                      static_cast<const int32_t *>(blk), rows, n_active);
}

}  // namespace gs
